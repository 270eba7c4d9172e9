// Chain TV-l2 by splitting at thresholds: the chain kernel of the 2D phases and of the
// batches of tv_chain_solve whose chains have at most kSplitMaxLen nodes.
//
// The dynamic program of Sec. 4.1 walks a chain node by node, and each node waits for the
// one before. Here a chain is cut top down instead. Take a run of neighbouring nodes whose
// boundary flows u (the edge terms w_i sign(x_{i+1} - x_i), prefix sums of x - y) are known,
// and let z be the mean it would have if it were one constant piece. For ONE threshold z the
// forward message of Algorithm 2 is a number per node,
//     t_i = m_{i-1} + (z - y_i),   m_i = clip(t_i, -w_i, w_i),
// and it tells on which side of z the minimiser lies: t_i > w_i puts x_i below z whatever
// follows, t_i < -w_i above it, and an undecided node goes with its right neighbour (the
// backward clip of Algorithm 2). Where neighbours end on different sides, the edge between
// them carries the flow +-w_i, so the run is cut there and the two parts are independent. A
// run on one side only is constant at z: its mean is z, so no part can lie above. Every round
// treats all runs of a chain at once; signals of the 1D experiment (Sec. 6.1) take 7 rounds
// at 1024 nodes, a ramp log2(n), and every round but the last adds a cut.
//
// Composed maps m -> clip(m + a, lo, hi) are closed under composition, so a round is not
// sequential: each lane holds L consecutive nodes in registers, composes its nodes' maps, a
// warp scan (across W warps: a shared-memory exchange) gives each lane its incoming m, a
// second walk gives the sides as two bit masks, and the undecided bits are filled from the
// right by one carry-propagating addition. The mean of every run comes from a walk from the
// right and a segmented scan over the lanes (join_runs). Cut flows are folded into the values at
// the cut (y_i += u, y_{i+1} -= u, w_i = 0), after which a cut needs no special case.
//
// Solutions are sums of the values of a run over its length: all nodes of a run are bitwise
// equal, and the rounding is that of one mean. The folded flows cost eps * |u| per run, so a
// chain that is to be cut at a flow above 16 max |y|, that has a NaN weight, or whose values are
// not finite or near the ends of FP32's range, goes to the warp's dynamic program
// (coop_solve_chain, records and reserve in the workspace) instead.
#pragma once
#include "tv2d_common.cuh"
#include "tv2d_gap.cuh"
#include "tv_coop.cuh"

namespace tvk {

constexpr int kSplitMaxLen = 4096;     // nodes of the longest chain (4 warps x 32 lanes x 32)
constexpr float kSplitHeavy = 16.f;
constexpr float kSplitTiny = 1e-37f;  // weights up to here decouple
// Largest |value| of a chain that is split. Above, the sums of 4096 values, each with two flows of
// up to 16 times as much folded in, could overflow; below, weights that decouple would count.
constexpr float kSplitMost = 1e32f, kSplitLeast = 1e-28f;

// What a chain's nodes are made of. PLAIN: c = y. INIT, ROW, COL: the set-up of the phases
// of eq. pd (x^0 rows, primal rows, dual columns).
enum SplitMode { SPLIT_PLAIN = 0, SPLIT_INIT = 1, SPLIT_ROW = 2, SPLIT_COL = 3 };

struct SplitView {
    int mode;
    bool cols;                 // chains are columns (node stride `stride`), else rows
    const float *p0, *p1, *p2; // PLAIN y; INIT f, y; ROW f, y, x^k; COL x^k, x^{k-1}, y
    const float *pw;           // edge weights, or NULL: lam
    float lam, ws;             // weight = ws * (pw or lam)
    float ca, cb, sg;          // ROW: c = ca (f - y) + cb x; COL: 1/sigma, theta, sigma
    float *o0, *o1;
    long long stride, wrow;    // columns: node stride (values and weights); rows: weight row
    float2 *rec, *spill;       // records and reserve of the fallback
    int maxlen;                // records of one chain

    __device__ __forceinline__ float unary(float a, float b, float c) const
    {
        if (mode == SPLIT_PLAIN) return a;
        if (mode == SPLIT_INIT) return a - b;
        if (mode == SPLIT_ROW) return ca * (a - b) + cb * c;
        return c * ca + (a + cb * (a - b));
    }
    __device__ __forceinline__ void emit(long long o, float xv, float c) const
    {
        if (mode == SPLIT_COL) {
            o0[o] = sg * (c - xv);
        } else {
            o0[o] = xv;
            if (mode == SPLIT_INIT) o1[o] = xv;
        }
    }
};

// The fallback's policy (coop_solve_chain): one chain of the view.
struct SplitCoopP {
    static constexpr bool CREC = false;
    struct Raw {
        float a, b, c, w;
    };
    struct Acc {};
    SplitView v;
    long long wstart;
    int n;

    __device__ int max_len() const { return v.maxlen; }
    __device__ long long at(long long start, int i) const { return start + (long long)i * v.stride; }
    __device__ void fetch(long long, long long start, int nn, int i, Raw &r) const
    {
        const bool in = i < nn;
        const long long o = at(start, i);
        r.a = in ? v.p0[o] : 0.f;
        r.b = in && v.p1 ? v.p1[o] : 0.f;
        r.c = in && v.p2 ? v.p2[o] : 0.f;
        r.w = v.lam;
        if (v.pw) r.w = i < nn - 1 ? v.pw[wstart + (long long)i * v.stride] : 0.f;
    }
    __device__ void unary(long long, long long, int, int, const Raw &r, float &c, float &w,
                          Acc &) const
    {
        c = v.unary(r.a, r.b, r.c);
        w = v.ws * r.w;
    }
    __device__ void emit(long long k, long long start, int i, float xv, float) const
    {
        float c = 0.f, w;
        if (v.mode == SPLIT_COL) unary_direct(i, n, k, start, c, w);
        v.emit(at(start, i), xv, c);
    }
    __device__ void unary_direct(int i, int nn, long long k, long long start, float &c,
                                 float &w) const
    {
        Raw r;
        Acc a;
        fetch(k, start, nn, i, r);
        unary(k, start, nn, i, r, c, w, a);
        if (i == nn - 1) w = 0.f;
    }
    __device__ void emit_direct(int i, long long k, long long start, float xv, float c) const
    {
        emit(k, start, i, xv, c);
    }
};

static __device__ __noinline__ void split_fallback(const SplitView &v, long long k,
                                                   long long start, long long wstart, int n,
                                                   int lane, float2 *spill, WsHeader *hdr)
{
    SplitCoopP p{v, wstart, n};
    SplitCoopP::Acc acc;
    coop_solve_chain(p, acc, k, start, n, lane, (float2 *)nullptr, (float *)nullptr, 0, v.rec,
                     (float *)nullptr, spill, hdr);
}

__device__ __forceinline__ float rcp_approx(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float clampw(float v, float lo, float hi)
{
    return fminf(fmaxf(v, lo), hi);
}

// s / k: the approximate reciprocal's quotient with one residual correction
__device__ __forceinline__ float mean_of(float s, float k)
{
    const float rc = rcp_approx(k), q = s * rc;
    return fmaf(fmaf(-q, k, s), rc, q);
}

// A sum carried in two floats: hi the running FP32 sum, lo what its roundings left out.
struct Sum2 {
    float hi, lo;
};
__device__ __forceinline__ Sum2 operator+(Sum2 a, Sum2 b)
{
    const float t = a.hi + b.hi, u = t - a.hi;
    return Sum2{t, ((a.hi - (t - u)) + (b.hi - u)) + (a.lo + b.lo)};
}
__device__ __forceinline__ Sum2 operator+(Sum2 a, float b)
{
    const float t = a.hi + b, u = t - a.hi;
    return Sum2{t, ((a.hi - (t - u)) + (b - u)) + a.lo};
}
__device__ __forceinline__ Sum2 pick(bool c, Sum2 a, Sum2 b)
{
    return Sum2{c ? a.hi : b.hi, c ? a.lo : b.lo};
}
__device__ __forceinline__ Sum2 shfl_down(Sum2 a, int o)
{
    return Sum2{__shfl_down_sync(FULL, a.hi, o), __shfl_down_sync(FULL, a.lo, o)};
}
__device__ __forceinline__ float pick(bool c, float a, float b) { return c ? a : b; }
__device__ __forceinline__ float shfl_down(float a, int o) { return __shfl_down_sync(FULL, a, o); }
// s / k to within a little over half an ulp: the residual takes up the low part
__device__ __forceinline__ float mean_of(Sum2 s, float k)
{
    const float rc = rcp_approx(k), q = s.hi * rc;
    return fmaf(fmaf(-q, k, s.hi) + s.lo, rc, q);
}

// Sums of the runs that leave a warp, for the other warps of its chain (W > 1).
template <int W, class T>
struct RunX {
    T R[W], St[W];        // head sum and tail sum of each warp
    float K[W], Kt[W];    // and their counts
    unsigned char cut[W];
};

// Exchange between the warps of one chain (W > 1).
template <int W>
struct SplitX {
    float a[W], lo[W], hi[W];     // composed map of each warp
    RunX<W, float> run;           // of a round
    RunX<W, Sum2> sum;            // of the solution
    float u[W], u2[W];            // flow of a (new) cut after the warp's last node
    float re[W];                  // r of that node
    unsigned amax[W];
    unsigned char side[W], more[W], heavy[W];  // heavy: 1; the stop flag: 2
    int bad;                      // the chain goes to the fallback, or was stopped
};

template <int W>
__device__ __forceinline__ void split_sync(int bar)
{
    if constexpr (W == 1) {
        __syncwarp();
    } else {
        // literal barrier names: with a name in a register the block would hold all 16, and
        // an SM only four such blocks
        if (bar == 0) asm volatile("bar.sync 1, %0;" ::"n"(W * WARP) : "memory");
        else if (bar == 1) asm volatile("bar.sync 2, %0;" ::"n"(W * WARP) : "memory");
        else if (bar == 2) asm volatile("bar.sync 3, %0;" ::"n"(W * WARP) : "memory");
        else asm volatile("bar.sync 4, %0;" ::"n"(W * WARP) : "memory");
    }
}

// The runs of one chain of lanes of L nodes, joined across its lanes and warps. C: the lane's
// cuts (node j is bit L-1-j, cut after it), bc the lanes of the warp with one; Sh the sum to the
// lane's first cut (or of all its nodes), St after its last one. mean(s, k): value of a run.
template <class T>
struct RunEnds {
    T Rn;          // sum and count from the next lane's first node to the end of its run
    float Kn;
    float zr, zt;  // value of the run at the lane's first node; of the one after its last cut
};
template <int L, int W, class T, class MEAN, class SYNC>
__device__ __forceinline__ RunEnds<T> join_runs(T Sh, T St, unsigned C, unsigned bc, int lane, int wi,
                                                RunX<W, T> *xc, MEAN mean, SYNC sync)
{
    const float kh = C ? (float)(__clz(C) - (31 - L)) : (float)L;  // nodes of the head
    const float kt = (float)(__ffs(C) - 1);                       // nodes after the last cut
    RunEnds<T> e;
    // R, K: sum and count from the lane's first node to the end of its run
    T R = Sh;
    float K = kh;
    int pe = lane;
    if (bc != FULL) {
        const unsigned ahead = bc >> lane;
        pe = ahead ? lane + __ffs(ahead) - 1 : WARP;  // lane where that run ends
#pragma unroll
        for (int o = 1; o < WARP; o <<= 1) {
            const T r2 = shfl_down(R, o);
            if (lane + o < WARP && lane + o <= pe) R = R + r2;
        }
        const float kp = __shfl_sync(FULL, kh, pe & (WARP - 1));
        K = pe < WARP ? (float)((pe - lane) * L) + kp : (float)((WARP - lane) * L);
    }
    const unsigned before = bc & ((1u << lane) - 1u);
    const int src = before ? 31 - __clz(before) : 0;
    if constexpr (W == 1) {
        e.Rn = shfl_down(R, 1);
        e.Kn = __shfl_down_sync(FULL, K, 1);
        e.zt = mean(St + e.Rn, kt + e.Kn);  // (unused in the last lane)
        const float zh = mean(R, K);        // of the lane's first node, if a run begins there
        e.zr = __shfl_sync(FULL, C ? e.zt : zh, src);
        if (lane == 0) e.zr = zh;
        if (lane == WARP - 1) {
            e.Rn = T{};
            e.Kn = 0.f;
        }
    } else {
        // Every warp forms the sum of a run that crosses warps in the same order (tail of
        // the warp it begins in, plus the head sums folded from the right), so that all its
        // nodes get the same bits.
        const int lq = bc ? 31 - __clz(bc) : 0;
        const T Rq = shfl_down(R, 1);
        const float Kq = __shfl_down_sync(FULL, K, 1);
        const T tS = pick(lane < WARP - 1, St + Rq, St);
        const float tK = lane < WARP - 1 ? kt + Kq : kt;
        if (lane == lq) {
            xc->St[wi] = tS;
            xc->Kt[wi] = tK;
        }
        if (lane == 0) {
            xc->R[wi] = R;
            xc->K[wi] = K;
            xc->cut[wi] = bc != 0;
        }
        sync();
        T Rin{}, rr{};               // the same for the next warp's first node; from warp q's
        float Kin = 0.f, kk = 0.f;   // first node to the end of its run
        float zprev = 0.f;           // value of the run that enters this warp
        bool enters = true;          // which is not found yet
#pragma unroll
        for (int q = W - 1; q >= 0; --q) {
            const bool c = xc->cut[q] != 0;
            if (q < wi && enters && c) {
                zprev = mean(xc->St[q] + rr, xc->Kt[q] + kk);
                enters = false;
            }
            rr = xc->R[q] + pick(c, T{}, rr);
            kk = xc->K[q] + (c ? 0.f : kk);
            if (q == wi + 1) {
                Rin = rr;
                Kin = kk;
            }
        }
        if (enters) zprev = mean(rr, kk);  // the chain's first run
        if (pe == WARP) {
            R = R + Rin;
            K += Kin;
        }
        e.Rn = shfl_down(R, 1);
        e.Kn = __shfl_down_sync(FULL, K, 1);
        if (lane == WARP - 1) {
            e.Rn = Rin;
            e.Kn = Kin;
        }
        const bool out = lane == lq;  // its last run leaves the warp
        e.zt = mean(pick(out, tS, St) + pick(out, Rin, e.Rn), (out ? tK : kt) + (out ? Kin : e.Kn));
        e.zr = __shfl_sync(FULL, e.zt, src);
        if (!before) e.zr = zprev;
    }
    return e;
}

// Lane slots of L nodes in shared memory, padded so that the lanes' 16-byte accesses do not
// share banks.
template <int L>
__host__ __device__ constexpr int split_lp()
{
    return (L / 4) % 2 == 1 ? L : L + 4;
}

// fma, clipped to [0, 1] by the instruction itself
__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// y0 += u, y1 -= u and w = 0 where bit is set: predicated, the lanes differ
__device__ __forceinline__ void cut_at(unsigned bit, float u, float &y0, float &y1, float &w)
{
    asm("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n @p add.f32 %0, %0, %3;\n"
        " @p sub.f32 %1, %1, %3;\n @p mov.f32 %2, 0f00000000;\n}"
        : "+f"(y0), "+f"(y1), "+f"(w)
        : "f"(u), "r"(bit));
}
__device__ __forceinline__ void cut_at_unit(unsigned bit, unsigned up, float &y0, float &y1,
                                            float &r)
{
    asm("{\n .reg .pred p, q;\n setp.ne.u32 p, %3, 0;\n setp.ne.u32 q, %4, 0;\n"
        " @q add.f32 %0, %0, 0f3F800000;\n @q add.f32 %1, %1, 0fBF800000;\n"
        " @p mov.f32 %2, 0f00000000;\n}"
        : "+f"(y0), "+f"(y1), "+f"(r)
        : "r"(bit), "r"(up));
}

// Solves one chain held as L nodes per lane in sc (values) and sx (weights if !UNI); writes
// the solution to sx. Returns (the same in every lane) whether it did, or the chain needs the
// fallback, or (STOP) *stop was raised meanwhile, which is looked at once a round.
//
// The walks are bound by issue and by the half-rate ALU pipe (minima, selects, logic), so
// what can be arithmetic on the FMA pipe is: with r = 1, or 0 where the chain is cut after a
// node, a sum that restarts at cuts is s = fma(s, r, y). Node j of a lane is bit L-1-j of
// its masks.
//
// UNI: one weight lamw for every edge. Values are divided by 2 lamw and messages shifted to
// v = m / (2 lamw) + 1/2 in [0, 1], so that a step m -> clip(m + z - y, -w, w) is one
// saturating fma, v -> sat(v r' + (z - y)), r' of the edge before the node. After a cut v
// restarts at 1/2: the half is folded into the values at the cut (with the flow +-1/2: both 0
// or both 1), and a node before a cut compares with 0 alone. The last sums take the values as
// they came, so that scaling costs no digits.
enum SplitEnd { SPLIT_DONE = 0, SPLIT_FALLBACK = 1, SPLIT_STOPPED = 2 };

template <int L, int W, bool UNI, bool STOP>
__device__ __forceinline__ int split_solve(const float *sc, float *sx, SplitX<W> *xc, int n,
                                           float lamw, int lane, int wi, int bar,
                                           [[maybe_unused]] const int *stop)
{
    constexpr int LP = split_lp<L>();
    constexpr unsigned ML = L == 32 ? 0xffffffffu : (1u << L) - 1u;
    const int base = (wi * WARP + lane) * L;
    const float4 *yp = reinterpret_cast<const float4 *>(sc + (wi * WARP + lane) * LP);
    float y[L], w[UNI ? 1 : L], r[UNI ? L : 1], z[L];
    unsigned C = 0;  // cuts (the edge after the node): chain end, padding, decoupled edges
    unsigned ab = 0;  // bits of the largest |y|
    const int last = n - 1 - base;  // the chain's last node, in the lane's numbering
#pragma unroll
    for (int q = 0; q < L / 4; ++q) {
        const float4 t = yp[q];
        y[4 * q] = t.x;
        y[4 * q + 1] = t.y;
        y[4 * q + 2] = t.z;
        y[4 * q + 3] = t.w;
    }
#pragma unroll
    for (int j = 0; j < L; ++j) ab = max(ab, __float_as_uint(y[j]) & 0x7fffffffu);
    if constexpr (UNI) {
        const int k = max(0, min(L, last));  // nodes with an edge to the next one
        C = k >= L ? 0u : ((1u << (L - k)) - 1u) & ML;
#pragma unroll
        for (int j = 0; j < L; ++j) r[j] = j < last ? 1.f : 0.f;
    } else {
        const float4 *wp = reinterpret_cast<const float4 *>(sx + (wi * WARP + lane) * LP);
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            const float4 e = wp[q];  // 0 from the chain's last node on
            w[4 * q] = e.x;
            w[4 * q + 1] = e.y;
            w[4 * q + 2] = e.z;
            w[4 * q + 3] = e.w;
        }
        float sum = 0.f;  // NaN if a weight is (weights are >= 0)
#pragma unroll
        for (int j = 0; j < L; ++j) sum += w[j];
        if (sum != sum) ab = 0x7fffffffu;
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const bool cut = !(w[j] > kSplitTiny);
            w[j] = cut ? 0.f : w[j];
            C = C << 1 | (cut ? 1u : 0u);
        }
    }
    ab = __reduce_max_sync(FULL, ab);
    if constexpr (W > 1) {
        if (lane == 0) xc->amax[wi] = ab;
        if (UNI && lane == WARP - 1) xc->re[wi] = r[UNI ? L - 1 : 0];
        split_sync<W>(bar);
#pragma unroll
        for (int q = 0; q < W; ++q) ab = max(ab, xc->amax[q]);
    }
    const float amax = __uint_as_float(ab);
    // not finite, or beyond what the sums hold: as the dynamic program has it
    if (!(amax <= kSplitMost && (amax >= kSplitLeast || amax == 0.f))) return SPLIT_FALLBACK;
    unsigned H = 0;   // edges whose flow would swamp the values
    unsigned UP = 0;  // UNI: cuts with flow +w
    if constexpr (UNI) {
        if (!(lamw > 1e-30f * amax && lamw > kSplitTiny)) {  // no weight to speak of: x = y
            float4 *xp = reinterpret_cast<float4 *>(sx + (wi * WARP + lane) * LP);
#pragma unroll
            for (int q = 0; q < L / 4; ++q) xp[q] = yp[q];
            return SPLIT_DONE;
        }
        if (lamw > kSplitHeavy * amax) H = ML;
        const float s = 0.5f / lamw;
        const bool head = wi == 0 && lane == 0;
#pragma unroll
        for (int j = 0; j < L; ++j) {
            y[j] *= s;
            if (j == 0 && head) y[j] -= 0.5f;
            if (j == last) y[j] += 0.5f;
        }
    } else {
#pragma unroll
        for (int j = 0; j < L; ++j)
            if (w[j] > kSplitHeavy * amax) H |= 1u << (L - 1 - j);
    }

    // 1, or 0 where the chain is cut after node j: kept for one weight, for a weight per edge
    // made from it (a register per node less, so 32 nodes a lane fit)
    auto keep = [&](int j) {
        if constexpr (UNI) return r[j];
        else return __saturatef(w[j] * 3e38f);
    };
    const bool any_heavy = __any_sync(FULL, H != 0);
    unsigned bc = __ballot_sync(FULL, C != 0);  // lanes with a cut
    float re = 0.f;  // UNI: r of the edge into the lane's first node
    if constexpr (UNI) {
        const float rq = __shfl_up_sync(FULL, r[L - 1], 1);
        if (lane > 0) re = rq;
        else if (W > 1 && wi > 0) re = xc->re[wi - 1];
    }
    auto sync = [&] { split_sync<W>(bar); };
    for (;;) {
        // ---- sums of the runs across lanes ----
        float Sh = 0.f, St = 0.f, b = 1.f;  // to the lane's first cut; after its last one
#pragma unroll
        for (int j = L - 1; j >= 0; --j) {
            const float rj = keep(j);
            Sh = fmaf(Sh, rj, y[j]);
            b *= rj;
            St = fmaf(b, y[j], St);
        }
        const RunEnds<float> run = join_runs<L, W>(
            Sh, St, C, bc, lane, wi, &xc->run, [](float s, float k) { return mean_of(s, k); }, sync);
        float zr = run.zr;

        // ---- mean of every run that begins in the lane, at its first node ----
        float s = run.Rn, k = run.Kn;
#pragma unroll
        for (int j = L - 1; j >= 0; --j) {
            const float rj = keep(j);
            s = fmaf(s, rj, y[j]);
            k = fmaf(k, rj, 1.f);
            z[j] = s * rcp_approx(k);
        }

        // ---- forward: z - y per node, and the lane's composed map ----
        float a = 0.f, lo = 0.f, hi = 0.f;
#pragma unroll
        for (int j = 0; j < L; ++j) {
            if (j > 0 && (UNI ? r : w)[j > 0 ? j - 1 : 0] == 0.f) zr = z[j];
            const float d = zr - y[j];
            z[j] = d;
            a += d;
            if constexpr (UNI) {
                const float rp = j == 0 ? re : r[j > 0 ? j - 1 : 0];
                if (j == 0) {
                    lo = __saturatef(d);
                    hi = __saturatef(rp + d);
                } else {
                    lo = fma_sat(lo, rp, d);
                    hi = fma_sat(hi, rp, d);
                }
            } else {
                if (j == 0) {
                    lo = -w[0];
                    hi = w[0];
                } else {
                    lo = clampw(lo + d, -w[j], w[j]);
                    hi = clampw(hi + d, -w[j], w[j]);
                }
            }
        }
        // m (UNI: v) into the lane's first node. A map with lo == hi forgets its input; from
        // such lanes the message walks through the few others, one lane a step, and only a
        // long row of those takes a scan of the composed maps.
        float m;
        const unsigned kn = __ballot_sync(FULL, lo == hi) | (W == 1 ? 1u : 0u);
        unsigned far = ~kn;
        far &= far << 1;
        far &= far << 2;  // rows of four and more
        if (far == 0 && (W == 1 || (kn & 1u))) {
            float out = W == 1 && lane == 0 ? clampw(a, lo, hi) : hi;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float in = __shfl_up_sync(FULL, out, 1);
                if (!((kn >> lane) & 1u)) out = clampw(in + a, lo, hi);
            }
            if constexpr (W > 1) {
                if (lane == WARP - 1) xc->a[wi] = 0.f, xc->lo[wi] = xc->hi[wi] = out;
                split_sync<W>(bar);
            }
            m = __shfl_up_sync(FULL, out, 1);
        } else {
#pragma unroll
            for (int o = 1; o < WARP; o <<= 1) {
                const float a2 = __shfl_up_sync(FULL, a, o);
                const float l2 = __shfl_up_sync(FULL, lo, o);
                const float h2 = __shfl_up_sync(FULL, hi, o);
                if (lane >= o) {
                    const float nl = clampw(l2 + a, lo, hi);
                    hi = clampw(h2 + a, lo, hi);
                    lo = nl;
                    a += a2;
                }
            }
            if constexpr (W > 1) {
                if (lane == WARP - 1) {
                    xc->a[wi] = a;
                    xc->lo[wi] = lo;
                    xc->hi[wi] = hi;
                }
                split_sync<W>(bar);
            }
            float mc = 0.f;
            if constexpr (W > 1) {
#pragma unroll
                for (int q = 0; q < W; ++q)
                    if (q < wi) mc = clampw(mc + xc->a[q], xc->lo[q], xc->hi[q]);
            }
            m = __shfl_up_sync(FULL, clampw(mc + a, lo, hi), 1);
        }
        if (lane == 0) {
            m = 0.f;
            if constexpr (W > 1) {
#pragma unroll
                for (int q = 0; q < W; ++q)
                    if (q < wi) m = clampw(m + xc->a[q], xc->lo[q], xc->hi[q]);
            }
        }

        int halt = 0;  // on its way while the sides are walked
        if constexpr (STOP) halt = *(const volatile int *)stop;

        // ---- sides: below z (t > w) and above (t < -w), one bit per node ----
        unsigned below = 0, above = 0;
#pragma unroll
        for (int j = 0; j < L; ++j) {
            if constexpr (UNI) {
                const float rp = j == 0 ? re : r[j > 0 ? j - 1 : 0];
                const float t = fmaf(m, rp, z[j]);
                m = fma_sat(m, rp, z[j]);
                below = __funnelshift_l(__float_as_uint(1.f - t), below, 1);
                above = __funnelshift_l(__float_as_uint(t), above, 1);
            } else {
                const float t = m + z[j];
                below = __funnelshift_l(__float_as_uint(w[j] - t), below, 1);
                above = __funnelshift_l(__float_as_uint(t + w[j]), above, 1);
                z[j] = m = clampw(t, -w[j], w[j]);  // the flow of a cut made here
            }
        }
        if constexpr (UNI) below |= C & ~above;
        const unsigned dec = below | above;
        const unsigned U = ~dec & ML;
        const bool first = dec != 0 && ((below >> (31 - __clz(dec | 1u))) & 1u);
        const unsigned bd = __ballot_sync(FULL, dec != 0), bl = __ballot_sync(FULL, first);
        unsigned carry;  // side of the next lane's first node
        {
            const unsigned nx = (bd >> lane) >> 1;
            const int q = lane + __ffs(nx);
            carry = nx ? (bl >> (q & 31)) & 1u : 0u;
            if constexpr (W > 1) {
                if (lane == 0) {
                    const int q0 = bd ? __ffs(bd) - 1 : 0;
                    xc->side[wi] = bd ? 2 + ((bl >> q0) & 1) : 0;
                }
                split_sync<W>(bar);
                if (!nx) {
                    unsigned sd = 0;
#pragma unroll
                    for (int q2 = W - 1; q2 >= 0; --q2)
                        if (q2 > wi && xc->side[q2]) sd = xc->side[q2] & 1u;
                    carry = sd;
                }
            }
        }
        const unsigned S = ((below << 1) | carry) & U;
        const unsigned low = below | (U & ~(U + S));
        const unsigned fresh = (low ^ ((low << 1) | carry)) & ~C & ML;

        // ---- new cuts: fold their flows into the values ----
        const unsigned upf = fresh & low;
        const unsigned bf = __ballot_sync(FULL, fresh != 0);
        bool more = bf != 0;
        bc |= bf;
        // the flow of a cut after the lane's last node (UNI: 2 with its half, 1 without)
        float ue;
        if constexpr (UNI) ue = (upf & 1u) ? 2.f : (float)(fresh & 1u);
        else ue = (fresh & 1u) ? z[L - 1] : 0.f;
        float up = __shfl_up_sync(FULL, ue, 1);
        if (more) {
            float dummy = 0.f;
#pragma unroll
            for (int j = 0; j < L; ++j) {
                const unsigned bit = 1u << (L - 1 - j);
                float &yn = j + 1 < L ? y[j + 1 < L ? j + 1 : 0] : dummy;
                if constexpr (UNI) cut_at_unit(fresh & bit, upf & bit, y[j], yn, r[j]);
                else cut_at(fresh & bit, z[j], y[j], yn, w[j]);
            }
        }
        C |= fresh;
        UP |= upf;
        bool hv = any_heavy && __any_sync(FULL, (fresh & H) != 0);
        if constexpr (W > 1) {
            if (lane == WARP - 1) {
                xc->u[wi] = ue;
                xc->more[wi] = more;
                xc->heavy[wi] = (hv ? 1 : 0) | (halt ? 2 : 0);
            }
            split_sync<W>(bar);
            more = hv = false;
            halt = 0;
#pragma unroll
            for (int q = 0; q < W; ++q) {
                more |= xc->more[q] != 0;
                hv |= (xc->heavy[q] & 1) != 0;
                halt |= xc->heavy[q] & 2;
            }
            if (lane == 0) up = wi > 0 ? xc->u[wi - 1] : 0.f;
        } else {
            if (lane == 0) up = 0.f;
            if constexpr (STOP) halt = __any_sync(FULL, halt);
        }
        if constexpr (UNI) {
            y[0] -= up > 1.f ? 1.f : 0.f;
            if (up > 0.f) re = 0.f;
        } else {
            y[0] -= up;
        }
        if (STOP && halt) return SPLIT_STOPPED;
        if (hv) return SPLIT_FALLBACK;
        if (!more) break;  // the runs are the solution
    }

    // ---- values of the runs: sums in two floats (in one, x was further off than the dynamic
    // program's: 4.7e-8 against 3.2e-8 for 512 x 256, now 2.3e-8). Loops of four nodes, the values
    // in shared memory: unrolled like the rounds this was 16 KB of code that runs once (1024 x 1024
    // with cold caches 30 us, now 26; 4096 x 1023 with weights per edge 65 us, now 62) ----
    float4 *slots = reinterpret_cast<float4 *>(sx + (wi * WARP + lane) * LP);
    unsigned F = 0;  // UNI: cuts that carry a flow; the values as they came, with the flows of all cuts
    float ul = 0.f;  // flow of the cut before the lane's first node
    if constexpr (UNI) {
        const unsigned ends = last >= L ? 0u : ML >> max(0, min(31, last));
        F = C & ~ends;
        const float u = (F & 1u) ? ((UP & 1u) ? lamw : -lamw) : 0.f;
        ul = __shfl_up_sync(FULL, u, 1);
        if (lane == 0) ul = 0.f;
        if constexpr (W > 1) {
            if (lane == WARP - 1) xc->u2[wi] = u;
            sync();
            if (lane == 0 && wi > 0) ul = xc->u2[wi - 1];
        }
    } else {
#pragma unroll
        for (int q = 0; q < L / 4; ++q)
            slots[q] = make_float4(y[4 * q], y[4 * q + 1], y[4 * q + 2], y[4 * q + 3]);
    }
    Sum2 Sh{0.f, 0.f}, St{0.f, 0.f};
    float k = 0.f;
    bool open = true;  // no cut at or after the node
#pragma unroll 1
    for (int q = L / 4 - 1; q >= 0; --q) {
        const int s4 = L - 4 - 4 * q;  // node 4 q + e is bit 3 - e
        const unsigned c4 = C >> s4, f4 = F >> s4, p4 = UP >> s4;
        const float4 t = UNI ? yp[q] : slots[q];
        const float v[4] = {t.x, t.y, t.z, t.w};
        float m[4], u = 0.f;
        auto flow = [&](unsigned bit) { return (f4 & bit) ? ((p4 & bit) ? lamw : -lamw) : 0.f; };
        if constexpr (UNI) u = flow(1u);
#pragma unroll
        for (int e = 3; e >= 0; --e) {
            float c = v[e];
            if constexpr (UNI) {
                const float before = e == 0 && q == 0 ? ul : flow(16u >> e);
                c += u - before;  // equal flows cancel exactly
                u = before;
            }
            const bool cut = c4 & (8u >> e);
            Sh = pick(cut, Sum2{0.f, 0.f}, Sh) + c;
            k = cut ? 1.f : k + 1.f;
            m[e] = mean_of(Sh, k);  // of a run that ends in the lane
            open = open && !cut;
            if (open) St = Sh;
        }
        slots[q] = make_float4(m[0], m[1], m[2], m[3]);
    }
    const RunEnds<Sum2> run = join_runs<L, W>(
        Sh, St, C, bc, lane, wi, &xc->sum, [](Sum2 a, float n) { return mean_of(a, n); }, sync);
    float zr = run.zr;
    const unsigned LC = C & (0u - C);
#pragma unroll 1
    for (int q = 0; q < L / 4; ++q) {
        const unsigned c4 = C >> (L - 4 - 4 * q), l4 = LC >> (L - 4 - 4 * q);
        const float4 t = slots[q];
        float v[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (c4 & (16u >> e)) zr = v[e];    // a run begins
            if (l4 & (16u >> e)) zr = run.zt;  // the bits other lanes have
            v[e] = zr;
        }
        slots[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
    return SPLIT_DONE;
}

struct UnitStride {  // of rows: known at compile time
    __device__ __forceinline__ operator long long() const { return 1; }
};

// Load, solve and store for the chains of one block: `nch` chains of W warps each. Rows are
// loaded by their own warps; columns by the whole block, nch neighbouring columns of a row at
// a time.
template <int L, int W, bool UNI, bool STOP>
__device__ __forceinline__ void split_chain(const SplitView &v, const int *stop, float *smem, SplitX<W> *xall,
                                            int nch, int cs, long long k0, int cnt, long long kc,
                                            long long start, long long wstart, int n,
                                            WsHeader *hdr, float2 *spill)
{
    constexpr int LP = split_lp<L>();
    constexpr int T = W * WARP;
    const int tid = threadIdx.x;
    const int lane = tid & (WARP - 1), warp = tid / WARP;
    const int g = warp / W, wi = warp % W;
    SplitX<W> *xc = xall + g;
    // the chain and the node lane that this thread loads and stores
    const int cc = v.cols ? tid & (nch - 1) : g;
    const int ll = v.cols ? tid / nch : wi * WARP + lane;
    const bool in = cc < cnt;
    const long long st = v.cols ? k0 + cc : start;
    const long long wst = v.cols ? st : wstart;
    float *lc = smem + (size_t)cc * cs, *lx = smem + (size_t)(nch + cc) * cs;
    // What counts here is the number of round trips to memory. With one weight a lane has the
    // registers for two: rows whose arrays all start on 16-byte boundaries go four nodes at a
    // time, and other chains L / 2 (1024 x 1024 rows 24.2 -> 22.2 us). With weights per edge the
    // same made the solve spill (4096 x 1024: 61 -> 69 us), so those take 8 at a time.
    const uintptr_t bits = (uintptr_t)(v.p0 + st) | (uintptr_t)(v.o0 + st) |
                           (v.p1 ? (uintptr_t)(v.p1 + st) : 0) | (v.p2 ? (uintptr_t)(v.p2 + st) : 0) |
                           (v.o1 ? (uintptr_t)(v.o1 + st) : 0);
    const bool vec = UNI && !v.cols && (bits & 15) == 0;
    auto load4 = [&] {
        constexpr int QL = L >= 16 ? 4 : L / 4;  // 16-byte pieces in flight
        const bool h1 = v.p1 != nullptr, h2 = v.p2 != nullptr;
        const int nn = in ? n : 0;
        auto ld = [nn](const float *q, int i) {
            if (i + 3 < nn) return *reinterpret_cast<const float4 *>(q + i);
            return make_float4(i < nn ? q[i] : 0.f, i + 1 < nn ? q[i + 1] : 0.f,
                               i + 2 < nn ? q[i + 2] : 0.f, 0.f);
        };
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int b0 = 0; b0 < L / 4; b0 += QL) {
            float4 a[QL], b[QL], c[QL];
#pragma unroll
            for (int u = 0; u < QL; ++u) {
                if (b0 + u >= L / 4) break;
                const int i = 4 * ((b0 + u) * T + ll);
                a[u] = ld(v.p0 + st, i);
                b[u] = h1 ? ld(v.p1 + st, i) : zero;
                c[u] = h2 ? ld(v.p2 + st, i) : zero;
            }
#pragma unroll
            for (int u = 0; u < QL; ++u) {
                if (b0 + u >= L / 4) break;
                const int i = 4 * ((b0 + u) * T + ll), p = i + (LP - L) * (i / L);
                *reinterpret_cast<float4 *>(lc + p) =
                    make_float4(v.unary(a[u].x, b[u].x, c[u].x), v.unary(a[u].y, b[u].y, c[u].y),
                                v.unary(a[u].z, b[u].z, c[u].z), v.unary(a[u].w, b[u].w, c[u].w));
            }
        }
    };
    constexpr int UL = UNI ? (L <= 16 ? L : L / 2) : L % 8 == 0 ? 8 : 4;
    auto load = [&](auto stride) {
        const long long step = T * (long long)stride, o0 = ll * (long long)stride;
        const float *q0 = v.p0 + st + o0, *q1 = v.p1 + st + o0, *q2 = v.p2 + st + o0,
                    *qw = v.pw + wst + o0;
        const bool h1 = v.p1 != nullptr, h2 = v.p2 != nullptr, hw = v.pw != nullptr;
        const int nn = in ? n : 0;
#pragma unroll 1
        for (int b0 = 0; b0 < L; b0 += UL) {
            float a[UL], b[UL], c[UL], e[UL];
#pragma unroll
            for (int u = 0; u < UL; ++u) {
                const int i = (b0 + u) * T + ll;
                const bool ok = i < nn;
                a[u] = ok ? q0[u * step] : 0.f;
                b[u] = ok && h1 ? q1[u * step] : 0.f;
                c[u] = ok && h2 ? q2[u * step] : 0.f;
                if constexpr (!UNI) e[u] = i < nn - 1 ? (hw ? qw[u * step] : v.lam) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < UL; ++u) {
                const int i = (b0 + u) * T + ll;
                const int p = i + (LP - L) * (i / L);
                lc[p] = v.unary(a[u], b[u], c[u]);
                if constexpr (!UNI) lx[p] = v.ws * e[u];
            }
            q0 += UL * step;
            q1 += UL * step;
            q2 += UL * step;
            qw += UL * step;
        }
    };
    if (v.cols) load(v.stride);
    else if (UNI && vec) load4();
    else load(UnitStride());
    if (tid % T == 0) xc->bad = 0;
    if (v.cols) __syncthreads();
    else split_sync<W>(g);
    int end = SPLIT_DONE;
    if (g < cnt) {
        end = split_solve<L, W, UNI, STOP>(smem + (size_t)g * cs, smem + (size_t)(nch + g) * cs, xc, n,
                                           v.ws * v.lam, lane, wi, g, stop);
        if (end != SPLIT_DONE && tid % T == 0) xc->bad = 1;
    }
    if (v.cols) __syncthreads();
    else split_sync<W>(g);
    if (in && !xall[cc].bad) {
        auto store = [&](auto stride) {
            long long o = st + ll * (long long)stride;
#pragma unroll 4
            for (int q = 0; q < L; ++q) {
                const int i = q * T + ll;
                const int p = i + (LP - L) * (i / L);
                if (i < n) v.emit(o, lx[p], lc[p]);
                o += T * (long long)stride;
            }
        };
        if (UNI && vec) {
#pragma unroll 4
            for (int q = 0; q < L / 4; ++q) {
                const int i = 4 * (q * T + ll), p = i + (LP - L) * (i / L);
                const float4 t = *reinterpret_cast<const float4 *>(lx + p);
                if (i + 3 < n) {
                    *reinterpret_cast<float4 *>(v.o0 + st + i) = t;
                    if (v.mode == SPLIT_INIT) *reinterpret_cast<float4 *>(v.o1 + st + i) = t;
                } else {
                    const float x[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (i + e < n) v.emit(st + i + e, x[e], 0.f);
                }
            }
        } else if (v.cols) {
            store(v.stride);
        } else {
            store(UnitStride());
        }
    }
    if (end == SPLIT_FALLBACK && wi == 0) {
        SplitView vv = v;
        split_fallback(vv, kc, v.cols ? kc : start, v.cols ? kc : wstart, n, lane, spill, hdr);
    }
}

// Nodes per lane for a chain of n nodes (0: longer than W warps hold). Three arrays of 32
// registers fit a lane.
template <int W>
__host__ __device__ constexpr int split_pick(int n)
{
    constexpr int T = 32 * W;
    if (W == 1 && n <= 4 * T) return 4;
    if (W == 1 && n <= 8 * T) return 8;
    if (W == 1 && n <= 12 * T) return 12;
    if (n <= 16 * T) return 16;
    if (n <= 20 * T) return 20;
    if (n <= 24 * T) return 24;
    if (n <= 28 * T) return 28;
    return n <= 32 * T ? 32 : 0;
}

// Floats of one chain's slot array (values; the weights or solutions take another).
template <int W>
__host__ __device__ constexpr int split_slots(int l, int nch)
{
    return 32 * W * ((l / 4) % 2 == 1 ? l : l + 4) + 32 / nch;
}

// Shared memory of the largest block of split_kernel<W>.
template <int W>
constexpr size_t split_smem_most()
{
    const int nch = W == 1 ? 8 : 4;
    return 2 * (size_t)nch * split_slots<W>(32, nch) * sizeof(float);
}

template <int W>
__host__ __device__ constexpr int split_threads()
{
    return W <= 2 ? 256 : 512;
}

// CSR batches: the node range [offsets[0], offsets[num_chains]) of x must not overlap
// that of y or of w (the host checks only x == y, since the offsets live on the device).
// Read by every thread at kernel entry; an overlap flags ERR_BAD_CHAIN and skips the
// whole launch.
__device__ __forceinline__ bool csr_disjoint(const float *x, const float *y, const float *w,
                                             long long off0, long long offn)
{
    if (offn <= off0) return true;
    const size_t len = (size_t)(offn - off0) * sizeof(float);
    auto apart = [&](const float *a) {
        if (a == nullptr) return true;
        const uintptr_t p = (uintptr_t)(x + off0), q = (uintptr_t)(a + off0);
        return p + len <= q || q + len <= p;
    };
    return apart(y) && apart(w);
}

// Chains of one array (tv_chain_solve, tv_chain_solve_columns) or of one image (the phases of
// the 2D solvers). The host fills the view, iterates and step sizes included: read from device
// state they cost each phase a chain of dependent loads and FP64 divisions.
struct SplitSrc {
    SplitView v;
    long long nchains;
    int len;                 // chain length, or with offsets the longest
    const int64_t *offsets;  // CSR rows, or NULL
    int n_lo;                // chains of more than n_lo nodes only
    int lanes;               // nodes a lane takes (0: by the chain's length)
    long long off0;
    const int *done;         // phases of eq. pd: the solve's stop flag, or NULL
    static constexpr bool GAP = false;

    __device__ bool bind(unsigned blk, int nch, SplitView &o, long long &k0, int &cnt,
                         WsHeader *hdr)
    {
        k0 = (long long)blk * nch;
        cnt = (int)min((long long)nch, nchains - k0);
        o = v;
        off0 = 0;
        if (offsets) {
            off0 = (long long)offsets[0];
            if (!csr_disjoint(v.o0, v.p0, v.pw, off0, (long long)offsets[nchains])) {
                if (threadIdx.x == 0) atomicOr(&hdr->status, ERR_BAD_CHAIN);
                return false;
            }
        }
        if (done && *done) return false;
        return true;
    }
    __device__ void chain(const SplitView &o, long long c, long long &start, long long &wstart,
                          int &n, WsHeader *hdr) const
    {
        n = len;
        if (o.cols) {
            start = wstart = c;
        } else if (offsets) {
            const long long a = offsets[c], b = offsets[c + 1];
            // monotone offsets keep every chain inside the first (c+1)*len nodes after
            // offsets[0]; that also bounds its slice of the reserve
            if (a < off0 || b < a || b - a > len || b - off0 > (c + 1) * (long long)len) {
                atomicOr(&hdr->status, ERR_BAD_CHAIN);
                n = 0;
                return;
            }
            start = wstart = a;
            n = (int)(b - a);
        } else {
            start = c * (long long)len;
            wstart = c * o.wrow;
        }
    }
    __device__ float2 *spill(const SplitView &o, long long c, long long start, int n) const
    {
        return o.spill + (offsets ? 2 * (start - off0) + 2 * c : c * (2LL * n + 2));
    }
};

// The column phase of a 2D solve with the gap pass of the iteration before in the first blocks
// of the grid. (A source of its own: with the look at the flag in every chain kernel the others
// were up to 4 % slower.)
struct SplitGapSrc : SplitSrc {  // (done is given)
    static constexpr bool GAP = true;
    GapView gap;
    int gap_blocks;
};

// SRC: bind(block, nch, view, k0, cnt) the chains k0 .. k0 + cnt - 1 of this block;
// chain(view, k, start, wstart, n) one of them (n = 0: skip); spill(view, k, start, n).
template <int W, bool UNI, class SRC>
__global__ void __launch_bounds__(split_threads<W>(), W <= 2 ? 2 : 1)
    split_kernel(SRC src, WsHeader *hdr, int nch, int cs)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ SplitX<W> xall[split_threads<W>() / (WARP * W)];
    float *smem = reinterpret_cast<float *>(smem_raw);
    SplitView v;
    long long k0;
    int cnt;
    unsigned blk = blockIdx.x;
    if constexpr (SRC::GAP) {
        if (blk < (unsigned)src.gap_blocks) {
            gap_pass(src.gap, blk, src.gap_blocks);
            return;
        }
        blk -= src.gap_blocks;
    }
    bool bound = src.bind(blk, nch, v, k0, cnt, hdr);
    // the gap pass may raise the flag meanwhile: the whole block sees it or none of it
    if constexpr (SRC::GAP) bound = !__syncthreads_or(!bound);
    if (!bound) return;
    const int g = threadIdx.x / (WARP * W);
    const long long kc = k0 + g;
    long long start = 0, wstart = 0;
    int n = 0;
    if (v.cols) src.chain(v, k0, start, wstart, n, hdr);
    else if (g < cnt) src.chain(v, kc, start, wstart, n, hdr);
    // chains that a launch for other lengths takes, and empty ones
    if (split_pick<W>(n) == 0 || n <= src.n_lo) n = 0;
    float2 *spill = src.spill(v, kc, start, n);
    const int *stop = nullptr;
    if constexpr (SRC::GAP) stop = src.done;
    if (n > 0) {
        const int l = src.lanes && n > 256 ? src.lanes : split_pick<W>(n);
        if constexpr (W == 1) {
            if (l == 4) split_chain<4, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
            if (l == 8) split_chain<8, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
            if (l == 12) split_chain<12, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
        }
        if (l == 16) split_chain<16, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
        if (l == 20) split_chain<20, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
        if (l == 24) split_chain<24, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
        if (l == 28) split_chain<28, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
        if (l == 32) split_chain<32, W, UNI, SRC::GAP>(v, stop, smem, xall, nch, cs, k0, cnt, kc, start, wstart, n, hdr, spill);
    }
}

}  // namespace tvk
