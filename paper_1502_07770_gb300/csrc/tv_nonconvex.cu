// Chains with continuous piecewise-linear unaries and truncated TV (Sec. 3):
//     x* in argmin_x sum_i f_i(x_i) + sum_{i<n} min(w_i |x_{i+1} - x_i|, C_i),
// f_i any continuous piecewise-linear function bounded below (a stereo matching cost,
// say), w_i >= 0, C_i >= 0 (C_i = +inf: plain TV). Dynamic programming on the chain
// (eq. Message:update): M^_i = f_i + M_{i-1,i}, M_{i,i+1} = M^_i (x) min(w_i|.|, C_i), the
// min-convolution taken as the three consecutive ones of Prop. ConsecutiveMinConvolution:
// with f^1 (Algorithm 1), with f^2 (Algorithm 1 on the mirrored function) and with f^3
// (min(h, min h + C)).
//
// Two warps per chain, one per half of a chain rooted at its middle node (see
// nc_chain_kernel). A message is a list of breakpoints (lambda_p, h(lambda_p)) in shared
// memory plus the slopes of its two ends; a warp goes over a list 32 points at a time, one
// point a lane, so that every lane works, shared accesses do not conflict and the record of
// M^_i is stored in whole lines.
//  - sum: the place of a point in the merged list is its own index plus its rank in the other
//    list (a binary search; for a grid of labels the rounded-up coordinate), every point
//    taking the other function's value by interpolation;
//  - Algorithm 1 as a scan: with g(z) = h(z) - w z, (h (x) f^1)(z) = w z + min_{y<=z} g(y),
//    so a prefix minimum of g decides which points stay (those on the running minimum) and
//    where a falling segment re-crosses it (the new breakpoint of Algorithm 1); votes give
//    each survivor its place. f^2 is the same pass run from the right end with g(z) = h(z) +
//    w z, its survivors written from the end of the buffer;
//  - f^3: values are relative to the minimum; points are clipped to C, crossings added.
// A node costs about 1700 warp instructions at 126 labels and 250 points. With a contiguous
// chunk of the list per lane (a counting and a writing walk each, 18.9 of 32 lanes active) it
// cost 3870, and 1000 x 1482 x 126 took 13.7 ms.
// Values are kept relative to the minimum of M^_i (the minimum is the same after every
// min-convolution, since each f^k >= 0 with f^k(0) = 0); the minima are summed in FP64 into
// the chain's optimum energy. Every M^_i goes to the workspace; the backward pass takes
// the root's x in argmin M^_root and, outwards, x_i = pi_i(x_j) (j the neighbour on the
// root side) from the definition of pi as an argmin of M^_i(z) + min(w |x_j - z|, C) over
// z, evaluated at every breakpoint of M^_i and at x_j, x_j - C/w, x_j + C/w (the first
// minimum in that order).
#include <cuda_runtime.h>

#include <algorithm>

#include "tv_launch.cuh"

using namespace tvk;
using namespace tvh;

namespace {

constexpr int kNcMaxWarps = 4;

// warps per block: as many as fit three message buffers each in ~220 KB of shared memory
// (at least the two warps of one chain: 2 * 24 * 4096 bytes fit)
constexpr int kNcMaxBuffers = 220 * 1024;
int nc_warps(int T) { return std::max(2, std::min(kNcMaxWarps, kNcMaxBuffers / (24 * T))); }

struct NcArgs {
    const int64_t *uoff;  // node -> first breakpoint (N + 1 entries), or NULL: grid unaries
    const float *ulam, *uval;
    int grid_len;         // grid unaries: breakpoints 0..grid_len-1, values uval[i * grid_len + l]
    const float *sl, *sr;
    float sl_s, sr_s;
    const float *w, *C;
    float w_s, C_s;
    const int64_t *offsets;
    long long nchains, nnodes;
    int maxlen;
    int T;                // breakpoints a message may hold
    float *x;
    double *energy;
    float2 *arena;        // chain k's M^_i at k * (maxlen + 1) * T, half 1 from ceil(maxlen/2) * T
    int2 *meta;           // per node: (offset in the chain's arena, count)
    float2 *tails;        // per node: end slopes of M^_i
};

// value of the list (P, t; end slopes sl, sr; constant c0 when t == 0) at z, on the
// segment left of index j (P[j-1] <= z <= P[j])
__device__ __forceinline__ float interp_at(const float2 *P, int t, float sl, float sr, float c0,
                                           int j, float z)
{
    if (t == 0) return c0;
    if (j <= 0) return P[0].y + sl * (z - P[0].x);
    if (j >= t) return P[t - 1].y + sr * (z - P[t - 1].x);
    const float2 a = P[j - 1], b = P[j];
    const float d = b.x - a.x;
    return d > 0.f ? a.y + (b.y - a.y) * ((z - a.x) / d) : a.y;
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}

__device__ __forceinline__ unsigned lanes_below(int lane) { return (1u << lane) - 1u; }

// Points of P (t of them, sorted) left of x: P[q].x < x, or <= x with EQ.
template <bool EQ>
__device__ __forceinline__ int rank_of(const float2 *P, int t, float x)
{
    int lo = 0;
    for (int s = t > 0 ? 1 << (31 - __clz(t)) : 0; s > 0; s >>= 1) {
        const int q = lo + s;
        if (q <= t) {
            const float v = P[q - 1].x;
            if (EQ ? v <= x : v < x) lo = q;
        }
    }
    return lo;
}

// merge A (ta) and B (tb) into O: O = A + B as functions; returns min of O's values (or
// the constant when ta + tb == 0). Ties: A's point first. GRID: B's points lie at 0, 1, ...
template <bool GRID>
__device__ float nc_merge(const float2 *A, int ta, float slA, float srA, float cA, const float2 *B,
                          int tb, float slB, float srB, float2 *O, int lane)
{
    float mn = INFINITY;
    for (int q = lane; q < ta; q += WARP) {
        const float2 e = A[q];
        const int j = GRID ? (int)fminf(fmaxf(ceilf(e.x), 0.f), (float)tb) : rank_of<false>(B, tb, e.x);
        const float v = e.y + interp_at(B, tb, slB, srB, 0.f, j, e.x);
        O[q + j] = make_float2(e.x, v);
        mn = fminf(mn, v);
    }
    for (int q = lane; q < tb; q += WARP) {
        const float2 e = B[q];
        const int i = rank_of<true>(A, ta, e.x);
        const float v = e.y + interp_at(A, ta, slA, srA, cA, i, e.x);
        O[q + i] = make_float2(e.x, v);
        mn = fminf(mn, v);
    }
    mn = warp_min(mn);
    return ta + tb ? mn : cA;
}

// Algorithm 1 as a scan: (H - m) (x) f^1 (REV = false) or (x) f^2 (REV = true), H of t points
// with end slopes sl, sr; values are shifted by -m on the way. With REV the list is read from
// its right end in mirrored coordinates (z -> -z). The result goes to O[0..] or, with REV, to
// the end of O (O[T - count..T)). Optionally copies the shifted input to `store` (the record of
// M^_i). Returns the output count (never above t); sets the output's end slopes.
template <bool REV>
__device__ int nc_mc12(const float2 *H, int t, float sl, float sr, float m, float w, float2 *O,
                       int T, float2 *store, int lane, float &osl, float &osr)
{
    const float vsl = REV ? -sr : sl, vsr = REV ? -sl : sr;  // end slopes of the view
    float Rc = INFINITY;            // minimum of g over the points before this block
    float px = 0.f, pg = INFINITY;  // last point before this block (first of its duplicates)
    float lastx = 0.f;              // x of the point before this block
    int cnt = 0;
    auto put = [&](int pos, float z, float v) {
        O[REV ? T - 1 - pos : pos] = make_float2(REV ? -z : z, v);
    };
    for (int b = 0; b < t; b += WARP) {
        const int q = b + lane;
        const bool in = q < t;
        float2 e = make_float2(0.f, 0.f);
        if (in) {
            const float2 h = H[REV ? t - 1 - q : q];
            e = make_float2(REV ? -h.x : h.x, h.y - m);
            if (store) store[q] = e;
        }
        // a point equal in z to its predecessor adds nothing
        float xb = __shfl_up_sync(FULL, e.x, 1);
        if (lane == 0) xb = lastx;
        const bool nd = in && !(q > 0 && xb == e.x);
        const float g = nd ? fmaf(-w, e.x, e.y) : INFINITY;
        float inc = g;
#pragma unroll
        for (int o = 1; o < WARP; o <<= 1) {
            const float u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc = fminf(inc, u);
        }
        const float ex = __shfl_up_sync(FULL, inc, 1);
        const float R = lane == 0 ? Rc : fminf(Rc, ex);  // minimum over the points before q
        const unsigned ndm = __ballot_sync(FULL, nd);
        const unsigned below = ndm & lanes_below(lane);
        const int src = below ? 31 - __clz(below) : 0;
        float qx = __shfl_sync(FULL, e.x, src), qg = __shfl_sync(FULL, g, src);
        if (!below) {
            qx = px;
            qg = pg;
        }
        // a falling segment re-crosses the running minimum between its ends
        bool cross = nd && q > 0 && qg > R && g < R;
        float z = 0.f;
        if (cross) {
            z = qx + (e.x - qx) * ((R - qg) / (g - qg));
            cross = z > qx && z < e.x;
        }
        const bool keep = nd && g <= R;
        const unsigned cm = __ballot_sync(FULL, cross), km = __ballot_sync(FULL, keep);
        const int pos = cnt + __popc(cm & lanes_below(lane)) + __popc(km & lanes_below(lane));
        if (cross) put(pos, z, fmaf(w, z, R));
        if (keep) put(pos + (cross ? 1 : 0), e.x, e.y);
        cnt += __popc(cm) + __popc(km);
        Rc = fminf(Rc, __shfl_sync(FULL, inc, WARP - 1));
        if (ndm) {
            const int l = 31 - __clz(ndm);
            px = __shfl_sync(FULL, e.x, l);
            pg = __shfl_sync(FULL, g, l);
        }
        lastx = __shfl_sync(FULL, e.x, WARP - 1);
    }
    // the right end of the view: its last point off the running minimum and g falling there:
    // the end re-crosses the minimum
    if (t > 0 && pg > Rc && vsr < w) {
        const float z = px + (Rc - pg) / (vsr - w);
        if (lane == 0) put(cnt, z, fmaf(w, z, Rc));
        ++cnt;
    }
    // end slopes: the left end keeps its slope (<= 0 <= w); the right end follows h where
    // g falls (slope < w), else rises with slope w
    const float nsr = vsr < w ? vsr : w;
    osl = REV ? -nsr : vsl;
    osr = REV ? -vsl : nsr;
    __syncwarp();
    return cnt;
}

// O = min(H, min H + C) for 0 < C < inf; H has minimum 0 (values relative). End slopes
// become 0. Points whose two neighbouring segments are both flat at the cap are dropped.
// Returns the output count, or -1 if it exceeds `cap_out` (then O is not complete).
__device__ int nc_mc3(const float2 *H, int t, float sl, float sr, float C, float2 *O, int cap_out,
                      int lane)
{
    const float cap = C;
    int cnt = 0;
    auto put = [&](int pos, float z, float v) {
        if (pos < cap_out) O[pos] = make_float2(z, v);
    };
    if (t > 0) {
        const float2 e = H[0];
        if (e.y < cap && sl < 0.f) {
            const float z = e.x + (cap - e.y) / sl;
            if (z < e.x) {
                if (lane == 0) put(0, z, cap);
                cnt = 1;
            }
        }
    }
    for (int b = 0; b < t; b += WARP) {
        const int p = b + lane;
        bool keep = false, cross = false;
        float2 e = make_float2(0.f, 0.f);
        float z = 0.f;
        if (p < t) {
            e = H[p];
            const bool lflat = p == 0 || H[p - 1].y >= cap;
            bool rflat = true;
            if (p + 1 < t) {
                const float2 f = H[p + 1];
                rflat = f.y >= cap;
                const float u = e.y - cap, v = f.y - cap;
                if ((u < 0.f && v > 0.f) || (u > 0.f && v < 0.f)) {
                    z = e.x + (f.x - e.x) * (u / (u - v));
                    cross = z > e.x && z < f.x;
                }
            }
            keep = !(e.y >= cap && lflat && rflat);
        }
        const unsigned km = __ballot_sync(FULL, keep), cm = __ballot_sync(FULL, cross);
        const int pos = cnt + __popc(km & lanes_below(lane)) + __popc(cm & lanes_below(lane));
        if (keep) put(pos, e.x, fminf(e.y, cap));
        if (cross) put(pos + (keep ? 1 : 0), z, cap);
        cnt += __popc(km) + __popc(cm);
    }
    if (t > 0) {
        const float2 e = H[t - 1];
        if (e.y < cap && sr > 0.f) {
            const float z = e.x + (cap - e.y) / sr;
            if (z > e.x) {
                if (lane == 0) put(cnt, z, cap);
                ++cnt;
            }
        }
    }
    __syncwarp();
    return cnt > cap_out ? -1 : cnt;
}

struct BestZ {
    float obj;
    int prio;
    float z;
};

__device__ __forceinline__ void best_of(BestZ &b, float obj, int prio, float z)
{
    if (obj < b.obj || (obj == b.obj && prio < b.prio)) b = BestZ{obj, prio, z};
}

__device__ __forceinline__ BestZ warp_best(BestZ b)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(FULL, b.obj, o);
        const int pr = __shfl_xor_sync(FULL, b.prio, o);
        const float z = __shfl_xor_sync(FULL, b.z, o);
        best_of(b, ob, pr, z);
    }
    return b;
}

// argmin over z of H(z) + min(w |xn - z|, C) (pair = true) or of H(z) (pair = false),
// candidates and order as in the file comment; H in shared memory. The points are shared out
// over the lanes; xn and xn -+ C/w, which may lie between them, take a lane each.
__device__ float nc_argmin(const float2 *H, int t, float sl, float sr, bool pair, float xn, float w,
                           float C, int lane)
{
    if (t == 0) return pair ? xn : 0.f;
    BestZ b{INFINITY, 0x7fffffff, 0.f};
    const bool trunc = pair && isfinite(C) && w > 0.f;
    auto pen = [&](float z) {
        if (!pair) return 0.f;
        return fminf(w * fabsf(xn - z), C);
    };
    if (pair && lane < (trunc ? 3 : 1)) {
        const float r = trunc ? C / w : 0.f;
        const float z = lane == 0 ? xn : (lane == 1 ? xn - r : xn + r);
        const int q = rank_of<true>(H, t, z);  // the segment left of point q, or an end
        float hz;
        if (q == 0) {
            hz = H[0].y + sl * (z - H[0].x);
        } else if (q == t) {
            const float2 e = H[t - 1];
            hz = e.y + sr * (z - e.x);
        } else {
            const float2 l = H[q - 1], e = H[q];
            const float d = e.x - l.x;
            hz = d > 0.f ? l.y + (e.y - l.y) * ((z - l.x) / d) : l.y;
        }
        best_of(b, hz + pen(z), lane == 0 ? 0 : t + lane, z);
    }
    for (int p = lane; p < t; p += WARP) {
        const float2 e = H[p];
        best_of(b, e.y + pen(e.x), 1 + p, e.x);
    }
    b = warp_best(b);
    return b.z;
}

// What the two warps of a chain tell each other at the root (shared memory).
struct NcPairXchg {
    double esum[2];   // each half's sum of message minima
    int ta[2], mi[2], at[2];  // each half's final message: count, buffer, first point
    float sl[2], sr[2], cA[2];
    int bad[2];
};

// (at most kNcMaxWarps / 2 = 2 pairs; literal names, or a block would hold all 16 barriers)
__device__ __forceinline__ void pair_bar(int pair)
{
    if (pair == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
    else asm volatile("bar.sync 2, 64;" ::: "memory");
}

// Two warps per chain, rooted at node mid = n/2 (Algorithm 2 may take any root): warp 0
// of the pair runs the forward pass over nodes 0..mid-1, warp 1 over nodes n-1..mid+1
// (the pairwise terms are symmetric, so the update is the same), each ending with the
// message into the root; after a pair barrier both warps form M^_mid = f_mid + M_L + M_R
// from the two messages and take the same x_mid in argmin M^_mid, then each clips its own
// half outwards. Shared memory per warp: three message buffers of T points.
// At most kNcMaxWarps warps a block; no launch bound, which capped the kernel at 72
// registers and spilled it.
__global__ void nc_chain_kernel(NcArgs p, WsHeader *hdr)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & (WARP - 1);
    const int warp = threadIdx.x / WARP;
    const int role = warp & 1;
    const int pair = warp >> 1;
    const int pairs = blockDim.x / (2 * WARP);
    const long long k = (long long)blockIdx.x * pairs + pair;
    const int T = p.T;
    NcPairXchg *xs = reinterpret_cast<NcPairXchg *>(smem_raw) + pair;
    float2 *buf0 = reinterpret_cast<float2 *>(smem_raw + ((pairs * sizeof(NcPairXchg) + 15) & ~(size_t)15));
    auto Pw = [&](int w, int b) { return buf0 + ((size_t)w * 3 + b) * T; };
    auto P = [&](int b) { return Pw(warp, b); };
    if (k >= p.nchains) return;  // both warps of the pair
    long long start = k * (long long)p.maxlen;
    int n = p.maxlen;
    if (p.offsets) {
        const long long off0 = p.offsets[0], lo = p.offsets[k], hi = p.offsets[k + 1];
        if (lo < off0 || hi < lo || hi - lo > p.maxlen || hi > p.nnodes) {
            if (lane == 0 && role == 0) atomicOr(&hdr->status, ERR_BAD_CHAIN);
            return;
        }
        start = lo;
        n = (int)(hi - lo);
    }
    if (n == 0) {
        if (lane == 0 && role == 0) p.energy[k] = 0.0;
        return;
    }
    const int mid = n >> 1;
    const int cnt = role == 0 ? mid : n - 1 - mid;
    const long long half_cap = (long long)((p.maxlen + 1) / 2) * T;
    float2 *arena = p.arena + k * (long long)(p.maxlen + 1) * T + role * half_cap;
    // node of step j and the node on the root side of its edge
    auto node_of = [&](int j) { return role == 0 ? j : n - 1 - j; };
    auto edge_of = [&](int i) { return role == 0 ? i : i - 1; };  // index of w / C of the edge

    // Grid unaries of up to kPre * 32 labels are fetched a node ahead (ahead[]).
    constexpr int kPre = 8;
    float ahead[kPre];
    const bool pre = !p.uoff && p.grid_len <= kPre * WARP;
    auto fetch = [&](long long node) {
        const float *v = p.uval + node * (long long)p.grid_len;
#pragma unroll
        for (int q = 0; q < kPre; ++q)
            if (q * WARP + lane < p.grid_len) ahead[q] = v[q * WARP + lane];
    };
    auto load_unary = [&](long long node, float2 *F, int &tf, float &slF, float &srF) -> bool {
        if (p.uoff) {
            const long long u0 = p.uoff[node], u1 = p.uoff[node + 1];
            tf = (int)max(0LL, u1 - u0);
            if (tf > T) return false;
            for (int q = lane; q < tf; q += WARP) F[q] = make_float2(p.ulam[u0 + q], p.uval[u0 + q]);
        } else {
            tf = p.grid_len;
            if (tf > T) return false;
            if (pre) {
#pragma unroll
                for (int q = 0; q < kPre; ++q)
                    if (q * WARP + lane < tf)
                        F[q * WARP + lane] = make_float2((float)(q * WARP + lane), ahead[q]);
            } else {
                for (int q = lane; q < tf; q += WARP)
                    F[q] = make_float2((float)q, p.uval[node * (long long)p.grid_len + q]);
            }
        }
        slF = p.sl ? p.sl[node] : p.sl_s;
        srF = p.sr ? p.sr[node] : p.sr_s;
        if (tf == 0) slF = srF = 0.f;
        return true;
    };
    auto merge = [&](const float2 *A, int tA, float slA, float srA, float cA, const float2 *B, int tB,
                     float slB, float srB, float2 *O) {
        return p.uoff ? nc_merge<false>(A, tA, slA, srA, cA, B, tB, slB, srB, O, lane)
                      : nc_merge<true>(A, tA, slA, srA, cA, B, tB, slB, srB, O, lane);
    };

    // ---------------- forward pass over this warp's half ----------------
    int mi = 0, ta = 0, at = 0;  // the message: ta points of buffer mi from point `at`
    if (pre && cnt > 0) fetch(start + node_of(0));
    float slA = 0.f, srA = 0.f, cA = 0.f;
    double energy = 0.0;
    unsigned aoff = 0;
    bool bad = false;
    for (int j = 0; j < cnt; ++j) {
        const int i = node_of(j);
        const long long node = start + i;
        const int fi = 1 - mi;
        float2 *F = P(fi);
        int tf;
        float slF, srF;
        if (!load_unary(node, F, tf, slF, srF) || ta + tf > T ||
            (long long)aoff + ta + tf > half_cap) {
            bad = true;
            break;
        }
        __syncwarp();
        if (pre) fetch(start + (j + 1 < cnt ? node_of(j + 1) : mid));
        float2 *Mh = P(2);
        const int th = ta + tf;
        const float m = merge(P(mi) + at, ta, slA, srA, cA, F, tf, slF, srF, Mh);
        const float slH = slA + slF, srH = srA + srF;
        energy += (double)m;
        __syncwarp();
        if (lane == 0) {
            p.meta[node] = make_int2((int)aoff, th);
            p.tails[node] = make_float2(slH, srH);
        }
        const int e = edge_of(i);
        const float wi = p.w ? p.w[start + e] : p.w_s;
        const float Ci = p.C ? p.C[start + e] : p.C_s;
        // (x) f^1 into F's buffer (free now), recording M^_i; (x) f^2 into mi's buffer
        float s1l, s1r, s2l, s2r;
        const int t1 = nc_mc12<false>(Mh, th, slH, srH, m, wi, F, T, arena + aoff, lane, s1l, s1r);
        aoff += (unsigned)th;
        const int t2 = nc_mc12<true>(F, t1, s1l, s1r, 0.f, wi, P(mi), T, nullptr, lane, s2l, s2r);
        at = T - t2;
        if (isfinite(Ci)) {
            if (Ci <= 0.f) {
                ta = 0;
                cA = 0.f;
                slA = srA = 0.f;
            } else {
                const int t3 = nc_mc3(P(mi) + at, t2, s2l, s2r, Ci, F, T, lane);
                if (t3 < 0) {
                    bad = true;
                    break;
                }
                mi = fi;
                at = 0;
                ta = t3;
                slA = srA = 0.f;
                cA = 0.f;
            }
        } else {
            ta = t2;
            slA = s2l;
            srA = s2r;
            cA = 0.f;
        }
        __syncwarp();
    }
    bad = __any_sync(FULL, bad);
    if (lane == 0) {
        xs->esum[role] = energy;
        xs->ta[role] = ta;
        xs->mi[role] = mi;
        xs->at[role] = at;
        xs->sl[role] = slA;
        xs->sr[role] = srA;
        xs->cA[role] = cA;
        xs->bad[role] = bad ? 1 : 0;
    }
    pair_bar(pair);

    // ---------------- root: M^_mid = M_L + M_R + f_mid, both warps alike ----------------
    const bool any_bad = xs->bad[0] || xs->bad[1];
    float xmid = 0.f;
    bool root_bad = any_bad;
    int tr = 0;
    float slr = 0.f, srr = 0.f, mr = 0.f;
    if (!any_bad) {
        const int tL = xs->ta[0], tR = xs->ta[1];
        const float2 *ML = Pw(2 * pair, xs->mi[0]) + xs->at[0],
                     *MR = Pw(2 * pair + 1, xs->mi[1]) + xs->at[1];
        const int other = 1 - xs->mi[role];  // my free message buffer
        if (tL + tR > T) {
            root_bad = true;
        } else {
            nc_merge<false>(ML, tL, xs->sl[0], xs->sr[0], xs->cA[0], MR, tR, xs->sl[1], xs->sr[1],
                            P(2), lane);
        }
        int tf = 0;
        float slF = 0.f, srF = 0.f;
        if (pre && cnt == 0) fetch(start + mid);
        if (!root_bad && !load_unary(start + mid, P(other), tf, slF, srF)) root_bad = true;
        if (!root_bad && tL + tR + tf > T) root_bad = true;
        __syncwarp();
        // both warps have read both messages before either overwrites its own
        pair_bar(pair);
        if (!root_bad) {
            const float cLR = (tL + tR == 0) ? xs->cA[0] + xs->cA[1] : 0.f;
            const float slLR = xs->sl[0] + xs->sl[1], srLR = xs->sr[0] + xs->sr[1];
            float2 *R = P(xs->mi[role]);
            mr = merge(P(2), tL + tR, slLR, srLR, cLR, P(other), tf, slF, srF, R);
            tr = tL + tR + tf;
            slr = slLR + slF;
            srr = srLR + srF;
            __syncwarp();
            xmid = nc_argmin(R, tr, slr, srr, false, 0.f, 0.f, 0.f, lane);
        }
    } else {
        pair_bar(pair);
    }
    if (root_bad) {
        if (role == 0) {
            if (lane == 0) {
                atomicOr(&hdr->status, ERR_CAPACITY);
                p.energy[k] = NAN;
            }
            for (int i = lane; i < n; i += WARP) p.x[start + i] = NAN;
        }
        return;
    }
    if (role == 0) {
        if (lane == 0) {
            p.energy[k] = xs->esum[0] + xs->esum[1] + (double)mr;
            p.x[start + mid] = xmid;
        }
    }
    __syncwarp();
    __threadfence_block();
    // ---------------- backward: clip this half outwards from the root ----------------
    // The records do not depend on x: they are copied a node ahead into two of the buffers, and
    // the places of the records two ahead.
    auto place = [&](int j, int2 &mt, float2 &tl) {
        if (j < 0) return;
        const long long node = start + node_of(j);
        mt = p.meta[node];
        tl = p.tails[node];
    };
    auto copy = [&](int j, const int2 &mt) {
        if (j >= 0)
            for (int q = lane; q < mt.y; q += WARP) cp_async8(P(j & 1) + q, arena + mt.x + q);
        cp_async_commit();
    };
    float xn = xmid;
    int2 m0 = make_int2(0, 0), m1 = m0;
    float2 t0 = make_float2(0.f, 0.f), t1 = t0;
    place(cnt - 1, m0, t0);
    place(cnt - 2, m1, t1);
    copy(cnt - 1, m0);
    for (int j = cnt - 1; j >= 0; --j) {
        copy(j - 1, m1);
        int2 m2 = make_int2(0, 0);
        float2 t2 = make_float2(0.f, 0.f);
        place(j - 2, m2, t2);
        cp_async_wait<1>();
        __syncwarp();
        const int i = node_of(j);
        const int e = edge_of(i);
        const float wi = p.w ? p.w[start + e] : p.w_s;
        const float Ci = p.C ? p.C[start + e] : p.C_s;
        const float xi = nc_argmin(P(j & 1), m0.y, t0.x, t0.y, true, xn, wi, Ci, lane);
        if (lane == 0) p.x[start + i] = xi;
        xn = xi;
        m0 = m1;
        t0 = t1;
        m1 = m2;
        t1 = t2;
        __syncwarp();
    }
    cp_async_wait<0>();
}

struct NcWs {
    WsHeader *hdr;
    float2 *arena;
    int2 *meta;
    float2 *tails;
    size_t bytes;
};

NcWs carve_nc(void *base, long long nodes, long long nchains, long long maxlen, int T)
{
    Carver cv(base);
    NcWs o;
    o.hdr = cv.take<WsHeader>(1);
    o.meta = cv.take<int2>((size_t)nodes);
    o.tails = cv.take<float2>((size_t)nodes);
    o.arena = cv.take<float2>((size_t)(nchains * (maxlen + 1) * (long long)T));
    o.bytes = align_up(cv.used, 256);
    return o;
}

}  // namespace

extern "C" {

size_t tv_chain_nonconvex_workspace_size(int64_t num_nodes, int64_t num_chains, int64_t max_len,
                                         int max_breakpoints)
{
    if (num_nodes < 0 || num_chains < 0 || max_len < 0 || max_breakpoints < 1) return 0;
    return carve_nc(nullptr, num_nodes, num_chains, max_len, max_breakpoints).bytes;
}

tv_status tv_chain_solve_nonconvex(const int64_t *d_uoff, const float *d_ulam,
                                   const float *d_uval, int grid_len, const float *d_sl,
                                   const float *d_sr, float sl, float sr, const float *d_w,
                                   float w, const float *d_C, float C, const int64_t *d_offsets,
                                   int64_t num_nodes, int64_t num_chains, int64_t max_len,
                                   int max_breakpoints, float *d_x, double *d_energy,
                                   void *d_workspace, size_t workspace_bytes, tv_stream_t stream)
{
    clear_error();
    if (num_chains < 0 || max_len < 0 || num_nodes < 0 || max_breakpoints < 1 ||
        max_breakpoints > 4096 || max_len > (1LL << 24)) {
        set_error("tv_chain_solve_nonconvex: need num_chains, max_len, num_nodes >= 0 and "
                  "1 <= max_breakpoints <= 4096");
        return TV_ERR_INVALID;
    }
    if (max_len * (long long)max_breakpoints >= (1LL << 31)) {
        set_error("tv_chain_solve_nonconvex: max_len * max_breakpoints must stay below 2^31");
        return TV_ERR_INVALID;
    }
    if (!d_offsets && num_nodes != num_chains * max_len) {
        set_error("tv_chain_solve_nonconvex: without offsets, num_nodes = num_chains * max_len");
        return TV_ERR_INVALID;
    }
    if (!d_uval || !d_x || !d_energy || !d_workspace || (d_uoff && !d_ulam) ||
        (!d_uoff && grid_len < 1)) {
        set_error("tv_chain_solve_nonconvex: uval, x, energy and workspace must not be NULL; "
                  "ulam with uoff, or grid_len >= 1 without");
        return TV_ERR_INVALID;
    }
    if (!d_uoff && grid_len > max_breakpoints) {
        set_error("tv_chain_solve_nonconvex: grid_len above max_breakpoints");
        return TV_ERR_INVALID;
    }
    if ((!d_sl && !(sl <= 0.f)) || (!d_sr && !(sr >= 0.f)) ||
        (!d_w && !(w >= 0.f && w < INFINITY)) || (!d_C && !(C >= 0.f))) {
        set_error("tv_chain_solve_nonconvex: need sl <= 0 <= sr, finite w >= 0, C >= 0");
        return TV_ERR_INVALID;
    }
    if (num_chains == 0 || max_len == 0) return TV_OK;
    NcWs ws = carve_nc(d_workspace, num_nodes, num_chains, max_len, max_breakpoints);
    if (workspace_bytes < ws.bytes) {
        set_error("tv_chain_solve_nonconvex: workspace of %zu bytes, %zu needed", workspace_bytes,
                  ws.bytes);
        return TV_ERR_NOMEM;
    }
    cudaStream_t s = (cudaStream_t)stream;
    tv_status st = check_cuda(cudaMemsetAsync(ws.hdr, 0, sizeof(WsHeader), s), "memset");
    if (st != TV_OK) return st;
    NcArgs p{d_uoff, d_ulam, d_uval, grid_len, d_sl, d_sr, sl, sr, d_w, d_C, w, C, d_offsets,
             num_chains, num_nodes, (int)max_len, max_breakpoints, d_x, d_energy, ws.arena,
             ws.meta, ws.tails};
    const int pairs = std::max(1, nc_warps(max_breakpoints) / 2);
    const int wpb = 2 * pairs;
    const size_t smem = ((pairs * sizeof(NcPairXchg) + 15) & ~(size_t)15) +
                        (size_t)wpb * 3 * max_breakpoints * sizeof(float2);
    // the most of any launch: the limit is the kernel's, and calls on other threads share it
    constexpr int most = kNcMaxBuffers + (kNcMaxWarps / 2 * (int)sizeof(NcPairXchg) + 15) / 16 * 16;
    st = check_cuda(cudaFuncSetAttribute(nc_chain_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, most),
                    "cudaFuncSetAttribute");
    if (st != TV_OK) return st;
    const long long blocks = (num_chains + pairs - 1) / pairs;
    const bool prof = prof_on();
    if (prof) prof_mark(PK_CHAIN, s, true);
    nc_chain_kernel<<<(unsigned)blocks, wpb * WARP, smem, s>>>(p, ws.hdr);
    st = check_cuda(cudaGetLastError(), "non-convex chain kernel launch");
    if (st == TV_OK) note_launch();
    if (prof) prof_mark(PK_CHAIN, s, false);
    return st;
}

}  // extern "C"
