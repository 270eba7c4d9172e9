// Vector-Jacobian product of the chain TV prox (the backward of a
// differentiable TV layer built on eq. 1D-ROF).
//
// Away from degenerate inputs the optimality conditions of eq. 1D-ROF fix the
// solution on every maximal run S = [l..r] of equal values ("segment") as
//     x_S = mean(y_S) + (u_r - u_{l-1}) / |S|,   u_e = w_e * sign(x_{e+1} - x_e)
// at the jump edges bounding S (u = 0 past the chain ends). Hence, for an
// upstream gradient g = dL/dx,
//     dL/dy_j = mean_{i in S(j)} g_i,
//     dL/dw_e = sign_e * (mean_{S left of e} g - mean_{S right of e} g) at a jump
//               edge e, and 0 on the edges inside a segment.
// Segments are read off the forward output: the backward clip of Algorithm 2
// copies x_{i+1} into x_i whenever the clip is inactive, so fused neighbours are
// bitwise equal.
//
// Chains of at most kSplitMaxLen nodes (run_means_kernel; not large batches of short ones): the
// chain lies in the shared memory of one warp (2 or 4 for more than 1024 nodes), L consecutive
// nodes a lane in padded slots, through which global accesses are whole lines. Run sums are walks
// that restart behind a run's last node, joined across lanes by one segmented scan (join_runs of
// tv_split.cuh), and are carried in two floats. The two reads and one or two writes bound the
// kernel from about 16384 chains on, before that the walks' latency. 4096 x 1024 with both
// gradients: 31 -> 14.4 us against the step-wise kernel (back to back; 16.2 with the walks
// unrolled over the chain in registers); 16384 x 1024 55 us (4.9 TB/s).
//
// Others (chain_vjp_kernel): one warp per chain, 32 nodes per step: a forward segmented
// scan of (sum, count) with a carry across steps yields each segment's mean at its last node;
// a reverse segmented scan spreads it over the segment. The loads of kGradUnroll steps are
// issued together before their scans run one after another: with one step's loads in flight
// per warp, the kernel was bound by memory latency.
#include <cuda_runtime.h>

#include "tv_launch.cuh"
#include "tv_split.cuh"

using namespace tvk;
using namespace tvh;

namespace {

constexpr int kGradWarps = 4;
constexpr int kGradUnroll = 4;        // steps whose loads are in flight together

struct GradArgs {
    const float *x, *g;
    const int64_t *offsets;
    long long nchains;
    int maxlen;
    float *gy, *gw;
    bool full;  // also write gw (0) at a chain's last node
};

// GW: with grad_w.
template <bool GW>
__global__ void __launch_bounds__(kGradWarps * WARP) chain_vjp_kernel(GradArgs a, WsHeader *hdr)
{
    const int lane = threadIdx.x & (WARP - 1);
    const int warp = threadIdx.x / WARP;
    const long long k = (long long)blockIdx.x * kGradWarps + warp;
    if (k >= a.nchains) return;
    long long start;
    int n;
    if (a.offsets) {
        const long long o0 = a.offsets[0], lo = a.offsets[k], hi = a.offsets[k + 1];
        if (lo < o0 || hi < lo || hi - lo > a.maxlen || hi - o0 > (k + 1) * (long long)a.maxlen) {
            if (lane == 0) atomicOr(&hdr->status, ERR_BAD_CHAIN);
            return;
        }
        start = lo;
        n = (int)(hi - lo);
    } else {
        start = k * (long long)a.maxlen;
        n = a.maxlen;
    }
    if (n == 0) return;
    const float *x = a.x + start, *g = a.g + start;
    float *gy = a.gy + start;
    float *mean = gy;  // segment means wait in grad_y itself
    const int nblk = (n + WARP - 1) / WARP;

    // ---- forward: segmented (sum, count); the mean lands on each segment's last node
    constexpr int U = kGradUnroll;
    float carry_s = 0.f;
    int carry_c = 0;  // open segment entering this block
    for (int b0 = 0; b0 < nblk; b0 += U) {
        float xv[U], xp[U], xn[U], gv[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int i = (b0 + q) * WARP + lane;
            const bool in = i < n;
            xv[q] = in ? x[i] : 0.f;
            xp[q] = (in && i > 0) ? x[i - 1] : 0.f;
            xn[q] = (i + 1 < n) ? x[i + 1] : 0.f;
            gv[q] = in ? g[i] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int b = b0 + q;
            if (b >= nblk) break;  // the same for every lane
            const int i = b * WARP + lane;
            const bool in = i < n;
            const float xi = xv[q];
            const float xprev = xp[q];
            const float xnext = xn[q];
            const bool head = in && (i == 0 || xi != xprev);
            const bool tail = in && (i == n - 1 || xi != xnext);
            float s = gv[q];
            // the segment of node i starts at lane hs of this step (-1: before it); the
            // sum over [max(hs, 0), lane] by the doubling scan, taking a partial sum only
            // from a lane inside the segment; the count from the lane index
            const unsigned hm = __ballot_sync(FULL, head) & (0xffffffffu >> (WARP - 1 - lane));
            const int hs = hm ? WARP - 1 - __clz(hm) : -1;
#pragma unroll
            for (int o = 1; o < WARP; o <<= 1) {
                const float s2 = __shfl_up_sync(FULL, s, o);
                if (lane - o >= (hs < 0 ? 0 : hs)) s += s2;
            }
            int c = hs < 0 ? lane + 1 + carry_c : lane - hs + 1;
            if (hs < 0) s += carry_s;
            if (tail) mean[i] = s / (float)c;
            carry_s = __shfl_sync(FULL, s, WARP - 1);
            carry_c = __shfl_sync(FULL, c, WARP - 1);
            // a segment that ended on the block's last node does not carry on
            const bool last_tail = __shfl_sync(FULL, (int)tail, WARP - 1);
            if (last_tail) {
                carry_s = 0.f;
                carry_c = 0;
            }
        }
    }
    __syncwarp();
    // ---- backward: every node takes the mean stored at its segment's last node
    // (a batch's tail means are read before any of its outputs is written: the means live in
    // grad_y itself, each at its segment's last node, inside the step that owns that node)
    float carry_m = 0.f;
    for (int b0 = nblk - 1; b0 >= 0; b0 -= U) {
        float xv[U], xn[U], mv[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int i = (b0 - q) * WARP + lane;
            const bool in = b0 - q >= 0 && i < n;
            xv[q] = in ? x[i] : 0.f;
            xn[q] = (in && i + 1 < n) ? x[i + 1] : 0.f;
            mv[q] = (in && (i == n - 1 || xv[q] != xn[q])) ? mean[i] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int b = b0 - q;
            if (b < 0) break;  // the same for every lane
            const int i = b * WARP + lane;
            const bool in = i < n;
            const float xi = xv[q];
            const float xnext = xn[q];
            const bool tail = in && (i == n - 1 || xi != xnext);
            // the mean sits at the segment's last node: lane te of this step, or (no tail
            // at or after this lane) a later step, whose mean is the carry
            const unsigned tm = __ballot_sync(FULL, tail) & (0xffffffffu << lane);
            const int te = tm ? __ffs(tm) - 1 : lane;
            float m = __shfl_sync(FULL, mv[q], te);
            if (!tm) m = carry_m;
            const float mn = __shfl_down_sync(FULL, m, 1);
            const float mright = (lane == WARP - 1) ? carry_m : mn;  // mean of node i+1
            __syncwarp();
            if (in) {
                gy[i] = m;
                // jump edge i -> i+1: sign * (mean left - mean right); fused edges: 0
                if (GW && i + 1 < n)
                    a.gw[start + i] = tail ? ((xnext > xi ? 1.f : -1.f) * (m - mright)) : 0.f;
            }
            carry_m = __shfl_sync(FULL, m, 0);
        }
    }
    if (GW && a.full && lane == 0) a.gw[start + n - 1] = 0.f;
}

// Exchange between the warps of one chain.
template <int W>
struct MeansX {
    RunX<W, Sum2> run;
    float z[W];
};

// Mean of a run. A sum that is not finite is the mean: the residual would turn an infinite one
// into NaN.
__device__ __forceinline__ float run_mean(Sum2 s, float k)
{
    return fabsf(s.hi) < INFINITY ? mean_of(s, k) : s.hi;
}

template <int L, int W, bool VEC>
__device__ __forceinline__ void run_means(const GradArgs &a, long long start, int n, float *sx,
                                          float *sg, MeansX<W> *xc)
{
    constexpr int LP = split_lp<L>();
    constexpr int T = W * WARP;
    const int lane = threadIdx.x & (WARP - 1), wi = W == 1 ? 0 : threadIdx.x / WARP;
    const int ll = wi * WARP + lane;
    auto sync = [&]() {  // W > 1: one chain per block
        if constexpr (W == 1) __syncwarp();
        else __syncthreads();
    };
    const float *x = a.x + start, *g = a.g + start;
    if constexpr (VEC) {
        float4 vx[L / 4], vg[L / 4];
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            const int i = 4 * (q * T + ll);
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            vx[q] = i < n ? *reinterpret_cast<const float4 *>(x + i) : zero;
            vg[q] = i < n ? *reinterpret_cast<const float4 *>(g + i) : zero;
        }
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            const int i = 4 * (q * T + ll), p = i + (LP - L) * (i / L);
            *reinterpret_cast<float4 *>(sx + p) = vx[q];
            *reinterpret_cast<float4 *>(sg + p) = vg[q];
        }
    } else {
        constexpr int U = L % 8 == 0 ? 8 : 4;
#pragma unroll 1
        for (int q0 = 0; q0 < L; q0 += U) {
            float vx[U], vg[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = (q0 + u) * T + ll;
                vx[u] = i < n ? x[i] : 0.f;
                vg[u] = i < n ? g[i] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = (q0 + u) * T + ll, p = i + (LP - L) * (i / L);
                sx[p] = vx[u];
                sg[p] = vg[u];
            }
        }
    }
    sync();
    // One walk from the right, restarting at cuts (selected, not multiplied by 0: an infinite or
    // NaN gradient stays in its own run), gives the sum to the lane's first cut, the one after
    // its last cut, and the means of the runs that lie in the lane, at their first nodes. Sums
    // are carried in two floats: node after node in one float a mean was off by a third more
    // than from the step-wise kernel's tree of sums. (Loops of four nodes, the values in shared
    // memory: unrolled, the code that runs once per chain took longer to fetch than to run.)
    // node j of the lane is bit L-1-j: C the runs' last nodes, UP where the solution rises
    float4 *xs = reinterpret_cast<float4 *>(sx + ll * LP), *gs = reinterpret_cast<float4 *>(sg + ll * LP);
    const int last = n - 1 - ll * L;
    const Sum2 zero{0.f, 0.f};
    Sum2 Sh = zero, St = zero;
    float k = 0.f;
    bool open = true;  // no cut at or after the node
    unsigned C = 0, UP = 0;
    float xn = ll + 1 < T ? sx[(ll + 1) * LP] : 0.f;
#pragma unroll 1
    for (int q = L / 4 - 1; q >= 0; --q) {
        const float4 xq = xs[q], gq = gs[q];
        const float xv[4] = {xq.x, xq.y, xq.z, xq.w}, g4[4] = {gq.x, gq.y, gq.z, gq.w};
        float m[4];
        unsigned c4 = 0, u4 = 0;
#pragma unroll
        for (int e = 3; e >= 0; --e) {
            const bool cut = 4 * q + e >= last || xv[e] != xn;
            c4 |= cut ? 8u >> e : 0u;
            u4 |= xn > xv[e] ? 8u >> e : 0u;
            xn = xv[e];
            Sh = pick(cut, zero, Sh) + g4[e];
            k = cut ? 1.f : k + 1.f;
            m[e] = run_mean(Sh, k);
            open = open && !cut;
            if (open) St = Sh;
        }
        C |= c4 << (L - 4 - 4 * q);
        UP |= u4 << (L - 4 - 4 * q);
        gs[q] = make_float4(m[0], m[1], m[2], m[3]);
    }
    const unsigned bc = __ballot_sync(FULL, C != 0);
    const RunEnds<Sum2> run = join_runs<L, W>(Sh, St, C, bc, lane, wi, &xc->run, run_mean, sync);
    float zr = run.zr;
    float zn = 0.f;  // mean of the node after the lane's last
    if (a.gw) {
        zn = __shfl_down_sync(FULL, zr, 1);
        if constexpr (W > 1) {
            if (lane == 0) xc->z[wi] = zr;
        }
        sync();  // every lane has read its neighbour's x, and the warps' first means are there
        if constexpr (W > 1) {
            if (lane == WARP - 1) zn = wi + 1 < W ? xc->z[wi + 1 < W ? wi + 1 : 0] : 0.f;
        }
    }
    const unsigned LC = C & (0u - C);
#pragma unroll 1
    for (int q = 0; q < L / 4; ++q) {
        const int s4 = L - 4 - 4 * q;
        const unsigned c4 = C >> s4, l4 = LC >> s4, u4 = UP >> s4;
        const float4 t = gs[q];
        float v[5] = {t.x, t.y, t.z, t.w, zn};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (c4 & (16u >> e)) zr = v[e];    // a run begins
            if (l4 & (16u >> e)) zr = run.zt;  // the bits other lanes have
            v[e] = zr;
        }
        gs[q] = make_float4(v[0], v[1], v[2], v[3]);
        if (!a.gw) continue;
        if (q + 1 < L / 4) v[4] = (l4 & 1u) ? run.zt : (c4 & 1u) ? gs[q + 1].x : zr;
        float d[4];  // a jump edge: sign * (mean left - mean right); fused edges: 0
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned bit = 8u >> e;
            const float h = v[e] - v[e + 1];
            d[e] = !(c4 & bit) || 4 * q + e >= last ? 0.f : (u4 & bit) ? h : -h;
        }
        xs[q] = make_float4(d[0], d[1], d[2], d[3]);
    }
    sync();
    float *gy = a.gy + start, *gw = a.gw ? a.gw + start : nullptr;
    if constexpr (VEC) {
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            const int i = 4 * (q * T + ll), p = i + (LP - L) * (i / L);
            if (i >= n) continue;
            *reinterpret_cast<float4 *>(gy + i) = *reinterpret_cast<const float4 *>(sg + p);
            if (!gw) continue;
            const float4 v = *reinterpret_cast<const float4 *>(sx + p);
            if (i + 4 < n || a.full) {
                *reinterpret_cast<float4 *>(gw + i) = v;
            } else {  // not the chain's last entry, which is no edge
                gw[i] = v.x;
                gw[i + 1] = v.y;
                gw[i + 2] = v.z;
            }
        }
    } else {
#pragma unroll 4
        for (int q = 0; q < L; ++q) {
            const int i = q * T + ll, p = i + (LP - L) * (i / L);
            if (i < n) gy[i] = sg[p];
            if (gw && i + (a.full ? 0 : 1) < n) gw[i] = sx[p];
        }
    }
}

// Nodes a lane of W warps holds for a chain of n nodes (0: too long).
template <int W>
__host__ __device__ constexpr int run_pick(int n)
{
    constexpr int T = 32 * W;
    if (W == 1 && n <= 8 * T) return 8;
    if (W == 1 && n <= 16 * T) return 16;
    if (n <= 24 * T) return 24;
    return n <= 32 * T ? 32 : 0;
}

// Rows of n_lo < n <= what W warps hold (CSR batches take one launch per class).
template <int W, bool VEC>
__global__ void __launch_bounds__(W <= 2 ? 64 : W * WARP)
    run_means_kernel(GradArgs a, WsHeader *hdr, int cs, int n_lo)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ MeansX<W> xc;
    const int warp = threadIdx.x / WARP;
    const long long k = W == 1 ? (long long)blockIdx.x * (blockDim.x / WARP) + warp : blockIdx.x;
    if (k >= a.nchains) return;
    long long start;
    int n;
    if (a.offsets) {
        const long long o0 = a.offsets[0], lo = a.offsets[k], hi = a.offsets[k + 1];
        if (lo < o0 || hi < lo || hi - lo > a.maxlen || hi - o0 > (k + 1) * (long long)a.maxlen) {
            if ((threadIdx.x & (WARP - 1)) == 0) atomicOr(&hdr->status, ERR_BAD_CHAIN);
            return;
        }
        start = lo;
        n = (int)(hi - lo);
    } else {
        start = k * (long long)a.maxlen;
        n = a.maxlen;
    }
    // uniform batches report no errors: the kernel clears the error word itself
    if (!a.offsets && k == 0 && threadIdx.x < sizeof(WsHeader) / sizeof(int))
        reinterpret_cast<int *>(hdr)[threadIdx.x] = 0;
    const int l = run_pick<W>(n);
    if (n <= n_lo || l == 0) return;
    float *sx = reinterpret_cast<float *>(smem_raw) + (W == 1 ? 2 * (size_t)warp * cs : 0);
    float *sg = sx + cs;
    if constexpr (W == 1) {
        if (l == 8) run_means<8, W, VEC>(a, start, n, sx, sg, &xc);
        if (l == 16) run_means<16, W, VEC>(a, start, n, sx, sg, &xc);
    }
    if (l == 24) run_means<24, W, VEC>(a, start, n, sx, sg, &xc);
    if (l == 32) run_means<32, W, VEC>(a, start, n, sx, sg, &xc);
}

template <int W>
tv_status launch_runs(const GradArgs &a, int nmax, bool vec, WsHeader *hdr, int n_lo, cudaStream_t s)
{
    const int cpb = W == 1 ? 2 : 1;  // chains per block
    const int l = run_pick<W>(nmax), cs = 32 * W * ((l / 4) % 2 == 1 ? l : l + 4);
    const size_t smem = 2 * sizeof(float) * (size_t)cs * cpb;
    // no opt-in (a limit that belongs to the kernel, which calls on other threads would move)
    static_assert(2 * sizeof(float) * 36 * 32 * W * (W == 1 ? 2 : 1) + sizeof(MeansX<W>) <= 48 * 1024,
                  "shared memory of the largest block");
    auto kern = vec ? run_means_kernel<W, true> : run_means_kernel<W, false>;
    kern<<<(unsigned)((a.nchains + cpb - 1) / cpb), cpb * W * WARP, smem, s>>>(a, hdr, cs, n_lo);
    tv_status st = check_cuda(cudaGetLastError(), "backward kernel launch");
    if (st == TV_OK) note_launch();
    return st;
}

// Every length class that the batch can hold.
tv_status launch_run_classes(const GradArgs &a, bool vec, WsHeader *hdr, cudaStream_t s)
{
    constexpr int N1 = 32 * WARP, N2 = 2 * N1;
    static_assert(kSplitMaxLen <= 4 * N1, "lengths");
    const int n = a.maxlen;
    const bool all = a.offsets != nullptr;
    tv_status st = TV_OK;
    if (all || n <= N1) st = launch_runs<1>(a, n <= N1 ? n : N1, vec, hdr, 0, s);
    if (st == TV_OK && n > N1 && (all || n <= N2))
        st = launch_runs<2>(a, n <= N2 ? n : N2, vec, hdr, all ? N1 : 0, s);
    if (st == TV_OK && n > N2) st = launch_runs<4>(a, n, vec, hdr, all ? N2 : 0, s);
    return st;
}

// Largest batch for the register kernel. A chain takes a warp (and its shared memory) however
// short it is, and a CSR batch a launch over all chains for every class of lengths, so the
// step-wise kernel is the faster one for large batches of short chains. Measured (us, step-wise /
// register kernel; chain_prox_backward called from Python, about 20 us of which are the call):
//  - rows: 20 nodes 21 / 24 for 20000 chains and 314 / 807 for a million, 60 nodes 22 / 24 for
//    20000 and 48 / 82 for 100000, 150 nodes 27 / 25 and 91 / 93, 400 nodes 49 / 35 and 194 / 146;
//  - CSR, lengths spread evenly up to 300 nodes 32 / 32 for 20000 chains and 106 / 119 for 100000,
//    800 nodes 24 / 24 for 3000 and 60 / 69 for 20000, 1600 nodes 35 / 31 and 127 / 131 (142 / 180
//    with grad_w), 4000 nodes 112 / 56 and 630 / 246; short chains but for one of 4096 nodes
//    67 / 58 for 20000 and 98 / 218 for 100000.
long long runs_max_chains(long long max_len, bool csr)
{
    if (!csr) return max_len < 128 ? 4096 : INT64_MAX;
    return max_len <= 1024 ? 2048 : max_len <= 2048 ? 4096 : 24000;
}

tv_status solve_backward(const float *d_x, const float *d_grad_x, const int64_t *d_offsets,
                         int64_t num_chains, int64_t max_len, float *d_grad_y, float *d_grad_w,
                         void *d_workspace, size_t workspace_bytes, tv_stream_t stream, bool full)
{
    clear_error();
    if (num_chains < 0 || max_len < 0 || max_len > (1LL << 24)) {
        set_error("tv_chain_solve_backward: num_chains and max_len must be >= 0");
        return TV_ERR_INVALID;
    }
    if (num_chains == 0) return TV_OK;
    if (!d_x || !d_grad_x || !d_grad_y || !d_workspace) {
        set_error("tv_chain_solve_backward: x, grad_x, grad_y and workspace must not be NULL");
        return TV_ERR_INVALID;
    }
    if (d_grad_y == d_x || d_grad_y == d_grad_x || (d_grad_w && (d_grad_w == d_x ||
                                                                 d_grad_w == d_grad_x ||
                                                                 d_grad_w == d_grad_y))) {
        set_error("tv_chain_solve_backward: outputs must not alias the inputs or each other");
        return TV_ERR_INVALID;
    }
    if (workspace_bytes < sizeof(WsHeader)) {
        set_error("tv_chain_solve_backward: workspace of %zu bytes, %zu needed", workspace_bytes,
                  sizeof(WsHeader));
        return TV_ERR_NOMEM;
    }
    cudaStream_t s = (cudaStream_t)stream;
    WsHeader *hdr = static_cast<WsHeader *>(d_workspace);
    tv_status st = TV_OK;
    const bool runs = max_len >= 1 && max_len <= kSplitMaxLen &&
                      num_chains <= runs_max_chains(max_len, d_offsets != nullptr);
    if (d_offsets || !runs) {
        st = check_cuda(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), s), "memset header");
        if (st != TV_OK) return st;
    }
    if (runs) {
        auto al = [](const void *q) { return ((uintptr_t)q & 15) == 0; };
        const bool vec = !d_offsets && max_len % 4 == 0 && al(d_x) && al(d_grad_x) &&
                         al(d_grad_y) && al(d_grad_w);
        GradArgs a{d_x, d_grad_x, d_offsets, num_chains, (int)max_len, d_grad_y, d_grad_w,
                   full};
        const bool prof = prof_on();
        if (prof) prof_mark(PK_GRAD, s, true);
        st = launch_run_classes(a, vec, hdr, s);
        if (prof) prof_mark(PK_GRAD, s, false);
        return st;
    }
    GradArgs a{d_x, d_grad_x, d_offsets, num_chains, (int)max_len, d_grad_y, d_grad_w, full};
    const long long blocks = (num_chains + kGradWarps - 1) / kGradWarps;
    const bool prof = prof_on();
    if (prof) prof_mark(PK_GRAD, s, true);
    auto kern = d_grad_w ? chain_vjp_kernel<true> : chain_vjp_kernel<false>;
    kern<<<(unsigned)blocks, kGradWarps * WARP, 0, s>>>(a, hdr);
    st = check_cuda(cudaGetLastError(), "backward kernel launch");
    if (st == TV_OK) note_launch();
    if (prof) prof_mark(PK_GRAD, s, false);
    return st;
}

}  // namespace

extern "C" tv_status tv_chain_solve_backward(const float *d_x, const float *d_grad_x,
                                             const int64_t *d_offsets, int64_t num_chains,
                                             int64_t max_len, float *d_grad_y, float *d_grad_w,
                                             void *d_workspace, size_t workspace_bytes,
                                             tv_stream_t stream)
{
    return solve_backward(d_x, d_grad_x, d_offsets, num_chains, max_len, d_grad_y, d_grad_w,
                          d_workspace, workspace_bytes, stream, false);
}

extern "C" tv_status tv_chain_solve_backward_full(const float *d_x, const float *d_grad_x,
                                                  const int64_t *d_offsets, int64_t num_chains,
                                                  int64_t max_len, float *d_grad_y,
                                                  float *d_grad_w, void *d_workspace,
                                                  size_t workspace_bytes, tv_stream_t stream)
{
    return solve_backward(d_x, d_grad_x, d_offsets, num_chains, max_len, d_grad_y, d_grad_w,
                          d_workspace, workspace_bytes, stream, true);
}
