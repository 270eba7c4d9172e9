// The duality gap of the 2D TV-l2 iteration and the device state that it drives.
#pragma once
#include "tv_launch.cuh"

namespace tvk {

struct Tv2dState {
    int k;                // completed primal (row) steps
    int done;             // per-pixel gap reached the tolerance
    unsigned ticket_col;  // warps finished in the running column phase
    unsigned ticket_row;  // warps finished in the running row phase
    int max_iters;
    int gap_k;            // index of the last gap written (-1: none yet)
    double tol;           // per-pixel tolerance; 0 never stops early
    double inv_N;         // 1 / (H W)
    double gap;           // last per-pixel gap G_{gap_k} / (H W)
};

// G_k after the primal step of iteration k: the per-pixel terms
// 1/2 (x - f)^2 + 1/2 (z - f)(z + f) with z = x^{k+1} + (x^{k+1} - x^k)/tau_k, plus
// w |difference| over the right and lower neighbour of every pixel. One pass over the image;
// FP32 within a thread, FP64 across threads; the last block reduces the block partials in a
// fixed order and raises the stop flag.
//
// A warp takes 32 columns of kGapRows consecutive rows and issues all their loads before it
// uses one; the lower neighbour is the next row's value, the right one the next lane's. What
// bounds it is latency (the loads, then the partials, the ticket and the last block's sums, one
// after the other): 12 us at 1024 x 1024 as a kernel between two phases, where its bytes take
// 2 us. The column phase of the next iteration does not depend on it and leaves most of the
// chip idle, so blocks of this pass ride in that phase's launch (see split_kernel), and
// the phase stops early if they raise the flag.
constexpr int kGapThreads = 256;  // of the pass as a kernel of its own
constexpr int kGapRows = 8;
constexpr int kGapMaxBlocks = 4096;

struct GapView {
    const float *f, *wh, *wv;
    float lam;
    int H, W;
    const float *x1, *x0;  // x^{k+1}, x^k
    int k;
    float inv_tau;
    long long ctiles, tiles;  // of 32 columns x kGapRows rows per warp of the block
    Tv2dState *st;
    double *partials, *gaps;
    unsigned *ticket;
};

// blocks of `warps` warps that take the pass
inline int gap_tiles(GapView &v, int warps)
{
    const int rows = warps * kGapRows;
    v.ctiles = (v.W + WARP - 1) / WARP;
    v.tiles = v.ctiles * ((v.H + rows - 1) / rows);
    return (int)(v.tiles < kGapMaxBlocks ? v.tiles : kGapMaxBlocks);
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = WARP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Sum over the block in a fixed order; valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double *red)
{
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & (WARP - 1)) == 0) red[threadIdx.x / WARP] = v;
    __syncthreads();
    double b = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x / WARP); ++w) b += red[w];
    return b;
}

// Block `blk` of the `blocks` that take the pass (gap_tiles for blockDim.x / 32 warps).
__device__ __forceinline__ void gap_pass(const GapView &v, unsigned blk, unsigned blocks)
{
    __shared__ double red[16];
    __shared__ bool last;
    if (v.st->done) return;
    const int lane = threadIdx.x & (WARP - 1), warp = threadIdx.x / WARP;
    const int H = v.H, W = v.W;
    const float *x1 = v.x1, *wh = v.wh, *wv = v.wv;
    const float inv_tau = v.inv_tau;
    double acc = 0.0;
    for (long long tile = blk; tile < v.tiles; tile += blocks) {
        const int c = (int)(tile % v.ctiles) * WARP + lane;
        const int r0 = ((int)(tile / v.ctiles) * (int)(blockDim.x / WARP) + warp) * kGapRows;
        float xv[kGapRows + 1], fv[kGapRows], xo[kGapRows], wd[kGapRows], wr[kGapRows], xe[kGapRows];
#pragma unroll
        for (int u = 0; u <= kGapRows; ++u) {
            const int r = r0 + u;
            const bool in = c < W && r < H;
            const long long q = (long long)r * W + c;
            xv[u] = in ? x1[q] : 0.f;
            if (u == kGapRows) break;
            fv[u] = in ? v.f[q] : 0.f;
            xo[u] = in ? v.x0[q] : 0.f;
            xe[u] = in && lane == WARP - 1 && c + 1 < W ? x1[q + 1] : 0.f;
            wr[u] = in && c + 1 < W ? (wh ? wh[q - r] : v.lam) : 0.f;
            wd[u] = in && r + 1 < H ? (wv ? wv[q] : v.lam) : 0.f;
        }
        float part = 0.f;
#pragma unroll
        for (int u = 0; u < kGapRows; ++u) {
            const float xn = __shfl_down_sync(FULL, xv[u], 1);
            const float xr = lane == WARP - 1 ? xe[u] : xn;
            const float z = xv[u] + (xv[u] - xo[u]) * inv_tau;
            float t = 0.5f * (xv[u] - fv[u]) * (xv[u] - fv[u]) + 0.5f * (z - fv[u]) * (z + fv[u]);
            if (wr[u] != 0.f) t += wr[u] * fabsf(xr - xv[u]);
            if (wd[u] != 0.f) t += wd[u] * fabsf(xv[u + 1] - xv[u]);
            part += t;
        }
        acc += (double)part;  // FP32 over a thread's 8 pixels, FP64 beyond
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) {
        v.partials[blk] = acc;
        __threadfence();
        last = atomicAdd(v.ticket, 1u) == blocks - 1;
    }
    __syncthreads();
    if (!last) return;
    // the last block sums the block partials in a fixed order
    __threadfence();
    double b = 0.0;
    for (unsigned bq = threadIdx.x; bq < blocks; bq += blockDim.x) b += __ldcg(v.partials + bq);
    b = block_sum(b, red);
    if (threadIdx.x == 0) {
        Tv2dState *st = v.st;
        const double g = b * st->inv_N;
        st->gap = g;
        st->gap_k = v.k;
        st->k = v.k + 1;
        v.gaps[v.k] = g;
        *v.ticket = 0;
        if (st->tol > 0.0 && g <= st->tol) st->done = 1;
    }
}

}  // namespace tvk
