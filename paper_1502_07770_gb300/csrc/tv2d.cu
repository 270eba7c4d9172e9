// 2D TV-l2 (ROF) denoising by Lagrangian decomposition (Sec. 6.1): the
// accelerated primal-dual iteration eq. pd on the saddle-point problem
// eq. rof-saddle, where both proximal maps are batches of chain problems.
//
// Per iteration k, two fused kernels solve the chains with the proximal arithmetic folded
// into their loads and stores: by threshold splitting (tv_split.cuh; sides of at most 4096
// pixels), else by the dynamic program of Algorithm 2 / Sec. 4.1 (one warp per chain for up
// to 2048 chains, else one thread):
//   column (dual) phase, one chain per image column:
//       eta = y + sigma_k (x^k + theta_{k-1} (x^k - x^{k-1}))
//       xhat = argmin TV_v(x) + sigma_k/2 ||x - eta/sigma_k||^2  (chains: c = eta/sigma_k,
//              w' = w_v/sigma_k)
//       y <- eta - sigma_k xhat                                   (eq. prox-tv-conj)
//   row (primal) phase, one chain per image row:
//       x^{k+1} = argmin TV_h(x) + (1+1/tau_k)/2 ||x - (f + (x^k - tau_k y)/tau_k)/(1+1/tau_k)||^2
//              (chains: c = (tau f + x^k - tau y)/(tau+1), w' = w_h tau/(tau+1)).
// Step sizes follow the accelerated variant: theta_k = 1/sqrt(1+2 tau_k),
// tau_{k+1} = theta_k tau_k, sigma_{k+1} = sigma_k/theta_k, tau_0 = sigma_0 = 1.
//
// Gap (the paper plots convergence but does not define its gap): with the edge
// fields p_h, p_v that the two chain solves certify (|p| <= w, D_v^T p_v = y^{k+1},
// f - D_h^T p_h - D_v^T p_v = x^{k+1} + (x^{k+1} - x^k)/tau_k),
//   G_k = P(x^{k+1}) - D(p) = 1/2||x^{k+1} - f||^2 + TV(x^{k+1}) - 1/2||f||^2
//         + 1/2||x^{k+1} + (x^{k+1} - x^k)/tau_k||^2 >= 0.
// The gap pass after each row phase (tv2d_gap.cuh) raises the stop flag on the device. Later
// kernels see it and return at once, so a batch of launched iterations costs little after it.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "tv2d_common.cuh"
#include "tv2d_gap.cuh"
#include "tv_launch.cuh"
#include "tv_split_launch.h"

using namespace tvk;
using namespace tvh;

namespace {

constexpr int kRing = 32;

__global__ void tv2d_init_state(Tv2dState *st, Tv2dParams *prm, int max_iters, double tol,
                                double inv_N, ParamChunk chunk)
{
    for (int q = threadIdx.x; q < chunk.count; q += blockDim.x) prm[chunk.first + q] = chunk.p[q];
    if (threadIdx.x != 0 || chunk.first != 0) return;
    st->k = 0;
    st->done = 0;
    st->ticket_col = 0;
    st->ticket_row = 0;
    st->max_iters = max_iters;
    st->gap_k = -1;
    st->tol = tol;
    st->inv_N = inv_N;
    st->gap = nan("");
}

__global__ void tv2d_start(Tv2dState *st, Tv2dState first, WsHeader *hdr)
{
    if (threadIdx.x == 0) *st = first;
    if (threadIdx.x < sizeof(WsHeader) / sizeof(int)) reinterpret_cast<int *>(hdr)[threadIdx.x] = 0;
}

// Warp-level completion counter: returns true in lane 0 of the last warp of the grid.
__device__ __forceinline__ bool last_warp_done(unsigned *ticket, int lane)
{
    bool last = false;
    if (lane == 0) {
        __threadfence();
        const unsigned total = gridDim.x * (blockDim.x / WARP);
        last = atomicAdd(ticket, 1u) == total - 1;
        if (last) {
            __threadfence();
            *ticket = 0;
        }
    }
    return last;
}

// ---------------------------------------------------------------- x^0 --------
// x^0 = argmin TV_h(x) + 1/2 ||x - (f - y^0)||^2: row chains with c = f - y, w = w_h.
template <bool HAS_WH>
struct InitRowsP {
    static constexpr bool COLS = false;
    static constexpr int NIN = HAS_WH ? 3 : 2;
    static constexpr bool NEIGH = false;
    static constexpr bool CREC = false;
    static constexpr int NOUT = 2;
    struct Acc {};

    const float *f, *y, *wh;
    float lam;
    long long H, W;
    float *x0, *x1;
    bool vec;

    __device__ bool resolve() { return true; }
    __device__ long long num_chains() const { return H; }
    __device__ int max_len() const { return (int)W; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k * W;
        n = (int)W;
        return true;
    }
    __device__ const float *in_ptr(int a) const { return a == 0 ? f : (a == 1 ? y : wh); }
    __device__ long long in_off(int a, long long k, long long start) const
    {
        return a == 2 ? k * (W - 1) : start;
    }
    __device__ int in_lim(int a, int n) const { return a == 2 ? n - 1 : n; }
    __device__ long long in_ld(int) const { return 1; }
    __device__ long long in_kmax(int) const { return H; }
    __device__ bool in_vec(int a) const { return vec && a < 2; }
    __device__ bool out_vec() const { return vec; }
    __device__ void unary(const float (&v)[NIN], float, int, int i, int n, long long, float &c,
                          float &w, Acc &) const
    {
        c = v[0] - v[1];
        if constexpr (HAS_WH) w = (i < n - 1) ? v[2] : 0.f;
        else w = (i < n - 1) ? lam : 0.f;
    }
    __device__ void unary_direct(int i, int n, long long k, long long start, float &c,
                                 float &w) const
    {
        c = f[start + i] - y[start + i];
        if constexpr (HAS_WH) w = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
        else w = (i < n - 1) ? lam : 0.f;
    }
    __device__ float *out_ptr(int o) const { return o == 0 ? x0 : x1; }
    __device__ long long out_off(int, long long, long long start) const { return start; }
    __device__ void emit_cols(int, long long, float, float) const {}
    __device__ void emit_direct(int i, long long, long long start, float xv, float) const
    {
        x0[start + i] = xv;
        x1[start + i] = xv;
    }
    __device__ long long spill_off(long long k, long long) const { return k * (2 * W + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void finish(Acc &) const {}
    __device__ void finish_empty() const {}
};

// ---------------------------------------------------------- primal step ------
template <bool HAS_WH>
struct RowPhaseP {
    static constexpr bool COLS = false;
    static constexpr int NIN = HAS_WH ? 4 : 3;
    static constexpr bool NEIGH = false;
    static constexpr bool CREC = false;
    static constexpr int NOUT = 1;
    struct Acc {};

    const float *f, *y, *wh;
    float lam;
    long long H, W;
    float *buf0, *buf1;
    Tv2dState *st;
    const Tv2dParams *prm;
    bool vec;
    // resolved per launch from the device state
    const float *xin;
    float *xout;
    float ca, cb;  // c = ca (f - y) + cb x^k, w' = ca w

    __device__ bool resolve()
    {
        const int k = st->k;
        if (st->done || k >= st->max_iters) return false;
        xin = (k & 1) ? buf1 : buf0;
        xout = (k & 1) ? buf0 : buf1;
        const double tau = prm[k].tau;
        ca = (float)(tau / (tau + 1.0));
        cb = (float)(1.0 / (tau + 1.0));
        return true;
    }
    __device__ long long num_chains() const { return H; }
    __device__ int max_len() const { return (int)W; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k * W;
        n = (int)W;
        return true;
    }
    __device__ const float *in_ptr(int a) const
    {
        return a == 0 ? f : (a == 1 ? xin : (a == 2 ? y : wh));
    }
    __device__ long long in_off(int a, long long k, long long start) const
    {
        return a == 3 ? k * (W - 1) : start;
    }
    __device__ int in_lim(int a, int n) const { return a == 3 ? n - 1 : n; }
    __device__ long long in_ld(int) const { return 1; }
    __device__ long long in_kmax(int) const { return H; }
    __device__ __forceinline__ void unary_vals(float fv, float xv, float yv, float wv, int i, int n,
                                               float &c, float &w) const
    {
        c = ca * (fv - yv) + cb * xv;
        w = (i < n - 1) ? ca * wv : 0.f;
    }
    __device__ bool in_vec(int a) const { return vec && a < 3; }
    __device__ bool out_vec() const { return vec; }
    __device__ void unary(const float (&v)[NIN], float, int, int i, int n, long long, float &c,
                          float &w, Acc &) const
    {
        float wv = lam;
        if constexpr (HAS_WH) wv = v[3];
        unary_vals(v[0], v[1], v[2], wv, i, n, c, w);
    }
    __device__ void unary_direct(int i, int n, long long k, long long start, float &c,
                                 float &w) const
    {
        float wv = lam;
        if constexpr (HAS_WH) wv = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
        unary_vals(f[start + i], xin[start + i], y[start + i], wv, i, n, c, w);
    }
    __device__ float *out_ptr(int) const { return xout; }
    __device__ long long out_off(int, long long, long long start) const { return start; }
    __device__ void emit_cols(int, long long, float, float) const {}
    __device__ void emit_direct(int i, long long, long long start, float xv, float) const
    {
        xout[start + i] = xv;
    }
    __device__ long long spill_off(long long k, long long) const { return k * (2 * W + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void count_done() const
    {
        const int lane = threadIdx.x & (WARP - 1);
        if (last_warp_done(&st->ticket_row, lane)) st->k = st->k + 1;
    }
    __device__ void finish(Acc &) const { count_done(); }
    __device__ void finish_empty() const { count_done(); }
};

// ------------------------------------------------------------ dual step ------
template <bool HAS_WV>
struct ColPhaseP {
    static constexpr bool COLS = true;
    static constexpr int NIN = HAS_WV ? 4 : 3;
    static constexpr bool NEIGH = false;
    static constexpr bool CREC = true;
    static constexpr int NOUT = 0;
    struct Acc {};

    const float *wv;
    float lam;
    long long H, W;
    float *buf0, *buf1, *y;
    Tv2dState *st;
    const Tv2dParams *prm;
    bool vec;
    // resolved per launch
    const float *xk, *xkm1;
    float sigma, inv_sigma, theta;

    __device__ bool resolve()
    {
        if (st->done) return false;
        const int k = st->k;
        xk = (k & 1) ? buf1 : buf0;
        xkm1 = (k & 1) ? buf0 : buf1;
        sigma = (float)prm[k].sigma;
        inv_sigma = (float)(1.0 / prm[k].sigma);
        theta = (float)prm[k].theta_prev;
        return true;
    }
    __device__ long long num_chains() const { return W; }
    __device__ int max_len() const { return (int)H; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k;
        n = (int)H;
        return true;
    }
    __device__ const float *in_ptr(int a) const
    {
        return a == 0 ? xk : (a == 1 ? xkm1 : (a == 2 ? y : wv));
    }
    __device__ long long in_off(int, long long, long long start) const { return start; }
    __device__ int in_lim(int a, int n) const { return a == 3 ? n - 1 : n; }
    __device__ long long in_ld(int) const { return W; }
    __device__ long long in_kmax(int) const { return W; }
    __device__ bool in_vec(int) const { return vec; }
    __device__ bool out_vec() const { return false; }
    __device__ void unary(const float (&v)[NIN], float, int, int i, int n, long long, float &c,
                          float &w, Acc &) const
    {
        float wvv = lam;
        if constexpr (HAS_WV) wvv = v[3];
        c = v[2] * inv_sigma + (v[0] + theta * (v[0] - v[1]));  // eta / sigma
        w = (i < n - 1) ? wvv * inv_sigma : 0.f;
    }
    __device__ void unary_direct(int i, int n, long long col, long long, float &c, float &w) const
    {
        (void)c;  // c comes from the forward-pass record (CREC)
        float wvv = lam;
        if constexpr (HAS_WV) wvv = (i < n - 1) ? wv[(long long)i * W + col] : 0.f;
        w = (i < n - 1) ? wvv * inv_sigma : 0.f;
    }
    __device__ float *out_ptr(int) const { return nullptr; }
    __device__ long long out_off(int, long long, long long) const { return 0; }
    __device__ void emit_cols(int i, long long col, float xhat, float c) const
    {
        if (col < W) y[(long long)i * W + col] = sigma * (c - xhat);
    }
    __device__ void emit_direct(int i, long long col, long long, float xhat, float c) const
    {
        y[(long long)i * W + col] = sigma * (c - xhat);
    }
    __device__ long long spill_off(long long col, long long) const { return col * (2 * H + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void finish(Acc &) const {}
    __device__ void finish_empty() const {}
};

// ============ the same three phases, one warp per chain (tv_coop.cuh) ============

template <bool HAS_WH>
struct CoopInitRowsP {
    static constexpr bool CREC = false;
    static constexpr bool UNIFORM_W = !HAS_WH;  // one weight (a scaled lambda) per chain
    struct Raw {
        float f, y, w;
    };
    struct Acc {};
    const float *f, *y, *wh;
    float lam;
    long long H, W;
    float *x0, *x1;

    __device__ bool resolve() { return true; }
    __device__ long long num_chains() const { return H; }
    __device__ int max_len() const { return (int)W; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k * W;
        n = (int)W;
        return true;
    }
    __device__ void fetch(long long k, long long start, int n, int i, Raw &r) const
    {
        r.f = (i < n) ? f[start + i] : 0.f;
        r.y = (i < n) ? y[start + i] : 0.f;
        if constexpr (HAS_WH) r.w = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
    }
    __device__ void unary(long long, long long, int, int, const Raw &r, float &c, float &w,
                          Acc &) const
    {
        c = r.f - r.y;
        if constexpr (HAS_WH) w = r.w;
        else w = lam;
    }
    __device__ void emit(long long, long long start, int i, float xv, float) const
    {
        x0[start + i] = xv;
        x1[start + i] = xv;
    }
    __device__ void unary_direct(int i, int n, long long k, long long start, float &c,
                                 float &w) const
    {
        c = f[start + i] - y[start + i];
        if constexpr (HAS_WH) w = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
        else w = (i < n - 1) ? lam : 0.f;
    }
    __device__ void emit_direct(int i, long long k, long long start, float xv, float c) const
    {
        emit(k, start, i, xv, c);
    }
    __device__ long long spill_off(long long k, long long) const { return k * (2 * W + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void finish(Acc &, int) const {}
    __device__ void finish_empty() const {}
};

template <bool HAS_WH>
struct CoopRowPhaseP {
    static constexpr bool CREC = false;
    static constexpr bool UNIFORM_W = !HAS_WH;  // one weight (a scaled lambda) per chain
    struct Raw {
        float f, x, y, w;
    };
    struct Acc {};
    const float *f, *y, *wh;
    float lam;
    long long H, W;
    float *buf0, *buf1;
    Tv2dState *st;
    const Tv2dParams *prm;
    const float *xin;
    float *xout;
    float ca, cb;

    __device__ bool resolve()
    {
        const int k = st->k;
        if (st->done || k >= st->max_iters) return false;
        xin = (k & 1) ? buf1 : buf0;
        xout = (k & 1) ? buf0 : buf1;
        const double tau = prm[k].tau;
        ca = (float)(tau / (tau + 1.0));
        cb = (float)(1.0 / (tau + 1.0));
        return true;
    }
    __device__ long long num_chains() const { return H; }
    __device__ int max_len() const { return (int)W; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k * W;
        n = (int)W;
        return true;
    }
    __device__ void fetch(long long k, long long start, int n, int i, Raw &r) const
    {
        const bool in = i < n;
        r.f = in ? f[start + i] : 0.f;
        r.x = in ? xin[start + i] : 0.f;
        r.y = in ? y[start + i] : 0.f;
        if constexpr (HAS_WH) r.w = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
    }
    __device__ void unary(long long, long long, int, int, const Raw &r, float &c, float &w,
                          Acc &) const
    {
        c = ca * (r.f - r.y) + cb * r.x;
        float wv = lam;
        if constexpr (HAS_WH) wv = r.w;
        w = ca * wv;
    }
    __device__ void emit(long long, long long start, int i, float xv, float) const
    {
        xout[start + i] = xv;
    }
    __device__ void unary_direct(int i, int n, long long k, long long start, float &c,
                                 float &w) const
    {
        float wv = lam;
        if constexpr (HAS_WH) wv = (i < n - 1) ? wh[k * (W - 1) + i] : 0.f;
        c = ca * (f[start + i] - y[start + i]) + cb * xin[start + i];
        w = (i < n - 1) ? ca * wv : 0.f;
    }
    __device__ void emit_direct(int i, long long k, long long start, float xv, float c) const
    {
        emit(k, start, i, xv, c);
    }
    __device__ long long spill_off(long long k, long long) const { return k * (2 * W + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void count_done() const
    {
        const int lane = threadIdx.x & (WARP - 1);
        if (last_warp_done(&st->ticket_row, lane)) st->k = st->k + 1;
    }
    __device__ void finish(Acc &, int) const { count_done(); }
    __device__ void finish_empty() const { count_done(); }
};

template <bool HAS_WV>
struct CoopColPhaseP {
    static constexpr bool CREC = true;
    static constexpr bool UNIFORM_W = !HAS_WV;  // one weight (a scaled lambda) per chain
    struct Raw {
        float x, xp, y, wv;
    };
    struct Acc {};
    const float *wv;
    float lam;
    long long H, W;
    float *buf0, *buf1, *y;
    Tv2dState *st;
    const Tv2dParams *prm;
    const float *xk, *xkm1;
    float sigma, inv_sigma, theta;

    __device__ bool resolve()
    {
        if (st->done) return false;
        const int k = st->k;
        xk = (k & 1) ? buf1 : buf0;
        xkm1 = (k & 1) ? buf0 : buf1;
        sigma = (float)prm[k].sigma;
        inv_sigma = (float)(1.0 / prm[k].sigma);
        theta = (float)prm[k].theta_prev;
        return true;
    }
    __device__ long long num_chains() const { return W; }
    __device__ int max_len() const { return (int)H; }
    __device__ bool chain(long long k, long long &start, int &n) const
    {
        start = k;
        n = (int)H;
        return true;
    }
    __device__ void fetch(long long col, long long, int n, int i, Raw &r) const
    {
        const bool in = i < n;
        const long long o = (long long)i * W + col;
        r.x = in ? xk[o] : 0.f;
        r.xp = in ? xkm1[o] : 0.f;
        r.y = in ? y[o] : 0.f;
        if constexpr (HAS_WV) r.wv = (i < n - 1) ? wv[o] : 0.f;
    }
    __device__ void unary(long long, long long, int, int, const Raw &r, float &c, float &w,
                          Acc &) const
    {
        float wvv = lam;
        if constexpr (HAS_WV) wvv = r.wv;
        c = r.y * inv_sigma + (r.x + theta * (r.x - r.xp));  // eta / sigma
        w = wvv * inv_sigma;
    }
    __device__ void emit(long long col, long long, int i, float xhat, float c) const
    {
        y[(long long)i * W + col] = sigma * (c - xhat);
    }
    __device__ void unary_direct(int i, int n, long long col, long long, float &c, float &w) const
    {
        (void)c;  // c comes from the forward-pass record
        float wvv = lam;
        if constexpr (HAS_WV) wvv = (i < n - 1) ? wv[(long long)i * W + col] : 0.f;
        w = (i < n - 1) ? wvv * inv_sigma : 0.f;
    }
    __device__ void emit_direct(int i, long long col, long long start, float xhat, float c) const
    {
        emit(col, start, i, xhat, c);
    }
    __device__ long long spill_off(long long col, long long) const { return col * (2 * H + 2); }
    __device__ void acc_init(Acc &) const {}
    __device__ void finish(Acc &, int) const {}
    __device__ void finish_empty() const {}
};

// The gap as a pass of its own (tv2d_gap.cuh): the last iteration of a batch, and the phases
// that are not on the splitting kernel.
__global__ void __launch_bounds__(kGapThreads) tv2d_gap_kernel(GapView v)
{
    pdl_enter();
    gap_pass(v, blockIdx.x, gridDim.x);
}

template <class P>
tv_status launch(const P &p, long long nchains, float2 *rec, float *crec, float2 *spill,
                 WsHeader *hdr, cudaStream_t s, int kind)
{
    return launch_chains<P, kRing>(p, nchains, rec, crec, spill, hdr, s, kind);
}

struct Tv2dWs {
    Tv2dState *st;
    Tv2dParams *prm;
    double *gaps, *partials;
    WsHeader *hdr;
    float *y, *buf1;
    const float *y0;  // where the first phases read the dual (NULL: 0)
    float2 *rec;
    float *crec;
    float2 *spill;
    size_t bytes;
    bool vec_rows, vec_cols;  // 16-byte copies: W % 4 == 0 and aligned image buffers
};

bool aligned16(const void *q) { return q == nullptr || ((uintptr_t)q & 15) == 0; }

Tv2dWs carve_tv2d(void *base, long long H, long long W, int max_iters)
{
    Carver cv(base);
    Tv2dWs o;
    const long long wr = (H + WARP - 1) / WARP, wc = (W + WARP - 1) / WARP;
    o.st = cv.take<Tv2dState>(1);
    o.prm = cv.take<Tv2dParams>((size_t)max_iters + 2);
    o.gaps = cv.take<double>((size_t)max_iters + 2);
    o.partials = cv.take<double>((size_t)kGapMaxBlocks);  // one per block of the gap kernel
    o.hdr = cv.take<WsHeader>(1);
    o.y = cv.take<float>((size_t)(H * W));
    o.y0 = o.y;
    o.buf1 = cv.take<float>((size_t)(H * W));
    const long long rec_rows = wr * W, rec_cols = wc * H;
    o.rec = cv.take<float2>((size_t)((rec_rows > rec_cols ? rec_rows : rec_cols) * WARP));
    o.crec = cv.take<float>((size_t)(rec_cols * WARP));
    const long long sp_rows = H * (2 * W + 2), sp_cols = W * (2 * H + 2);
    o.spill = cv.take<float2>((size_t)(sp_rows > sp_cols ? sp_rows : sp_cols));
    o.bytes = align_up(cv.used, 256);
    o.vec_rows = o.vec_cols = false;
    return o;
}

// One iteration's step sizes and place in the schedule (the host's copy of Tv2dParams).
struct Step {
    int k = 0;
    double tau = 1.0, sigma = 1.0, theta_prev = 0.0;
    void next()
    {
        const double theta = 1.0 / sqrt(1.0 + 2.0 * tau);
        tau *= theta;
        sigma /= theta;
        theta_prev = theta;
        ++k;
    }
};

// The phases on the threshold-splitting kernel (tv_split.cuh): rows or columns of the image.
SplitSrc split_src(SplitMode mode, const float *img, const float *w, float lam, long long H,
                   long long W, const Step &it, float *x0, const Tv2dWs &ws)
{
    SplitSrc src{};
    SplitView &v = src.v;
    const bool cols = mode == SPLIT_COL;
    float *xc = (it.k & 1) ? ws.buf1 : x0, *xo = (it.k & 1) ? x0 : ws.buf1;
    v.mode = mode;
    v.cols = cols;
    v.pw = w;
    v.lam = lam;
    v.ws = 1.f;
    if (mode == SPLIT_INIT) {
        v.p0 = img;
        v.p1 = ws.y0;
        v.o0 = x0;
        v.o1 = ws.buf1;
    } else if (mode == SPLIT_ROW) {
        v.p0 = img;
        v.p1 = ws.y;
        v.p2 = xc;
        v.o0 = xo;
        v.ca = v.ws = (float)(it.tau / (it.tau + 1.0));
        v.cb = (float)(1.0 / (it.tau + 1.0));
    } else {
        v.p0 = xc;
        v.p1 = xo;
        v.p2 = it.k == 0 ? ws.y0 : ws.y;
        v.o0 = ws.y;
        v.ca = v.ws = (float)(1.0 / it.sigma);
        v.cb = (float)it.theta_prev;
        v.sg = (float)it.sigma;
    }
    v.stride = cols ? W : 1;
    v.wrow = W - 1;
    v.rec = ws.rec;
    v.spill = ws.spill;
    v.maxlen = (int)(cols ? H : W);
    src.nchains = cols ? W : H;
    src.len = v.maxlen;
    src.done = &ws.st->done;  // (clear before the first phase)
    return src;
}

// Rows: the phases' thread kernel is slower than tv_chain_solve's, so the splitting kernel is the
// faster one for larger batches (ms, four iterations, thread / splitting kernel: 16384 x 1024
// 8.9 / 5.4, 65536 x 1024 26.5 / 20.9, 32768 x 512 9.8 / 8.2, 30000 x 200 6.6 / 6.7; with edge
// weights 65536 x 512 25.6 / 22.4, 30000 x 200 9.6 / 9.2).
bool split_rows(long long H, long long W, const float *wh)
{
    long long most = INT64_MAX;
    if (W < 64) most = W < 32 ? 2048 : kCoopMaxChainsDefault;
    else if (wh) most = W < 192 ? 150 * W : INT64_MAX;
    else if (W < 640) most = W < 400 ? std::max(2048LL, 23 * W) : 32768;
    return split_takes(W, H, most);
}
// Columns: for short ones too, as the phases are fewer launches here (8 x 8, six iterations 120 us
// against 147 on the old phases, 20 x 1500 222 against 565), and beyond what chains alone take
// (1000 x 20000, four iterations 9.4 / 6.7 ms).
bool split_cols(long long H, long long W, const float *)
{
    return split_takes(H, W, H < 64 ? kCoopMaxChainsDefault : H < 256 ? 16384 : INT64_MAX);
}

template <bool HAS_WH>
tv_status launch_init(const float *img, const float *wh, float lam, long long H, long long W,
                      float *x0, const Tv2dWs &ws, cudaStream_t s)
{
    if (split_rows(H, W, wh))
        return launch_split(split_src(SPLIT_INIT, img, wh, lam, H, W, Step(), x0, ws), ws.hdr, s,
                            PK_INIT);
    if (H <= coop_max_chains()) {
        CoopInitRowsP<HAS_WH> p{img, ws.y, wh, lam, H, W, x0, ws.buf1};
        return launch_coop(p, H, (int)W, ws.rec, nullptr, ws.spill, ws.hdr, s, PK_INIT);
    }
    InitRowsP<HAS_WH> p{img, ws.y, wh, lam, H, W, x0, ws.buf1, ws.vec_rows};
    return launch(p, H, ws.rec, nullptr, ws.spill, ws.hdr, s, PK_INIT);
}

template <bool HAS_WH>
tv_status launch_row(const float *img, const float *wh, float lam, long long H, long long W,
                     const Step &it, float *x0, const Tv2dWs &ws, cudaStream_t s)
{
    if (split_rows(H, W, wh))
        return launch_split(split_src(SPLIT_ROW, img, wh, lam, H, W, it, x0, ws), ws.hdr, s, PK_ROW);
    if (H <= coop_max_chains()) {
        CoopRowPhaseP<HAS_WH> p{img, ws.y, wh, lam, H, W, x0, ws.buf1, ws.st, ws.prm,
                                nullptr, nullptr, 0.f, 0.f};
        return launch_coop(p, H, (int)W, ws.rec, nullptr, ws.spill, ws.hdr, s, PK_ROW);
    }
    RowPhaseP<HAS_WH> p{img, ws.y, wh, lam, H, W, x0, ws.buf1, ws.st, ws.prm, ws.vec_rows,
                        nullptr, nullptr, 0.f, 0.f};
    return launch(p, H, ws.rec, nullptr, ws.spill, ws.hdr, s, PK_ROW);
}

template <bool HAS_WV>
tv_status launch_col(const float *wv, float lam, long long H, long long W, const Step &it,
                     float *x0, const Tv2dWs &ws, const GapView *gap, cudaStream_t s)
{
    if (split_cols(H, W, wv)) {
        const SplitSrc src = split_src(SPLIT_COL, nullptr, wv, lam, H, W, it, x0, ws);
        return gap ? launch_split_gap(src, *gap, ws.hdr, s, PK_COL) : launch_split(src, ws.hdr, s, PK_COL);
    }
    if (W <= coop_max_chains()) {
        CoopColPhaseP<HAS_WV> p{wv, lam, H, W, x0, ws.buf1, ws.y, ws.st, ws.prm,
                                nullptr, nullptr, 0.f, 0.f, 0.f};
        return launch_coop(p, W, (int)H, ws.rec, ws.crec, ws.spill, ws.hdr, s, PK_COL);
    }
    ColPhaseP<HAS_WV> p{wv, lam, H, W, x0, ws.buf1, ws.y, ws.st, ws.prm,
                        ws.vec_cols && aligned16(wv), nullptr, nullptr, 0.f, 0.f, 0.f};
    return launch(p, W, ws.rec, ws.crec, ws.spill, ws.hdr, s, PK_COL);
}

tv_status launch_col_any(const float *wv, float lam, long long H, long long W, const Step &it,
                         float *x0, const Tv2dWs &ws, const GapView *gap, cudaStream_t s)
{
    return wv ? launch_col<true>(wv, lam, H, W, it, x0, ws, gap, s)
              : launch_col<false>(wv, lam, H, W, it, x0, ws, gap, s);
}

// the gap of iteration it.k
GapView gap_view(const float *img, const float *wh, const float *wv, float lam, long long H, long long W,
                 const Step &it, const float *x0, const Tv2dWs &ws)
{
    const float *xn = (it.k & 1) ? x0 : ws.buf1, *xp = (it.k & 1) ? ws.buf1 : x0;
    return GapView{img, wh, wv, lam, (int)H, (int)W, xn, xp, it.k, (float)(1.0 / it.tau), 0, 0,
                   ws.st, ws.partials, ws.gaps, &ws.st->ticket_col};
}

tv_status launch_gap(GapView v, cudaStream_t s)
{
    const int blocks = gap_tiles(v, kGapThreads / WARP);
    tv_status st = check_cuda(launch_k(tv2d_gap_kernel, dim3(blocks), dim3(kGapThreads), 0, s, v),
                              "gap kernel launch");
    if (st == TV_OK) note_launch();
    return st;
}

// Once the solve has finished (converged or out of iterations) with x^k in the second
// buffer (k odd), copy it to x; a no-op otherwise. Enqueued after every batch of
// iterations, so the host's one state read per batch also covers the result.
__global__ void tv2d_final_copy(const Tv2dState *st, const float4 *buf1, float4 *x, long long n4,
                                const float *buf1s, float *xs, long long n)
{
    pdl_enter();
    const int k = st->k;
    const bool finished = st->done || k >= st->max_iters;
    if (!finished || !(k & 1)) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += stride)
        x[q] = buf1[q];
    for (long long q = 4 * n4 + (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride)
        xs[q] = buf1s[q];
}

tv_status read_state(const Tv2dWs &ws, cudaStream_t s, Tv2dState &out)
{
    tv_status st = check_cuda(cudaMemcpyAsync(&out, ws.st, sizeof(out), cudaMemcpyDeviceToHost, s),
                              "read state");
    if (st != TV_OK) return st;
    return check_cuda(cudaStreamSynchronize(s), "synchronize");
}

}  // namespace

extern "C" {

size_t tv2d_workspace_size(int64_t H, int64_t W, int max_iters)
{
    if (H < 1 || W < 1 || max_iters < 0) return 0;
    return carve_tv2d(nullptr, H, W, max_iters).bytes;
}

tv_status tv2d_denoise(const float *d_img, int64_t H, int64_t W, const float *d_wh,
                       const float *d_wv, float lambda, const float *d_y0, int max_iters,
                       double gap_tol, float *d_x, int *iters_out, double *gap_out,
                       void *d_workspace, size_t workspace_bytes, tv_stream_t stream)
{
    clear_error();
    if (H < 1 || W < 1 || H > (1LL << 24) || W > (1LL << 24) || max_iters < 0 ||
        max_iters > (1 << 24)) {
        set_error("tv2d_denoise: need H, W >= 1 and 0 <= max_iters <= 2^24");
        return TV_ERR_INVALID;
    }
    if (!d_img || !d_x || !d_workspace) {
        set_error("tv2d_denoise: img, x and workspace must not be NULL");
        return TV_ERR_INVALID;
    }
    if (!(gap_tol >= 0.0 && gap_tol < INFINITY)) {
        set_error("tv2d_denoise: gap_tol must be finite and >= 0");
        return TV_ERR_INVALID;
    }
    if ((!d_wh || !d_wv) && !(lambda >= 0.f && lambda < INFINITY)) {
        set_error("tv2d_denoise: lambda must be finite and >= 0");
        return TV_ERR_INVALID;
    }
    const size_t npx = (size_t)(H * W) * sizeof(float);
    const void *ins[4] = {d_img, d_wh, d_wv, d_y0};
    const size_t insz[4] = {npx, (size_t)(H * (W - 1)) * sizeof(float),
                            (size_t)((H - 1) * W) * sizeof(float), npx};
    for (int q = 0; q < 4; ++q) {
        const char *a = (const char *)d_x, *b = (const char *)ins[q];
        if (b && insz[q] && a < b + insz[q] && b < a + npx) {
            set_error("tv2d_denoise: x must not overlap the inputs");
            return TV_ERR_INVALID;
        }
    }
    Tv2dWs ws = carve_tv2d(d_workspace, H, W, max_iters);
    if (workspace_bytes < ws.bytes) {
        set_error("tv2d_denoise: workspace of %zu bytes, %zu needed", workspace_bytes, ws.bytes);
        return TV_ERR_NOMEM;
    }
    ws.vec_rows = ws.vec_cols = (W % 4 == 0) && aligned16(d_img) && aligned16(d_x);
    cudaStream_t s = (cudaStream_t)stream;
    tv_status st;
    const bool split = split_rows(H, W, d_wh) && split_cols(H, W, d_wv);
    if (split) {
        // the phases take step sizes from the host, and the first ones read d_y0 itself, or 0
        ws.y0 = d_y0;
        Tv2dState first{};
        first.max_iters = max_iters;
        first.gap_k = -1;
        first.tol = gap_tol;
        first.inv_N = 1.0 / ((double)H * W);
        first.gap = NAN;
        tv2d_start<<<1, WARP, 0, s>>>(ws.st, first, ws.hdr);
        if ((st = check_cuda(cudaGetLastError(), "start")) != TV_OK) return st;
        note_launch();
    } else {
        // step sizes of eq. pd, FP64 on the host
        static thread_local ParamChunk chunk;
        for (int first = 0; first <= max_iters; first += kParamChunk) {
            fill_params(chunk, first, std::min(kParamChunk, max_iters + 1 - first));
            tv2d_init_state<<<1, 128, 0, s>>>(ws.st, ws.prm, max_iters, gap_tol,
                                              1.0 / ((double)H * W), chunk);
            if ((st = check_cuda(cudaGetLastError(), "init state")) != TV_OK) return st;
            note_launch();
        }
        if ((st = check_cuda(cudaMemsetAsync(ws.hdr, 0, sizeof(WsHeader), s), "memset")) != TV_OK)
            return st;
        st = d_y0 ? check_cuda(cudaMemcpyAsync(ws.y, d_y0, npx, cudaMemcpyDeviceToDevice, s), "copy y0")
                  : check_cuda(cudaMemsetAsync(ws.y, 0, npx, s), "zero y");
        if (st != TV_OK) return st;
    }
    // launches of the two phases timed before this call (benchmark profiling only)
    const bool prof = prof_on();
    const size_t prof_col0 = prof ? prof_pending(PK_COL) : 0;
    const size_t prof_row0 = prof ? prof_pending(PK_ROW) : 0;
    // from here on each kernel may become resident while its predecessor finishes
    PdlScope pdl(true);
    st = d_wh ? launch_init<true>(d_img, d_wh, lambda, H, W, d_x, ws, s)
              : launch_init<false>(d_img, d_wh, lambda, H, W, d_x, ws, s);
    if (st != TV_OK) return st;

    // Each iteration: column (dual) phase, row (primal) phase, gap. Iterations go out in
    // batches, each followed by the conditional result copy and one read of the device state
    // (the only host synchronisation): a first batch of 6 (the usual iteration count of 1e-4
    // solves is 3 to 7; the device stop flag turns iterations launched after convergence into
    // immediate returns), then batches of 3.
    const long long N = H * W;
    const int copy_blocks = (int)std::min<long long>((N / 4 + 255) / 256 + 1, 4LL * sm_count_current());
    auto launch_copy = [&]() -> tv_status {
        tv_status r = check_cuda(
            launch_k(tv2d_final_copy, dim3(copy_blocks), dim3(256), 0, s, (const Tv2dState *)ws.st,
                     reinterpret_cast<const float4 *>(ws.buf1), reinterpret_cast<float4 *>(d_x),
                     aligned16(d_x) && aligned16(ws.buf1) ? N / 4 : 0, (const float *)ws.buf1,
                     d_x, N),
            "result copy");
        if (r == TV_OK) note_launch();
        return r;
    };
    // On the splitting kernel the gap of an iteration rides in the next one's column phase;
    // the last of a batch is a kernel of its own. 1024 x 1024 at 5 iterations: 353 us
    // against 374 with a gap kernel after every iteration; 297 x 401 at 6: 229 against 247.
    const bool fused = split_cols(H, W, d_wv);
    GapView gap;
    Tv2dState hs;
    Step it;
    int launched = 0;
    bool done = false;
    while (launched < max_iters && !done) {
        const int batch = launched == 0 ? 6 : 3;
        const int u = (max_iters - launched) < batch ? (max_iters - launched) : batch;
        for (int t = 0; t < u; ++t) {
            st = launch_col_any(d_wv, lambda, H, W, it, d_x, ws, fused && t > 0 ? &gap : nullptr, s);
            if (st != TV_OK) return st;
            st = d_wh ? launch_row<true>(d_img, d_wh, lambda, H, W, it, d_x, ws, s)
                      : launch_row<false>(d_img, d_wh, lambda, H, W, it, d_x, ws, s);
            if (st != TV_OK) return st;
            gap = gap_view(d_img, d_wh, d_wv, lambda, H, W, it, d_x, ws);
            if (!fused || t + 1 == u)
                if ((st = launch_gap(gap, s)) != TV_OK) return st;
            it.next();
        }
        launched += u;
        if ((st = launch_copy()) != TV_OK) return st;
        if ((st = read_state(ws, s, hs)) != TV_OK) return st;
        done = hs.done != 0;
    }
    if (max_iters == 0 && (st = read_state(ws, s, hs)) != TV_OK) return st;
    if (prof) {
        // phases of iterations after the k-th returned at once: keep only the k timed
        // launches of each phase that did the work
        prof_drop_from(PK_COL, prof_col0 + (size_t)hs.k);
        prof_drop_from(PK_ROW, prof_row0 + (size_t)hs.k);
    }
    if (iters_out) *iters_out = hs.k;
    if (gap_out) *gap_out = hs.gap;
    return done ? TV_OK : TV_ERR_NOT_CONVERGED;
}

}  // extern "C"
