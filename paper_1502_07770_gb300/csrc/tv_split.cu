// Launch of the threshold-splitting chain kernel (tv_split.cuh).
#include <cuda_runtime.h>

#include "tv_split_launch.h"

using namespace tvk;

namespace tvh {

namespace {

template <int W, bool UNI>
tv_status launch_w(SplitSrc src, int lmax, int nch, WsHeader *hdr, cudaStream_t s)
{
    const int cs = split_slots<W>(lmax, nch);
    const size_t smem = 2 * (size_t)nch * cs * sizeof(float);
    auto kern = split_kernel<W, UNI, SplitSrc>;
    tv_status st = check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem),
                              "cudaFuncSetAttribute");
    if (st != TV_OK) return st;
    const long long blocks = (src.nchains + nch - 1) / nch;
    st = check_cuda(launch_k(kern, dim3((unsigned)blocks), dim3(nch * W * WARP), smem, s, src, hdr,
                             nch, cs),
                    "chain kernel launch");
    if (st == TV_OK) note_launch();
    return st;
}

template <bool UNI>
tv_status launch_u(SplitSrc src, WsHeader *hdr, cudaStream_t s)
{
    const int sms = sm_count_current();
    tv_status st = TV_OK;
    const int n = src.len;
    src.n_lo = 0;
    src.lanes = 0;
    constexpr int N1 = 32 * WARP, N2 = 2 * N1;  // what one warp and two hold
    static_assert(kSplitMaxLen <= 4 * N1, "lengths");
    if (src.v.cols) {
        // neighbouring columns share a block: 16- to 32-byte pieces of each row, unless there
        // are too few columns to occupy every SM that way
        int nch = n <= N1 ? 8 : 4;
        while (nch > 2 && src.nchains < 3LL * sms * nch / 2) nch /= 2;
        if (n <= N1) return launch_w<1, UNI>(src, split_pick<1>(n), nch, hdr, s);
        if (n <= N2) return launch_w<2, UNI>(src, split_pick<2>(n), nch, hdr, s);
        return launch_w<4, UNI>(src, split_pick<4>(n), nch, hdr, s);
    }
    const int nch = src.nchains <= 16LL * sms ? 1 : 2;
    if (!src.offsets) {
        if (n <= N1) return launch_w<1, UNI>(src, split_pick<1>(n), nch, hdr, s);
        if (n <= N2) return launch_w<2, UNI>(src, split_pick<2>(n), 1, hdr, s);
        return launch_w<4, UNI>(src, split_pick<4>(n), 1, hdr, s);
    }
    // Lengths vary: one launch per number of warps, each with the one variant that holds its
    // longest chain (and 4 or 8 nodes a lane up to 256). The unrolled loop of a variant (up to
    // 20 KB) fits the instruction cache and several do not: 6000 chains of 1 to 2500 nodes, each
    // with the variant of its own length, took 239-415 us, most of it waiting for instructions.
    auto place = [&](int n_lo, int lanes) {
        src.n_lo = n_lo;
        src.lanes = lanes;
    };
    if (n > N2) {
        place(N2, split_pick<4>(n));
        st = launch_w<4, UNI>(src, src.lanes, 1, hdr, s);
    }
    if (st == TV_OK && n > N1) {
        place(N1, split_pick<2>(n <= N2 ? n : N2));
        st = launch_w<2, UNI>(src, src.lanes, 1, hdr, s);
    }
    place(0, split_pick<1>(n <= N1 ? n : N1));
    if (st == TV_OK) st = launch_w<1, UNI>(src, src.lanes, nch, hdr, s);
    return st;
}

}  // namespace

tv_status launch_split(SplitSrc src, WsHeader *hdr, cudaStream_t s, int kind)
{
    if (src.nchains <= 0 || src.len <= 0) return TV_OK;
    const bool prof = prof_on();
    if (prof) prof_mark(kind, s, true);
    const tv_status st = src.v.pw ? launch_u<false>(src, hdr, s) : launch_u<true>(src, hdr, s);
    if (prof) prof_mark(kind, s, false);
    return st;
}

}  // namespace tvh
