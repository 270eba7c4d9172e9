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
    // warps per chain: what one, two and four hold (eight: 16 nodes a lane)
    constexpr int N1 = (UNI ? 32 : 24) * WARP, N2 = 2 * N1, N4 = 4 * N1;
    static_assert(N4 >= kSplitMaxLen || !UNI, "lengths");
    if (src.v.cols) {
        // neighbouring columns share a block: 16- to 32-byte pieces of each row, unless there
        // are too few columns to occupy every SM that way
        int nch = n <= N1 ? 8 : (n <= N4 ? 4 : 2);
        while (nch > 2 && src.nchains < 3LL * sms * nch / 2) nch /= 2;
        if (n <= N1) return launch_w<1, UNI>(src, split_pick<1, UNI>(n), nch, hdr, s);
        if (n <= N2) return launch_w<2, UNI>(src, split_pick<2, UNI>(n), nch, hdr, s);
        if (n <= N4) return launch_w<4, UNI>(src, split_pick<4, UNI>(n), nch, hdr, s);
        if constexpr (!UNI) return launch_w<8, UNI>(src, split_pick<8, UNI>(n), nch, hdr, s);
        return TV_OK;
    }
    const int nch = src.nchains <= 16LL * sms ? 1 : 2;
    const bool all = src.offsets != nullptr;  // lengths vary: one launch per length class
    if (all || n <= N1)
        st = launch_w<1, UNI>(src, split_pick<1, UNI>(n <= N1 ? n : N1), nch, hdr, s);
    if (st == TV_OK && n > N1 && (all || n <= N2)) {
        src.n_lo = all ? N1 : 0;
        st = launch_w<2, UNI>(src, split_pick<2, UNI>(n <= N2 ? n : N2), 1, hdr, s);
    }
    if (st == TV_OK && n > N2 && (all || n <= N4)) {
        src.n_lo = all ? N2 : 0;
        st = launch_w<4, UNI>(src, split_pick<4, UNI>(n <= N4 ? n : N4), 1, hdr, s);
    }
    if constexpr (!UNI) {
        if (st == TV_OK && n > N4) {
            src.n_lo = all ? N4 : 0;
            st = launch_w<8, UNI>(src, split_pick<8, UNI>(n), 1, hdr, s);
        }
    }
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
