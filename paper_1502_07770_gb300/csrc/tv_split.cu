// Launch of the threshold-splitting chain kernel (tv_split.cuh).
#include <cuda_runtime.h>

#include "tv_split_grid.cuh"

using namespace tvk;

namespace tvh {

namespace {

// chains of one length
template <bool UNI>
tv_status launch_rows(const SplitSrc &src, WsHeader *hdr, cudaStream_t s)
{
    const int n = src.len;
    if (n <= N1) return launch_w<1, UNI>(src, split_pick<1>(n), src.nchains <= 16LL * sm_count_current() ? 1 : 2, hdr, s);
    if (n <= N2) return launch_w<2, UNI>(src, split_pick<2>(n), 1, hdr, s);
    return launch_w<4, UNI>(src, split_pick<4>(n), 1, hdr, s);
}

template <bool UNI>
tv_status launch_u(SplitSrc src, WsHeader *hdr, cudaStream_t s)
{
    tv_status st = TV_OK;
    const int n = src.len;
    src.n_lo = 0;
    src.lanes = 0;
    if (src.v.cols) return launch_cols<UNI>(src, hdr, s);
    if (!src.offsets) return launch_rows<UNI>(src, hdr, s);
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
    if (st == TV_OK) st = launch_w<1, UNI>(src, src.lanes, src.nchains <= 16LL * sm_count_current() ? 1 : 2, hdr, s);
    return st;
}

}  // namespace

tv_status launch_split(SplitSrc src, WsHeader *hdr, cudaStream_t s, int kind)
{
    if (src.nchains <= 0 || src.len <= 0) return TV_OK;
    return profiled(kind, s, [&] {
        return src.v.pw ? launch_u<false>(src, hdr, s) : launch_u<true>(src, hdr, s);
    });
}

}  // namespace tvh
