// Grids of the threshold-splitting chain kernel.
#pragma once
#include <algorithm>

#include "tv_split_launch.h"

namespace tvh {
namespace {

using namespace tvk;

template <int W, bool UNI, class SRC>
tv_status launch_w(SRC src, int lmax, int nch, WsHeader *hdr, cudaStream_t s)
{
    const int cs = split_slots<W>(lmax, nch);
    const size_t smem = 2 * (size_t)nch * cs * sizeof(float);
    auto kern = split_kernel<W, UNI, SRC>;
    tv_status st = TV_OK;
    // Beyond what needs no opt-in (with the exchange; a call less, 1 us). The limit is the kernel's,
    // not the launch's: always the most, so that no other thread's call lowers it meanwhile.
    static_assert(sizeof(SplitX<W>) * (split_threads<W>() / (WARP * W)) <= 1536, "static shared memory");
    if (smem > 46 * 1024)
        st = check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)split_smem_most<W>()),
                        "cudaFuncSetAttribute");
    if (st != TV_OK) return st;
    long long blocks = (src.nchains + nch - 1) / nch;
    if constexpr (SRC::GAP) {
        // two per SM, which leaves room for chains beside them from the start: with a block per
        // tile behind the chains the flag came 8 us later at 1024 x 1024
        src.gap_blocks = std::min(gap_tiles(src.gap, nch * W), 2 * sm_count_current());
        blocks += src.gap_blocks;
    }
    st = check_cuda(launch_k(kern, dim3((unsigned)blocks), dim3(nch * W * WARP), smem, s, src, hdr,
                             nch, cs),
                    "chain kernel launch");
    if (st == TV_OK) note_launch();
    return st;
}

constexpr int N1 = 32 * WARP, N2 = 2 * N1;  // what one warp and two hold
static_assert(kSplitMaxLen <= 4 * N1, "lengths");

template <bool UNI, class SRC>
tv_status launch_cols(const SRC &src, WsHeader *hdr, cudaStream_t s)
{
    // neighbouring columns share a block: 16- to 32-byte pieces of each row, unless there
    // are too few columns to occupy every SM that way
    const int n = src.len;
    int nch = n <= N1 ? 8 : 4;
    while (nch > 2 && src.nchains < 3LL * sm_count_current() * nch / 2) nch /= 2;
    if (n <= N1) return launch_w<1, UNI>(src, split_pick<1>(n), nch, hdr, s);
    if (n <= N2) return launch_w<2, UNI>(src, split_pick<2>(n), nch, hdr, s);
    return launch_w<4, UNI>(src, split_pick<4>(n), nch, hdr, s);
}

template <class F>
tv_status profiled(int kind, cudaStream_t s, F launch)
{
    const bool prof = prof_on();
    if (prof) prof_mark(kind, s, true);
    const tv_status st = launch();
    if (prof) prof_mark(kind, s, false);
    return st;
}

}  // namespace
}  // namespace tvh
