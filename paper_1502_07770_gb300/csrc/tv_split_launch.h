// Host entry of the threshold-splitting chain kernel.
#pragma once
#include "tv_launch.cuh"
#include "tv_split.cuh"

namespace tvh {

// Chains of at most kSplitMaxLen nodes, on `s`; the source's fields as tv_split.cuh says.
tv_status launch_split(tvk::SplitSrc src, tvk::WsHeader *hdr, cudaStream_t s, int kind);
// The columns of `src`, a phase of a 2D solve, with the gap pass `gap` of the iteration before
// in the same launch.
tv_status launch_split_gap(const tvk::SplitSrc &src, const tvk::GapView &gap, tvk::WsHeader *hdr,
                           cudaStream_t s, int kind);

// Whether a batch of chains runs on it. It is the warp-per-chain kernel of TV-l2 chains that
// fit its registers, unless another was asked for (tv_set_coop_split); a batch above the
// largest one for warp-per-chain kernels (`max_chains`, or the value that
// tv_set_coop_max_chains set) goes to the thread-per-chain kernels.
inline bool split_takes(long long max_len, long long chains, long long max_chains)
{
    return max_len >= 2 && max_len <= tvk::kSplitMaxLen && coop_split() == 1 &&
           chains <= (coop_max_auto() ? max_chains : coop_max_chains());
}

// Crossovers, measured (us, splitting / thread kernel):
//  - rows that the fixed-shape thread kernel stages 16 bytes at a time: at 1024 nodes 49 / 113
//    for 4096 chains and 166 / 176 for 16384, at 256 nodes 24 / 35 and 69 / 49, at 4096 nodes
//    220 / 453 and 819 / 675; with a weight per edge, at 1024 nodes 75 / 119 and 263 / 193, at
//    4096 nodes 353 / 471 and 1362 / 737;
//  - other rows: at 1023 nodes 166 / 234 for 16384 chains and 623 / 890 for 65536, with weights
//    262 / 543 and 1004 / 1281; chains of under 64 nodes leave most of a warp idle;
//  - columns (the thread kernel runs one thread per chain): at 1024 nodes 57 / 889 for 4096 and
//    650 / 1119 for 65536, at 100 nodes 56 / 93 for 16384 and 195 / 114 for 65536.
constexpr long long kSplitMaxChainsVec = 8192, kSplitMaxChainsVecW = 6144;
inline long long split_max_chains(long long len, bool cols, bool vec, bool has_w)
{
    if (len < 64) return kCoopMaxChainsDefault;
    if (vec && !cols) return has_w ? kSplitMaxChainsVecW : kSplitMaxChainsVec;
    return cols && len < 256 ? 16384 : INT64_MAX;
}

}  // namespace tvh
