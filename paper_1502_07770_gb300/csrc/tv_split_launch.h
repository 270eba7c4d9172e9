// Host entry of the threshold-splitting chain kernel.
#pragma once
#include <algorithm>

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

// Largest batch for the splitting kernel. Crossovers, measured (us, splitting / thread kernel;
// chain_prox called from Python, about 15 us of which are the call):
//  - rows that the fixed-shape thread kernel stages 16 bytes at a time (vec). Splitting costs
//    about the same for any short chain, the thread kernel in proportion to its length, so the
//    line goes with the length: 64 nodes 17 / 18 for 2048 chains and 21 / 16 for 4096, 128 nodes
//    22 / 22 for 4096 and 28 / 23 for 6144, 192 nodes 25 / 29 and 32 / 30 for 6000, 256 nodes
//    35 / 39 for 6000, 300 nodes 40 / 44 for 6000 and 50 / 44 for 8192, 400 nodes 46 / 54 and
//    58 / 54. Long ones: at 512 nodes 57 / 66 for 8192 and 95 / 91 for 16384, at 1024 nodes
//    101 / 127 and 180 / 177, at 4096 nodes 470 / 484 and 853 / 675. With a weight per edge as
//    above up to 256 nodes, then at 1024 nodes 92 / 129 for 6000 and 129 / 129 for 8192.
//  - other rows, one weight: 130 nodes 24 / 23 for 3072 chains, 201 nodes 27 / 31 for 4096 and
//    36 / 35 for 6144, 257 nodes 45 / 44 for 6000, 385 nodes 52 / 61 for 6000 and 66 / 62 for
//    8192, 514 nodes 155 / 190 for 20000 and 469 / 449 for 65536, 770 nodes 563 / 582 for 50000.
//    Just above what one warp or two hold the kernel pays for half-empty warps: 1027 nodes
//    126 / 145 for 6000, 168 / 152 for 8192 and 984 / 752 for 50000, 2050 nodes 245 / 278 and
//    328 / 292; 3001 nodes 870 / 1170 for 20000.
//  - other rows with a weight per edge (the thread kernel stages those worst): 65 nodes 31 / 39
//    for 8192 and 51 / 41 for 16384, 130 nodes 66 / 78 for 16384 and 120 / 91 for 32768, 201
//    nodes 86 / 122 for 20000 and 198 / 175 for 50000, 257 nodes 104 / 156 and 246 / 213, 385
//    nodes 313 / 313 for 50000 and 916 / 881 for 150000, 1023 nodes 65 / 167 for 4096;
//  - columns (the thread kernel runs one thread per chain): at 1024 nodes 57 / 889 for 4096 and
//    650 / 1119 for 65536, at 300 nodes 180 / 258 for 40000 and 638 / 554 for 150000, at 100
//    nodes 56 / 93 for 16384 and 195 / 114 for 65536.
// Chains of under 64 nodes leave most of a warp idle. There, and up to 4096 chains otherwise, the
// alternative is a warp per chain by the dynamic program, whose time goes with the length (us,
// splitting / dynamic program, device time of a call): rows of 8 nodes 8.2 / 6.2 for 20 to 1000
// chains and 14.4 / 8.4 for 4000, 16 nodes 8.3 / 8.2 and 14.4 / 12.3, 24 nodes 8.3 / 9.0 and
// 14.7 / 16.4, 63 nodes 9.0 / 16.4 and 16.4 / 33.0; columns of 16 nodes 8.2 / 6.4 and 16.3 / 11.2, 24
// nodes 8.3 / 8.2 and 16.4 / 14.4, 32 nodes 8.5 / 8.4 and 16.4 / 17.6, 63 nodes 8.3 / 12.4 and
// 17.1 / 30.7.
//
// CSR batches (`csr`; `len` is their longest chain): a short chain still takes its warps, and one
// of more than 256 nodes is solved at the longest chain's nodes a lane, while the thread kernels
// take the time of the longest chain or that of all nodes. The line is the lowest crossover over
// lengths spread evenly up to `len`, all near it, or far below it but for one (us, splitting /
// thread kernel): 260 nodes 38 / 42 for 5000 chains and 73 / 54 for 10000, 400 nodes 60 / 57 for
// 5000, 600 nodes 61 / 80 and 127 / 108, 1000 nodes 130 / 126 for 7000 and 196 / 182 for 10000,
// 1600 nodes 240 / 286 for 10000 and 384 / 292 for 14000, 2400 nodes 335 / 416 and 485 / 443, 4096
// nodes (1200 on average) 360 / 480 and 523 / 487. With a weight per edge, where the thread
// kernels are slower: 150 nodes 73 / 87 for 20000 and 163 / 119 for 50000, 400 nodes 231 / 220
// for 20000, 600 nodes 341 / 330 for 28000, 1000 nodes 311 / 536 for 20000, 1600 nodes 484 / 617
// and 732 / 646 for 28000, 4096 nodes (1200 on average) 702 / 995 and 1051 / 953 for 28000.
// (Limits from rows of the longest length sent 65536 chains of up to 900 nodes, 400 on average,
// here: 1258 us for 494, and a million of 20 nodes but for one of 700: 2455 for 319.)
inline long long split_max_chains(long long len, bool cols, bool vec, bool has_w, bool csr = false)
{
    if (csr && len >= 64) {
        if (has_w) return len <= 256 ? 120 * len : std::min(47 * len, 22000LL);
        return std::max(4096LL, len <= 256 ? 23 * len : len <= 1024 ? 9 * len : std::min(2 * len + 7000, 13500LL));
    }
    if (len < 64) return len < (cols ? 32 : 20) ? 0 : kCoopMaxChainsDefault;
    if (cols) return len < 256 ? 16384 : len < 512 ? 250 * len : INT64_MAX;
    if (vec) return std::max(2048LL, std::min(28 * len, has_w ? 6144LL : len < 512 ? 6800LL : 8192LL));
    if (has_w) return len < 384 ? 150 * len : INT64_MAX;
    if (len < 400) return std::max(2048LL, std::min(23 * len, 7000LL));
    if ((len > 1024 && len <= 1536) || (len > 2048 && len <= 2560)) return 7000;
    return len < 640 ? 32768 : INT64_MAX;
}

}  // namespace tvh
