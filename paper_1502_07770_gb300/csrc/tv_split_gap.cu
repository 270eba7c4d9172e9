// The column phase of a 2D solve with the gap pass of the iteration before in the same launch
// (a unit of its own: the kernel's variants take most of a minute to compile).
#include <cuda_runtime.h>

#include "tv_split_grid.cuh"

namespace tvh {

tv_status launch_split_gap(const SplitSrc &src, const GapView &gap, WsHeader *hdr, cudaStream_t s,
                           int kind)
{
    if (!src.done) {
        set_error("column phase without a stop flag");
        return TV_ERR_INVALID;
    }
    const SplitGapSrc g{src, gap, 0};
    return profiled(kind, s, [&] {
        return src.v.pw ? launch_cols<false>(g, hdr, s) : launch_cols<true>(g, hdr, s);
    });
}

}  // namespace tvh
