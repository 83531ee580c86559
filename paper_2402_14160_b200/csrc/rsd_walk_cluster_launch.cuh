// Launch of the cluster walk for one element type.
#pragma once
#include "rsd_api_common.h"
#include "rsd_walk_cluster.cuh"

namespace rsd {
namespace walk_cluster {

template <typename T, int NT, int WARPS, int MODE>
void launch_shape(const ClusterArgs& a, int B, int C, cudaStream_t s) {
    constexpr size_t smem = draft_tiles_bytes<NT, WARPS>();
    if (smem > 0 && !rsd_host::raise_shared_memory<walk_cluster_kernel<T, NT, WARPS, MODE>>((int)smem)) return;
    rsd_host::launch_overlapped(walk_cluster_kernel<T, NT, WARPS, MODE>, (unsigned)(B * C), (WARPS + 1) * 32, smem, s, C, a);
}
template <typename T, int MODE>
void launch_mode(const ClusterArgs& a, int B, const Shape& c, cudaStream_t s) {
    if (c.W == 16) launch_shape<T, 2, 16, MODE>(a, B, c.C, s);
    else if (c.NT == 4) launch_shape<T, 4, 8, MODE>(a, B, c.C, s);
    else if (c.NT == 2) launch_shape<T, 2, 8, MODE>(a, B, c.C, s);
    else launch_shape<T, 1, 8, MODE>(a, B, c.C, s);
}
template <typename T>
void launch_of(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s) {
    if (a.resample) launch_mode<T, kResample>(a, B, c, s);
    else if (extra) launch_mode<T, kRuleWalk>(a, B, c, s);
    else launch_mode<T, kPlainWalk>(a, B, c, s);
}

}  // namespace walk_cluster
}  // namespace rsd
