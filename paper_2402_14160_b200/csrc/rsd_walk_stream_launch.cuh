// Launch of the streaming walk for one element type.
#pragma once
#include "rsd_api_common.h"
#include "rsd_draw.cuh"
#include "rsd_walk_stream.cuh"

namespace rsd {
namespace walk_cluster {

template <typename T, int MODE>
void launch_stream_mode(const ClusterArgs& a, int B, int C, int per_sm, cudaStream_t s) {
    auto launch = [&](auto kernel) { rsd_host::launch_overlapped(kernel, (unsigned)(B * C), kStreamThreads, 0, s, C, a); };
    if (C != 1) {
        launch(walk_stream_kernel<T, kClasses, MODE, 2>);
    } else if constexpr (sizeof(T) == 2) {
        launch(per_sm == 3 ? walk_stream_kernel<T, 1, MODE, 3> : walk_stream_kernel<T, 1, MODE, 2>);
    } else {
        launch(walk_stream_kernel<T, 1, MODE, 2>);
    }
}
template <typename T>
void launch_stream_of(const ClusterArgs& a, bool extra, int B, int C, int per_sm, cudaStream_t s) {
    if (a.resample) launch_stream_mode<T, kResample>(a, B, C, per_sm, s);
    else if (extra) launch_stream_mode<T, kRuleWalk>(a, B, C, per_sm, s);
    else launch_stream_mode<T, kPlainWalk>(a, B, C, per_sm, s);
}

template <typename T>
void launch_draw_of(const ResampleArgs& a, int B, cudaStream_t s) {
    rsd_host::launch_overlapped(draw_target_kernel<T>, (unsigned)B, kDrawWarps * 32, 0, s, 0, a);
}

}  // namespace walk_cluster
}  // namespace rsd
