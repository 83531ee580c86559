#include "rsd_walk_stream_launch.cuh"

namespace rsd {
namespace walk_cluster {
void launch_stream_f32(const ClusterArgs& a, bool extra, int B, int C, int per_sm, cudaStream_t s) { launch_stream_of<float>(a, extra, B, C, per_sm, s); }
void launch_draw_f32(const ResampleArgs& a, int B, cudaStream_t s) { launch_draw_of<float>(a, B, s); }
}  // namespace walk_cluster
}  // namespace rsd
