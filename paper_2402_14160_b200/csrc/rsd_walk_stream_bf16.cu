#include "rsd_walk_stream_launch.cuh"

namespace rsd {
namespace walk_cluster {
void launch_stream_bf16(const ClusterArgs& a, bool extra, int B, int C, int per_sm, cudaStream_t s) { launch_stream_of<__nv_bfloat16>(a, extra, B, C, per_sm, s); }
}  // namespace walk_cluster
}  // namespace rsd
