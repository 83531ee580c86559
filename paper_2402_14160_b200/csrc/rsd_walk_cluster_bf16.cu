#include "rsd_walk_cluster_launch.cuh"

namespace rsd {
namespace walk_cluster {
void launch_bf16(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s) { launch_of<__nv_bfloat16>(a, extra, B, c, s); }
}  // namespace walk_cluster
}  // namespace rsd
