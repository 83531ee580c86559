#include "rsd_walk_cluster_launch.cuh"

namespace rsd {
namespace walk_cluster {
void launch_f32(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s) { launch_of<float>(a, extra, B, c, s); }
}  // namespace walk_cluster
}  // namespace rsd
