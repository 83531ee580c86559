// What the host hands to the cluster walk (rsd_walk_cluster.cuh), and its launch per element type
// (rsd_walk_cluster_f32.cu, rsd_walk_cluster_bf16.cu).
#pragma once
#include "rsd_verify.cuh"

namespace rsd {
namespace walk_cluster {

struct ClusterArgs {
    VerifyArgs v;
    ResampleArgs r;      // resample != 0: the stand-alone draw (v: rows, V and random stream only)
    int resample;
    int off_boundaries;  // a base or stride of the rows is not a multiple of 16 bytes
};

// C blocks of W working warps with NT tiles of 512 entries each
struct Shape {
    int C, W, NT;
    float waves;         // sequences asked for over sequences resident at a time
};

// extra: the baseline rules, the Gumbel-Top-1 draw or the stand-alone residual draw
void launch_f32(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s);
void launch_bf16(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s);

}  // namespace walk_cluster
}  // namespace rsd
