// What the host hands to the cluster walk (rsd_walk_cluster.cuh, rsd_walk_stream.cuh), and its launches per element type
// (rsd_walk_cluster_*.cu, rsd_walk_stream_*.cu).
#pragma once
#include "rsd_verify.cuh"

namespace rsd {
namespace walk_cluster {

struct ClusterArgs {
    VerifyArgs v;
    ResampleArgs r;      // resample != 0: the stand-alone draw (v: rows, V and random stream only)
    int resample;
    int ring_rows;       // a plain walk over rows that the ring walk takes in large batches
};

// C blocks of W working warps with NT tiles of 512 entries each
struct Shape {
    int C, W, NT;
    float waves;         // sequences asked for over sequences resident at a time
};

// How many clusters of such a shape the current device holds at a time (asked once per device).
int resident_clusters(int C, int W, int NT);

// extra: the baseline rules, the Gumbel-Top-1 draw or the stand-alone residual draw
void launch_f32(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s);
void launch_bf16(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s);
// The same with rows that are read in every pass; C: blocks per sequence, 1 or 8; per_sm: blocks per SM (3: 2-byte rows, C = 1).
void launch_stream_f32(const ClusterArgs& a, bool extra, int B, int C, int per_sm, cudaStream_t s);
void launch_stream_bf16(const ClusterArgs& a, bool extra, int B, int C, int per_sm, cudaStream_t s);

// The residual draw without a rejected token, one block per sequence (rsd_draw.cuh).
void launch_draw_f32(const ResampleArgs& a, int B, cudaStream_t s);
void launch_draw_bf16(const ResampleArgs& a, int B, cudaStream_t s);

}  // namespace walk_cluster
}  // namespace rsd
