#include <algorithm>

#include "rsd_walk_cluster_launch.cuh"

namespace rsd {
namespace walk_cluster {
namespace {
template <int NT, int WARPS>
int ask_resident(int C) {
    constexpr size_t smem = draft_tiles_bytes<NT, WARPS>();
    const auto kernel = walk_cluster_kernel<float, NT, WARPS, kPlainWalk>;
    if (smem > 0 && !rsd_host::raise_shared_memory<walk_cluster_kernel<float, NT, WARPS, kPlainWalk>>((int)smem)) return 0;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C);
    cfg.blockDim = dim3((WARPS + 1) * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess ? n : 0;
}
}  // namespace

// (The other element type and modes are compiled for as many blocks per SM.  Clusters stay within a GPC, so there are fewer of them than
// blocks per SM, SMs and cluster size give: 71 of 74 clusters of four at two blocks per SM, 33 of 37 of eight.)
int resident_clusters(int C, int W, int NT) {
    static std::atomic<int> known[64][4][4];             // [device][shape][log2 C]
    const int shape = W == 16 ? 3 : NT == 4 ? 2 : NT - 1, size = C == 8 ? 3 : C / 2;
    int dev = 0;
    const bool keep = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
    int n = keep ? known[dev][shape][size].load(std::memory_order_relaxed) : 0;
    if (n > 0) return n;
    n = shape == 3 ? ask_resident<2, 16>(C) : shape == 2 ? ask_resident<4, 8>(C) : shape == 1 ? ask_resident<2, 8>(C) : ask_resident<1, 8>(C);
    if (n <= 0) {
        (void)cudaGetLastError();                        // (a rule of thumb, not an error of the call)
        n = std::max(rsd_host::sm_count() * (shape == 3 ? 1 : shape == 0 ? 3 : 2) / C, 1);
    }
    if (keep) known[dev][shape][size].store(n, std::memory_order_relaxed);
    return n;
}

void launch_f32(const ClusterArgs& a, bool extra, int B, const Shape& c, cudaStream_t s) { launch_of<float>(a, extra, B, c, s); }
}  // namespace walk_cluster
}  // namespace rsd
