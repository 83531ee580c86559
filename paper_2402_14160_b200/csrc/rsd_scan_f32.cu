#include "rsd_scan_launch.cuh"

namespace rsd {
void launch_scan_f32(int threads, bool aligned, bool need_lse, int blocks, const ScanArgs& a, cudaStream_t s) {
    launch_scan_of<float>(threads, aligned, need_lse, blocks, a, s);
}
void launch_level_f32(int threads, bool aligned, bool need_lse, int blocks, const ScanArgs& a, const SbsEpilogueArgs& e, cudaStream_t s) {
    launch_level_of<float>(threads, aligned, need_lse, blocks, a, e, s);
}
}  // namespace rsd
