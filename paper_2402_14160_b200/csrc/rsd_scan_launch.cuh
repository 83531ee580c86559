// Launch of the row scan for one element type; each type is a translation unit of its own (rsd_scan_f32.cu,
// rsd_scan_bf16.cu), which keeps the compiles short.
#pragma once
#include <atomic>

#include "../../include/rsd.h"
#include "rsd_api_common.h"
#include "rsd_scan.cuh"

namespace rsd {

template <typename T, bool ALIGNED, bool NEED_LSE, bool TEMP, int NT, bool SPLIT>
void launch_scan_threads(int blocks, const ScanArgs& a, cudaStream_t s) {
    const auto kernel = scan_topk_kernel<T, ALIGNED, NEED_LSE, TEMP, NT, SPLIT>;
    constexpr size_t kBuffer = NT == 128 ? 0 : scan_buffer_bytes<T, NT>();   // (128 threads: a static one)
    const size_t smem = scan_bounds_bytes(a.V) + kBuffer;
    if (smem > (NT == 128 ? 32 : 40) * 1024) {   // (with the static arrays beside it close to the 48 KB that need no attribute)
        // The attribute belongs to the (function, device) pair: raised once per device to what the longest row needs.
        static std::atomic<bool> raised[64];
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return;   // the error stays pending: the caller's check_launch() reports it
        if (dev < 0 || dev >= 64 || !raised[dev].load(std::memory_order_acquire)) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(scan_bounds_bytes(RSD_MAX_VOCAB) + kBuffer)) != cudaSuccess)
                return;
            if (dev >= 0 && dev < 64) raised[dev].store(true, std::memory_order_release);
        }
    }
    if (NT == 128 && a.wait_first) kernel<<<blocks, NT, smem, s>>>(a);
    else rsd_host::launch_overlapped(kernel, (unsigned)blocks, NT, smem, s, a.cluster_status ? a.R : 0, a);
}
template <typename T, bool ALIGNED, bool NEED_LSE, bool TEMP>
void launch_scan_temp(int threads, int blocks, const ScanArgs& a, cudaStream_t s) {
    if (NEED_LSE) {   // (512 threads would sum in another order: see scan_threads())
        if (threads == 256 && a.V <= kScanSplitVocab) launch_scan_threads<T, ALIGNED, NEED_LSE, TEMP, 256, NEED_LSE>(blocks, a, s);
        else if (threads == 256) launch_scan_threads<T, ALIGNED, NEED_LSE, TEMP, 256, false>(blocks, a, s);
        else launch_scan_threads<T, ALIGNED, NEED_LSE, TEMP, 128, false>(blocks, a, s);
    } else {
        if (threads == 512) launch_scan_threads<T, ALIGNED, false, TEMP, 512, false>(blocks, a, s);
        else if (threads == 256) launch_scan_threads<T, ALIGNED, false, TEMP, 256, false>(blocks, a, s);
        else launch_scan_threads<T, ALIGNED, false, TEMP, 128, false>(blocks, a, s);
    }
}
template <typename T, bool ALIGNED, bool NEED_LSE>
void launch_scan_lse(int threads, int blocks, const ScanArgs& a, cudaStream_t s) {
    if (a.temp != 1.0f) launch_scan_temp<T, ALIGNED, NEED_LSE, true>(threads, blocks, a, s);
    else launch_scan_temp<T, ALIGNED, NEED_LSE, false>(threads, blocks, a, s);
}
template <typename T>
void launch_scan_of(int threads, bool aligned, bool need_lse, int blocks, const ScanArgs& a, cudaStream_t s) {
    if (need_lse) {
        if (aligned) launch_scan_lse<T, true, true>(threads, blocks, a, s);
        else launch_scan_lse<T, false, true>(threads, blocks, a, s);
    } else {
        if (aligned) launch_scan_lse<T, true, false>(threads, blocks, a, s);
        else launch_scan_lse<T, false, false>(threads, blocks, a, s);
    }
}

// A beam search level: rows few enough for one of the kernels of few rows.
template <typename T, bool ALIGNED, bool NEED_LSE, bool TEMP, int NT, bool SPLIT>
void launch_level_threads(int blocks, const ScanArgs& a, const SbsEpilogueArgs& e, cudaStream_t s) {
    constexpr size_t kBuffer = NT == 128 ? 0 : scan_buffer_bytes<T, NT>();
    constexpr auto kernel = scan_level_kernel<T, ALIGNED, NEED_LSE, TEMP, NT, SPLIT>;
    if (!rsd_host::raise_shared_memory<kernel>((int)(scan_bounds_bytes(RSD_MAX_VOCAB) + kBuffer))) return;
    rsd_host::launch_overlapped(kernel, (unsigned)blocks, NT, scan_bounds_bytes(a.V) + kBuffer, s, a.R, a, e);
}
template <typename T, bool ALIGNED>
void launch_level_aligned(int threads, bool need_lse, int blocks, const ScanArgs& a, const SbsEpilogueArgs& e, cudaStream_t s) {
    if (!need_lse) {                                     // (log-probabilities as they are: no temperature)
        if (threads == 512) launch_level_threads<T, ALIGNED, false, false, 512, false>(blocks, a, e, s);
        else launch_level_threads<T, ALIGNED, false, false, 256, false>(blocks, a, e, s);
    } else if (a.temp != 1.0f) {
        if (threads == 256 && a.V > kScanSplitVocab) launch_level_threads<T, ALIGNED, true, true, 256, false>(blocks, a, e, s);
        else if (threads == 256) launch_level_threads<T, ALIGNED, true, true, 256, true>(blocks, a, e, s);
        else launch_level_threads<T, ALIGNED, true, true, 128, false>(blocks, a, e, s);
    } else {
        if (threads == 256 && a.V > kScanSplitVocab) launch_level_threads<T, ALIGNED, true, false, 256, false>(blocks, a, e, s);
        else if (threads == 256) launch_level_threads<T, ALIGNED, true, false, 256, true>(blocks, a, e, s);
        else launch_level_threads<T, ALIGNED, true, false, 128, false>(blocks, a, e, s);
    }
}
template <typename T>
void launch_level_of(int threads, bool aligned, bool need_lse, int blocks, const ScanArgs& a, const SbsEpilogueArgs& e, cudaStream_t s) {
    if (aligned) launch_level_aligned<T, true>(threads, need_lse, blocks, a, e, s);
    else launch_level_aligned<T, false>(threads, need_lse, blocks, a, e, s);
}

}  // namespace rsd
