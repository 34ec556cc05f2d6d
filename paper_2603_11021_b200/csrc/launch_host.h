// What the host settles with the runtime ahead of a launch.  Plain C++: no device code.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>

namespace llvq {

// How much dynamic shared memory the kernels may use on the device of one context, per kernel (numbered as they are first launched);
// 0 = not asked for yet.  The runtime keeps the last value it was given, so every thread and context gives it the same one, the most
// that the kernel can have: whoever comes first or last, no launch finds less than it needs.  Kept with the context and not with
// the process, like the device memory that the launch needs: both go with the device's state.
constexpr int kMaxKernels = 256;
struct SmemLimits {
    std::atomic<uint32_t> bytes[kMaxKernels] = {};
};

inline std::atomic<int> next_kernel_number{0};

template <auto kKernel>
int kernel_number()
{
    static const int number = next_kernel_number.fetch_add(1);
    return number;
}

// Whether a launch of the kernel on the current device can have `bytes` of dynamic shared memory; most = what a block may have there in all.
template <auto kKernel>
bool allow_smem(SmemLimits& limits, size_t most, size_t bytes)
{
    const int number = kernel_number<kKernel>();
    std::atomic<uint32_t>* const kept = number < kMaxKernels ? &limits.bytes[number] : nullptr;
    uint32_t limit = kept ? kept->load(std::memory_order_acquire) : 0u;
    if (limit == 0u) {
        cudaFuncAttributes attr;
        if (cudaFuncGetAttributes(&attr, reinterpret_cast<const void*>(kKernel)) != cudaSuccess || attr.sharedSizeBytes >= most) return false;
        limit = (uint32_t)(most - attr.sharedSizeBytes);
        if (cudaFuncSetAttribute(reinterpret_cast<const void*>(kKernel), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess) return false;
        if (kept) kept->store(limit, std::memory_order_release);
    }
    return bytes <= limit;
}

}  // namespace llvq
