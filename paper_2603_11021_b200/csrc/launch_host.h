// What the host settles with the runtime ahead of a launch.  Plain C++: no device code.
#pragma once
#include <cuda.h>
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

// The driver's function that encodes tensor maps, without linking against the driver library; null when it cannot be had, which is asked
// again by the next call.
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                 const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiled encode_tiled()
{
    static std::atomic<EncodeTiled> kept{nullptr};
    EncodeTiled f = kept.load(std::memory_order_acquire);
    if (!f) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) return nullptr;
        f = reinterpret_cast<EncodeTiled>(fn);
        kept.store(f, std::memory_order_release);
    }
    return f;
}

// The tensor map of X [batch][k_in] bf16 (16-byte aligned, k_in a multiple of 8): boxes of 64 columns x npad rows, 128-byte swizzle.
// The driver's function asks for a current context, which a thread has only once a runtime call has bound the device's: a thread whose first
// such call this is binds it here (the calls before it, of PyTorch's allocator and stream included, need none).
inline bool make_x_map(int device, const uint16_t* d_x, int64_t k_in, int batch, int npad, CUtensorMap* map)
{
    const EncodeTiled encode = encode_tiled();
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)k_in, (cuuint64_t)batch}, strides[1] = {(cuuint64_t)k_in * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)npad}, steps[2] = {1, 1};
    auto made = [&] {
        return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(d_x), dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    return made() || (cudaSetDevice(device) == cudaSuccess && made());
}

}  // namespace llvq
