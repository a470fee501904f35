// elbm_copy.cu -- copies of populations between device buffers.
#include <cuda.h>
#include <cuda_runtime.h>

#include "elbm_device.cuh"
#include "elbm_launch.h"

namespace eelbm {
namespace {

constexpr int kCopyBlock = 256;
constexpr int kCopyVectors = 2; // 16-byte vectors per thread

// Bound by memory, or by the launch where the state is small.  Two 16-byte loads in flight per
// thread with full occupancy reach the rate of a plain copy, and a kernel of our own overlaps
// its launch with the kernels before and after it, which cudaMemcpyAsync does not.  us per
// copy, back to back, cudaMemcpyAsync and this kernel: 0.15 to 2.4 MB 4.1, 1.4; 14.8 MB 8.2,
// 3.3; 151 MB 52.3, 44.6; 1.81 GB 539, 508 (7.1 TB/s).  One vector per thread is slower from
// 9 MB on (1.81 GB: 523), four and eight are the same, streaming policies too.
__global__ void __launch_bounds__(kCopyBlock) k_copy(const uint4 *src, uint4 *dst, int64_t n, int tail)
{
    wait_previous_kernel();
    const int64_t k0 = int64_t(blockIdx.x) * (kCopyBlock * kCopyVectors) + threadIdx.x;
    uint4 v[kCopyVectors];
#pragma unroll
    for (int k = 0; k < kCopyVectors; ++k)
        if (k0 + k * kCopyBlock < n) v[k] = __ldca(src + k0 + k * kCopyBlock);
#pragma unroll
    for (int k = 0; k < kCopyVectors; ++k)
        if (k0 + k * kCopyBlock < n) dst[k0 + k * kCopyBlock] = v[k];
    if (blockIdx.x == 0 && int(threadIdx.x) < tail) // the bytes behind the last whole vector
        reinterpret_cast<unsigned char *>(dst + n)[threadIdx.x] =
            __ldca(reinterpret_cast<const unsigned char *>(src + n) + threadIdx.x);
}

using PointerGetAttributes = CUresult (*)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
PointerGetAttributes pointer_get_attributes()
{
    static const PointerGetAttributes fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &p, 12000, cudaEnableDefault, &q) != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<PointerGetAttributes>(p);
    }();
    return fn;
}

// Whether [p, p + bytes) lies in one device allocation of `device` (0.05 us).
bool plain_device_range(const void *p, size_t bytes, int device)
{
    const PointerGetAttributes get = pointer_get_attributes();
    unsigned type = 0, managed = 1;
    int owner = -1;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL,
                                   CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                   CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *into[5] = {&type, &owner, &managed, &start, &size};
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    if (!get || get(5, what, into, at) != CUDA_SUCCESS) return false;
    return type == CU_MEMORYTYPE_DEVICE && !managed && owner == device && at >= start && bytes <= size &&
           at - start <= size - bytes;
}

} // namespace

// The kernel takes what it can address as cudaMemcpyAsync would: the caller's range within one
// allocation of this device, both ends on 16 bytes.  Anything else (another device's memory,
// managed or pinned memory, odd addresses, ranges that the driver refuses) is left to
// cudaMemcpyAsync.
cudaError_t copy_device(void *dst, const void *src, const void *outer, size_t bytes, int device, cudaStream_t s)
{
    const int64_t n = int64_t(bytes / 16), per = kCopyBlock * kCopyVectors;
    const int64_t blocks = n > 0 ? (n + per - 1) / per : 1;
    const bool aligned = ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0;
    if (!aligned || blocks > 0x7fffffff || !plain_device_range(outer, bytes, device))
        return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, s);
    return launch(k_copy, dim3(unsigned(blocks)), kCopyBlock, s, static_cast<const uint4 *>(src), static_cast<uint4 *>(dst), n,
                  int(bytes % 16));
}

} // namespace eelbm
