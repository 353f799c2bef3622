// Hand a frame's denoised map and flags to a caller's device buffers in one
// launch.  Two device-to-device copies take a launch each and run one after
// the other (10 us at 1920 x 1080).  Here a thread moves 16 pixels: four 16-byte
// loads of alpha and one of flags, all in flight together (5.2 us).
#include "internal.h"

namespace esim {
namespace {

constexpr int kMapThreads = 256;

template <class V>
__device__ __forceinline__ void copy16(const void* src, void* dst, size_t first, int n)
{
    V v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < n) v[k] = __ldg(static_cast<const V*>(src) + first + k);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < n) static_cast<V*>(dst)[first + k] = v[k];
}

__global__ void __launch_bounds__(kMapThreads) copy_maps_kernel(const float* alpha, float* alpha_out,
                                                                const uint8_t* flag, uint8_t* flag_out, size_t n)
{
    const size_t i = ((size_t)blockIdx.x * kMapThreads + threadIdx.x) * 16;
    if (i >= n) return;
    if (i + 16 <= n) {
        const uint4 f = flag_out ? __ldg(reinterpret_cast<const uint4*>(flag + i)) : make_uint4(0, 0, 0, 0);
        if (alpha_out) copy16<float4>(alpha, alpha_out, i / 4, 4);
        if (flag_out) *reinterpret_cast<uint4*>(flag_out + i) = f;
    } else {
        for (size_t k = i; k < n; ++k) {
            if (alpha_out) alpha_out[k] = alpha[k];
            if (flag_out) flag_out[k] = flag[k];
        }
    }
}

typedef CUresult (*AddressRangeFn)(CUdeviceptr*, size_t*, CUdeviceptr);

AddressRangeFn address_range_fn()
{
    static const AddressRangeFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<AddressRangeFn>(f);
    }();
    return fn;
}

// Memory of this device that 16-byte accesses can reach, `bytes` of it within one
// allocation (a copy call checks that; the kernel would write past it).
bool reachable(const void* p, size_t bytes, int device)
{
    if (reinterpret_cast<uintptr_t>(p) & 15u) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type != cudaMemoryTypeDevice || a.device != device) return false;
    const AddressRangeFn range = address_range_fn();
    CUdeviceptr base = 0;
    size_t size = 0;
    const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    return range && range(&base, &size, at) == CUDA_SUCCESS && at - base <= size && size - (at - base) >= bytes;
}

}  // namespace

cudaError_t copy_maps(const float* alpha, float* alpha_out, const uint8_t* flag, uint8_t* flag_out, size_t n,
                      bool to_device, int device, cudaStream_t s)
{
    if (!alpha_out && !flag_out) return cudaSuccess;
    if (to_device && (!alpha_out || reachable(alpha_out, n * sizeof(float), device)) &&
        (!flag_out || reachable(flag_out, n, device))) {
        const size_t blocks = (n + 16 * kMapThreads - 1) / (16 * kMapThreads);
        copy_maps_kernel<<<(unsigned)blocks, kMapThreads, 0, s>>>(alpha, alpha_out, flag, flag_out, n);
        return cudaGetLastError();
    }
    // host buffers, another device's, unaligned ones, or ones that are too small (refused)
    const cudaMemcpyKind k = to_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    cudaError_t e = alpha_out ? cudaMemcpyAsync(alpha_out, alpha, n * sizeof(float), k, s) : cudaSuccess;
    if (e == cudaSuccess && flag_out) e = cudaMemcpyAsync(flag_out, flag, n, k, s);
    return e;
}

}  // namespace esim
