// Activations between pinned host memory and the workspace, for the call on host buffers: a kernel that reads or writes the
// host's memory over the link, in the place of a copy by the copy engine.
//
// The link bounds a large copy and the hand-overs around it a small one: between a copy engine's copy and a kernel lie about
// 5 us each way, between two kernels of a stream 1 - 3, and a kernel that is launched dependent has the layer's first
// weights on their way while x still arrives.  us per call with the engine / with this kernel, one stream, calls in a row:
// 4096 -> 4096 at 1 token 24.6 / 16.4, at 32 36.1 / 34.6; 4096 -> 14336 at 8 48.6 / 39.6.  16 calls over four streams, where copies of both
// directions share the link: 188 / 135 at 1 token, 257 / 204 at 32, 379 / 332 at 64 (512 KB each way), but 569 / 628 at 128: there
// the engine's larger packets count, so copies of more than 512 KB stay with it, and so does memory that the device cannot
// address.  The price: beside another stream's launch that fills the device a copy waits for SMs, where the engine would not.
// 148 CTAs, four 16-byte loads of a thread in flight: at 64 KB all SMs are ahead of 16 (5.3 against 7.2 us).
#include <cuda.h>

#include <algorithm>

#include "common.cuh"

namespace meteora {

constexpr int kCopyThreads = 256, kCopyVecs = 4;
constexpr size_t kCopyMaxBytes = (size_t)512 << 10;

__global__ void __launch_bounds__(kCopyThreads) k_host_copy(const uint4* src, uint4* dst, size_t n) {
    // (the kernel behind reads only weights before it has waited for this one)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const size_t step = (size_t)gridDim.x * kCopyThreads;
    for (size_t i = (size_t)blockIdx.x * kCopyThreads + threadIdx.x; i < n; i += step * kCopyVecs) {
        uint4 v[kCopyVecs];
#pragma unroll
        for (int q = 0; q < kCopyVecs; ++q)
            if (i + q * step < n) v[q] = __ldcv(src + i + q * step);
#pragma unroll
        for (int q = 0; q < kCopyVecs; ++q)
            if (i + q * step < n) dst[i + q * step] = v[q];
    }
}

typedef CUresult (*PointerAttributesFn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);

// The device's address of a host buffer, nullptr unless all of it is one piece of pinned memory and moves as 16-byte vectors.
static void* device_view(const void* host, size_t bytes) {
    static const PointerAttributesFn fn = []() -> PointerAttributesFn {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &sym, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
            return nullptr;
        return (PointerAttributesFn)sym;
    }();
    if (!fn || bytes % 16 != 0 || bytes > kCopyMaxBytes) return nullptr;
    unsigned int type = 0, managed = 0;
    CUdeviceptr dev = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                   CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* out[5] = {&type, &managed, &dev, &start, &size};
    if (fn(5, what, out, (CUdeviceptr)host) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || managed || !dev || dev % 16 != 0) return nullptr;
    const CUdeviceptr at = (CUdeviceptr)host;
    if (at < start || bytes > size || at - start > size - bytes) return nullptr;
    return (void*)dev;
}

// Between the host buffer and a device buffer (16-byte aligned) of the workspace.
int launch_host_copy(void* dst, const void* src, size_t bytes, bool to_device, cudaStream_t st) {
    void* const host = device_view(to_device ? src : dst, bytes);
    if (!host) return cuda_status(cudaMemcpyAsync(dst, src, bytes, to_device ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost, st));
    const size_t n = bytes / 16;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min<size_t>(148, (n + kCopyThreads - 1) / kCopyThreads));
    cfg.blockDim = dim3(kCopyThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = tuning().pdl ? 1 : 0;
    return cuda_status(cudaLaunchKernelEx(&cfg, k_host_copy, (const uint4*)(to_device ? host : src), (uint4*)(to_device ? dst : host), n));
}

}  // namespace meteora
