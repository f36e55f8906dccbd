// Short copies between a pinned host view and device memory, by a kernel. A copy engine moves
// the bytes as fast, but every hand-over between it and a kernel costs microseconds (a
// semaphore between two engines), which a short DAG that writes, computes and reads pays
// twice.  Two writes of B bytes on two streams, a kernel, a read of 4 bytes and the host's
// wait, by the copy engines and by kernels: 62.5 KB 25.0 and 19.3 us, 500 KB 30.5 and 22.4 us,
// 4 MB 66.9 and 57.4 us (16-byte pieces).  Longer copies are bound by the host link either way
// and stay with the copy engines.  So do copies beside kernels of the same context that they
// do not follow: 4 MB by a kernel beside an iteration of HITS at 4e6 vertices (166 us) add 16
// us to it, by an engine nothing.  And copies beside more than one other: kernels share the
// link, engines do one copy after another, so that what follows the first overlaps the rest
// (ten writes, B&S launches and reads of 5e5 options each: 225 us, 258 us with every write by
// a kernel).  The one-byte pieces of unaligned copies end at 64 KB (write, kernel and 64-byte
// read of 1 MB 31.5 us, with the write by an engine 24.3; of 4 MB 71.7 and 46; of 64 KB 19.6
// either way); four-byte ones take 24.4, 45.5 and 19.6 us.
#include <cuda.h>  // pointer attributes (the query comes from the runtime's driver entry point)
#include <cuda_runtime.h>

#include <cstdint>

#include "host_range.h"
#include "kcommon.cuh"

namespace gdag {

constexpr size_t kHostCopyMax = (size_t)4 << 20, kHostCopyByteMax = (size_t)64 << 10;

// T-sized pieces, one a thread, then the bytes that are left.
template <class T>
__global__ void __launch_bounds__(kThreads) host_copy_kernel(unsigned char *__restrict__ dst,
                                                             const unsigned char *__restrict__ src, size_t bytes)
{
    const size_t n = bytes / sizeof(T), i = (size_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < n) reinterpret_cast<T *>(dst)[i] = __ldcg(reinterpret_cast<const T *>(src) + i);
    if (blockIdx.x == 0 && threadIdx.x < bytes % sizeof(T))
        dst[n * sizeof(T) + threadIdx.x] = __ldcg(src + n * sizeof(T) + threadIdx.x);
}

namespace {

// The driver's pointer query (several attributes in one call), through the runtime.
typedef CUresult (*PointerAttributes)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
PointerAttributes pointer_attributes()
{
    static const PointerAttributes fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        const bool ok = cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &p, 12000, cudaEnableDefault, &q) ==
                            cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<PointerAttributes>(p) : nullptr;
    }();
    return fn;
}

// The device's address of [host, host + bytes) if one pinned allocation or
// registration holds all of it, else null.
unsigned char *device_view(const void *host, size_t bytes)
{
    const PointerAttributes query = pointer_attributes();
    if (!query) return nullptr;
    CUmemorytype type = (CUmemorytype)0;
    unsigned managed = 0;
    CUdeviceptr dev = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED,
                                  CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *to[] = {&type, &managed, &dev, &start, &size};
    if (query(5, what, to, (CUdeviceptr)(uintptr_t)host) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || managed || !dev) return nullptr;
    // the range is given in host or in device addresses; under unified addressing
    // they are the same
    if (!range_holds(start, size, (uint64_t)(uintptr_t)host, bytes) && !range_holds(start, size, (uint64_t)dev, bytes))
        return nullptr;
    return reinterpret_cast<unsigned char *>((uintptr_t)dev);
}

// At the highest priority: its blocks take the first slots that come free, as a copy
// engine would take its turn, beside kernels of other contexts that fill the
// device.  64 KB behind 20 B&S launches of 1e7 options: 16 us, by a copy engine 16,
// at the default priority 122 (it waits for the last launch's blocks to start).
template <class T> cudaError_t launch_copy(unsigned char *d, const unsigned char *f, size_t bytes, cudaStream_t s)
{
    static const int priority = [] {
        int least = 0, greatest = 0;
        return cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess ? greatest : 0;
    }();
    cudaLaunchConfig_t cfg = {};
    const size_t n = bytes / sizeof(T);
    cfg.gridDim = dim3((unsigned)ceil_div((int64_t)(n > 0 ? n : 1), kThreads));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributePriority;
    at[0].val.priority = priority;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, host_copy_kernel<T>, d, f, bytes);
}

}  // namespace

// Copy by a kernel if `host` (the source or the destination) is pinned memory
// that the device can reach, the copy is short and no kernel or second copy of the
// context may be running `beside` it; *done tells.
cudaError_t host_copy(void *dst, const void *src, size_t bytes, const void *host, bool beside, cudaStream_t s, bool *done)
{
    *done = false;
    if (beside || bytes == 0 || bytes > kHostCopyMax) return cudaSuccess;
    unsigned char *const view = device_view(host, bytes);
    if (!view) return cudaSuccess;
    unsigned char *d = host == dst ? view : static_cast<unsigned char *>(dst);
    const unsigned char *f = host == src ? view : static_cast<const unsigned char *>(src);
    const uintptr_t al = reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(f);
    if (al % 4 != 0 && bytes > kHostCopyByteMax) return cudaSuccess;
    *done = true;
    if (al % 16 == 0) return launch_copy<uint4>(d, f, bytes, s);
    if (al % 4 == 0) return launch_copy<uint32_t>(d, f, bytes, s);
    return launch_copy<unsigned char>(d, f, bytes, s);
}

}  // namespace gdag
