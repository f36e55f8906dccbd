// Short copies between a pinned host view and device memory, by a kernel.
// A copy engine moves the bytes as fast, but every hand-over between it and a
// kernel costs microseconds (a semaphore between two engines), which a short DAG
// that writes, computes and reads pays twice.  Two writes of B bytes on two
// streams, a kernel, a read of 4 bytes and the host's wait, by the copy engines and
// by kernels: 62.5 KB 25.0 and 19.3 us, 500 KB 30.5 and 22.4 us, 4 MB 66.9 and
// 57.4 us.  Longer copies are bound by the host link either way and stay with the
// copy engines, which leave the SMs to the kernels that they overlap with.
#include <cuda_runtime.h>

#include <cstdint>

#include "kcommon.cuh"

namespace gdag {

constexpr size_t kHostCopyMax = (size_t)4 << 20;

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

// Copy by a kernel if `host` (the source or the destination) is pinned memory
// that the device can reach and the copy is short; *done tells.
cudaError_t host_copy(void *dst, const void *src, size_t bytes, const void *host, cudaStream_t s, bool *done)
{
    *done = false;
    if (bytes == 0 || bytes > kHostCopyMax) return cudaSuccess;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host) != cudaSuccess) {
        cudaGetLastError();
        return cudaSuccess;
    }
    if (at.type != cudaMemoryTypeHost || !at.devicePointer) return cudaSuccess;
    unsigned char *d = static_cast<unsigned char *>(host == dst ? at.devicePointer : dst);
    const unsigned char *f = static_cast<const unsigned char *>(host == src ? at.devicePointer : src);
    const uintptr_t al = reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(f);
    auto grid = [&](size_t piece) { return (unsigned)ceil_div((int64_t)(bytes / piece > 0 ? bytes / piece : 1), kThreads); };
    if (al % 16 == 0) host_copy_kernel<uint4><<<grid(16), kThreads, 0, s>>>(d, f, bytes);
    else if (al % 4 == 0) host_copy_kernel<uint32_t><<<grid(4), kThreads, 0, s>>>(d, f, bytes);
    else host_copy_kernel<unsigned char><<<grid(1), kThreads, 0, s>>>(d, f, bytes);
    *done = true;
    return cudaGetLastError();
}

}  // namespace gdag
