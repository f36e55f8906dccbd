// Device code shared by the IMG kernels: the per-launch ones (k_img.cu) and the
// merged form of a whole image program (k_img_merge.cu), which must compute
// the same bits.
#pragma once

#include "kcommon.cuh"

namespace gdag {

constexpr int kMmMaxBlocks = 4096;  // (min, max) pairs that a minmax node's scratch holds

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Warp-strip stencils.  Each warp owns a strip of image columns, four per
// lane (one 128-bit load per row and lane), and slides down a band of rows:
// the vertical taps come from a window of rows kept in registers (each input
// row is loaded once), the horizontal taps from the neighbouring lanes'
// registers by warp shuffles, so there is no shared memory and no block
// barrier.  The HL lanes at each end of a warp are halo lanes: they load
// and filter the columns next to the strip (replicated at the image edge)
// but store nothing, so a strip is 4 (32 - 2 HL) columns wide.  Rows and
// columns outside the image take the nearest edge value (clamp-to-edge).
constexpr int kStWarps = 4;
constexpr int kStThreads = 32 * kStWarps;
constexpr unsigned kFull = 0xffffffffu;

// Pixels x .. x+3 of row y, clamped to the image; one 128-bit load when the
// four lie inside the image and rows are 16-byte aligned (vec).
__device__ __forceinline__ float4 load4_clamped(const float *__restrict__ in, int rows, int cols, bool vec, int y, int x)
{
    const float *row = in + (size_t)clampi(y, 0, rows - 1) * cols;
    if (vec && x >= 0 && x + 3 < cols) return __ldg(reinterpret_cast<const float4 *>(row + x));
    return make_float4(__ldg(row + clampi(x, 0, cols - 1)), __ldg(row + clampi(x + 1, 0, cols - 1)),
                       __ldg(row + clampi(x + 2, 0, cols - 1)), __ldg(row + clampi(x + 3, 0, cols - 1)));
}

// Store pixels x .. x+3 (x >= 0) of row y, those inside the image.
__device__ __forceinline__ void store4(float *__restrict__ out, int rows, int cols, bool vec, int y, int x, float4 v)
{
    if (y >= rows || x >= cols) return;
    float *o = out + (size_t)y * cols + x;
    if (vec && x + 3 < cols) {
        *reinterpret_cast<float4 *>(o) = v;
    } else {
        o[0] = v.x;
        if (x + 1 < cols) o[1] = v.y;
        if (x + 2 < cols) o[2] = v.z;
        if (x + 3 < cols) o[3] = v.w;
    }
}

__device__ __forceinline__ bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// sqrt(gx^2 + gy^2) with the single-instruction approximate square root
// (relative error about 1e-7, far inside the 1e-5 tolerance; the outputs
// that are compared bit for bit downstream are min/max of these values
// themselves); exactly 0 for a flat neighbourhood.
__device__ __forceinline__ float sobel_mag(float gx, float gy)
{
    const float g2 = fmaf(gx, gx, gy * gy);
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(g2));
    return g2 > 0.f ? r : 0.f;
}

__device__ __forceinline__ float unsharp1(float a, float b, float alpha) { return fmaf(alpha, a - b, a); }

__device__ __forceinline__ float combine1(float s, float b5, float b9, float e5, float e9)
{
    return e5 * s + (1.f - e5) * (e9 * b5 + (1.f - e9) * b9);
}

}  // namespace gdag
