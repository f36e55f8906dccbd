// Merged form of the IMG program (Section IV-B, IMG): ten launches
//   b1 = gauss_blur(img), b2 = gauss_blur(img), e1 = sobel(b1), e2 = sobel(b2),
//   mm1 = minmax(e1), mm2 = minmax(e2), extend(e1, mm1), extend(e2, mm2),
//   s = unsharp(img, b1), out = combine(s, b1, b2, e1, e2)
// that gdag_issue finds in one run are issued as one unit of two kernels.
// Launch by launch the program moves 23 images through HBM (1.54 GB at
// 4096 x 4096); the unit moves 10:
//   stage 1  reads img, writes b1, b2 and s, and only measures the raw edge
//            maps (their (min, max) pairs per block);
//   stage 2  combines the pairs into mm1 and mm2, reads b1, b2 and s, computes
//            each edge map again in its stretched form, and writes e1, e2 and
//            out.
// Measured at 4096 x 4096, steps one after another: 113 us a step, from 220 us as
// ten launches (0.88 of the measured HBM rate for the unit's 671 MB); 9 us
// from 46 us at 512 x 512, where ten launches cost the host 4 us each; 38 us from
// 53 us at 1300 x 3001, whose rows allow no 128-bit access.
// Computing Sobel twice costs arithmetic that both stages have to spare (they
// stay near the memory rate) and saves writing the raw maps and reading them
// back three times.  Every value is computed by the operations of the single
// kernels in their order (img.cuh), so b1, b2, s, mm1, mm2, e1 and e2 are the
// same bits.
#include <initializer_list>
#include <type_traits>

#include "catalog.h"
#include "kcommon.cuh"
#include "img.cuh"

namespace gdag {

constexpr int kMergeMaxR = 4;                // larger radii need two halo lanes a side
constexpr int kMgHL = 2;                     // halo lanes per side: one for the blurs, one for Sobel
constexpr int kMgCols = 4 * (32 - 2 * kMgHL);  // columns a warp stores

// Horizontal pass of a blur on the vertical sums (lo, hi) of a lane's four
// columns: gauss_blur's operations in its order, neighbour columns by shuffles
// (only those within R).
template <int R> __device__ __forceinline__ float4 blur_horizontal(float2 lo, float2 hi, const float (&wr)[2 * R + 1])
{
    constexpr int W = 2 * R + 1, HALO = 4;
    float v[4 + 2 * HALO];
    v[HALO] = lo.x;
    v[HALO + 1] = lo.y;
    v[HALO + 2] = hi.x;
    v[HALO + 3] = hi.y;
    const float c[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
    for (int k = 0; k < R; ++k) {
        v[HALO - 1 - k] = __shfl_up_sync(kFull, c[3 - k], 1);
        v[HALO + 4 + k] = __shfl_down_sync(kFull, c[k], 1);
    }
    float2 a01 = make_float2(0.f, 0.f), a23 = a01, mid = a01;
    float e0 = 0.f, e3 = 0.f;
#pragma unroll
    for (int k = 0; k < W; ++k) {
        const int o = HALO - R + k;
        const float2 wk = make_float2(wr[k], wr[k]);
        // (HALO - R + k) has the parity that gauss_blur's offset of the same
        // tap has, its halo being a multiple of four columns too
        if ((o & 1) == 0) {
            a01 = __ffma2_rn(wk, make_float2(v[o], v[o + 1]), a01);
            a23 = __ffma2_rn(wk, make_float2(v[o + 2], v[o + 3]), a23);
        } else {
            mid = __ffma2_rn(wk, make_float2(v[o + 1], v[o + 2]), mid);
            e0 = fmaf(wr[k], v[o], e0);
            e3 = fmaf(wr[k], v[o + 3], e3);
        }
    }
    return make_float4(a01.x + e0, a01.y + mid.x, a23.x + mid.y, a23.y + e3);
}

// The columns past the image's last one repeat it (a lane that holds the last
// column; lanes wholly outside are never read, sobel_row stops at the edge).
__device__ __forceinline__ float4 repeat_last(float4 v, int x, int cols)
{
    const int k = cols - 1 - x;  // the lane's index of the last column
    if (k >= 0 && k < 3) {
        if (k < 1) v.y = v.x;
        if (k < 2) v.z = v.y;
        v.w = v.z;
    }
    return v;
}

__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// sobel_mag of two pixels: max(r, 0) is r, or 0 for a NaN, as its comparison
__device__ __forceinline__ float2 sobel_mag2(float2 gx, float2 gy)
{
    const float2 g2 = __ffma2_rn(gx, gx, __fmul2_rn(gy, gy));
    float2 r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(g2.x));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(g2.y));
    return make_float2(fmaxf(r.x, 0.f), fmaxf(r.y, 0.f));
}

// Sobel magnitudes of a lane's four columns from the rows above, at and below:
// sobel_kernel's operations, two pixels an instruction where their operands sit
// in aligned register pairs (both stages are bound by instruction issue).  At
// the left or right edge of the image (`edge`, for the warp) a lane takes its
// own edge column in the place of the missing neighbour.
__device__ __forceinline__ float4 sobel_row(float4 a, float4 b, float4 c, bool edge, int x, int cols)
{
    const float2 two = make_float2(2.f, 2.f), neg = make_float2(-1.f, -1.f);
    const float2 s01 = __ffma2_rn(two, lo2(b), __fadd2_rn(lo2(a), lo2(c)));
    const float2 s23 = __ffma2_rn(two, hi2(b), __fadd2_rn(hi2(a), hi2(c)));
    const float2 d01 = __ffma2_rn(neg, lo2(a), lo2(c)), d23 = __ffma2_rn(neg, hi2(a), hi2(c));  // c - a
    float svl = __shfl_up_sync(kFull, s23.y, 1), svr = __shfl_down_sync(kFull, s01.x, 1);
    float dvl = __shfl_up_sync(kFull, d23.y, 1), dvr = __shfl_down_sync(kFull, d01.x, 1);
    if (edge) {  // the whole warp
        if (x <= 0) {
            svl = s01.x;
            dvl = d01.x;
        }
        if (x + 4 >= cols) {
            svr = s23.y;
            dvr = d23.y;
        }
    }
    // columns 1 and 2, and 0 and 3, as pairs
    const float2 gx12 = __ffma2_rn(neg, s01, s23), t12 = __fadd2_rn(d01, d23);
    const float2 gx03 = make_float2(s01.y - svl, svr - s23.x);
    const float2 gy12 = make_float2(fmaf(2.f, d01.y, t12.x), fmaf(2.f, d23.x, t12.y));
    const float2 gy03 = make_float2(fmaf(2.f, d01.x, dvl + d01.y), fmaf(2.f, d23.y, d23.x + dvr));
    const float2 m12 = sobel_mag2(gx12, gy12), m03 = sobel_mag2(gx03, gy03);
    return make_float4(m03.x, m12.x, m12.y, m03.y);
}

struct Range {
    float lo = INFINITY, hi = -INFINITY;
    __device__ __forceinline__ void add(float v)
    {
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    // three-operand minimum and maximum: two instructions for four values
    __device__ __forceinline__ void add4(float4 v)
    {
        asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(v.x), "f"(v.y));
        asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(v.z), "f"(v.w));
        asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(v.x), "f"(v.y));
        asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(v.z), "f"(v.w));
    }
};

// The block's ranges from its threads', in every thread.
__device__ __forceinline__ void block_ranges(Range &a, Range &b, float (&red)[4][kStWarps])
{
    const float v[4] = {warp_min(a.lo), warp_max(a.hi), warp_min(b.lo), warp_max(b.hi)};
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) red[q][threadIdx.x >> 5] = v[q];
    __syncthreads();
    a.lo = red[0][0];
    a.hi = red[1][0];
    b.lo = red[2][0];
    b.hi = red[3][0];
#pragma unroll
    for (int w = 1; w < kStWarps; ++w) {
        a.lo = fminf(a.lo, red[0][w]);
        a.hi = fmaxf(a.hi, red[1][w]);
        b.lo = fminf(b.lo, red[2][w]);
        b.hi = fmaxf(b.hi, red[3][w]);
    }
}

// Stage 1.  Warp strips as in gauss_blur: a warp slides down a band of rows and
// keeps the last two rows of each blur for Sobel.  It is bound by instruction
// issue, so the form is the one with the fewest instructions a row:
//  - the image rows come through a ring of four groups of four rows in shared
//    memory, by asynchronous copies one group ahead; a lane reads only what it
//    copied itself, so no barrier is needed.  (A ring in registers, as
//    gauss_blur's, needs the row loop unrolled by its length; with two blurs and
//    two Sobels that code, 44 KB, runs from beyond the instruction caches.)
//  - four blurred rows an iteration, in two pairs: a pair shares its reads of
//    the ring (WB + 1 rows for two outputs), the groups' addresses change hands
//    once an iteration, and the rows kept for Sobel are never moved;
//  - the rows and columns at the image's edges are repeated in branches that the
//    whole warp takes or skips.
// A band of TH output rows takes TH + 2 blurred ones; the warps of a block take
// bands below one another.  57 us at 4096 x 4096 (268 MB, 0.69 of the HBM rate;
// 52 us with Sobel left out, so its arithmetic is mostly hidden), from 83 us in
// the first form, with the ring in registers.
constexpr int kS1Group = 4;       // rows
constexpr int kS1MaxBand = 512;   // output rows
static_assert(2 * kMergeMaxR + 4 <= 3 * kS1Group, "an iteration's rows lie in three groups");

// The four columns a lane moves: with whole 128-bit groups (`vec`, for the grid)
// a lane outside the image moves the group at the image's edge, else each column
// is clamped on its own.  Either way the whole warp takes one path: with a slow
// path for the lanes at the edge, the first and last strips' warps, all resident
// from the start, ended a quarter later than the others.
__device__ __forceinline__ void copy4_row(float4 *dst, const float *__restrict__ in, int rows, int cols, bool vec, int y,
                                          int x)
{
    const float *row = in + (size_t)clampi(y, 0, rows - 1) * cols;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (vec) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(row + clampi(x, 0, cols - 4)) : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * k), "l"(row + clampi(x + k, 0, cols - 1))
                         : "memory");
    }
}

__device__ __forceinline__ float4 load4_row(const float *in, int rows, int cols, bool vec, int y, int x)
{
    const float *row = in + (size_t)clampi(y, 0, rows - 1) * cols;
    if (vec) return load_dep(reinterpret_cast<const float4 *>(row + clampi(x, 0, cols - 4)));
    return make_float4(load_dep(row + clampi(x, 0, cols - 1)), load_dep(row + clampi(x + 1, 0, cols - 1)),
                       load_dep(row + clampi(x + 2, 0, cols - 1)), load_dep(row + clampi(x + 3, 0, cols - 1)));
}

// The vertical sums (lo, hi) of a lane outside the image, which moved whole
// groups: the edge column's in all four places.
__device__ __forceinline__ void splat_outside(float2 &lo, float2 &hi, int x, int cols)
{
    if (x < 0) {
        lo.y = lo.x;
        hi = lo;
    } else if (x >= cols) {
        hi.x = hi.y;
        lo = hi;
    }
}

template <int RA, int RB, bool VEC>
__global__ void __launch_bounds__(kStThreads, 4)
    img_stage1_kernel(const float *__restrict__ img, float *__restrict__ ba, float *__restrict__ bb,
                      float *__restrict__ sh, const float *__restrict__ wa, const float *__restrict__ wb,
                      float2 *__restrict__ part_a, float2 *__restrict__ part_b, float alpha, int rows, int cols, int th)
{
    static_assert(RA < RB && RB <= kMergeMaxR, "the second blur is the wider one, within one halo lane");
    constexpr int WA = 2 * RA + 1, WB = 2 * RB + 1;
    // stage 2 may become resident from now on: it waits for this grid
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ float4 ring[kStWarps][4][kS1Group][32];
    __shared__ float red[4][kStWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * kMgCols + 4 * (lane - kMgHL);
    const int y0 = (blockIdx.y * kStWarps + warp) * th;  // th is even
    const bool stores = lane >= kMgHL && lane < 32 - kMgHL && x < cols;
    // warps of the first and last strips see the image's left or right edge: lane 31
    // holds columns (blockIdx.x + 1) * kMgCols + 4 .. + 7, and lane 30's blur reads them
    const bool edge = blockIdx.x == 0 || (int)(blockIdx.x + 1) * kMgCols + 8 > cols;
    Range ra, rb;
    if (y0 < rows) {  // the whole warp
        const int yend = min(y0 + th, rows);
        float wra[WA], wrb[WB];
#pragma unroll
        for (int k = 0; k < WA; ++k) wra[k] = __ldg(wa + k);
#pragma unroll
        for (int k = 0; k < WB; ++k) wrb[k] = __ldg(wb + k);
        // group g holds input rows y0 - 1 - RB + 4g .. + 3 in slot g % 4
        const int yi = y0 - 1 - RB;
        auto copy_group = [&](float4 *dst, int yy) {
#pragma unroll
            for (int k = 0; k < kS1Group; ++k) copy4_row(dst + 32 * k, img, rows, cols, VEC, yy + k, x);
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float4 *g0 = &ring[warp][0][0][lane], *g1 = &ring[warp][1][0][lane], *g2 = &ring[warp][2][0][lane],
               *g3 = &ring[warp][3][0][lane];
        copy_group(g0, yi);
        copy_group(g1, yi + kS1Group);
        copy_group(g2, yi + 2 * kS1Group);
        float4 a0, a1, b0, b1;  // blurred rows y - 2 and y - 1 of both
        a0 = a1 = b0 = b1 = make_float4(0.f, 0.f, 0.f, 0.f);
        // Blurred rows y and y + 1 (J of this iteration's four) and the Sobel
        // rows y - 1 and y.
        auto pair = [&](auto jc, int y) {
            constexpr int J = decltype(jc)::value;
            float2 la0 = make_float2(0.f, 0.f), ha0 = la0, la1 = la0, ha1 = la0, lb0 = la0, hb0 = la0, lb1 = la0, hb1 = la0;
            float4 c0, c1;
#pragma unroll
            for (int j = 0; j <= WB; ++j) {  // input row y - RB + j
                const int q = J + j;
                const float4 p = (q < 4 ? g0 : (q < 8 ? g1 : g2))[32 * (q % 4)];
                if (j == RB) c0 = p;
                if (j == RB + 1) c1 = p;
                if (j < WB) {
                    const float2 w = make_float2(wrb[j], wrb[j]);
                    lb0 = __ffma2_rn(w, lo2(p), lb0);
                    hb0 = __ffma2_rn(w, hi2(p), hb0);
                }
                if (j > 0) {
                    const float2 w = make_float2(wrb[j - 1], wrb[j - 1]);
                    lb1 = __ffma2_rn(w, lo2(p), lb1);
                    hb1 = __ffma2_rn(w, hi2(p), hb1);
                }
                const int ja = j - (RB - RA);
                if (ja >= 0 && ja < WA) {
                    const float2 w = make_float2(wra[ja], wra[ja]);
                    la0 = __ffma2_rn(w, lo2(p), la0);
                    ha0 = __ffma2_rn(w, hi2(p), ha0);
                }
                if (ja >= 1 && ja <= WA) {
                    const float2 w = make_float2(wra[ja - 1], wra[ja - 1]);
                    la1 = __ffma2_rn(w, lo2(p), la1);
                    ha1 = __ffma2_rn(w, hi2(p), ha1);
                }
            }
            if (edge && VEC) {
                splat_outside(la0, ha0, x, cols);
                splat_outside(la1, ha1, x, cols);
                splat_outside(lb0, hb0, x, cols);
                splat_outside(lb1, hb1, x, cols);
            }
            float4 va0 = blur_horizontal<RA>(la0, ha0, wra), va1 = blur_horizontal<RA>(la1, ha1, wra);
            float4 vb0 = blur_horizontal<RB>(lb0, hb0, wrb), vb1 = blur_horizontal<RB>(lb1, hb1, wrb);
            if (edge && !VEC) {
                va0 = repeat_last(va0, x, cols);
                va1 = repeat_last(va1, x, cols);
                vb0 = repeat_last(vb0, x, cols);
                vb1 = repeat_last(vb1, x, cols);
            }
            auto store_row = [&](int yy, float4 va, float4 vb, float4 c) {
                const float4 u = make_float4(unsharp1(c.x, va.x, alpha), unsharp1(c.y, va.y, alpha),
                                             unsharp1(c.z, va.z, alpha), unsharp1(c.w, va.w, alpha));
                if (VEC) {
                    const size_t i = (size_t)yy * cols + x;
                    *reinterpret_cast<float4 *>(ba + i) = va;
                    *reinterpret_cast<float4 *>(bb + i) = vb;
                    *reinterpret_cast<float4 *>(sh + i) = u;
                } else {
                    store4(ba, rows, cols, false, yy, x, va);
                    store4(bb, rows, cols, false, yy, x, vb);
                    store4(sh, rows, cols, false, yy, x, u);
                }
            };
            if (stores && y >= y0 && y < yend) store_row(y, va0, vb0, c0);
            if (stores && y + 1 < yend) store_row(y + 1, va1, vb1, c1);
            if (y < 0 || y + 1 >= rows) {
                // rows outside the image repeat its first and last blurred row
                if (y < 0) {
                    va0 = va1;
                    vb0 = vb1;
                } else if (y == rows) {
                    va0 = a1;
                    vb0 = b1;
                } else {
                    va1 = va0;
                    vb1 = vb0;
                }
            }
            float4 ma0 = sobel_row(a0, a1, va0, edge, x, cols), ma1 = sobel_row(a1, va0, va1, edge, x, cols);
            float4 mb0 = sobel_row(b0, b1, vb0, edge, x, cols), mb1 = sobel_row(b1, vb0, vb1, edge, x, cols);
            if (edge && !VEC) {  // columns past the last one count as the last one
                ma0 = repeat_last(ma0, x, cols);
                ma1 = repeat_last(ma1, x, cols);
                mb0 = repeat_last(mb0, x, cols);
                mb1 = repeat_last(mb1, x, cols);
            }
            if (stores && y > y0 && y <= yend) {  // row y - 1 is of this band
                ra.add4(ma0);
                rb.add4(mb0);
            }
            if (stores && y >= y0 && y < yend) {  // so is row y
                ra.add4(ma1);
                rb.add4(mb1);
            }
            a0 = va0;
            a1 = va1;
            b0 = vb0;
            b1 = vb1;
        };
        // blurred rows y .. y + 3, y odd; the last one that counts is yend
#pragma unroll 1
        for (int y = y0 - 1; y <= yend; y += 4) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            copy_group(g3, y - RB + 3 * kS1Group);
            pair(std::integral_constant<int, 0>{}, y);
            pair(std::integral_constant<int, 2>{}, y + 2);
            float4 *g = g0;
            g0 = g1;
            g1 = g2;
            g2 = g3;
            g3 = g;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    block_ranges(ra, rb, red);
    if (threadIdx.x == 0) {
        const int b = blockIdx.y * gridDim.x + blockIdx.x;
        part_a[b] = make_float2(ra.lo, ra.hi);
        part_b[b] = make_float2(rb.lo, rb.hi);
    }
}

// Stage 2.  Warp strips as in sobel (one halo lane a side, the rows loaded two
// ahead of their use) over both blurred images at once.  Each block first
// combines stage 1's pairs by itself (a few hundred, from L2), which is quicker
// than a kernel of its own between the two; min and max round nothing, so every
// block gets the same range.  Launched as a programmatic dependent of stage 1.
// Bound by HBM: 63 us alone at 4096 x 4096 (403 MB, 0.94 of the rate), 67 us with
// full divisions in the stretch.
constexpr int kS2Cols = 4 * 30;

// (m - mn) / span, correctly rounded, 0 for a flat map, as extend.  Three
// instructions (div_by) instead of a full division while span lies well inside
// the normal range (`quick`): then mn and every m are finite, a magnitude is 0 or
// at least 2^-63 (its square is 0 or normal), so a difference of two is 0 or at
// least 2^-86, and neither the quotient (2^-126 at least) nor its residual
// leaves the range in which div_by rounds correctly.
__device__ __forceinline__ float4 stretch4(float4 m, float mn, float span, float rspan, bool quick, bool flat)
{
    const float4 d = make_float4(m.x - mn, m.y - mn, m.z - mn, m.w - mn);
    if (quick)
        return make_float4(div_by(d.x, span, rspan), div_by(d.y, span, rspan), div_by(d.z, span, rspan),
                           div_by(d.w, span, rspan));
    if (flat) return make_float4(0.f, 0.f, 0.f, 0.f);
    return make_float4(__fdiv_rn(d.x, span), __fdiv_rn(d.y, span), __fdiv_rn(d.z, span), __fdiv_rn(d.w, span));
}

struct Stretch {
    float mn, span, rspan;
    bool quick, flat;
    __device__ __forceinline__ explicit Stretch(Range r)
    {
        mn = r.lo;
        span = r.hi - mn;
        rspan = (float)(1.0 / (double)span);
        flat = !(r.hi > mn);
        quick = span >= 0x1p-60f && span <= 0x1p40f;
    }
    __device__ __forceinline__ float4 operator()(float4 m) const { return stretch4(m, mn, span, rspan, quick, flat); }
};

template <bool VEC>
__global__ void __launch_bounds__(kStThreads)
    img_stage2_kernel(const float *ba, const float *bb, const float *sh, const float2 *part_a, const float2 *part_b,
                      int pairs,
                      float *__restrict__ mm_a, float *__restrict__ mm_b, float *__restrict__ ea,
                      float *__restrict__ eb, float *__restrict__ out, int rows, int cols, int th)
{
    __shared__ float red[4][kStWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * kS2Cols + 4 * (lane - 1);
    const int y0 = (blockIdx.y * kStWarps + warp) * th;
    const int yend = min(y0 + th, rows);
    const bool edge = blockIdx.x == 0 || (int)(blockIdx.x + 1) * kS2Cols + 4 > cols;
    const bool stores = lane >= 1 && lane < 31 && x < cols;
    // stage 1 has completed and its writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    Range ra, rb;
    for (int b = threadIdx.x; b < pairs; b += kStThreads) {
        const float2 pa = load_dep(part_a + b), pb = load_dep(part_b + b);
        ra.lo = fminf(ra.lo, pa.x);
        ra.hi = fmaxf(ra.hi, pa.y);
        rb.lo = fminf(rb.lo, pb.x);
        rb.hi = fmaxf(rb.hi, pb.y);
    }
    block_ranges(ra, rb, red);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        mm_a[0] = ra.lo;
        mm_a[1] = ra.hi;
        mm_b[0] = rb.lo;
        mm_b[1] = rb.hi;
    }
    if (y0 >= rows) return;  // the whole warp
    const Stretch sa(ra), sb(rb);
    float4 a0 = load4_row(ba, rows, cols, VEC, y0 - 1, x), a1 = load4_row(ba, rows, cols, VEC, y0, x);
    float4 b0 = load4_row(bb, rows, cols, VEC, y0 - 1, x), b1 = load4_row(bb, rows, cols, VEC, y0, x);
    float4 a2 = load4_row(ba, rows, cols, VEC, y0 + 1, x), b2 = load4_row(bb, rows, cols, VEC, y0 + 1, x);
    float4 s0 = load4_row(sh, rows, cols, VEC, y0, x);
    for (int y = y0; y < yend; ++y) {
        const float4 a3 = load4_row(ba, rows, cols, VEC, y + 2, x), b3 = load4_row(bb, rows, cols, VEC, y + 2, x);
        const float4 s1 = load4_row(sh, rows, cols, VEC, y + 1, x);
        const float4 p = sa(sobel_row(a0, a1, a2, edge, x, cols));
        const float4 q = sb(sobel_row(b0, b1, b2, edge, x, cols));
        if (stores) {
            const float4 o = make_float4(combine1(s0.x, a1.x, b1.x, p.x, q.x), combine1(s0.y, a1.y, b1.y, p.y, q.y),
                                         combine1(s0.z, a1.z, b1.z, p.z, q.z), combine1(s0.w, a1.w, b1.w, p.w, q.w));
            const size_t i = (size_t)y * cols + x;
            if (VEC) {
                *reinterpret_cast<float4 *>(ea + i) = p;
                *reinterpret_cast<float4 *>(eb + i) = q;
                *reinterpret_cast<float4 *>(out + i) = o;
            } else {
                store4(ea, rows, cols, false, y, x, p);
                store4(eb, rows, cols, false, y, x, q);
                store4(out, rows, cols, false, y, x, o);
            }
        }
        a0 = a1;
        a1 = a2;
        a2 = a3;
        b0 = b1;
        b1 = b2;
        b2 = b3;
        s0 = s1;
    }
}

namespace {

// the unit's launches, in the order the launcher takes them
enum { kBlurA, kBlurB, kSobelA, kSobelB, kMmA, kMmB, kExtA, kExtB, kUnsharp, kCombine, kRoles };

// Band height for a grid of `strips` columns of warps: of the multiples of
// `unit`, the one whose waves of resident warps cost the fewest rows
// (each band pays `prime` rows of loads before its first output) in at most
// kMmMaxBlocks blocks; the tallest if none is few enough.
int band_height(int strips, int rows, int unit, int prime, int warps_per_wave, int max_m)
{
    int64_t best = INT64_MAX;
    int th_best = unit * max_m;
    for (int m = 1; m <= max_m; ++m) {
        const int th = unit * m;
        const int64_t blocks = (int64_t)strips * ceil_div(ceil_div(rows, th), kStWarps);
        const int64_t waves = ceil_div(blocks * kStWarps, warps_per_wave);
        const int64_t cost = waves * (th + prime);
        if (blocks <= kMmMaxBlocks && cost < best) {
            best = cost;
            th_best = th;
        }
    }
    return th_best;
}

bool aligned_all(std::initializer_list<const void *> ps)
{
    uintptr_t u = 0;
    for (const void *p : ps) u |= (uintptr_t)p;
    return (u & 15) == 0;
}

// Warps that one wave of kernel `fn` (kStThreads a block) holds.
int wave_warps(const void *fn, int &per_sm)
{
    if (per_sm < 1 &&
        (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kStThreads, 0) != cudaSuccess || per_sm < 1))
        per_sm = 1;
    return sm_count() * per_sm * kStWarps;
}

template <int RA, int RB, bool VEC> int launch_stage1(const LaunchArgs *const *m, cudaStream_t s, int &blocks)
{
    const LaunchArgs &l = *m[kBlurA];
    const int rows = l.i32(3), cols = l.i32(4);
    static int per_sm = 0;
    const int strips = (int)ceil_div(cols, kMgCols);
    const int th = band_height(strips, rows, 8, 12, wave_warps((const void *)img_stage1_kernel<RA, RB, VEC>, per_sm),
                               kS1MaxBand / 8);
    const dim3 g((unsigned)strips, (unsigned)ceil_div(ceil_div(rows, th), kStWarps));
    blocks = (int)(g.x * g.y);
    img_stage1_kernel<RA, RB, VEC><<<g, kStThreads, 0, s>>>(
        l.p<float>(0), l.p<float>(1), m[kBlurB]->p<float>(1), m[kUnsharp]->p<float>(2), l.p<float>(2),
        m[kBlurB]->p<float>(2), m[kMmA]->p<float2>(2), m[kMmB]->p<float2>(2), m[kUnsharp]->f32(3), rows, cols, th);
    return cudaGetLastError();
}

template <bool VEC> int launch_stages(const LaunchArgs *const *m, cudaStream_t s)
{
    const int rows = m[kBlurA]->i32(3), cols = m[kBlurA]->i32(4), ra = m[kBlurA]->i32(5), rb = m[kBlurB]->i32(5);
    int blocks = 0, e = cudaErrorInvalidValue;
    switch (ra * 8 + rb) {
    case 1 * 8 + 2: e = launch_stage1<1, 2, VEC>(m, s, blocks); break;
    case 1 * 8 + 3: e = launch_stage1<1, 3, VEC>(m, s, blocks); break;
    case 1 * 8 + 4: e = launch_stage1<1, 4, VEC>(m, s, blocks); break;
    case 2 * 8 + 3: e = launch_stage1<2, 3, VEC>(m, s, blocks); break;
    case 2 * 8 + 4: e = launch_stage1<2, 4, VEC>(m, s, blocks); break;
    case 3 * 8 + 4: e = launch_stage1<3, 4, VEC>(m, s, blocks); break;
    }
    if (e != cudaSuccess) return e;
    static int per_sm = 0;
    const int strips = (int)ceil_div(cols, kS2Cols);
    const int th = band_height(strips, rows, 4, 6, wave_warps((const void *)img_stage2_kernel<VEC>, per_sm), 64);
    return launch_dependent(img_stage2_kernel<VEC>,
                            dim3((unsigned)strips, (unsigned)ceil_div(ceil_div(rows, th), kStWarps)), kStThreads, s,
                            (const float *)m[kBlurA]->p<float>(1), (const float *)m[kBlurB]->p<float>(1),
                            (const float *)m[kUnsharp]->p<float>(2), (const float2 *)m[kMmA]->p<float2>(2),
                            (const float2 *)m[kMmB]->p<float2>(2), blocks, m[kMmA]->p<float>(1),
                            m[kMmB]->p<float>(1), m[kSobelA]->p<float>(1), m[kSobelB]->p<float>(1),
                            m[kCombine]->p<float>(5), rows, cols, th);
}

int launch_img_merged(const LaunchArgs *const *m, int, void *sv)
{
    // 128-bit groups need rows and arrays on 16-byte boundaries
    const bool vec = m[kBlurA]->i32(4) % 4 == 0 &&
                     aligned_all({m[kBlurA]->ptr[0], m[kBlurA]->ptr[1], m[kBlurB]->ptr[1], m[kUnsharp]->ptr[2],
                                  m[kSobelA]->ptr[1], m[kSobelB]->ptr[1], m[kCombine]->ptr[5]});
    return vec ? launch_stages<true>(m, (cudaStream_t)sv) : launch_stages<false>(m, (cudaStream_t)sv);
}

// the first launch of `kernel` among the run's first n whose array arguments named by
// (index, handle) pairs match; -1 if there is none
template <size_t N> int find(Run &run, int n, const char (&kernel)[N], int i0, int h0, int i1, int h1)
{
    for (int j = 0; j < n; ++j) {
        const RunLaunch &l = *run.at(j);
        if (l.array[i0] == h0 && (i1 < 0 || l.array[i1] == h1) && is(l.k, kernel)) return j;
    }
    return -1;
}

}  // namespace

// The IMG program around the combine launch of the run: found by its data
// flow, whatever the order of its independent launches.
bool merge_img(Run &run, Merge &out)
{
    int c = 1;
    while (run.kernel(c) && !is(run.kernel(c), "combine")) ++c;
    if (c + 1 < kRoles || !run.kernel(c) || !run.at(c)) return false;
    const int n = c + 1;
    auto at = [&](int j) -> const RunLaunch & { return *run.at(j); };
    const int32_t s = at(c).array[0], ba = at(c).array[1], bb = at(c).array[2], ea = at(c).array[3],
                  eb = at(c).array[4];
    int *r = out.member;
    r[kCombine] = c;
    r[kUnsharp] = find(run, n, "unsharp", 1, ba, 2, s);
    if (r[kUnsharp] < 0) return false;
    const int32_t img = at(r[kUnsharp]).array[0];
    r[kBlurA] = find(run, n, "gauss_blur", 0, img, 1, ba);
    r[kBlurB] = find(run, n, "gauss_blur", 0, img, 1, bb);
    r[kSobelA] = find(run, n, "sobel", 0, ba, 1, ea);
    r[kSobelB] = find(run, n, "sobel", 0, bb, 1, eb);
    r[kMmA] = find(run, n, "minmax", 0, ea, -1, 0);
    r[kMmB] = find(run, n, "minmax", 0, eb, -1, 0);
    for (int q = 0; q < kRoles; ++q)
        if (q != kExtA && q != kExtB && r[q] < 0) return false;
    r[kExtA] = find(run, n, "extend", 0, ea, 1, at(r[kMmA]).array[1]);
    r[kExtB] = find(run, n, "extend", 0, eb, 1, at(r[kMmB]).array[1]);
    if (r[kExtA] < 0 || r[kExtB] < 0) return false;
    // each launch after those whose results it takes, before those that
    // overwrite what it reads
    static const int before[][2] = {{kBlurA, kSobelA}, {kBlurB, kSobelB}, {kSobelA, kMmA},   {kSobelB, kMmB},
                                    {kMmA, kExtA},     {kMmB, kExtB},     {kExtA, kCombine}, {kExtB, kCombine},
                                    {kBlurA, kUnsharp}, {kUnsharp, kCombine}};
    for (const auto &p : before)
        if (r[p[0]] >= r[p[1]]) return false;
    // what is written is written once, and is none of the inputs
    const int32_t w[] = {ba, bb, ea, eb, s, at(c).array[5], at(r[kMmA]).array[1], at(r[kMmB]).array[1],
                         at(r[kMmA]).array[2], at(r[kMmB]).array[2], img, at(r[kBlurA]).array[2],
                         at(r[kBlurB]).array[2]};
    for (int i = 0; i < 10; ++i)
        for (int j = i + 1; j < 13; ++j)
            if (w[i] == w[j]) return false;
    // one image size, and radii that stage 1 is built for
    const LaunchArgs &l = at(r[kBlurA]).a;
    const int rows = l.i32(3), cols = l.i32(4);
    const int64_t px = (int64_t)rows * cols;
    for (int q : {kBlurB})
        if (at(r[q]).a.i32(3) != rows || at(r[q]).a.i32(4) != cols) return false;
    for (int q : {kSobelA, kSobelB})
        if (at(r[q]).a.i32(2) != rows || at(r[q]).a.i32(3) != cols) return false;
    if (at(r[kMmA]).a.i64(3) != px || at(r[kMmB]).a.i64(3) != px || at(r[kExtA]).a.i64(2) != px ||
        at(r[kExtB]).a.i64(2) != px || at(r[kUnsharp]).a.i64(4) != px || at(c).a.i64(6) != px)
        return false;
    const int ra = l.i32(5), rb = at(r[kBlurB]).a.i32(5);
    if (ra >= rb || rb > kMergeMaxR) return false;
    // the pairs of the tallest bands fit the minmax scratch
    if (ceil_div(cols, kMgCols) * ceil_div(ceil_div(rows, kS1MaxBand), kStWarps) > kMmMaxBlocks) return false;
    out.count = kRoles;
    out.launch = launch_img_merged;
    return true;
}

}  // namespace gdag
