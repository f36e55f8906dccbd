// DL nodes (Section IV-B, DL): a convolutional network projects two images to
// low-dimensional embeddings and combines them with a dense layer.
//   conv3x3_relu_pool  3x3 convolution (3 -> 64 channels, zero padding 1) +
//                      bias + ReLU + 2x2 max-pool, bf16 NCHW in and out, fp32
//                      accumulation on the tcgen05 tensor cores
//   avgpool_global     mean of every (image, channel) plane -> f32 embedding
//   concat_dense       out = [e1 e2] wd + bd, fp32
//
// conv3x3_relu_pool is an implicit GEMM on a persistent grid of one
// 576-thread CTA per SM that holds all 512 tensor-memory columns: two sets of
// accumulators, so that the tensor cores fill one set while the epilogue
// drains the other.  A tile is two input rows x 256 input columns of one
// image; its 512 pixels form four M = 128 operands, one per position in the
// 2x2 pooling window: accumulator a = 2*dy + p holds the pixels of row y0+dy
// and column parity p, so row m of every accumulator belongs to pooled column
// x0/2 + m and the pooling maximum is taken inside one thread, with no
// exchange.  N = 64 output channels, K = 27 taps padded to 32, fp32
// accumulation in tensor memory (four 128-lane x 64-column accumulators per
// set).  A launch does one convolution, or the two of a merged launch, whose
// tiles follow one another in one grid.
//
// K order.  A thread builds its im2col row from three aligned 32-bit words of
// each staged input row: L = columns (2m-2, 2m-1), C = (2m, 2m+1) and
// R = (2m+2, 2m+3) relative to x0.  The pixel of parity 0 takes taps
// (hi L, lo C, hi C), the pixel of parity 1 (lo C, hi C, lo R), so for both
// parities the word C supplies two taps as they are, and the third taps of the
// nine (channel, tap row) pairs are packed two per word.  K positions 0..17
// are the nine C words, 18..26 the nine lone taps, 27 and 28 carry the bias
// (A = 1, B = the bias split into a bf16 high part and a bf16 remainder, so
// the fp32 accumulator receives it to about 2^-18 relative), 29..31 are zero;
// the weight operand B_p is laid out in the same order, one per parity.  Operands use
// the canonical K-major layout without swizzle (8-row x 16-byte core
// matrices, 128 B between K-adjacent and 512 B between M/N-adjacent ones).
//
// Warp roles, per tile t (set s = t % 2).  What bounds a tile is the latency of the
// chain that it goes through in each role, not a rate, so the producers and the
// epilogue work in two teams, one per set: each has two tiles' time for its chain.
//   warp 17 (loader, one lane): keeps the halo copies (3 channels x 4 rows x
//     272 columns per tile, two cp.async.bulk.tensor boxes, zeros outside
//     the image, box slots padded to 128-byte boundaries) eight tiles ahead
//     in a ring of buffers, each completing on its own mbarrier, and refills a
//     buffer once its producers have read it ("halo empty").
//   warps 1-4 and 5-8 (producers, team s): wait for the tile's halo and for the
//     MMAs of tile t-2 to have read A set s, build A set s (thread m writes row m
//     of the four operands), and arrive on "A full" and "halo empty", one arrival
//     per warp.
//   warp 0 (control, one lane): once A set s is written ("A full") and the
//     epilogue has drained accumulator set s ("empty", tile t-2), issues eight
//     tcgen05.mma.cta_group::1.kind::f16 (K = 16 each) and commits them to
//     the set's "full" mbarrier.
//   warps 9-12 and 13-16 (epilogue, team s): all stage the weights once (one round
//     of loads of the raw weights and bias into a staging buffer, then the two B
//     operands of each convolution in the K order, one 16-byte core-matrix row per
//     store); per tile wait for "full", read the accumulators with
//     tcgen05.ld (warp w reads lanes 32*(w%4).., 16 channels a round),
//     signal "empty", take the maximum of the four (bias included; ReLU
//     commutes with the maximum), convert channel pairs to bf16 with ReLU in
//     one instruction and stage the pooled tile (64 channels x 128 columns, two
//     buffers a team) in shared memory, from where one thread writes it
//     with one TMA tensor store (8-byte vector stores by the team's 128 threads
//     when a pooled row is not a multiple of 8 values).
// Two convolutions of 16 x 3 x 256 x 256 take 22.4 us (0.68 us a tile beside about
// 4 us of start-up), from 34.4 us as two launches of a form with one team in each
// role, the halo copies issued by the control lane, and 1.0 us a tile.
// Every wait is bounded (about one second) and also ends when another role
// raises the shared abort flag; a warp or role decides to stop with a vote
// (__all_sync, or a barrier that ANDs its threads' results), so no barrier is
// left half-arrived.
// On an abort the CTA records status[0] = 1, lets its copies and MMAs in
// flight land (bounded), frees its tensor memory and returns.
#include <cuda.h>  // CUtensorMap and its enums (the encoder comes from the runtime's driver entry point)
#include <cuda_bf16.h>

#include <cstring>
#include <initializer_list>
#include <mutex>
#include <vector>

#include "catalog.h"
#include "kcommon.cuh"
#include "tcgen05.cuh"

namespace gdag {

constexpr int kConvM = 128, kConvN = 64, kConvK = 32, kConvTaps = 27;
constexpr int kCtlThreads = 32;                      // warp 0: MMA issue (one lane)
constexpr int kTeamThreads = 128;                    // a team of producers or of the epilogue
constexpr int kProdThreads = 2 * kTeamThreads;       // warps 1-8: im2col
constexpr int kEpiThreads = 2 * kTeamThreads;        // warps 9-16: epilogue and stores
constexpr int kLoadThreads = 32;                     // warp 17: halo copies (one lane)
constexpr int kConvThreads = kCtlThreads + kProdThreads + kEpiThreads + kLoadThreads;
constexpr int kTileCols = 256;                       // input columns per tile
constexpr int kHaloBox = 136;                        // columns per TMA box (two boxes: x0-8 .. x0+263)
constexpr int kHaloBoxBytes = kHaloBox * 4 * 3 * 2;  // 3 channels x 4 rows, bf16: the bytes one box moves
constexpr int kHaloBoxStride = (kHaloBoxBytes + 127) / 128 * 128;  // TMA destinations are 128-byte aligned
constexpr int kHaloBytes = 2 * kHaloBoxStride;       // one halo buffer
constexpr int kHaloBufs = 8;                         // halo ring depth: copies run this many tiles ahead
constexpr int kOpABytes = kConvM * kConvK * 2;       // 8 KB per accumulator
constexpr int kOpASet = 4 * kOpABytes;               // the four A operands of one tile
constexpr int kOpBBytes = kConvN * kConvK * 2;       // 4 KB per parity
constexpr int kAccCols = 4 * kConvN;                 // one accumulator set: 256 columns
constexpr int kTmemCols = 2 * kAccCols;              // two sets: the SM's 512 columns
constexpr int kStageBytes = kConvN * (kTileCols / 2) * 2;  // pooled tile [64][128] bf16
constexpr int kOffB = 2 * kOpASet;
constexpr int kOpBConv = 2 * kOpBBytes;              // the two B operands of one convolution
constexpr int kOffHalo = kOffB + 2 * kOpBConv;
constexpr int kOffStage = kOffHalo + kHaloBufs * kHaloBytes;
constexpr int kOffBars = kOffStage + 4 * kStageBytes;
// halo full and halo empty x kHaloBufs, A full x2, accumulator full x2, accumulator empty x2
constexpr int kNumBars = 2 * kHaloBufs + 6;
// more than half of the SM's 228 KB, so that one CTA (holding all 512
// tensor-memory columns) owns an SM
constexpr size_t kConvSmem = kOffBars + kNumBars * 8 + 16;
static_assert(kConvSmem > 114 * 1024 && kConvSmem <= 227 * 1024, "conv shared memory");
static_assert(kConvSmem < (size_t)(0x4000 << 4), "shared addresses fit a matrix descriptor's 14-bit start field");
static_assert(2 * kConvN * kConvTaps + 4 * kConvN <= kStageBytes, "raw weights must fit one staging buffer");
static_assert((2 * kConvN * (kConvK / 8)) % kEpiThreads == 0, "B rows split evenly over the epilogue");
static_assert(kOffHalo % 128 == 0 && kHaloBoxStride % 128 == 0 && kHaloBytes % 128 == 0 && kOffStage % 128 == 0 &&
                  kStageBytes % 128 == 0 && (kHaloBox * 2) % 16 == 0,
              "TMA shared-memory addresses must be 128-byte aligned, box rows multiples of 16 bytes");

// One convolution of a launch.
struct Conv {
    CUtensorMap tin, tout;
    const __nv_bfloat16 *wt;
    const float *bias;
    __nv_bfloat16 *out;
    int *status;
    int h, w, tma_store;
    int tiles_x, rows2, ntiles;
};
struct ConvPair {
    Conv m[2];
};

// byte offset of (row, k) in the canonical K-major, no-swizzle layout
__device__ __forceinline__ int umma_off(int row, int k)
{
    return ((row >> 3) * (kConvK / 8) + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// shared-memory matrix descriptor (sm_100): start >> 4, leading byte offset
// (between K-adjacent core matrices) >> 4 at bit 16, stride byte offset
// (between M/N-adjacent core matrices) >> 4 at bit 32, version 1 at bit 46,
// no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)((kConvK / 8) * 128 >> 4) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: D f32, A and B bf16, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t kConvIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kConvN >> 3) << 17) | ((uint32_t)(kConvM >> 4) << 24);

// weight index ci*9 + ky*3 + kx held at K position k of parity p's operand,
// -1 for the bias and zero positions 27..31 (the K order above)
__host__ __device__ __forceinline__ int conv_tap(int p, int k)
{
    const int i = k >> 1, half = k & 1;
    if (i < 9) return (i / 3) * 9 + (i % 3) * 3 + (p == 0 ? 1 : 0) + half;
    if (i < 14) {
        const int q = 2 * (i - 9) + half;
        return q < 9 ? (q / 3) * 9 + (q % 3) * 3 + (p == 0 ? 0 : 2) : -1;
    }
    return -1;
}

__device__ __forceinline__ void conv_tile_coords(int tile, int tiles_x, int rows2, int &b, int &y0, int &x0)
{
    const int xt = tile % tiles_x;
    const int r2 = (tile / tiles_x) % rows2;
    b = tile / (tiles_x * rows2);
    y0 = 2 * r2;
    x0 = xt * kTileCols;
}

// halo of one tile by TMA: two boxes of 136 columns x 4 rows x 3 channels
// starting at (x0 - 8, y0 - 1, 3b) of the image tensor (columns, rows,
// image*3 + channel); the hardware fills zeros outside the image, including
// the negative first column and row.  Issued by one thread; completion is
// counted in bytes on `bar`.
__device__ __forceinline__ void conv_issue_halo(const Conv &m, unsigned char *dst, uint32_t bar, int tile)
{
    int b, y0, x0;
    conv_tile_coords(tile, m.tiles_x, m.rows2, b, y0, x0);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2 * kHaloBoxBytes) : "memory");
#pragma unroll
    for (int half = 0; half < 2; ++half)
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
                smem_addr(dst + half * kHaloBoxStride)),
            "l"(reinterpret_cast<uint64_t>(&m.tin)), "r"(x0 - 8 + half * kHaloBox), "r"(y0 - 1), "r"(3 * b), "r"(bar)
            : "memory");
}

// The raw weights and bias of one convolution into `raw` (one round of loads),
// then the two B operands in the K order from there, one 16-byte core-matrix row
// (eight K positions of one channel) per store.  Thread etid builds the rows
// of channel etid % 64 at K chunk etid / 64 (uniform over a warp) for both
// parities: the chunk is matched against compile-time values, so every tap
// index is a constant.
constexpr int kRawWeights = kConvN * kConvTaps;
constexpr int kRawPer = (kRawWeights + kEpiThreads - 1) / kEpiThreads;
__device__ __forceinline__ void conv_load_raw(const Conv &m, unsigned char *raw, int etid)
{
    uint16_t *wraw = reinterpret_cast<uint16_t *>(raw);
    float *braw = reinterpret_cast<float *>(raw + 2 * kRawWeights);
    const unsigned short *wsrc = reinterpret_cast<const unsigned short *>(m.wt);
    unsigned short wl[kRawPer];
#pragma unroll
    for (int r = 0; r < kRawPer; ++r) {
        const int i = etid + r * kEpiThreads;
        wl[r] = i < kRawWeights ? __ldg(wsrc + i) : (unsigned short)0;
    }
    const float bl = etid < kConvN ? __ldg(m.bias + etid) : 0.f;
#pragma unroll
    for (int r = 0; r < kRawPer; ++r) {
        const int i = etid + r * kEpiThreads;
        if (i < kRawWeights) wraw[i] = wl[r];
    }
    if (etid < kConvN) braw[etid] = bl;
}

__device__ __forceinline__ void conv_build_b(const unsigned char *raw, unsigned char *sb, int etid)
{
    const uint16_t *wraw = reinterpret_cast<const uint16_t *>(raw);
    const float *braw = reinterpret_cast<const float *>(raw + 2 * kRawWeights);
    constexpr int kKc = kConvK / 8;
    static_assert(kEpiThreads == kConvN * kKc, "one channel and K chunk per epilogue thread");
    const int co = etid % kConvN, kq = etid / kConvN;
    const float bb = braw[co];
    const __nv_bfloat16 bhi = __float2bfloat16_rn(bb);
    const uint32_t bias_hi = __bfloat16_as_ushort(bhi);
    const uint32_t bias_lo = __bfloat16_as_ushort(__float2bfloat16_rn(bb - __bfloat162float(bhi)));
#pragma unroll
    for (int kc = 0; kc < kKc; ++kc) {
        if (kc != kq) continue;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            uint32_t q[4];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                uint32_t two = 0;
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const int k = 8 * kc + j + h2, tap = conv_tap(p, k);
                    const uint32_t v = tap >= 0 ? (uint32_t)wraw[co * kConvTaps + tap]
                                                : (k == 27 ? bias_hi : (k == 28 ? bias_lo : 0u));
                    two |= v << (16 * h2);
                }
                q[j / 2] = two;
            }
            *reinterpret_cast<uint4 *>(sb + p * kOpBBytes + umma_off(co, 8 * kc)) = make_uint4(q[0], q[1], q[2], q[3]);
        }
    }
}

__global__ void __launch_bounds__(kConvThreads, 1) conv3x3_relu_pool_kernel(const __grid_constant__ ConvPair pair)
{
    extern __shared__ __align__(1024) unsigned char conv_smem[];
    unsigned char *sa = conv_smem;                  // two sets of four A operands
    unsigned char *sb = conv_smem + kOffB;          // two B operands of each convolution
    unsigned char *halo = conv_smem + kOffHalo;     // halo buffers [box][ci][row][136]
    unsigned char *stage = conv_smem + kOffStage;   // two pooled tiles [64][128] a team
    uint64_t *bars = reinterpret_cast<uint64_t *>(conv_smem + kOffBars);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kNumBars);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int n0 = pair.m[0].ntiles, ntiles = n0 + pair.m[1].ntiles;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // every CTA is resident: the pools' start-up may pass

    // the TMA copies need a 128-byte aligned window: check before any copy
    // or tensor-memory use (uniform over the CTA)
    if ((smem_addr(conv_smem) & 127u) != 0) {
        if (threadIdx.x == 0)
            for (int q = 0; q < 2; ++q)
                if (pair.m[q].ntiles > 0) atomicExch(pair.m[q].status, 2);
        return;
    }
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t halo_bar = smem_addr(&bars[0]);                // + 8 * buffer: the tile's halo landed
    const uint32_t hempty_bar = smem_addr(&bars[kHaloBufs]);      // + 8 * buffer: the producers read it
    const uint32_t afull_bar = smem_addr(&bars[2 * kHaloBufs]);   // + 8 * set: A written
    const uint32_t full_bar = afull_bar + 16;                     // + 8 * set: MMAs done (A read, accumulators ready)
    const uint32_t empty_bar = afull_bar + 32;                    // + 8 * set: epilogue done reading the accumulators

    if (warp == 0) {
        if (lane == 0) {
            *abort = 0;
            for (int j = 0; j < kHaloBufs; ++j) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(halo_bar + 8 * j));
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(hempty_bar + 8 * j), "r"(kTeamThreads / 32));
            }
            for (int s = 0; s < 2; ++s) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(afull_bar + 8 * s), "r"(kTeamThreads / 32));
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full_bar + 8 * s));
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty_bar + 8 * s), "r"(kTeamThreads / 32));
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "n"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();  // barriers initialised, tensor memory allocated
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;
    const int stride = (int)gridDim.x;

    if (warp == 0) {
        // ---- control (one lane): MMA issue
        // the whole warp meets the epilogue warps, which staged the weights
        asm volatile("bar.sync 3, %0;" ::"n"(kCtlThreads + kEpiThreads) : "memory");
        if (lane == 0) {
            const uint64_t a_desc0 = umma_desc(smem_addr(sa)), b_desc0 = umma_desc(smem_addr(sb));
            uint32_t it = 0;
            int issued_mma = 0;  // tiles of this CTA (in order) whose MMAs were issued
            for (int tile = blockIdx.x; tile < ntiles; tile += stride, ++it) {
                const int s = it & 1;
                // A set s written; accumulator set s drained by the epilogue of tile it-2
                if (!mbar_wait_bounded(afull_bar + 8 * s, (it >> 1) & 1, abort) ||
                    (it >= 2 && !mbar_wait_bounded(empty_bar + 8 * s, ((it >> 1) - 1) & 1, abort))) {
                    *abort = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                // descriptors differ from the first one only in their start
                // address field (no carry: shared addresses stay below 256 KB)
                const uint64_t a_set = a_desc0 + (uint64_t)(s * (kOpASet >> 4));
                const uint64_t b_set = b_desc0 + (uint64_t)(tile >= n0 ? kOpBConv >> 4 : 0);
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int ks = 0; ks < kConvK / 16; ++ks) {
                        const uint64_t ad = a_set + (uint64_t)((a * kOpABytes + ks * 256) >> 4);
                        const uint64_t bd = b_set + (uint64_t)(((a & 1) * kOpBBytes + ks * 256) >> 4);
                        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                                     " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
                                         tmem + s * kAccCols + a * kConvN),
                                     "l"(ad), "l"(bd), "r"(kConvIdesc), "r"((uint32_t)ks));
                    }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    full_bar + 8 * s));
                ++issued_mma;
            }
            if (*abort && issued_mma > 0) {
                // the MMAs in flight finish before the CTA frees tensor memory
                // (a bounded wait that ignores the abort flag)
                const volatile int no_abort = 0;
                const int last = issued_mma - 1;
                mbar_wait_bounded(full_bar + 8 * (last & 1), (last >> 1) & 1, &no_abort);
            }
        }
        __syncwarp();
    } else if (warp <= kProdThreads / 32) {
        // ---- producers, team s: row m of the four A operands of its tiles
        const int s = (tid - kCtlThreads) / kTeamThreads, m = (tid - kCtlThreads) % kTeamThreads;
        int woff[3];  // byte offsets of halo words m+3, m+4, m+5 (L, C, R), each in its box
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int wq = m + 3 + q, box = wq >= kHaloBox / 2;
            woff[q] = box * kHaloBoxStride + (wq - box * (kHaloBox / 2)) * 4;
        }
        unsigned char *As = sa + s * kOpASet;
        uint32_t it = s;
        for (int tile = blockIdx.x + s * stride; tile < ntiles; tile += 2 * stride, it += 2) {
            const int hb = it % kHaloBufs;
            const bool hok = mbar_wait_bounded(halo_bar + 8 * hb, (it / kHaloBufs) & 1, abort);
            // A set s was last read by the MMAs of tile it-2
            const bool aok = it < 2 || mbar_wait_bounded(full_bar + 8 * s, ((it >> 1) - 1) & 1, abort);
            if (!__all_sync(0xffffffffu, hok && aok)) {  // warp-uniform: the warp meets at __syncwarp below
                if (lane == 0) *abort = 1;
                break;
            }
            const unsigned char *hbuf = halo + hb * kHaloBytes;
            uint32_t Lw[12], Cw[12], Rw[12];  // [ci][row 0..3]
#pragma unroll
            for (int ci = 0; ci < 3; ++ci)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const unsigned char *row = hbuf + (ci * 4 + r) * (kHaloBox * 2);
                    Lw[ci * 4 + r] = *reinterpret_cast<const uint32_t *>(row + woff[0]);
                    Cw[ci * 4 + r] = *reinterpret_cast<const uint32_t *>(row + woff[1]);
                    Rw[ci * 4 + r] = *reinterpret_cast<const uint32_t *>(row + woff[2]);
                }
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    uint32_t wd[16];
#pragma unroll
                    for (int i = 0; i < 9; ++i) wd[i] = Cw[(i / 3) * 4 + dy + i % 3];
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const int q0 = 2 * i, q1 = 2 * i + 1;
                        const int r0 = (q0 / 3) * 4 + dy + q0 % 3, r1 = q1 < 9 ? (q1 / 3) * 4 + dy + q1 % 3 : 0;
                        if (p == 0)
                            wd[9 + i] = __byte_perm(Lw[r0], q1 < 9 ? Lw[r1] : 0u, 0x7632);
                        else
                            wd[9 + i] = __byte_perm(Rw[r0], q1 < 9 ? Rw[r1] : 0u, 0x5410);
                    }
                    wd[13] |= 0x3F800000u;  // K 27: 1.0 (bias, high part)
                    wd[14] = 0x00003F80u;    // K 28: 1.0 (bias, remainder)
                    wd[15] = 0u;
                    unsigned char *A = As + (2 * dy + p) * kOpABytes;
#pragma unroll
                    for (int kc = 0; kc < 4; ++kc)
                        *reinterpret_cast<uint4 *>(A + umma_off(m, 8 * kc)) =
                            make_uint4(wd[4 * kc], wd[4 * kc + 1], wd[4 * kc + 2], wd[4 * kc + 3]);
                }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic stores -> tensor-core reads
            __syncwarp();
            if (lane == 0) {
                // every value read from the halo has been written to A above
                mbar_arrive(afull_bar + 8 * s);
                mbar_arrive(hempty_bar + 8 * hb);
            }
        }
    } else if (warp == kConvThreads / 32 - 1) {
        // ---- loader (one lane): halo copies kHaloBufs tiles ahead
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&pair.m[0].tin)) : "memory");
            uint32_t it = 0;
            for (int tile = blockIdx.x; tile < ntiles; tile += stride, ++it) {
                const int hb = it % kHaloBufs;
                if (it >= kHaloBufs && !mbar_wait_bounded(hempty_bar + 8 * hb, ((it / kHaloBufs) - 1) & 1, abort)) {
                    *abort = 1;
                    break;
                }
                const bool second = tile >= n0;
                conv_issue_halo(pair.m[second], halo + hb * kHaloBytes, halo_bar + 8 * hb, tile - (second ? n0 : 0));
            }
            if (*abort) {
                // the copies in flight land before the CTA frees its memory
                // (bounded waits that ignore the abort flag): the last copy
                // into buffer j was tile index jl, the largest below `it` that
                // is j modulo kHaloBufs
                const volatile int no_abort = 0;
                for (uint32_t j = 0; j < (uint32_t)kHaloBufs && j < it; ++j) {
                    const uint32_t jl = j + (it - 1 - j) / kHaloBufs * kHaloBufs;
                    mbar_wait_bounded(halo_bar + 8 * j, (jl / kHaloBufs) & 1, &no_abort);
                }
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: stage the weights once, then team s reads TMEM lanes
        // 32*quad.. of its tiles' accumulators, pooled column x0/2 + mo
        const int etid = tid - kCtlThreads - kProdThreads;
        {
            // raw copies in the team buffers that are written last (tiles 2 and 3)
            unsigned char *raw0 = stage + kStageBytes, *raw1 = stage + 3 * kStageBytes;
            conv_load_raw(pair.m[0], raw0, etid);
            if (ntiles > n0) conv_load_raw(pair.m[1], raw1, etid);
            asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads) : "memory");
            conv_build_b(raw0, sb, etid);
            if (ntiles > n0) conv_build_b(raw1, sb + kOpBConv, etid);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // B: generic stores -> tensor-core reads
            asm volatile("bar.sync 3, %0;" ::"n"(kCtlThreads + kEpiThreads) : "memory");
        }
        const int s = etid / kTeamThreads, et = etid % kTeamThreads, quad = warp & 3;
        const int mo = quad * 32 + lane;
        unsigned char *sg0 = stage + 2 * s * kStageBytes;
        uint32_t it = s;
        for (int tile = blockIdx.x + s * stride; tile < ntiles; tile += 2 * stride, it += 2) {
            const bool second = tile >= n0;
            const Conv &m = pair.m[second];
            int b, y0, x0;  // the tile's coordinates, computed while its MMAs may still run
            conv_tile_coords(tile - (second ? n0 : 0), m.tiles_x, m.rows2, b, y0, x0);
            const bool fok = mbar_wait_bounded(full_bar + 8 * s, (it >> 1) & 1, abort);
            asm volatile("tcgen05.fence::after_thread_sync;");
            unsigned char *sg = sg0 + ((it >> 1) & 1) * kStageBytes;
#pragma unroll
            for (int chunk = 0; chunk < kConvN / 16; ++chunk) {
                const int c0 = 16 * chunk;
                uint32_t v[4][16];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + s * kAccCols + a * kConvN + c0;
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                        : "=r"(v[a][0]), "=r"(v[a][1]), "=r"(v[a][2]), "=r"(v[a][3]), "=r"(v[a][4]), "=r"(v[a][5]),
                          "=r"(v[a][6]), "=r"(v[a][7]), "=r"(v[a][8]), "=r"(v[a][9]), "=r"(v[a][10]), "=r"(v[a][11]),
                          "=r"(v[a][12]), "=r"(v[a][13]), "=r"(v[a][14]), "=r"(v[a][15])
                        : "r"(taddr));
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (chunk == kConvN / 16 - 1) {
                    // this warp is done with accumulator set s
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty_bar + 8 * s);
                }
                uint16_t *st = reinterpret_cast<uint16_t *>(sg) + c0 * (kTileCols / 2) + mo;
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    float m0, m1;
                    asm("max.f32 %0, %1, %2, %3;"
                        : "=f"(m0)
                        : "f"(__uint_as_float(v[0][j])), "f"(__uint_as_float(v[1][j])), "f"(__uint_as_float(v[2][j])));
                    asm("max.f32 %0, %1, %2, %3;"
                        : "=f"(m1)
                        : "f"(__uint_as_float(v[0][j + 1])), "f"(__uint_as_float(v[1][j + 1])),
                          "f"(__uint_as_float(v[2][j + 1])));
                    m0 = fmaxf(m0, __uint_as_float(v[3][j]));
                    m1 = fmaxf(m1, __uint_as_float(v[3][j + 1]));
                    uint32_t pk;  // channel c0+j in the low half, c0+j+1 in the high half
                    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(pk) : "f"(m1), "f"(m0));
                    st[j * (kTileCols / 2)] = (uint16_t)(pk & 0xFFFFu);
                    st[(j + 1) * (kTileCols / 2)] = (uint16_t)(pk >> 16);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // staging writes -> TMA store reads
            // the store of the team's previous tile must be done reading its
            // buffer before the team's next tile writes it
            if (et == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            if (!bar_and(4 + s, kTeamThreads, fok && !*abort)) {
                if (et == 0) *abort = 1;
                break;
            }
            if (m.tma_store) {
                // one TMA store of the 128 x 1 x 64 box at (x0/2, y0/2, 64b);
                // the hardware drops the columns past the image edge
                if (et == 0) {
                    asm volatile(
                        "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                            reinterpret_cast<uint64_t>(&m.tout)),
                        "r"(x0 >> 1), "r"(y0 >> 1), "r"(kConvN * b), "r"(smem_addr(sg))
                        : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            } else {
                // pooled rows not a multiple of 8 values: 8-byte stores of
                // whole vectors (the valid width, wo - x0/2 capped at 128, is
                // a multiple of 4); the team's next tile writes the other buffer
                const int ho = m.h / 2, wo = m.w / 2;
                const int valid = min(kTileCols / 2, wo - (x0 >> 1));
                __nv_bfloat16 *orow = m.out + (((size_t)b * kConvN) * ho + (y0 >> 1)) * wo + (x0 >> 1);
                const size_t plane = (size_t)ho * wo;
                const uint2 *src = reinterpret_cast<const uint2 *>(sg);
                for (int i = et; i < kConvN * (kTileCols / 8); i += kTeamThreads) {
                    const int ch = i / (kTileCols / 8), j = i % (kTileCols / 8);
                    if (4 * j < valid) *reinterpret_cast<uint2 *>(orow + ch * plane + 4 * j) = src[i];
                }
            }
        }
        if (et == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    if (tid == 0 && *abort)
        for (int q = 0; q < 2; ++q)
            if (pair.m[q].ntiles > 0) atomicExch(pair.m[q].status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols));
}

// e[p] = mean of plane p (hw bf16 values), fp32 per thread, fixed-order
// block tree; one block per plane.  128-bit loads when every plane starts on
// a 16-byte boundary (hw % 8 == 0 and an aligned base), eight of a thread in
// flight, each one's eight values summed as a tree; scalar loads otherwise.
// A launch does one input, or the two of a merged launch (blocks [0, planes)
// of the grid the first).
struct AvgPool {
    const __nv_bfloat16 *p;
    float *e;
    int hw, vec, planes;
};
struct AvgPoolPair {
    AvgPool m[2];
};

__global__ void __launch_bounds__(256) avgpool_global_kernel(const __grid_constant__ AvgPoolPair pair)
{
    __shared__ double sh[256 / 32];
    const bool second = (int)blockIdx.x >= pair.m[0].planes;
    const AvgPool &m = pair.m[second];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");  // in a unit, the convolutions' outputs are visible
    const int plane = (int)blockIdx.x - (second ? pair.m[0].planes : 0), hw = m.hw;
    float s = 0.f;
    if (m.vec) {
        const uint4 *q = reinterpret_cast<const uint4 *>(m.p + (size_t)plane * hw);
        constexpr int kV = 8;
        for (int i = threadIdx.x; i < hw / 8; i += kV * 256) {
            uint4 v[kV];
#pragma unroll
            for (int k = 0; k < kV; ++k) v[k] = i + k * 256 < hw / 8 ? load_dep(q + i + k * 256) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int k = 0; k < kV; ++k) {
                const uint32_t u[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
                float t[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) t[j] = __uint_as_float(u[j] << 16) + __uint_as_float(u[j] & 0xFFFF0000u);
                s += (t[0] + t[1]) + (t[2] + t[3]);
            }
        }
    } else {
        const uint16_t *q = reinterpret_cast<const uint16_t *>(m.p) + (size_t)plane * hw;
        for (int i = threadIdx.x; i < hw; i += 256) s += __uint_as_float((uint32_t)load_dep(q + i) << 16);
    }
    const double t = block_sum((double)s, sh);
    if (threadIdx.x == 0) m.e[plane] = (float)(t / hw);
}

// out[b][j] = bd[j] + sum_i e1[b][i] wd[i][j] + sum_i e2[b][i] wd[c+i][j]:
// one block per image, one warp per class (strided), the 2c products of a
// logit split over the lanes and summed by a fixed shuffle tree.
__global__ void __launch_bounds__(256) concat_dense_kernel(const float *e1, const float *e2,
                                                           const float *__restrict__ wd, const float *__restrict__ bd,
                                                           float *__restrict__ out, int c, int classes)
{
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");  // in a unit, the embeddings are visible
    for (int j = warp; j < classes; j += 256 / 32) {
        float s = 0.f;
        for (int i = lane; i < 2 * c; i += 32) {
            const float e = load_dep(i < c ? e1 + (size_t)b * c + i : e2 + (size_t)b * c + (i - c));
            s = fmaf(e, wd[(size_t)i * classes + j], s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[(size_t)b * classes + j] = s + bd[j];
    }
}

namespace {

const char *validate_conv(const LaunchArgs &a)
{
    const int n = a.i32(5), h = a.i32(6), w = a.i32(7);
    if (n < 1 || h < 2 || w < 8) return "n >= 1, h >= 2, w >= 8 required";
    if (h % 2 || w % 8) return "h must be even and w a multiple of 8";
    if ((int64_t)n * (h / 2) * ceil_div(w, kTileCols) > INT32_MAX) return "too many tiles";
    if (a.bytes[0] / 2 / 3 / (size_t)h / (size_t)w < (size_t)n) return "x smaller than n x 3 x h x w bf16";
    if (a.bytes[1] < (size_t)kConvN * kConvTaps * 2) return "weights smaller than 64 x 3 x 3 x 3 bf16";
    if (a.bytes[2] < (size_t)kConvN * 4) return "bias smaller than 64 floats";
    if (a.bytes[3] / 2 / kConvN / (size_t)(h / 2) / (size_t)(w / 2) < (size_t)n)
        return "out smaller than n x 64 x h/2 x w/2 bf16";
    if (a.bytes[4] < 4) return "status smaller than one int32";
    if ((reinterpret_cast<uintptr_t>(a.ptr[0]) & 15) != 0 || (reinterpret_cast<uintptr_t>(a.ptr[3]) & 15) != 0)
        return "x and out must be 16-byte aligned";
    return nullptr;
}

// rank-3 bf16 tensor map, dims innermost first, dense; zeros outside
bool encode_bf16_3d(CUtensorMap *m, void *base, uint64_t d0, uint64_t d1, uint64_t d2, uint32_t b0, uint32_t b1,
                    uint32_t b2)
{
    EncodeTiled fn = tma_encoder();
    if (!fn) return false;
    const cuuint64_t dims[3] = {d0, d1, d2};
    const cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
    const cuuint32_t box[3] = {b0, b1, b2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct ConvMaps {
    const void *x = nullptr, *out = nullptr;
    int n = 0, h = 0, w = 0;
    CUtensorMap tin, tout;
};

// The tensor maps of one convolution.  Per process: raise the dynamic
// shared-memory limit once (no attribute calls on later launches, so the launch
// can be stream-captured), and keep the tensor maps of the last few (buffer,
// shape) combinations.
cudaError_t conv_maps(const LaunchArgs &a, Conv &out)
{
    const int n = a.i32(5), h = a.i32(6), w = a.i32(7);
    const int wo = w / 2, tma_store = wo % 8 == 0;
    static std::mutex mu;
    static bool configured = false;
    static ConvMaps cache[8];
    static int cache_next = 0;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(conv3x3_relu_pool_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kConvSmem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    int hit = -1;
    for (int i = 0; i < 8; ++i)
        if (cache[i].x == a.ptr[0] && cache[i].out == a.ptr[3] && cache[i].n == n && cache[i].h == h && cache[i].w == w)
            hit = i;
    if (hit < 0) {
        ConvMaps m;
        m.x = a.ptr[0];
        m.out = a.ptr[3];
        m.n = n;
        m.h = h;
        m.w = w;
        std::memset(&m.tin, 0, sizeof m.tin);
        std::memset(&m.tout, 0, sizeof m.tout);
        if (!encode_bf16_3d(&m.tin, a.ptr[0], (uint64_t)w, (uint64_t)h, (uint64_t)3 * n, kHaloBox, 4, 3))
            return cudaErrorNotSupported;
        if (tma_store && !encode_bf16_3d(&m.tout, a.ptr[3], (uint64_t)wo, (uint64_t)(h / 2), (uint64_t)kConvN * n,
                                         kTileCols / 2, 1, kConvN))
            return cudaErrorNotSupported;
        hit = cache_next;
        cache[hit] = m;
        cache_next = (cache_next + 1) % 8;
    }
    out.tin = cache[hit].tin;
    out.tout = cache[hit].tout;
    return cudaSuccess;
}

// One convolution, or the two of a merged launch.
int launch_conv_run(const LaunchArgs *const *m, int count, void *s)
{
    ConvPair pair;
    std::memset(&pair, 0, sizeof pair);
    int64_t tiles = 0;
    for (int i = 0; i < count; ++i) {
        const LaunchArgs &a = *m[i];
        const int n = a.i32(5), h = a.i32(6), w = a.i32(7);
        Conv &c = pair.m[i];
        const cudaError_t e = conv_maps(a, c);
        if (e != cudaSuccess) return e;
        c.wt = a.p<__nv_bfloat16>(1);
        c.bias = a.p<float>(2);
        c.out = a.p<__nv_bfloat16>(3);
        c.status = a.p<int>(4);
        c.h = h;
        c.w = w;
        c.tma_store = (w / 2) % 8 == 0;
        c.tiles_x = (int)ceil_div(w, kTileCols);
        c.rows2 = h / 2;
        c.ntiles = n * c.rows2 * c.tiles_x;
        tiles += c.ntiles;
    }
    const unsigned grid = (unsigned)(tiles < sm_count() ? tiles : sm_count());
    conv3x3_relu_pool_kernel<<<grid, kConvThreads, kConvSmem, (cudaStream_t)s>>>(pair);
    return cudaGetLastError();
}

int launch_conv(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_conv_run(m, 1, s);
}

const char *validate_avgpool(const LaunchArgs &a)
{
    const int planes = a.i32(2), hw = a.i32(3);
    if (planes < 1 || hw < 1) return "planes >= 1 and hw >= 1 required";
    if (a.bytes[0] / 2 / (size_t)hw < (size_t)planes) return "input smaller than planes x hw bf16";
    if (a.bytes[1] / 4 < (size_t)planes) return "e smaller than planes floats";
    return nullptr;
}

AvgPoolPair avgpool_pair(const LaunchArgs *const *m, int count, unsigned *grid)
{
    AvgPoolPair pair = {};
    int blocks = 0;
    for (int i = 0; i < count; ++i) {
        const LaunchArgs &a = *m[i];
        const int hw = a.i32(3);
        pair.m[i] = AvgPool{a.p<__nv_bfloat16>(0), a.p<float>(1), hw,
                            hw % 8 == 0 && (reinterpret_cast<uintptr_t>(a.ptr[0]) & 15) == 0, a.i32(2)};
        blocks += pair.m[i].planes;
    }
    *grid = (unsigned)blocks;
    return pair;
}

int launch_avgpool_run(const LaunchArgs *const *m, int count, void *s)
{
    unsigned grid;
    const AvgPoolPair pair = avgpool_pair(m, count, &grid);
    avgpool_global_kernel<<<grid, 256, 0, (cudaStream_t)s>>>(pair);
    return cudaGetLastError();
}

int launch_avgpool(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_avgpool_run(m, 1, s);
}

const char *validate_dense(const LaunchArgs &a)
{
    const int n = a.i32(5), c = a.i32(6), k = a.i32(7);
    if (n < 1 || c < 1 || k < 1) return "n, c and classes must be >= 1";
    if (a.bytes[0] / 4 / (size_t)c < (size_t)n || a.bytes[1] / 4 / (size_t)c < (size_t)n)
        return "e1 or e2 smaller than n x c floats";
    if (a.bytes[2] / 4 / (size_t)k < (size_t)2 * c) return "wd smaller than 2c x classes floats";
    if (a.bytes[3] / 4 < (size_t)k) return "bd smaller than classes floats";
    if (a.bytes[4] / 4 / (size_t)k < (size_t)n) return "out smaller than n x classes floats";
    return nullptr;
}

int launch_dense(const LaunchArgs &a, void *s)
{
    const int n = a.i32(5), k = a.i32(7);
    concat_dense_kernel<<<(unsigned)n, 256, 0, (cudaStream_t)s>>>(a.p<float>(0), a.p<float>(1), a.p<float>(2),
                                                                  a.p<float>(3), a.p<float>(4), a.i32(6), k);
    return cudaGetLastError();
}

// Whether two launches may run in either order: neither writes an array of the other.
bool apart(const RunLaunch &f, const RunLaunch &g)
{
    for (int p = 0; p < f.a.nargs; ++p)
        for (int q = 0; q < g.a.nargs; ++q)
            if (f.k->spec[p].kind == GDAG_ARG_ARRAY && g.k->spec[q].kind == GDAG_ARG_ARRAY && f.array[p] == g.array[q] &&
                (f.k->spec[p].mode != GDAG_MODE_IN || g.k->spec[q].mode != GDAG_MODE_IN))
                return false;
    return true;
}

// The same kernel on two inputs, the two branches of the DL program: the next
// launch of it that shares nothing written with the first.  One grid pays one
// start-up and one part-filled last round (4096 tiles over 152 CTAs make 27
// rounds, 2048 make 14), and the host one launch.
template <MergeLaunchFn LAUNCH> bool merge_branches(Run &run, Merge &out)
{
    const RunLaunch &f = *run.at(0);
    // work items (tiles or planes), which one grid counts in 32 bits
    auto items = [](const LaunchArgs &a) {
        return a.nargs == 8 ? (int64_t)a.i32(5) * (a.i32(6) / 2) * ceil_div(a.i32(7), kTileCols) : (int64_t)a.i32(2);
    };
    for (int j = 1; run.kernel(j); ++j) {
        if (run.kernel(j) != f.k) continue;
        if (!run.at(j)) return false;
        const RunLaunch &g = *run.at(j);
        if (items(f.a) + items(g.a) > INT32_MAX / 2 || !apart(f, g)) return false;
        out.count = out.apart = 2;
        out.member[0] = 0;
        out.member[1] = j;
        out.launch = LAUNCH;
        return true;
    }
    return false;
}

// Two convolutions, the pools of their outputs and the dense layer over these: the
// two pairs and the dense layer, each a programmatic dependent of the launch
// before it, so that its start-up passes while that one still runs.
// 16 x 3 x 256 x 256 twice, a step: 35.5 us, from 37.7 us as two pairs and a launch.
int launch_branches(const LaunchArgs *const *m, int, void *s)
{
    int r = launch_conv_run(m, 2, s);
    if (r) return r;
    unsigned grid;
    const AvgPoolPair pools = avgpool_pair(m + 2, 2, &grid);
    r = launch_dependent(avgpool_global_kernel, dim3(grid), 256, (cudaStream_t)s, pools);
    if (r) return r;
    const LaunchArgs &d = *m[4];
    return launch_dependent(concat_dense_kernel, dim3((unsigned)d.i32(5)), 256, (cudaStream_t)s,
                            (const float *)d.p<float>(0), (const float *)d.p<float>(1), (const float *)d.p<float>(2),
                            (const float *)d.p<float>(3), d.p<float>(4), d.i32(6), d.i32(7));
}

// The five launches in a row (either order of the branches), the pools after both
// convolutions; other programs keep the pairs.
bool merge_dl(Run &run, Merge &out)
{
    if (!merge_branches<launch_conv_run>(run, out)) return false;
    if (out.member[1] != 1 || !is(run.kernel(2), "avgpool_global") || run.kernel(3) != run.kernel(2) ||
        !is(run.kernel(4), "concat_dense") || !run.at(4))
        return true;
    const RunLaunch &a = *run.at(0), &b = *run.at(1);
    const int pool0 = run.at(2)->array[0] == a.array[3] ? 2 : 3, pool1 = 5 - pool0;
    const RunLaunch &p = *run.at(pool0), &q = *run.at(pool1), &d = *run.at(4);
    if (p.array[0] != a.array[3] || q.array[0] != b.array[3] || !apart(p, q)) return true;
    if (!((d.array[0] == p.array[1] && d.array[1] == q.array[1]) || (d.array[0] == q.array[1] && d.array[1] == p.array[1])))
        return true;
    if ((int64_t)p.a.i32(2) + q.a.i32(2) > INT32_MAX / 2) return true;
    out.count = 5;
    const int order[5] = {0, 1, pool0, pool1, 4};
    for (int k = 0; k < 5; ++k) out.member[k] = order[k];
    out.launch = launch_branches;
    return true;
}

KernelEntry entry(const char *name, const void *fn, std::initializer_list<gdag_argspec> spec, ValidateFn v,
                  LauncherFn l)
{
    KernelEntry e;
    e.name = name;
    e.fn = fn;
    e.nargs = (int)spec.size();
    int i = 0;
    for (const auto &sp : spec) e.spec[i++] = sp;
    e.validate = v;
    e.launcher = l;
    return e;
}

}  // namespace

void append_dl_kernels(std::vector<KernelEntry> &v)
{
    v.push_back(entry("conv3x3_relu_pool", (const void *)conv3x3_relu_pool_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT),
                       arr(GDAG_MODE_INOUT), scal(4), scal(4), scal(4)},
                      validate_conv, launch_conv));
    v.back().merge = merge_dl;
    v.push_back(entry("avgpool_global", (const void *)avgpool_global_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT), scal(4), scal(4)}, validate_avgpool, launch_avgpool));
    v.back().merge = merge_branches<launch_avgpool_run>;
    v.push_back(entry("concat_dense", (const void *)concat_dense_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT),
                       scal(4), scal(4), scal(4)},
                      validate_dense, launch_dense));
}

}  // namespace gdag
