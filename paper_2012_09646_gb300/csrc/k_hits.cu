// HITS nodes (Section IV-B, HITS: hubs and authorities by repeated sparse
// matrix-vector products with a matrix and its transpose).
//   spmv_partition  split points of the merge path of a CSR matrix
//   spmv_csr        y = A x for CSR A (the transpose is passed as its own CSR)
//   l2norm          norm[0] = ||x||_2
//   scale           x := x / norm[0]  (unchanged if norm is 0)
//   seg_l2norm      norms[g] = ||x[seg[g] .. seg[g+1])||_2 for G segments
//   seg_scale       x[seg[g] .. seg[g+1]) := ... / norms[g]  (unchanged if 0)
// The seg_ kernels serve a batch of independent graphs stored
// block-diagonally (one CSR whose diagonal blocks are the graphs): the SpMV
// needs nothing new, and the per-graph norms and scaling are one launch each
// for the whole batch instead of one per graph.
//
// spmv_csr balances power-law rows (one row may hold ~1e6 nonzeros) with
// the merge-path decomposition of Merrill and Garland ("Merge-based parallel
// sparse matrix-vector multiplication", SC 2016), restated here: the
// sequence that merges the n row ends with the nnz nonzeros is cut into
// tiles of equal length (kSpmvTile items), so every block does the same work
// whatever the row lengths.  A block stages its tile's products
// val[j] * x[col[j]] in shared memory; then each thread sums a row of the tile
// (a warp a long row), and the part of the last row that goes on in the next
// tile is carried; a second kernel adds the carries to the rows that cross
// tiles.  No atomics and a fixed order: the result is the same on every run.
// Bytes per product: 4 (col) + 4 (val) + 4 (x gather), plus 4 per row for
// rowptr and 4 for y.
#include <climits>
#include <initializer_list>
#include <vector>

#include "catalog.h"
#include "kcommon.cuh"

namespace gdag {

constexpr int kSpmvThreads = 128;
constexpr int kSpmvTile = 1280;  // items: at five nonzeros a row, 1067 products and 213 rows

inline int64_t spmv_tiles(int64_t nrows, int64_t nnz) { return ceil_div(nrows + nnz > 0 ? nrows + nnz : 1, kSpmvTile); }

// part[b] = (rows, nonzeros) consumed before merge-path diagonal b * tile:
// the first i with rowptr[i+1] > d - i - 1, i.e. row end i is not yet
// consumed while nonzero d - i is.
__global__ void spmv_partition_kernel(const int *__restrict__ rowptr, int2 *__restrict__ part, int nrows, int nnz,
                                      int tiles)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > tiles) return;
    const int64_t total = (int64_t)nrows + nnz;
    int64_t d = (int64_t)b * kSpmvTile;
    if (d > total) d = total;
    int64_t lo = d - nnz > 0 ? d - nnz : 0, hi = d < nrows ? d : nrows;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)rowptr[mid + 1] <= d - mid - 1)
            lo = mid + 1;
        else
            hi = mid;
    }
    part[b] = make_int2((int)lo, (int)(d - lo));
}

// One product y = A x: of a launch, or of one of the two that a merged launch does.
struct Spmv {
    const int *rowptr, *col;
    const float *val, *x;
    const int2 *part;
    float *y, *carry;
    int nrows, tiles;
};
struct SpmvPair {
    Spmv m[2];
};

// What bounds it: the gathers.  A plain grid-stride loop over val[j] * x[col[j]]
// alone, no rows and no output, takes 162 us on the benchmark's A (1e7 rows, 5e7
// nonzeros, uniform columns) and 136 us on its transpose, an L1 tag lookup a clock
// and SM; whatever else a block asks of the load-store unit adds to that.  So the
// part after the products is kept short: a thread sums its row from shared memory
// (the row ends are loaded before the products, so they wait with them), with no
// search, no scan and one barrier.  210 us and 183 us (with the carries, launches
// back to back on one vector), from 247 us and 227 us for a form in which each thread
// walked seven items of the merged sequence (a binary search, a dependent chain of
// shared-memory reads and a block-wide segmented scan).  Tiles of 640 to 1536 items
// measured within 2%; 64 threads x 640 the same.  The order of a row's sum is chosen
// for its error: groups of four as a tree, four sums taking the groups in turn, the
// one to three products left added to the smallest of these (Sums4).  Rows of k
// uniform products are then off (root mean square, relative) by 0.89 to 1.01 times
// what chains of seven and a tree give, for every k up to 64; groups added to one sum,
// by 1.3 to 1.7 times from 31, and 218 us and 201 us.  Five iterations of HITS at 1e7
// vertices, mean of 60 graphs: a is off by 6.04e-8 (6.33e-8 in the seven-item form),
// h by 4.54e-8 (4.90e-8).
// col and val are streamed once (evict-first); x is gathered through L1 and L2: in
// the transpose of a power-law graph the high-degree vertices recur (L2-only
// gathers: 471 us).  More loads of a thread in flight before its products (two or
// all), the next columns ahead, or an evict-last policy for x measured slower.
constexpr int kSpmvLong = 64;  // products of a row in a tile beyond which a warp sums it

// Four partial sums that take the terms in turn; z[0] is the next one's.
struct Sums4 {
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    __device__ __forceinline__ void add(float v)
    {
        const float next = z[0] + v;
        z[0] = z[1];
        z[1] = z[2];
        z[2] = z[3];
        z[3] = next;
    }
    __device__ __forceinline__ float total() const { return (z[0] + z[1]) + (z[2] + z[3]); }
};

__global__ void __launch_bounds__(kSpmvThreads) spmv_tile_kernel(const __grid_constant__ SpmvPair pair)
{
    // the kernel that adds the carries may become resident from now on
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ float s_prod[kSpmvTile];
    const bool second = (int)blockIdx.x >= pair.m[0].tiles;
    const Spmv &m = pair.m[second];
    const int b = (int)blockIdx.x - (second ? pair.m[0].tiles : 0);
    const int2 p0 = __ldg(m.part + b), p1 = __ldg(m.part + b + 1);
    const int i0 = p0.x, j0 = p0.y;
    const int tile_rows = p1.x - i0, tile_nnz = p1.y - j0;
    // rows t of the tile; row tile_rows is the one that goes on in the next
    int t = threadIdx.x, lo = 0, hi = 0;
    auto bounds = [&] {
        lo = hi = 0;
        if (t <= tile_rows) {
            lo = __ldg(m.rowptr + i0 + t);
            hi = t < tile_rows ? __ldg(m.rowptr + i0 + t + 1) : p1.y;
        }
    };
    bounds();
    const int *__restrict__ col = m.col + j0;
    const float *__restrict__ val = m.val + j0, *__restrict__ x = m.x;
    for (int q = threadIdx.x; q < tile_nnz; q += kSpmvThreads) s_prod[q] = __ldcs(val + q) * __ldg(x + __ldcs(col + q));
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int t0 = threadIdx.x - lane; t0 <= tile_rows; t0 += kSpmvThreads) {  // the whole warp
        if (t0 >= kSpmvThreads) {
            t = t0 + lane;
            bounds();
        }
        const int a = max(lo - j0, 0), e = min(hi - j0, tile_nnz);
        const bool lng = e - a > kSpmvLong;
        Sums4 z;
        if (!lng) {
            int q = a;
            for (; q + 4 <= e; q += 4) z.add((s_prod[q] + s_prod[q + 1]) + (s_prod[q + 2] + s_prod[q + 3]));
            float rest = 0.f;
            for (; q < e; ++q) rest += s_prod[q];
            z.z[0] += rest;
        }
        float sum = z.total();
        unsigned lm = __ballot_sync(0xffffffffu, lng);
        while (lm) {
            const int src = __ffs(lm) - 1;
            lm &= lm - 1;
            const int ra = __shfl_sync(0xffffffffu, a, src), re = __shfl_sync(0xffffffffu, e, src);
            Sums4 y;
            for (int q = ra + lane; q < re; q += 32) y.add(s_prod[q]);
            float part = y.total();
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            if (lane == src) sum = part;
        }
        if (t < tile_rows) m.y[i0 + t] = sum;
        else if (t == tile_rows) m.carry[b] = sum;
    }
}

// Rows crossing tiles: tile b carries row part[b+1].x into tile b + 1.  The
// first tile carrying a row (its chain head) adds all the chain's carries to
// the value the finishing tile wrote.  How long a chain is follows from where its
// row ends in the merged sequence, so no tile is looked at to find out: one
// thread per tile, a head whose chain has at most kFixShort tiles sums it alone,
// in tile order (almost every chain); of the longer ones, the power-law rows that
// span up to a thousand tiles, a block's warps take one each, and the block
// together those beyond kFixLong.  The order of every sum is fixed.  Launched as
// a programmatic dependent: it waits on the device for the tiles.  4 us on the
// benchmark's A with its rows of up to 5e6 nonzeros, 2 us on the transpose; 17 and
// 4 us when a warp walked each chain, 128 tiles a round trip, to find its end.
constexpr int kFixShort = 4, kFixLong = 512, kFixThreads = 256;

__global__ void __launch_bounds__(kFixThreads) spmv_fixup_kernel(const __grid_constant__ SpmvPair pair, int blocks0)
{
    // heads of longer chains are more than kFixShort tiles apart
    constexpr int kQueue = kFixThreads / kFixShort;
    __shared__ int q_tile[kQueue], q_row[kQueue], q_len[kQueue], q_n;
    __shared__ float red[kFixThreads / 32];
    const bool second = (int)blockIdx.x >= blocks0;
    const Spmv &m = pair.m[second];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = ((int)blockIdx.x - (second ? blocks0 : 0)) * kFixThreads + threadIdx.x;
    int r = -1, len = 0;
    if (threadIdx.x == 0) q_n = 0;
    if (b < m.tiles) {
        r = __ldg(&m.part[b + 1].x);
        const bool head = r < m.nrows && (b == 0 || __ldg(&m.part[b].x) != r);
        // row r's end is item r + rowptr[r + 1] of the merged sequence
        if (head) len = min((int)(((int64_t)r + __ldg(m.rowptr + r + 1)) / kSpmvTile), m.tiles) - b;
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the tiles' sums and carries are visible
    if (len > 0 && len <= kFixShort) {
        float z = 0.f;
#pragma unroll
        for (int k = 0; k < kFixShort; ++k)
            if (k < len) z += m.carry[b + k];
        m.y[r] = z + m.y[r];
    } else if (len > kFixShort) {
        const int i = atomicAdd(&q_n, 1);
        if (i < kQueue) {
            q_tile[i] = b;
            q_row[i] = r;
            q_len[i] = len;
        }
    }
    __syncthreads();
    const int n = min(q_n, kQueue);
    // eight carries a lane in flight
    auto chain = [&](const float *c, int len, int first, int stride) {
        float z = 0.f;
        for (int k = first; k < len; k += 8 * stride)
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int kk = k + u * stride;
                z += kk < len ? c[kk] : 0.f;
            }
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        return z;
    };
    for (int i = warp; i < n; i += kFixThreads / 32) {
        if (q_len[i] > kFixLong) continue;
        const float z = chain(m.carry + q_tile[i], q_len[i], lane, 32);
        if (lane == 0) m.y[q_row[i]] = z + m.y[q_row[i]];
    }
    for (int i = 0; i < n; ++i) {  // uniform over the block
        if (q_len[i] <= kFixLong) continue;
        const float z = chain(m.carry + q_tile[i], q_len[i], threadIdx.x, kFixThreads);
        if (lane == 0) red[warp] = z;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int w = 0; w < kFixThreads / 32; ++w) t += red[w];
            m.y[q_row[i]] = t + m.y[q_row[i]];
        }
        __syncthreads();
    }
}

// norm[0] = sqrt(sum x_i^2), as two kernels on the node's stream.  The first:
// each 128-thread block takes chunks of 2048 float4 (32 KB) and issues all
// sixteen 128-bit loads of a thread at once, so a vector of a few tens of MB
// is requested in about one memory latency (blocks that walked a grid-stride
// loop waited for several rounds); a thread sums its 64 squares as a fixed
// pairwise tree in fp32 (error a few ulp of the chunk's sum, and no
// dependent chain as in compensated summation) and its chunks in fp64; each
// block sums its threads in an fp64 tree and writes its partial.  The
// second, one block, adds the partials in a fixed order and writes the norm.
// It is launched as a programmatic dependent of the first: it becomes
// resident while the first runs and waits (griddepcontrol.wait) for the
// first grid to complete and its writes to be visible, so no block of the
// first takes an arrival atomic and the combine starts as the last partial
// lands.  The grid depends only on n: the same sum on every run.
constexpr int kL2Threads = 128;
constexpr int kL2V = 16;                               // float4 per thread per chunk
constexpr int kL2Chunk4 = kL2Threads * kL2V;           // 2048 float4
constexpr int kL2MaxBlocks = 4096;
constexpr int kL2CombineThreads = 256;
// scratch: the block partials (doubles)
constexpr size_t kL2ScratchBytes = (size_t)kL2MaxBlocks * 8 + 16;

inline unsigned l2norm_grid(int64_t n)
{
    const int64_t chunks = ceil_div(n >> 2, kL2Chunk4);
    return (unsigned)(chunks < 1 ? 1 : (chunks < kL2MaxBlocks ? chunks : kL2MaxBlocks));
}

// One vector of a launch, or of the two that a merged launch does (blocks
// [0, blocks) of the grid the first, the others the second).
struct L2Norm {
    const float *x;
    double *part;
    float *norm;
    int64_t n;
    int blocks;
};
struct L2NormPair {
    L2Norm m[2];
};

__global__ void __launch_bounds__(kL2Threads) l2norm_kernel(const __grid_constant__ L2NormPair pair)
{
    // the combine kernel may start now: it waits for this grid to finish
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool second = (int)blockIdx.x >= pair.m[0].blocks;
    const L2Norm &m = pair.m[second];
    const int block = (int)blockIdx.x - (second ? pair.m[0].blocks : 0), blocks = m.blocks;
    const float *__restrict__ x = m.x;
    const int64_t n = m.n;
    __shared__ double sh[kL2Threads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const int64_t n4 = n >> 2, chunks = (n4 + kL2Chunk4 - 1) / kL2Chunk4;
    double acc = 0.0;
    if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {
        for (int64_t c = block; c < chunks; c += blocks) {
            float4 v[kL2V];
#pragma unroll
            for (int u = 0; u < kL2V; ++u) {
                const int64_t i = c * kL2Chunk4 + threadIdx.x + (int64_t)u * kL2Threads;
                v[u] = i < n4 ? __ldcs(x4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float q[kL2V];
#pragma unroll
            for (int u = 0; u < kL2V; ++u) q[u] = (v[u].x * v[u].x + v[u].y * v[u].y) + (v[u].z * v[u].z + v[u].w * v[u].w);
#pragma unroll
            for (int w = kL2V / 2; w > 0; w >>= 1)
#pragma unroll
                for (int u = 0; u < w; ++u) q[u] += q[u + w];
            acc += (double)q[0];
        }
        if (block == 0 && threadIdx.x < (n & 3)) {
            const float t = x[(n4 << 2) + threadIdx.x];
            acc += (double)(t * t);
        }
    } else {
        for (int64_t i = (int64_t)block * kL2Threads + threadIdx.x; i < n; i += (int64_t)blocks * kL2Threads)
            acc += (double)(x[i] * x[i]);
    }
    acc = warp_sum(acc);
    if (lane == 0) sh[warp] = acc;
    __syncthreads();
    if (warp == 0) {
        double b = lane < kL2Threads / 32 ? sh[lane] : 0.0;
        b = warp_sum(b);
        if (lane == 0) m.part[block] = b;
    }
}

__global__ void __launch_bounds__(kL2CombineThreads) l2norm_combine_kernel(const __grid_constant__ L2NormPair pair)
{
    const L2Norm &m = pair.m[blockIdx.x];
    __shared__ double sh[kL2CombineThreads / 32];
    // the partial-sum grid has completed and its writes are visible
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double t = 0.0;
    for (int b = threadIdx.x; b < m.blocks; b += kL2CombineThreads) t += m.part[b];
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        double q = threadIdx.x < kL2CombineThreads / 32 ? sh[threadIdx.x] : 0.0;
        q = warp_sum(q);
        if (threadIdx.x == 0) m.norm[0] = (float)sqrt(q);
    }
}

size_t l2norm_scratch_bytes() { return kL2ScratchBytes; }

// x := x / norm[0], correctly rounded (div_by); a zero norm leaves x
// unchanged.
struct Scale {
    float *x;
    const float *norm;
    int64_t n;
    int blocks;
};
struct ScalePair {
    Scale m[2];
};

__global__ void __launch_bounds__(kThreads) scale_kernel(const __grid_constant__ ScalePair pair)
{
    const bool second = (int)blockIdx.x >= pair.m[0].blocks;
    const Scale &m = pair.m[second];
    const int block = (int)blockIdx.x - (second ? pair.m[0].blocks : 0), blocks = m.blocks;
    float *__restrict__ x = m.x;
    const int64_t n = m.n;
    const float nr = m.norm[0];
    if (!(nr > 0.f)) return;
    const float rr = (float)(1.0 / (double)nr);
    if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {
        float4 *x4 = reinterpret_cast<float4 *>(x);
        const int64_t n4 = n >> 2, bd = kThreads, tile = bd * kUnroll;
        for (int64_t base = (int64_t)block * tile; base < n4; base += (int64_t)blocks * tile) {
            float4 v[kUnroll];
#pragma unroll
            for (int k = 0; k < kUnroll; ++k) {
                int64_t i = base + threadIdx.x + k * bd;
                if (i < n4) v[k] = x4[i];
            }
#pragma unroll
            for (int k = 0; k < kUnroll; ++k) {
                int64_t i = base + threadIdx.x + k * bd;
                if (i < n4)
                    x4[i] = make_float4(div_by(v[k].x, nr, rr), div_by(v[k].y, nr, rr), div_by(v[k].z, nr, rr),
                                        div_by(v[k].w, nr, rr));
            }
        }
        if (block == 0 && threadIdx.x < (n & 3)) {
            int64_t i = (n4 << 2) + threadIdx.x;
            x[i] = div_by(x[i], nr, rr);
        }
    } else {
        for (int64_t i = (int64_t)block * kThreads + threadIdx.x; i < n; i += (int64_t)blocks * kThreads)
            x[i] = div_by(x[i], nr, rr);
    }
}

size_t seg_norm_scratch_bytes(int64_t G);

// Segments are cut into equal slices, as many as give each at least kSegSlice
// elements, kSegSlices at most; block (slice, g) handles one slice of segment g,
// and the blocks past a segment's slices end at once.  (kSegSlices slices of
// every segment, a few elements a thread where the segments are short, cost a
// block's barriers and arrival for each: 64 segments of 1e4 to 1e5 elements take
// 12 us, from 14 us.)  Segment bounds are clamped to
// [0, n], so a malformed seg array cannot index outside x.
constexpr int kSegSlices = 32, kSegSlice = 4096;

// The slice's elements [lo, hi) and the segment's number of slices; false past it.
__device__ __forceinline__ bool seg_slice(const int *__restrict__ seg, int g, int sl, int n, int &lo, int &hi,
                                          int &slices)
{
    int b = seg[g], e = seg[g + 1];
    b = b < 0 ? 0 : (b > n ? n : b);
    e = e < b ? b : (e > n ? n : e);
    const int64_t len = e - b;
    slices = min(kSegSlices, max(1, (int)((len + kSegSlice - 1) / kSegSlice)));
    lo = b + (int)(len * sl / slices);
    hi = b + (int)(len * (sl + 1) / slices);
    return sl < slices;
}

// norms[g] = sqrt(sum of x_i^2 over segment g): per thread, rounds of eight
// 128-bit loads in flight, each round's 32 squares summed as a fixed fp32
// pairwise tree and the rounds in fp64; fp64 block tree per slice; the last
// slice of a segment to arrive adds the slices' partials in slice order (the
// result does not depend on timing) and resets the segment's arrival
// counter.
constexpr int kSegV = 8;  // float4 in flight per thread

// One batch of a launch, or of the two that a merged launch does (blockIdx.z).
struct SegNorm {
    float *x;
    const int *seg;
    float *norms;
    double *scratch;  // seg_l2norm only
    int G, n;
};
struct SegNormPair {
    SegNorm m[2];
};

__global__ void __launch_bounds__(kThreads) seg_l2norm_kernel(const __grid_constant__ SegNormPair pair)
{
    __shared__ double sh[kThreads / 32];
    __shared__ bool last;
    const SegNorm &m = pair.m[blockIdx.z];
    const float *__restrict__ x = m.x;
    const int *__restrict__ seg = m.seg;
    float *__restrict__ norms = m.norms;
    double *scratch = m.scratch;
    const int G = m.G, n = m.n;
    const int g = blockIdx.y, sl = blockIdx.x;
    if (g >= G) return;
    int lo, hi, slices;
    if (!seg_slice(seg, g, sl, n, lo, hi, slices)) return;
    double acc = 0.0;
    // scalar head up to a 16-byte boundary, float4 body, scalar tail (x
    // itself is 16-byte aligned: checked on the host)
    const int a0 = min(hi, (lo + 3) & ~3), a1 = max(a0, hi & ~3);
    for (int i = lo + threadIdx.x; i < a0; i += kThreads) acc += (double)(x[i] * x[i]);
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    for (int j = (a0 >> 2) + threadIdx.x; j < (a1 >> 2); j += kSegV * kThreads) {
        float4 v[kSegV];
#pragma unroll
        for (int u = 0; u < kSegV; ++u) {
            const int q = j + u * kThreads;
            v[u] = q < (a1 >> 2) ? x4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float qs[kSegV];
#pragma unroll
        for (int u = 0; u < kSegV; ++u) qs[u] = (v[u].x * v[u].x + v[u].y * v[u].y) + (v[u].z * v[u].z + v[u].w * v[u].w);
#pragma unroll
        for (int w = kSegV / 2; w > 0; w >>= 1)
#pragma unroll
            for (int u = 0; u < w; ++u) qs[u] += qs[u + w];
        acc += (double)qs[0];
    }
    for (int i = a1 + threadIdx.x; i < hi; i += kThreads) acc += (double)(x[i] * x[i]);
    const double bs = block_sum(acc, sh);
    double *part = scratch + (size_t)g * kSegSlices;
    unsigned *counter = reinterpret_cast<unsigned *>(scratch + (size_t)G * kSegSlices) + g;
    if (threadIdx.x == 0) part[sl] = bs;
    __threadfence();  // the partial visible device-wide before the arrival
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == (unsigned)(slices - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();  // every slice's partial visible
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < slices; ++k) t += ((volatile double *)part)[k];
        norms[g] = (float)sqrt(t);
        *counter = 0u;
    }
}

// x := x / norms[g] over segment g, correctly rounded (div_by); a zero norm
// leaves the segment unchanged.
__global__ void __launch_bounds__(kThreads) seg_scale_kernel(const __grid_constant__ SegNormPair pair)
{
    const SegNorm &m = pair.m[blockIdx.z];
    float *__restrict__ x = m.x;
    const int *__restrict__ seg = m.seg;
    const int n = m.n;
    const int g = blockIdx.y, sl = blockIdx.x;
    if (g >= m.G) return;
    const float nr = m.norms[g];
    if (!(nr > 0.f)) return;
    const float rr = (float)(1.0 / (double)nr);
    int lo, hi, slices;
    if (!seg_slice(seg, g, sl, n, lo, hi, slices)) return;
    const int a0 = min(hi, (lo + 3) & ~3), a1 = max(a0, hi & ~3);
    for (int i = lo + threadIdx.x; i < a0; i += kThreads) x[i] = div_by(x[i], nr, rr);
    float4 *x4 = reinterpret_cast<float4 *>(x);
    for (int j = (a0 >> 2) + threadIdx.x; j < (a1 >> 2); j += kThreads) {
        const float4 u = x4[j];
        x4[j] = make_float4(div_by(u.x, nr, rr), div_by(u.y, nr, rr), div_by(u.z, nr, rr), div_by(u.w, nr, rr));
    }
    for (int i = a1 + threadIdx.x; i < hi; i += kThreads) x[i] = div_by(x[i], nr, rr);
}

namespace {

const char *validate_partition(const LaunchArgs &a)
{
    const int nrows = a.i32(2), nnz = a.i32(3);
    if (nrows < 0 || nnz < 0) return "nrows and nnz must be >= 0";
    if ((int64_t)nrows + nnz > INT_MAX - kSpmvTile) return "nrows + nnz too large for int32 indexing";
    if (a.bytes[0] / 4 < (size_t)nrows + 1) return "rowptr smaller than nrows + 1 int32";
    if (a.bytes[1] < (size_t)(spmv_tiles(nrows, nnz) + 1) * 8) return "part smaller than gdag_scratch_bytes()";
    return nullptr;
}

int launch_partition(const LaunchArgs &a, void *s)
{
    const int nrows = a.i32(2), nnz = a.i32(3);
    const int tiles = (int)spmv_tiles(nrows, nnz);
    spmv_partition_kernel<<<(unsigned)ceil_div(tiles + 1, 256), 256, 0, (cudaStream_t)s>>>(
        a.p<int>(0), a.p<int2>(1), nrows, nnz, tiles);
    return cudaGetLastError();
}

const char *validate_spmv(const LaunchArgs &a)
{
    const int nrows = a.i32(7), nnz = a.i32(8);
    if (nrows < 0 || nnz < 0) return "nrows and nnz must be >= 0";
    if ((int64_t)nrows + nnz > INT_MAX - kSpmvTile) return "nrows + nnz too large for int32 indexing";
    const int64_t tiles = spmv_tiles(nrows, nnz);
    if (a.bytes[0] / 4 < (size_t)nrows + 1) return "rowptr smaller than nrows + 1 int32";
    if (a.bytes[1] / 4 < (size_t)nnz || a.bytes[2] / 4 < (size_t)nnz) return "col or val smaller than nnz";
    if (a.bytes[4] < (size_t)(tiles + 1) * 8) return "part smaller than gdag_scratch_bytes(\"spmv_partition\")";
    if (a.bytes[5] / 4 < (size_t)nrows) return "y smaller than nrows floats";
    if (a.bytes[3] / 4 < (size_t)nrows) return "x smaller than nrows floats (square matrices)";
    if (a.bytes[6] < (size_t)tiles * 4) return "carry smaller than gdag_scratch_bytes(\"spmv_csr\")";
    return nullptr;
}

Spmv spmv_of(const LaunchArgs &a)
{
    const int nrows = a.i32(7), nnz = a.i32(8);
    return Spmv{a.p<int>(0), a.p<int>(1), a.p<float>(2), a.p<float>(3), a.p<int2>(4), a.p<float>(5), a.p<float>(6),
                nrows, nrows > 0 ? (int)spmv_tiles(nrows, nnz) : 0};
}

// One or two products in one launch each of the two kernels.
int launch_spmv_run(const LaunchArgs *const *m, int count, void *sv)
{
    cudaStream_t s = (cudaStream_t)sv;
    SpmvPair pair = {};
    int64_t tiles = 0, fix[2] = {0, 0};
    for (int i = 0; i < count; ++i) {
        pair.m[i] = spmv_of(*m[i]);
        tiles += pair.m[i].tiles;
        fix[i] = ceil_div(pair.m[i].tiles, kFixThreads);
    }
    if (tiles == 0) return cudaSuccess;
    spmv_tile_kernel<<<(unsigned)tiles, kSpmvThreads, 0, s>>>(pair);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_dependent(spmv_fixup_kernel, dim3((unsigned)(fix[0] + fix[1])), kFixThreads, s, pair, (int)fix[0]);
}

int launch_spmv(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_spmv_run(m, 1, s);
}

const char *validate_l2norm(const LaunchArgs &a)
{
    const int64_t n = a.i64(3);
    if (n < 0) return "n < 0";
    if (a.bytes[0] / 4 < (size_t)n) return "x smaller than n floats";
    if (a.bytes[1] < 4) return "norm smaller than one float";
    if (a.bytes[2] < kL2ScratchBytes) return "scratch smaller than gdag_scratch_bytes()";
    return nullptr;
}

// Each launcher below takes one launch, or two that a merged launch does.
int launch_l2norm_run(const LaunchArgs *const *m, int count, void *s)
{
    L2NormPair pair = {};
    int blocks = 0;
    for (int i = 0; i < count; ++i) {
        const int64_t n = m[i]->i64(3);
        pair.m[i] = L2Norm{m[i]->p<float>(0), m[i]->p<double>(2), m[i]->p<float>(1), n, (int)l2norm_grid(n)};
        blocks += pair.m[i].blocks;
    }
    l2norm_kernel<<<(unsigned)blocks, kL2Threads, 0, (cudaStream_t)s>>>(pair);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the combine as a programmatic dependent of the partial sums
    return launch_dependent(l2norm_combine_kernel, dim3((unsigned)count), kL2CombineThreads, (cudaStream_t)s, pair);
}

int launch_l2norm(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_l2norm_run(m, 1, s);
}

const char *validate_scale(const LaunchArgs &a)
{
    const int64_t n = a.i64(2);
    if (n < 0) return "n < 0";
    if (a.bytes[0] / 4 < (size_t)n) return "x smaller than n floats";
    if (a.bytes[1] < 4) return "norm smaller than one float";
    return nullptr;
}

int launch_scale_run(const LaunchArgs *const *m, int count, void *s)
{
    ScalePair pair = {};
    int blocks = 0;
    for (int i = 0; i < count; ++i) {
        const int64_t n = m[i]->i64(2);
        pair.m[i] = Scale{m[i]->p<float>(0), m[i]->p<float>(1), n, n > 0 ? (int)stream_grid(n >> 2) : 0};
        blocks += pair.m[i].blocks;
    }
    if (blocks == 0) return cudaSuccess;
    scale_kernel<<<(unsigned)blocks, kThreads, 0, (cudaStream_t)s>>>(pair);
    return cudaGetLastError();
}

int launch_scale(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_scale_run(m, 1, s);
}

const char *validate_seg_common(const LaunchArgs &a, int gi, int ni)
{
    const int G = a.i32(gi), n = a.i32(ni);
    if (G < 0 || n < 0) return "G and n must be >= 0";
    if (G > 65535) return "at most 65535 segments";
    if (a.bytes[0] / 4 < (size_t)n) return "x smaller than n floats";
    if (a.bytes[1] / 4 < (size_t)G + 1) return "seg smaller than G + 1 int32";
    if (a.bytes[2] / 4 < (size_t)G) return "norms smaller than G floats";
    if ((reinterpret_cast<uintptr_t>(a.ptr[0]) & 15) != 0) return "x must be 16-byte aligned";
    return nullptr;
}

const char *validate_seg_l2norm(const LaunchArgs &a)
{
    if (const char *m = validate_seg_common(a, 4, 5)) return m;
    if (a.bytes[3] < seg_norm_scratch_bytes(a.i32(4))) return "scratch smaller than gdag_scratch_bytes(\"seg_l2norm\", G)";
    return nullptr;
}

template <bool NORM> int launch_seg_run(const LaunchArgs *const *m, int count, void *s)
{
    SegNormPair pair = {};
    int G = 0;
    for (int i = 0; i < count; ++i) {
        const LaunchArgs &a = *m[i];
        pair.m[i] = SegNorm{a.p<float>(0), a.p<int>(1), a.p<float>(2), NORM ? a.p<double>(3) : nullptr,
                            a.i32(NORM ? 4 : 3), a.i32(NORM ? 5 : 4)};
        if (pair.m[i].G > G) G = pair.m[i].G;
    }
    if (G == 0) return cudaSuccess;
    const dim3 grid(kSegSlices, (unsigned)G, (unsigned)count);
    if (NORM) seg_l2norm_kernel<<<grid, kThreads, 0, (cudaStream_t)s>>>(pair);
    else seg_scale_kernel<<<grid, kThreads, 0, (cudaStream_t)s>>>(pair);
    return cudaGetLastError();
}

int launch_seg_l2norm(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_seg_run<true>(m, 1, s);
}

const char *validate_seg_scale(const LaunchArgs &a) { return validate_seg_common(a, 3, 4); }

int launch_seg_scale(const LaunchArgs &a, void *s)
{
    const LaunchArgs *m[1] = {&a};
    return launch_seg_run<false>(m, 1, s);
}

// Two independent launches of one kernel as one, the two branches of a HITS
// iteration, while the launches are what bounds it: up to 2^22 rows and nonzeros
// for the products, 2^20 elements for the vectors.  Five iterations, merged and not,
// of one program and of three in turn: 20000 vertices 113 and 70 us against 171 and
// 174; 156250 139 and 73 against 192 and 198; 600000 228 and 140 against 215 and 185.
// On larger graphs the two branches on two streams are the quicker form where one
// program has the device (700000: 222 us against 247, 1e6: 280 against 306, 1e7: 2045
// against 2118): a branch's norm and scaling run beside the other's product.
// A pair waits for short host writes of either: the first products of a program
// whose vectors the host writes would otherwise part its branches to the end (with
// the writes and the reads, merged and parted: 20000 vertices 163 and 180 us, 156250 238
// and 248; 300000, 1.2 MB each, 281 and 285).  The vector kernels wait for one
// another's products too, while these are short (64 MB of arrays, 20 to 25 us):
// above the products' line they still halve their launches, which bound three programs in
// turn (800000 vertices, waiting and not: one program 256 and 247 us, three 185 and 217).
constexpr uint32_t kWaitsFor = 1u << 20, kWaitsForKernels = 64u << 20;
template <MergeLaunchFn LAUNCH> bool merge_two(Run &run, Merge &out)
{
    const RunLaunch &f = *run.at(0);
    auto small = [](const RunLaunch &l) {
        if (is(l.k, "spmv_csr")) return (int64_t)l.a.i32(7) + l.a.i32(8) <= (1 << 22);
        return (is(l.k, "l2norm")  ? l.a.i64(3)
                : is(l.k, "scale") ? l.a.i64(2)
                                   : (int64_t)l.a.i32(is(l.k, "seg_l2norm") ? 5 : 4)) <= (1 << 20);
    };
    if (!small(f)) return false;
    for (int j = 1; run.kernel(j); ++j) {
        if (run.kernel(j) != f.k) continue;
        if (!run.at(j)) return false;
        const RunLaunch &g = *run.at(j);
        if (!small(g)) return false;
        // what either writes, the other does not touch
        bool apart = true;
        for (int p = 0; p < f.a.nargs; ++p)
            for (int q = 0; q < g.a.nargs; ++q)
                if (f.array[p] >= 0 && f.array[p] == g.array[q])
                    apart = apart && f.k->spec[p].mode == GDAG_MODE_IN && g.k->spec[q].mode == GDAG_MODE_IN;
        if (!apart) return false;
        out.count = out.apart = 2;
        out.waits_for = kWaitsFor;
        out.waits_for_kernels = is(f.k, "spmv_csr") ? 0 : kWaitsForKernels;
        out.member[0] = 0;
        out.member[1] = j;
        out.launch = LAUNCH;
        return true;
    }
    return false;
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

size_t seg_norm_scratch_bytes(int64_t G) { return (size_t)(G > 0 ? G : 0) * (kSegSlices * 8 + 4) + 16; }
size_t spmv_part_bytes(int64_t rows_plus_nnz) { return (size_t)(ceil_div(rows_plus_nnz > 0 ? rows_plus_nnz : 1, kSpmvTile) + 1) * 8; }
size_t spmv_carry_bytes(int64_t rows_plus_nnz) { return (size_t)ceil_div(rows_plus_nnz > 0 ? rows_plus_nnz : 1, kSpmvTile) * 4 + 16; }

void append_hits_kernels(std::vector<KernelEntry> &v)
{
    v.push_back(entry("spmv_partition", (const void *)spmv_partition_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT), scal(4), scal(4)}, validate_partition,
                      launch_partition));
    v.push_back(entry("spmv_csr", (const void *)spmv_tile_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN),
                       arr(GDAG_MODE_OUT), arr(GDAG_MODE_INOUT), scal(4), scal(4)},
                      validate_spmv, launch_spmv));
    v.back().merge = merge_two<launch_spmv_run>;
    v.push_back(entry("l2norm", (const void *)l2norm_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT), arr(GDAG_MODE_INOUT), scal(8)}, validate_l2norm,
                      launch_l2norm));
    v.back().merge = merge_two<launch_l2norm_run>;
    v.push_back(entry("scale", (const void *)scale_kernel, {arr(GDAG_MODE_INOUT), arr(GDAG_MODE_IN), scal(8)},
                      validate_scale, launch_scale));
    v.back().merge = merge_two<launch_scale_run>;
    v.push_back(entry("seg_l2norm", (const void *)seg_l2norm_kernel,
                      {arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), arr(GDAG_MODE_OUT), arr(GDAG_MODE_INOUT), scal(4), scal(4)},
                      validate_seg_l2norm, launch_seg_l2norm));
    v.back().merge = merge_two<launch_seg_run<true>>;
    v.push_back(entry("seg_scale", (const void *)seg_scale_kernel,
                      {arr(GDAG_MODE_INOUT), arr(GDAG_MODE_IN), arr(GDAG_MODE_IN), scal(4), scal(4)}, validate_seg_scale,
                      launch_seg_scale));
    v.back().merge = merge_two<launch_seg_run<false>>;
}

}  // namespace gdag
