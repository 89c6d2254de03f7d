// Training data of the learned surrogate, built on the device: transitions of the plain
// integrator (the 41 network inputs of a state and its RPMs, the 13-d state change over one
// control step) and the standardisation of a set of transitions (the trimming of its tails,
// the mean and standard deviation of the kept set, the out-of-distribution box, and the
// standardised inputs and targets the training GEMMs read).
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "mdg.h"
#include "mdg_internal.cuh"

namespace {

namespace cg = cooperative_groups;

constexpr int kIn = MDG_MLP_IN, kOut = MDG_MLP_OUT, kCols = kIn + kOut;
static_assert(kCols % 6 == 0, "the sample's rounds of six columns");
constexpr int kTile = 1024;  // rows of one block of the finite test and the sampling
constexpr int kSampleMax = 262144;

int fail(int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    mdg::set_last_error(buf);
    return code;
}

int cuda_fail(cudaError_t e, const char* what)
{
    return fail(MDG_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// The 13-d state [p, q, v, w] of drone g from the state planes.
__device__ __forceinline__ void state13(const float4* S, long long n, long long g, float x[13])
{
    const float4 a = S[g], b = S[n + g], c = S[2 * n + g], d = S[3 * n + g];
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    x[8] = c.x; x[9] = c.y; x[10] = c.z; x[11] = c.w;
    x[12] = d.x;
}

// After the step: delta = x_after - x_before, x_before being the first 13 of the drone's 41 inputs.
// A block's rows of 52 bytes leave as one contiguous span.
__global__ void __launch_bounds__(256) transition_delta_kernel(const float4* __restrict__ S, long long n,
                                                               const float* __restrict__ raw, float* __restrict__ delta)
{
    __shared__ float s_delta[256 * kOut];
    const long long g0 = (long long)blockIdx.x * 256, g = g0 + threadIdx.x;
    if (g < n) {
        float x[13];
        state13(S, n, g, x);
#pragma unroll
        for (int k = 0; k < 13; ++k) s_delta[kOut * threadIdx.x + k] = x[k] - raw[kIn * g + k];
    }
    __syncthreads();
    const int m = (int)min(256LL, n - g0) * kOut;
    for (int i = threadIdx.x; i < m; i += 256) delta[kOut * g0 + i] = s_delta[i];
}

// Column c of row i of the transition set: the inputs, then the targets.
__device__ __forceinline__ float column(const float* raw, const float* delta, long long i, int c)
{
    return c < kIn ? raw[i * kIn + c] : delta[i * kOut + (c - kIn)];
}

// Keys that order floats as unsigned integers (finite values; -0 before +0).
__device__ __forceinline__ uint32_t float_key(float v)
{
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__host__ __device__ inline float key_float(uint32_t k)
{
    const uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}

// The standardisation of a transition set reads the set five times, each time as contiguous tiles
// of rows copied into shared memory (or, for the finite test, straight through registers), and
// keeps its decisions as one bit a row: finite; inside the trim box (with the sums of the rows
// that are); those rows' squared deviations from the means; inside the z limits (with their range);
// the training set written out. Bytes of the reads bound it, but for the sums: 216 B a row each,
// and 256 B a row written. Every number that a later kernel needs stays on the device, so the host
// waits once, at the end. 2,000,003 rows: 7.1 ms with a thread per row or per element (32 counting
// passes for the quantiles, FP64 shared-memory atomics for the moments, 15 allocations and 8
// waits), 1.1 ms now: finite 74 us (5.8 TB/s), sample 58, selection 97, box and sums 140, deviations
// 157 (both their arithmetic), z limits 76 (5.7 TB/s), training set 141 (5.9 TB/s, both ways), the
// two scans, means and statistics 35; the rest is the one allocation and its release (150 us) and
// the host's copies. (One pass for sum and square about the middle of the box took 179 us instead of
// the 297 of two, but lost deviations to cancellation and overflow where the box is wide: without a
// limit, margin = inf, one of 0.05 about 1e4 came out 8e-5 of itself off and a column of size 1e25 as constant.)

// Counts of the set: finite rows, rows inside the trim box, rows kept.
struct Counts {
    long long finite, box, kept;
};

struct Stats {
    float box_lo[kCols], box_hi[kCols];  // the trim box of every column
    uint32_t box_min[kCols], box_max[kCols];  // range of the rows inside it, as float keys
    double mean64[kCols];
    float pivot[kCols], scale[kCols];  // the deviations' frame
    float mean[kCols], inv_std[kCols], std_[kCols];
    float limit[kCols];  // the largest |v - mean| that passes: |v - mean| / std <= the column's z limit
    uint32_t key_min[kIn], key_max[kIn];  // range of the kept rows, as float keys
    Counts n;
};

__device__ __forceinline__ bool finite4(float4 v)
{
    // x * 0 is NaN for an infinite or NaN x, else a zero
    return fmaf(v.x, 0.f, v.y * 0.f) + fmaf(v.z, 0.f, v.w * 0.f) == 0.f;
}

// One bit a row: every input and target is finite; and the number of such rows of each tile.
template <bool kVec>
__global__ void __launch_bounds__(256) finite_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                     long long N, uint32_t* __restrict__ bits, int* __restrict__ counts)
{
    __shared__ uint32_t s_bits[kTile / 32];
    const long long r0 = (long long)blockIdx.x * kTile;
    const int rows = (int)min((long long)kTile, N - r0);
    if (threadIdx.x < kTile / 32) {
        const int left = rows - 32 * (int)threadIdx.x;
        s_bits[threadIdx.x] = left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u;
    }
    __syncthreads();
    auto clear = [&](int i, int cols) { atomicAnd(&s_bits[(i / cols) >> 5], ~(1u << ((i / cols) & 31))); };
    auto scan = [&](const float* src, int cols) {
        const int n = rows * cols, n4 = kVec ? n / 4 : 0;
        const float4* v4 = reinterpret_cast<const float4*>(src);
#pragma unroll 4
        for (int i = threadIdx.x; i < n4; i += 256) {
            const float4 v = v4[i];
            if (!finite4(v)) {  // rare
                const float e[4] = {v.x, v.y, v.z, v.w};
                for (int k = 0; k < 4; ++k)
                    if (!isfinite(e[k])) clear(4 * i + k, cols);
            }
        }
        for (int i = 4 * n4 + threadIdx.x; i < n; i += 256)
            if (!isfinite(src[i])) clear(i, cols);
    };
    scan(raw + r0 * kIn, kIn);
    scan(delta + r0 * kOut, kOut);
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t w = s_bits[threadIdx.x];
        bits[(long long)blockIdx.x * (kTile / 32) + threadIdx.x] = w;
        const int c = __reduce_add_sync(0xffffffffu, __popc(w));
        if (threadIdx.x == 0) counts[blockIdx.x] = c;
    }
}

// Exclusive prefix sum of the tiles' counts in place, and their total: one block, 16 consecutive
// counts a thread, so that the 15,626 counts of two million rows take one round.
__global__ void __launch_bounds__(1024) scan_kernel(int* __restrict__ counts, int n, long long* __restrict__ total)
{
    __shared__ int s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long carry = 0;
    for (int base = 0; base < n; base += 16 * 1024) {
        const int i0 = base + 16 * (int)threadIdx.x;
        int v[16], mine = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = i0 + k < n ? counts[i0 + k] : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) mine += v[k];
        int x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            x += lane >= o ? y : 0;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll 8
        for (int w = 0; w < 32; ++w) {
            const int t = s_warp[w];
            before += w < warp ? t : 0;
            all += t;
        }
        int at = (int)carry + before + x - mine;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (i0 + k < n) counts[i0 + k] = at;
            at += v[k];
        }
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// The evenly strided sample of the finite rows for the trim quantiles: finite row number
// s * stride is sample row s.
struct Sampling {
    long long stride, n;
};
__device__ __forceinline__ Sampling sampling(long long n_finite)
{
    Sampling s;
    s.stride = n_finite / kSampleMax > 1 ? n_finite / kSampleMax : 1;
    s.n = (n_finite + s.stride - 1) / s.stride;
    return s;
}

// Copies `cols` columns from c0 of the sampled rows, as float keys, column by column:
// sample[(c - c0) * pitch + s]. Rows are read whole and turned in shared memory (a pitch of 55
// words: no bank conflict either way).
constexpr int kSampleRows = 128;
__global__ void __launch_bounds__(256) sample_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                     const uint32_t* __restrict__ bits, const int* __restrict__ offsets,
                                                     const Stats* __restrict__ st, int c0, int cols,
                                                     uint32_t* __restrict__ sample, long long pitch)
{
    __shared__ int s_row[kTile];  // tile row of each sampled row
    __shared__ uint32_t s_keys[kSampleRows][kCols + 1];
    const uint32_t stride = (uint32_t)sampling(st->n.finite).stride;
    const uint32_t off = (uint32_t)offsets[blockIdx.x];
    const uint32_t first = (off + stride - 1) / stride;  // the tile's first sample row
    const int lane = threadIdx.x & 31;
    // every warp's lanes hold the tile's 32 words, with the rows before each word
    const uint32_t word = bits[(long long)blockIdx.x * (kTile / 32) + lane];
    int before = __popc(word);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, before, o);
        before += lane >= o ? y : 0;
    }
    const int total = __shfl_sync(0xffffffffu, before, 31);
    before -= __popc(word);
    for (int w = threadIdx.x >> 5; w < kTile / 32; w += 8) {
        const uint32_t u = __shfl_sync(0xffffffffu, word, w);
        const uint32_t rank = off + __shfl_sync(0xffffffffu, before, w) + __popc(u & ((1u << lane) - 1u));
        if (((u >> lane) & 1u) && rank % stride == 0) s_row[rank / stride - first] = 32 * w + lane;
    }
    __syncthreads();
    const uint32_t end = off + (uint32_t)total;
    const int n = (int)((end + stride - 1) / stride - first);
    const long long r0 = (long long)blockIdx.x * kTile;
    const int warp = threadIdx.x >> 5;
    for (int k0 = 0; k0 < n; k0 += kSampleRows) {
        const int m = min(n - k0, kSampleRows);
#pragma unroll 4
        for (int k = warp; k < m; k += 8) {
            const long long r = r0 + s_row[k0 + k];
            s_keys[k][lane] = float_key(raw[r * kIn + lane]);
            if (lane < kCols - 32) s_keys[k][32 + lane] = float_key(column(raw, delta, r, 32 + lane));
        }
        __syncthreads();
        for (int c = warp; c < cols; c += 8)
            for (int k = lane; k < m; k += 32) sample[c * pitch + first + k0 + k] = s_keys[k][c0 + c];
        __syncthreads();
    }
}

// The trim box: per column the quantiles trim_frac and 1 - trim_frac of the sample by linear
// interpolation between order statistics, widened by margin times their distance. The four order
// statistics by radix selection on the keys, 11 + 11 + 10 bits: each pass counts the digits of
// the keys that share a statistic's prefix, and the digit that holds its rank extends the prefix.
// A cluster of four blocks takes a column: each counts a quarter of the keys in its own shared
// memory, the first adds the four histograms up over distributed shared memory. Three reads of
// the 62 MB sample, two of them from L2, in place of 32 passes over the rows (1.0 ms): 97 us; one
// block a column took 230 us, clusters of eight 194 us.
constexpr int kSelBlocks = 4, kSelThreads = 512;
__global__ void __cluster_dims__(kSelBlocks, 1, 1) __launch_bounds__(kSelThreads, 2)
    select_kernel(const uint32_t* __restrict__ sample, long long pitch, int c0, float trim_frac, float margin,
                  Stats* __restrict__ st)
{
    __shared__ unsigned s_hist[4][2048];
    __shared__ uint32_t s_prefix[4];
    __shared__ unsigned s_rank[4];
    cg::cluster_group cluster = cg::this_cluster();
    const int c = c0 + blockIdx.x / kSelBlocks, part = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long n = st->n.finite > 0 ? sampling(st->n.finite).n : 0;
    if (part == 0 && threadIdx.x == 0) st->box_min[c] = 0xffffffffu, st->box_max[c] = 0u;
    if (n == 0) {  // no finite row: an empty box (every block of the cluster leaves)
        if (part == 0 && threadIdx.x == 0) st->box_lo[c] = 1.f, st->box_hi[c] = -1.f;
        return;
    }
    const double hq[2] = {(n - 1) * (double)trim_frac, (n - 1) * (1.0 - (double)trim_frac)};
    if (threadIdx.x < 4) {
        const long long k0 = (long long)floor(hq[threadIdx.x >> 1]);
        s_rank[threadIdx.x] = (unsigned)((threadIdx.x & 1) ? min(k0 + 1, n - 1) : k0);
        s_prefix[threadIdx.x] = 0;
    }
    // this block's quarter, in 16-byte pieces; the last block also takes the keys beyond whole pieces
    const uint32_t* key = sample + (c - c0) * pitch;
    const uint4* key4 = reinterpret_cast<const uint4*>(key);
    const int n4 = (int)(n / 4), per = (n4 + kSelBlocks - 1) / kSelBlocks;
    const int i0 = min(n4, part * per), i1 = min(n4, i0 + per);
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0, bits = pass == 2 ? 10 : 11;
        for (int i = threadIdx.x; i < 4 * 2048; i += kSelThreads) (&s_hist[0][0])[i] = 0;
        __syncthreads();
        // statistics that share a prefix share the first one's histogram; the others never match
        uint32_t pre[4];
        int slot[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            pre[j] = s_prefix[j];
            slot[j] = j;
#pragma unroll
            for (int i = 3; i >= 0; --i)
                if (i < j && pre[i] == pre[j]) slot[j] = i;
        }
#pragma unroll
        for (int j = 1; j < 4; ++j)
            if (slot[j] != j) pre[j] = 0xffffffffu;  // prefixes have at most 22 bits
        const uint32_t mask = (1u << bits) - 1u;
        unsigned* hist = &s_hist[0][0];
        auto count = [&](uint32_t k, bool valid) {
            if (pass == 0) {  // one histogram, as four copies: most values share a few exponents
                if (valid) atomicAdd(hist + ((lane & 3) * 2048 + (k >> 21)), 1u);
                return;
            }
            const uint32_t top = k >> (shift + bits);
            int at = top == pre[0] ? 0 : top == pre[1] ? 2048 : top == pre[2] ? 4096 : top == pre[3] ? 6144 : -1;
            at = valid ? at : -1;
            const unsigned hits = __ballot_sync(0xffffffffu, at >= 0);
            if (!hits) return;
            at += (int)((k >> shift) & mask);  // not used where at was -1
            // a column of equal values (padded neighbours) would serialise 32 ways
            const int lead = __shfl_sync(0xffffffffu, at, __ffs(hits) - 1);
            const bool hit = (hits >> lane) & 1u;
            if (__all_sync(0xffffffffu, !hit || at == lead)) {
                if (lane == 0) atomicAdd(hist + lead, (unsigned)__popc(hits));
            } else if (hit) {
                atomicAdd(hist + at, 1u);
            }
        };
        for (int b = i0; b < i1; b += 4 * kSelThreads) {
            uint4 v[4];
            bool ok[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int i = b + m * kSelThreads + (int)threadIdx.x;
                ok[m] = i < i1;
                v[m] = ok[m] ? key4[i] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                count(v[m].x, ok[m]);
                count(v[m].y, ok[m]);
                count(v[m].z, ok[m]);
                count(v[m].w, ok[m]);
            }
        }
        if (part == kSelBlocks - 1 && warp == 0) count(4 * n4 + lane < n ? key[4 * n4 + lane] : 0u, 4 * n4 + lane < n);
        if (pass == 0) {
            __syncthreads();
            for (int i = threadIdx.x; i < 2048; i += kSelThreads)
                s_hist[0][i] += s_hist[1][i] + s_hist[2][i] + s_hist[3][i];
        }
        cluster.sync();
        if (part == 0) {
#pragma unroll
            for (int r = 1; r < kSelBlocks; ++r) {
                const unsigned* far = cluster.map_shared_rank(&s_hist[0][0], r);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (slot[j] == j)
                        for (int i = threadIdx.x; i < 2048; i += kSelThreads) s_hist[j][i] += far[2048 * j + i];
            }
            __syncthreads();
            if (warp < 4) {  // warp j: the digit that holds statistic j's rank
                const int sj = warp == 0 ? slot[0] : warp == 1 ? slot[1] : warp == 2 ? slot[2] : slot[3];
                const unsigned* h = s_hist[sj];
                unsigned mine = 0;
#pragma unroll 16
                for (int b = 0; b < 64; ++b) mine += h[64 * lane + ((b + lane) & 63)];
                unsigned upto = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, upto, o);
                    upto += lane >= o ? y : 0u;
                }
                const unsigned rank = s_rank[warp];
                __syncwarp();
                if (upto > rank && upto - mine <= rank) {  // exactly one lane
                    unsigned before = upto - mine;
                    int b = 64 * lane;
                    while (before + h[b] <= rank) before += h[b++];
                    const uint32_t prefix = (s_prefix[warp] << bits) | (uint32_t)b;
                    s_rank[warp] = rank - before;
                    for (int r = 0; r < kSelBlocks; ++r) *cluster.map_shared_rank(&s_prefix[warp], r) = prefix;
                }
            }
        }
        cluster.sync();  // the prefixes are everywhere; the histograms may be cleared
    }
    if (part == 0 && threadIdx.x == 0) {
        float qv[2];
        for (int q = 0; q < 2; ++q) {
            const float x0 = key_float(s_prefix[2 * q]), x1 = key_float(s_prefix[2 * q + 1]);
            qv[q] = fmaf((float)(hq[q] - floor(hq[q])), x1 - x0, x0);
        }
        const float r = qv[1] - qv[0];
        st->box_lo[c] = fmaf(-margin, r, qv[0]);
        st->box_hi[c] = fmaf(margin, r, qv[1]);
    }
}

// ---- tiles of rows in shared memory ----

constexpr int kSub = 128;  // rows of a shared-memory tile
constexpr int kSubFloats = kSub * kCols;

// Starts the copy of rows [r0, r0 + rows) to `dst`: the inputs [row][41], then, kSub * 41 floats
// on, the targets [row][13]. kVec: the sets are 16-byte aligned, and so is every tile's start.
template <bool kVec>
__device__ __forceinline__ void load_rows(float* dst, const float* raw, const float* delta, long long r0, int rows)
{
    auto part = [&](float* d, const float* src, int n) {
        const uint32_t s = (uint32_t)__cvta_generic_to_shared(d);
        const int n4 = kVec ? n / 4 : 0;
        for (int i = threadIdx.x; i < n4; i += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s + 16u * i), "l"(src + 4 * i));
        for (int i = 4 * n4 + threadIdx.x; i < n; i += blockDim.x)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s + 4u * i), "l"(src + i));
    };
    part(dst, raw + r0 * kIn, rows * kIn);
    part(dst + kSub * kIn, delta + r0 * kOut, rows * kOut);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// The block's tiles in turn, the next one's copy in flight: body(tile, rows, shared tile), called
// by all threads with the tile complete.
template <bool kVec, class Body>
__device__ __forceinline__ void for_tiles(float* smem, const float* raw, const float* delta, long long N, Body body)
{
    const long long tiles = (N + kSub - 1) / kSub;
    auto rows_of = [&](long long t) { return (int)min((long long)kSub, N - t * kSub); };
    long long t = blockIdx.x;
    if (t < tiles) load_rows<kVec>(smem, raw, delta, t * kSub, rows_of(t));
    for (int k = 0; t < tiles; t += gridDim.x, ++k) {
        const long long next = t + gridDim.x;
        if (next < tiles) {
            load_rows<kVec>(smem + ((k + 1) & 1) * kSubFloats, raw, delta, next * kSub, rows_of(next));
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        body(t, rows_of(t), smem + (k & 1) * kSubFloats);
        __syncthreads();  // the tile's buffer is filled again two tiles on
    }
}

__device__ __forceinline__ const float& tile_value(const float* tile, int row, int c)
{
    return c < kIn ? tile[row * kIn + c] : tile[kSub * kIn + row * kOut + (c - kIn)];
}

// The tile's rows that pass test(value, column) in every column and whose bit of `bits` is set,
// as four words in `words` (shared). Two threads a row, half of the columns each; consecutive
// lanes take consecutive rows (41 and 13 are odd: no bank conflict).
template <class Test>
__device__ __forceinline__ void row_words(const float* tile, int rows, const uint32_t* bits, long long t,
                                          uint32_t (*part)[4], uint32_t* words, Test test)
{
    const int row = threadIdx.x & (kSub - 1), half = threadIdx.x / kSub;
    bool ok = row < rows;
    if (ok) {
        if (half == 0) {
#pragma unroll 9
            for (int c = 0; c < kCols / 2; ++c) ok = ok & test(tile[row * kIn + c], c);
        } else {
#pragma unroll 7
            for (int c = kCols / 2; c < kIn; ++c) ok = ok & test(tile[row * kIn + c], c);
#pragma unroll
            for (int c = 0; c < kOut; ++c) ok = ok & test(tile[kSub * kIn + row * kOut + c], kIn + c);
        }
    }
    const uint32_t w = __ballot_sync(0xffffffffu, ok);
    if ((threadIdx.x & 31) == 0) part[half][row >> 5] = w;
    __syncthreads();
    if (threadIdx.x < 4) words[threadIdx.x] = part[0][threadIdx.x] & part[1][threadIdx.x] & bits[t * 4 + threadIdx.x];
    __syncthreads();
}

// The sums of a column are FP64 sums in effect: GB300's FP64 pipe (about 2 operations a clock and SM) took
// 1.2 ms for the two passes over 2,000,003 rows, so each thread adds in three floats a row, two rows an
// instruction in the packed float2 forms, with the rounding error of every addition carried into the
// next word (Knuth's two-sum), and hands them to an FP64 sum every 64 rows. Against exact sums of 2 million
// rows (normal about 0, 2 and 1e4, log-normal, uniform of size 1e-9) the relative error is at most 1.7e-15,
// mostly that of the blocks' FP64 partial sums; all in FP64 it is up to 6.9e-15, with two words instead
// of three 1.2e-14.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void two_sum(float2 a, float2 b, float2& s, float2& e)
{
    s = __fadd2_rn(a, b);
    const float2 bb = sub2(s, a);
    e = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
}
struct ColumnSum {
    static constexpr int kTiles = 4;  // of 32 rows each, between hand-overs
    float2 h = {}, l = {}, g = {};
    double sum = 0.0;
    int tiles = 0;
    __device__ __forceinline__ void low(float2 e)
    {
        float2 e2;
        two_sum(l, e, l, e2);
        g = __fadd2_rn(g, e2);
    }
    __device__ __forceinline__ void add(float2 x)
    {
        float2 e;
        two_sum(h, x, h, e);
        low(e);
    }
    __device__ __forceinline__ void hand_over()
    {
        sum += ((double)h.x + ((double)l.x + (double)g.x)) + ((double)h.y + ((double)l.y + (double)g.y));
        h = l = g = make_float2(0.f, 0.f);
        tiles = 0;
    }
    __device__ __forceinline__ void end_tile()
    {
        if (++tiles == kTiles) hand_over();
    }
};

// The block's sum of every column (four threads each, one for 32 rows of a tile), as its own partial sum:
// partial[block][column].
__device__ __forceinline__ void store_partial(double (*s_sum)[kCols], ColumnSum& s, int group, int c, double* partial)
{
    s.hand_over();
    if (group < 4) s_sum[group][c] = s.sum;
    __syncthreads();
    if (threadIdx.x < kCols)
        partial[(long long)blockIdx.x * kCols + threadIdx.x] = (s_sum[0][threadIdx.x] + s_sum[1][threadIdx.x]) +
                                                               (s_sum[2][threadIdx.x] + s_sum[3][threadIdx.x]);
}

// The blocks' partial sums of column c, added up by a block of 128 threads (one block for all columns
// would take 17 us).
__device__ __forceinline__ double column_total(const double* partial, int blocks, int c)
{
    __shared__ double s_sum[4];
    double s = 0.0;
    for (int b = threadIdx.x; b < blocks; b += 128) s += partial[(long long)b * kCols + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    return (s_sum[0] + s_sum[1]) + (s_sum[2] + s_sum[3]);
}

// Bound of a trim box within which no run of 64 rows overflows; wider columns are added in FP64 as they are.
constexpr float kHuge = 0x1p100f;

// keep1 (finite and inside the trim box in every column) and, over those rows, every column's sum and
// range. Four threads a column and tile; 54 x 4 of the 256 threads add.
template <bool kVec>
__global__ void __launch_bounds__(256) box_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                  long long N, const uint32_t* __restrict__ finite, Stats* __restrict__ st,
                                                  uint32_t* __restrict__ keep, double* __restrict__ partial,
                                                  long long* __restrict__ box_rows)
{
    extern __shared__ __align__(16) float s_tile[];  // [2][kSubFloats], filled 16 bytes at a time
    __shared__ float2 s_box[kCols];
    __shared__ uint32_t s_part[2][4], s_words[4];
    __shared__ double s_sum[4][kCols];
    for (int c = threadIdx.x; c < kCols; c += 256) s_box[c] = make_float2(st->box_lo[c], st->box_hi[c]);
    __syncthreads();
    const int c = threadIdx.x % kCols, group = threadIdx.x / kCols;  // group 4: idle
    const bool wide = !(fmaxf(fabsf(s_box[c].x), fabsf(s_box[c].y)) <= kHuge);
    ColumnSum sum;
    float lo = INFINITY, hi = -INFINITY;
    int kept = 0;
    for_tiles<kVec>(s_tile, raw, delta, N, [&](long long t, int rows, const float* tile) {
        row_words(tile, rows, finite, t, s_part, s_words,
                  [&](float v, int k) { return v >= s_box[k].x && v <= s_box[k].y; });
        if (threadIdx.x < 4) {
            keep[t * 4 + threadIdx.x] = s_words[threadIdx.x];
            kept += __popc(s_words[threadIdx.x]);
        }
        if (group < 4) {
            const uint32_t word = s_words[group];
            const float* src = &tile_value(tile, 32 * group, c);
            const int step = c < kIn ? kIn : kOut;
            auto row = [&](int r, float& v) {
                v = src[r * step];
                const bool in = (word >> r) & 1u;
                lo = in ? fminf(lo, v) : lo;
                hi = in ? fmaxf(hi, v) : hi;
                v = in ? v : 0.f;
            };
            float2 x;
            if (wide) {
                for (int r = 0; r < 32; ++r) row(r, x.x), sum.sum += (double)x.x;
            } else {
#pragma unroll 8
                for (int r = 0; r < 32; r += 2) {
                    row(r, x.x);
                    row(r + 1, x.y);
                    sum.add(x);
                }
            }
            sum.end_tile();
        }
    });
    store_partial(s_sum, sum, group, c, partial);
    if (group < 4 && lo <= hi) {
        atomicMin(&st->box_min[c], float_key(lo));
        atomicMax(&st->box_max[c], float_key(hi));
    }
    if (threadIdx.x < 4 && kept) atomicAdd(reinterpret_cast<unsigned long long*>(box_rows), (unsigned long long)kept);
}

// Mean of every column over the box rows, and the frame of its deviations: the power of two that brings
// the largest to between 1 and 2 (so that no square overflows, and none that counts vanishes) and the
// mean in that scale, as the pivot that rows are taken about.
__global__ void __launch_bounds__(128) mean_kernel(const double* __restrict__ partial, int blocks, Stats* __restrict__ st)
{
    const int c = blockIdx.x;
    const double sum = column_total(partial, blocks, c);
    if (threadIdx.x != 0) return;
    double mean = 0.0;
    float pivot = 0.f, scale = 1.f;
    if (st->n.box > 0) {
        mean = sum / (double)st->n.box;
        const double far = fmax((double)key_float(st->box_max[c]) - mean, mean - (double)key_float(st->box_min[c]));
        // to +-126, so that the power of two is a normal float
        scale = ldexpf(1.f, far > 0.0 ? -min(max(ilogb(far), -126), 126) : 0);
        pivot = (float)mean * scale;
    }
    st->mean64[c] = mean;
    st->pivot[c] = pivot;
    st->scale[c] = scale;
}

// Every column's sum of squared deviations from its pivot over the box rows, in its scale. A deviation is
// a pair of floats exactly; its square goes in as the rounded product and what that leaves out.
template <bool kVec>
__global__ void __launch_bounds__(256) deviation_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                        long long N, const uint32_t* __restrict__ box,
                                                        const Stats* __restrict__ st, double* __restrict__ partial)
{
    extern __shared__ __align__(16) float s_tile[];
    __shared__ double s_sum[4][kCols];
    const int c = threadIdx.x % kCols, group = threadIdx.x / kCols;
    const float2 sc = make_float2(st->scale[c], st->scale[c]);
    const float pivot = st->pivot[c];
    const float2 off = make_float2(-pivot, -pivot);
    ColumnSum sum;
    for_tiles<kVec>(s_tile, raw, delta, N, [&](long long t, int, const float* tile) {
        if (group >= 4) return;
        const uint32_t word = box[t * 4 + group];
        const float* src = &tile_value(tile, 32 * group, c);
        const int step = c < kIn ? kIn : kOut;
#pragma unroll 8
        for (int r = 0; r < 32; r += 2) {
            const float2 v = __fmul2_rn(make_float2(src[r * step], src[(r + 1) * step]), sc);
            // a row that is out counts as the pivot: it adds exact zeros
            const float2 x = make_float2((word >> r) & 1u ? v.x : pivot, (word >> r) & 2u ? v.y : pivot);
            float2 d, e;
            two_sum(x, off, d, e);
            const float2 p = __fmul2_rn(d, d);
            sum.add(p);
            sum.low(__ffma2_rn(__fadd2_rn(d, d), e, __ffma2_rn(d, d, make_float2(-p.x, -p.y))));
        }
        sum.end_tile();
    });
    store_partial(s_sum, sum, group, c, partial);
}

// Unbiased standard deviation of every column over the box rows (a column whose deviation is below
// 1e-6 max(|mean|, 1) is scaled by 1) and the z limits as limits of |v - mean|. The pivot is the mean to
// a float's rounding, 2^-24 of it, so that what the sum has to be corrected by for it is at most 2^-8 of a
// variance that counts.
__global__ void __launch_bounds__(128) stats_kernel(const double* __restrict__ partial, int blocks, float ood_z,
                                                    float target_clip, Stats* __restrict__ st)
{
    const int c = blockIdx.x;
    const double sum = column_total(partial, blocks, c);
    if (threadIdx.x != 0) return;
    if (c < kIn) st->key_min[c] = 0xffffffffu, st->key_max[c] = 0u;
    const double mean = st->mean64[c], n = (double)st->n.box, scale = (double)st->scale[c];
    const double off = mean * scale - (double)st->pivot[c];
    const double sd = n >= 2.0 ? sqrt(fmax(0.0, sum - n * off * off) / (n - 1.0)) / scale : 0.0;
    const float sf = sd > 1e-6 * fmax(fabs(mean), 1.0) ? (float)sd : 1.f;
    const float z = c < kIn ? ood_z : target_clip;
    float a = z * sf;
    for (int k = 0; k < 64 && !(a / sf <= z); ++k) a = nextafterf(a, 0.f);
    for (int k = 0; k < 64 && nextafterf(a, INFINITY) / sf <= z; ++k) a = nextafterf(a, INFINITY);
    st->mean[c] = (float)mean;
    st->std_[c] = sf;
    st->inv_std[c] = 1.f / sf;
    st->limit[c] = a;
}

// keep2: among the box rows, every standardised input within +-ood_z and every standardised
// target within +-target_clip; the number of such rows of each tile, and their inputs' range.
template <bool kVec>
__global__ void __launch_bounds__(256) zbox_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                   long long N, const uint32_t* __restrict__ box, Stats* __restrict__ st,
                                                   uint32_t* __restrict__ keep, int* __restrict__ counts)
{
    extern __shared__ __align__(16) float s_tile[];
    __shared__ float2 s_lim[kCols];
    __shared__ uint32_t s_part[2][4], s_words[4];
    for (int c = threadIdx.x; c < kCols; c += 256) s_lim[c] = make_float2(st->mean[c], st->limit[c]);
    __syncthreads();
    const int c = threadIdx.x % kIn, group = threadIdx.x / kIn;  // groups 4-6: idle
    float lo = INFINITY, hi = -INFINITY;
    for_tiles<kVec>(s_tile, raw, delta, N, [&](long long t, int rows, const float* tile) {
        row_words(tile, rows, box, t, s_part, s_words,
                  [&](float v, int k) { return fabsf(v - s_lim[k].x) <= s_lim[k].y; });
        if (threadIdx.x < 4) keep[t * 4 + threadIdx.x] = s_words[threadIdx.x];
        if (threadIdx.x == 0)
            counts[t] = __popc(s_words[0]) + __popc(s_words[1]) + __popc(s_words[2]) + __popc(s_words[3]);
        if (group < 4) {
            const uint32_t word = s_words[group];
            const float* src = tile + 32 * group * kIn + c;
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
                const float v = src[r * kIn];
                const bool in = (word >> r) & 1u;
                lo = in ? fminf(lo, v) : lo;
                hi = in ? fmaxf(hi, v) : hi;
            }
        }
    });
    if (group < 4 && lo <= hi) {
        atomicMin(&st->key_min[c], float_key(lo));
        atomicMax(&st->key_max[c], float_key(hi));
    }
}

// The training set: kept row j (below the kept number rounded down to 128) is row j of the
// output, inputs standardised to bf16 (zero padded to 64), targets standardised (zero padded to
// 32). Eight threads write a row's eight 16-byte pieces: those of warps 0-3 the inputs, those of
// warps 4-7 the targets, each thread always the same columns, so that their statistics stay in
// registers.
template <bool kVec>
__global__ void __launch_bounds__(256) emit_kernel(const float* __restrict__ raw, const float* __restrict__ delta,
                                                   long long N, const uint32_t* __restrict__ keep,
                                                   const int* __restrict__ offsets, const Stats* __restrict__ st,
                                                   uint4* __restrict__ x, float4* __restrict__ t_out)
{
    extern __shared__ __align__(16) float s_tile[];
    __shared__ uint8_t s_row[kSub];
    const int piece = threadIdx.x & 7, first = (threadIdx.x >> 3) & 15;
    const bool input = threadIdx.x < 128;
    float mean[8], div[8];  // inputs: 1 / std; targets: std
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = input ? 8 * piece + k : kIn + 4 * piece + k;
        const bool used = input ? c < kIn : (k < 4 && c < kCols);
        mean[k] = used ? st->mean[c] : 0.f;
        div[k] = used ? (input ? st->inv_std[c] : st->std_[c]) : 0.f;
    }
    const long long n_out = st->n.kept / 128 * 128;
    for_tiles<kVec>(s_tile, raw, delta, N, [&](long long t, int, const float* tile) {
        const uint32_t w[4] = {keep[4 * t], keep[4 * t + 1], keep[4 * t + 2], keep[4 * t + 3]};
        const int n0 = __popc(w[0]), n1 = n0 + __popc(w[1]), n2 = n1 + __popc(w[2]), n_keep = n2 + __popc(w[3]);
        if (threadIdx.x < kSub) {
            const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
            const uint32_t u = q == 0 ? w[0] : q == 1 ? w[1] : q == 2 ? w[2] : w[3];
            const int before = q == 0 ? 0 : q == 1 ? n0 : q == 2 ? n1 : n2;
            if ((u >> lane) & 1u) s_row[before + __popc(u & ((1u << lane) - 1u))] = (uint8_t)threadIdx.x;
        }
        __syncthreads();
        const long long j0 = offsets[t];
        const int n = (int)min((long long)n_keep, n_out - j0);
        if (input) {
            for (int i = first; i < n; i += 16) {
                const float* src = tile + s_row[i] * kIn + 8 * piece;
                float z[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) z[k] = 8 * piece + k < kIn ? (src[k] - mean[k]) * div[k] : 0.f;
                uint32_t o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __nv_bfloat162 b = __floats2bfloat162_rn(z[2 * k], z[2 * k + 1]);
                    o[k] = *reinterpret_cast<const uint32_t*>(&b);
                }
                x[(j0 + i) * (MDG_MLP_IN_PAD / 8) + piece] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        } else {
            for (int i = first; i < n; i += 16) {
                const float* src = tile + kSub * kIn + s_row[i] * kOut + 4 * piece;
                float z[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) z[k] = 4 * piece + k < kOut ? (src[k] - mean[k]) / div[k] : 0.f;
                t_out[(j0 + i) * (MDG_MLP_OUT_PAD / 4) + piece] = make_float4(z[0], z[1], z[2], z[3]);
            }
        }
    });
}

}  // namespace

extern "C" {

int mdg_transition(mdg_handle h, float* state, const float* rpm, const float* rpm_scale, float* applied, float* raw,
                   float* delta, int32_t n_substeps, void* stream)
{
    if (!h) return fail(MDG_ERR_ARG, "mdg_transition: NULL handle");
    const long long n = mdg_num_drones(h);
    if (n == 0) return MDG_OK;
    if (!state || !rpm || !applied || !raw || !delta) return fail(MDG_ERR_ARG, "mdg_transition: NULL buffer");
    const uintptr_t a16 = reinterpret_cast<uintptr_t>(state) | reinterpret_cast<uintptr_t>(rpm) |
                          reinterpret_cast<uintptr_t>(rpm_scale) | reinterpret_cast<uintptr_t>(applied);
    if (a16 & 15u) return fail(MDG_ERR_ARG, "mdg_transition: state, rpm, rpm_scale and applied must be 16-byte aligned");
    if ((reinterpret_cast<uintptr_t>(raw) | reinterpret_cast<uintptr_t>(delta)) & 3u)
        return fail(MDG_ERR_ARG, "mdg_transition: raw and delta must be 4-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    // the device of the handle current for the launches, as in the calls that make the transition up
    int prev = -1;
    cudaError_t e = cudaGetDevice(&prev);
    if (e == cudaSuccess && prev != h->device) e = cudaSetDevice(h->device);
    if (e == cudaSuccess) e = mdg::transition_features(h, state, rpm, rpm_scale, applied, raw, s);
    int rc = e == cudaSuccess ? mdg_step(h, state, applied, MDG_ACT_RPM, n_substeps, stream)
                              : cuda_fail(e, "mdg_transition");
    if (rc == MDG_OK) {
        transition_delta_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(reinterpret_cast<const float4*>(state), n, raw,
                                                                            delta);
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "mdg_transition");
    }
    if (prev >= 0 && prev != h->device) cudaSetDevice(prev);
    return rc;
}

int mdg_mlp_fit_normalization(mdg_mlp m, const float* raw, const float* delta, int64_t N, float trim_frac, float margin,
                              float ood_z, float target_clip, uint16_t* x_out, float* t_out, int64_t* n_finite,
                              int64_t* n_kept, void* stream)
{
    if (!m || !raw || !delta || !x_out || !t_out) return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: NULL argument");
    if (N <= 0 || N > 0x7fffffffLL) return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: N = %lld", (long long)N);
    if (!(trim_frac >= 0.f && trim_frac < 0.5f) || !(margin >= 0.f) || !(ood_z > 0.f) || !(target_clip > 0.f))
        return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: trim_frac in [0, 0.5), margin >= 0, ood_z and "
                                 "target_clip > 0");
    if ((reinterpret_cast<uintptr_t>(x_out) & 15u) || (reinterpret_cast<uintptr_t>(t_out) & 15u))
        return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: x_out and t_out must be 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    const int tiles = (int)((N + kTile - 1) / kTile);        // tiles of the finite test
    const long long subs = (N + kSub - 1) / kSub;            // shared-memory tiles
    const long long words = (long long)tiles * (kTile / 32);  // bit words, whole tiles
    const long long pitch = (std::min<long long>(N, 2LL * kSampleMax) + 3) / 4 * 4 + 132;  // below 2 kSampleMax rows; no power of two
    int dev = 0, n_sm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int blocks = (int)std::min<long long>(subs, 4LL * n_sm);
    // one allocation, carved up: with the sample of all columns, or of six, or of one at a time where
    // there is no room for it (113 MB of it above half a million rows)
    size_t at_st = 0, at_bits = 0, at_keep = 0, at_counts = 0, at_partial = 0, at_sample = 0;
    uint8_t* ws = nullptr;
    int cols = kCols;
    cudaError_t e;
    for (;;) {
        size_t bytes = 0;
        auto place = [&bytes](size_t n) {
            const size_t at = bytes;
            bytes += (n + 255) / 256 * 256;
            return at;
        };
        at_st = place(sizeof(Stats));
        at_bits = place(words * 4);
        at_keep = place(words * 4);
        at_counts = place((size_t)std::max<long long>(tiles, subs) * 4);
        at_partial = place((size_t)blocks * kCols * 8);
        at_sample = place((size_t)pitch * cols * 4);
#ifdef MDG_DEBUG
        e = cols == kCols ? cudaErrorMemoryAllocation : cudaMalloc(&ws, bytes);  // as if there were no room
#else
        e = cudaMalloc(&ws, bytes);
#endif
        if (e != cudaErrorMemoryAllocation || cols == 1) break;
        cudaGetLastError();
        cols = cols > 6 ? 6 : 1;
    }
    if (e != cudaSuccess) return cuda_fail(e, "mdg_mlp_fit_normalization");
    Stats* d_st = reinterpret_cast<Stats*>(ws + at_st);
    uint32_t *bits = reinterpret_cast<uint32_t*>(ws + at_bits), *keep = reinterpret_cast<uint32_t*>(ws + at_keep);
    int* counts = reinterpret_cast<int*>(ws + at_counts);
    double* partial = reinterpret_cast<double*>(ws + at_partial);
    uint32_t* sample = reinterpret_cast<uint32_t*>(ws + at_sample);
    Stats st{};
    auto run = [&](auto vec) {
        constexpr bool kVec = decltype(vec)::value;
        constexpr int smem = 2 * kSubFloats * (int)sizeof(float);
        cudaError_t r = cudaMemsetAsync(&d_st->n, 0, sizeof(Counts), s);
        for (const void* f : {(const void*)box_kernel<kVec>, (const void*)deviation_kernel<kVec>, (const void*)zbox_kernel<kVec>,
                              (const void*)emit_kernel<kVec>})
            if (r == cudaSuccess) r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r != cudaSuccess) return r;
        finite_kernel<kVec><<<tiles, 256, 0, s>>>(raw, delta, N, bits, counts);
        scan_kernel<<<1, 1024, 0, s>>>(counts, tiles, &d_st->n.finite);
        for (int c = 0; c < kCols; c += cols) {
            sample_kernel<<<tiles, 256, 0, s>>>(raw, delta, bits, counts, d_st, c, cols, sample, pitch);
            select_kernel<<<cols * kSelBlocks, kSelThreads, 0, s>>>(sample, pitch, c, trim_frac, margin, d_st);
        }
        box_kernel<kVec><<<blocks, 256, smem, s>>>(raw, delta, N, bits, d_st, keep, partial, &d_st->n.box);
        mean_kernel<<<kCols, 128, 0, s>>>(partial, blocks, d_st);
        deviation_kernel<kVec><<<blocks, 256, smem, s>>>(raw, delta, N, keep, d_st, partial);
        stats_kernel<<<kCols, 128, 0, s>>>(partial, blocks, ood_z, target_clip, d_st);
        // the z test reads the box rows' words from `keep` and leaves the kept rows' in `bits`
        zbox_kernel<kVec><<<blocks, 256, smem, s>>>(raw, delta, N, keep, d_st, bits, counts);
        scan_kernel<<<1, 1024, 0, s>>>(counts, (int)subs, &d_st->n.kept);
        emit_kernel<kVec><<<blocks, 256, smem, s>>>(raw, delta, N, bits, counts, d_st, reinterpret_cast<uint4*>(x_out),
                                                    reinterpret_cast<float4*>(t_out));
        return cudaGetLastError();
    };
    const bool vec = ((reinterpret_cast<uintptr_t>(raw) | reinterpret_cast<uintptr_t>(delta)) & 15u) == 0;
    e = vec ? run(std::true_type{}) : run(std::false_type{});
    if (e == cudaSuccess) e = cudaMemcpyAsync(&st, d_st, sizeof(Stats), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(ws);
    if (e != cudaSuccess) return cuda_fail(e, "mdg_mlp_fit_normalization");
    const long long n_fin = st.n.finite, n2 = st.n.kept, n_out = n2 / 128 * 128;
    if (n_fin == 0 || st.n.box < 2) return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: too few usable rows");
    if (n2 == 0) return fail(MDG_ERR_ARG, "mdg_mlp_fit_normalization: no row passes the trim");
    // the out-of-distribution box: the kept inputs' range, widened by 10% of it plus 1e-6
    float in_lo[kIn], in_hi[kIn];
    for (int c = 0; c < kIn; ++c) {
        const float a = key_float(st.key_min[c]), b = key_float(st.key_max[c]);
        const float pad = 0.1f * (b - a) + 1e-6f;
        in_lo[c] = a - pad;
        in_hi[c] = b + pad;
    }
    std::vector<float> out_std(kOut), in_std(kIn);
    for (int k = 0; k < kIn; ++k) in_std[k] = st.std_[k];
    for (int k = 0; k < kOut; ++k) out_std[k] = st.std_[kIn + k];
    const int rc = mdg_mlp_set_normalization(m, st.mean, in_std.data(), st.mean + kIn, out_std.data(), in_lo, in_hi);
    if (rc != MDG_OK) return rc;
    if (n_finite) *n_finite = n_fin;
    if (n_kept) *n_kept = n_out;
    return MDG_OK;
}

}  // extern "C"
