// Device primitives: exclusive prefix sums and a stable LSD radix sort.
#include "internal.cuh"

namespace mce {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

// Block-wide exclusive scan of one value per thread; returns the block total.
template <class T>
__device__ T block_exclusive_scan(T x, T *warp_sums, T &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T ws = lane < (kScanThreads / 32) ? warp_sums[lane] : T(0);
        T wi = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < (kScanThreads / 32)) warp_sums[lane] = wi - ws;
        if (lane == (kScanThreads / 32) - 1) warp_sums[kScanThreads / 32] = wi;
    }
    __syncthreads();
    T r = warp_sums[warp] + incl - x;
    total = warp_sums[kScanThreads / 32];
    __syncthreads();
    return r;
}

template <class T>
__global__ void k_scan_reduce(const T *in, int64_t n, T *block_sums) {
    __shared__ T ws[kScanThreads / 32 + 1];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i)
        if (base + i < n) s += in[base + i];
    T total;
    block_exclusive_scan<T>(s, ws, total);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

template <class T>
__global__ void k_scan_apply(const T *in, T *out, int64_t n, const T *block_offsets) {
    __shared__ T ws[kScanThreads / 32 + 1];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = (base + i < n) ? in[base + i] : T(0);
        s += v[i];
    }
    T total;
    T run = block_exclusive_scan<T>(s, ws, total) + (block_offsets ? block_offsets[blockIdx.x] : T(0));
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        if (base + i < n) out[base + i] = run;
        run += v[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = run;
}

// Scans of up to this many items run in one launch of one block: three
// launches of the tiled scan cost more than the one block takes.
constexpr int64_t kScanOne = 16384;
constexpr int kScanOneThreads = 1024;

template <class T>
__global__ void __launch_bounds__(kScanOneThreads) k_scan_one(const T *in, T *out, int32_t n) {
    __shared__ T ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (n + kScanOneThreads - 1) / kScanOneThreads;
    const int i0 = threadIdx.x * per, i1 = i0 + per < n ? i0 + per : n;
    T s = 0;
    for (int i = i0; i < i1; ++i) s += in[i];
    T incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    const T w = ws[lane];
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += y;
    }
    T run = __shfl_sync(0xffffffffu, wi - w, warp) + incl - s;
    const T total = __shfl_sync(0xffffffffu, wi, 31);
    for (int i = i0; i < i1; ++i) {
        const T x = in[i];
        out[i] = run;
        run += x;
    }
    if (threadIdx.x == 0) out[n] = total;
}

template <class T>
mce_status exclusive_scan(const T *in, T *out, int64_t n, cudaStream_t s) {
    if (n <= 0) {
        return cuda_status(cudaMemsetAsync(out, 0, sizeof(T), s), "scan memset");
    }
    if (n <= kScanOne) {
        MCE_LAUNCH(k_scan_one<T>, 1, kScanOneThreads, 0, s, in, out, (int32_t)n);
        return MCE_OK;
    }
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    DevBuf sums;
    MCE_TRY(sums.alloc((size_t)(tiles + 1) * sizeof(T), s));
    MCE_LAUNCH(k_scan_reduce<T>, (unsigned)tiles, kScanThreads, 0, s, in, n, sums.as<T>());
    MCE_TRY(exclusive_scan<T>(sums.as<T>(), sums.as<T>(), tiles, s));
    MCE_LAUNCH(k_scan_apply<T>, (unsigned)tiles, kScanThreads, 0, s, in, out, n, (const T *)sums.as<T>());
    return MCE_OK;
}

// ------------------------------------------------------------------ radix sort

constexpr int kRadix = 256;

// Rank of this lane's key among the keys of its digit that its warp has seen
// (earlier rounds, then earlier lanes of this round); digit = kRadix for a
// lane without a key.  wcnt: the warp's digit counters.
__device__ __forceinline__ int radix_rank(int32_t *wcnt, uint32_t digit) {
    // lanes with the same digit, bit by bit: nine ballots.  One match_any runs
    // digit by digit on GB300: with it the five scatter passes of an R-MAT 18
    // ingest took 357 us, with the ballots 217 us
    uint32_t peers = __ballot_sync(0xffffffffu, digit < kRadix);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (digit >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, set);
        peers &= set ? m : ~m;
    }
    const int before = __popc(peers & lanemask_lt());
    const int seen = digit < kRadix ? wcnt[digit] : 0;
    __syncwarp();
    if (before == 0 && digit < kRadix) wcnt[digit] = seen + __popc(peers);
    __syncwarp();
    return seen + before;
}

// Exclusive scan over the first 256 threads of a block (one value a digit).
__device__ __forceinline__ int32_t digit_scan(int32_t x, int32_t *ws) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (warp < kRadix / 32 && lane == 31) ws[warp] = incl;
    __syncthreads();
    int32_t r = incl - x;
    for (int w = 0; w < warp && w < kRadix / 32; ++w) r += ws[w];
    __syncthreads();
    return r;
}

// All passes of a small sort in one block, the keys in registers and, between
// passes, in shared memory.  Three launches a pass cost more than the work
// below a few thousand keys.
constexpr int kOneThreads = 1024;
constexpr int kOneItems = 8;
constexpr int64_t kOneKeys = kOneThreads * kOneItems;
constexpr int kOneWarps = kOneThreads / 32;
constexpr size_t kOneSmem = kOneKeys * 8 + (size_t)kOneWarps * kRadix * 4 + kRadix * 4 + 64;

__global__ void __launch_bounds__(kOneThreads) k_radix_one(uint64_t *keys, int32_t n, int lo, int hi, int width) {
    extern __shared__ __align__(16) unsigned char smem_one[];
    uint64_t *sk = reinterpret_cast<uint64_t *>(smem_one);
    int32_t *cnt = reinterpret_cast<int32_t *>(sk + kOneKeys);   // [warp][digit]
    int32_t *start = cnt + kOneWarps * kRadix;
    int32_t *ws = start + kRadix;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rounds = (n + kOneThreads - 1) / kOneThreads;   // a warp holds 32 * rounds consecutive keys
    uint64_t key[kOneItems];
    int rank[kOneItems];
    const int w0 = warp * 32 * rounds;
#pragma unroll
    for (int r = 0; r < kOneItems; ++r) {
        const int i = w0 + r * 32 + lane;
        key[r] = r < rounds && i < n ? keys[i] : 0ULL;
    }
    for (int shift = lo; shift < hi; shift += width) {
        const uint32_t mask = (1u << (hi - shift < width ? hi - shift : width)) - 1u;
        for (int i = t; i < kOneWarps * kRadix; i += kOneThreads) cnt[i] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOneItems; ++r)
            if (r < rounds) {
                const bool valid = w0 + r * 32 + lane < n;
                rank[r] = radix_rank(cnt + warp * kRadix, valid ? (uint32_t)(key[r] >> shift) & mask : kRadix);
            }
        __syncthreads();
        int32_t run = 0;
        if (t < kRadix)
            for (int w = 0; w < kOneWarps; ++w) {
                const int32_t c = cnt[w * kRadix + t];
                cnt[w * kRadix + t] = run;
                run += c;
            }
        const int32_t base = digit_scan(run, ws);
        if (t < kRadix) start[t] = base;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOneItems; ++r)
            if (r < rounds && w0 + r * 32 + lane < n) {
                const uint32_t d = (uint32_t)(key[r] >> shift) & mask;
                sk[start[d] + cnt[warp * kRadix + d] + rank[r]] = key[r];
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kOneItems; ++r) {
            const int i = w0 + r * 32 + lane;
            if (r < rounds && i < n) key[r] = sk[i];
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < kOneItems; ++r) {
        const int i = w0 + r * 32 + lane;
        if (r < rounds && i < n) keys[i] = key[r];
    }
}

// Larger sorts: per pass the digit counts of every tile, their scan along each
// digit's row, and a stable scatter.  Bound: the scatter by shared memory (75 %
// of its throughput) and instructions (68 %), the counts by the latency of their
// loads (37 % of HBM; 24 B a key and pass in all).
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;

// counts[d * tiles + t] = keys of tile t whose digit is d
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint64_t *__restrict__ keys, int64_t n, int shift,
                                                             uint32_t mask, int32_t *counts, int32_t tiles) {
    __shared__ int32_t h[kSortWarps][kRadix];   // per warp: a frequent digit would serialise one counter
    const int t = threadIdx.x;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) h[w][t] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (kSortThreads * ITEMS);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t i = base + (int64_t)r * kSortThreads + t;
        if (i < n) atomicAdd(&h[t >> 5][(uint32_t)(keys[i] >> shift) & mask], 1);
    }
    __syncthreads();
    int32_t s = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) s += h[w][t];
    counts[(int64_t)t * tiles + blockIdx.x] = s;
}

// row d of the counts: exclusive scan over the tiles in place, total[d] = its sum
__global__ void __launch_bounds__(kSortThreads) k_radix_rows(int32_t *counts, int32_t tiles, int32_t *total) {
    __shared__ int32_t ws[kRadix / 32];
    __shared__ int32_t last;
    int32_t *row = counts + (int64_t)blockIdx.x * tiles;
    int32_t carry = 0;
    for (int32_t i0 = 0; i0 < tiles; i0 += kSortThreads) {
        const int32_t i = i0 + threadIdx.x;
        const int32_t x = i < tiles ? row[i] : 0;
        const int32_t r = digit_scan(x, ws);
        if (i < tiles) row[i] = carry + r;
        if (threadIdx.x == kSortThreads - 1) last = r + x;
        __syncthreads();
        carry += last;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Stable scatter: a warp ranks its consecutive keys, the block adds the
// counters of the warps before it, and the tile is put in digit order in
// shared memory first, so that a digit's keys leave as one run.
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(const uint64_t *__restrict__ in,
                                                                uint64_t *__restrict__ out, int64_t n, int shift,
                                                                uint32_t mask, const int32_t *__restrict__ rows,
                                                                int32_t tiles, const int32_t *__restrict__ total) {
    constexpr int TILE = kSortThreads * ITEMS;
    __shared__ uint64_t sk[TILE];
    __shared__ int32_t cnt[kSortWarps][kRadix];
    __shared__ int32_t start[kRadix], dst[kRadix], ws[kRadix / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    const int have = (int)(n - base < TILE ? n - base : TILE);
    uint64_t key[ITEMS];
    int rank[ITEMS];
    const int w0 = warp * 32 * ITEMS;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int i = w0 + r * 32 + lane;
        key[r] = i < have ? in[base + i] : 0ULL;
    }
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) cnt[w][t] = 0;
    const int32_t digit0 = digit_scan(total[t], ws);   // keys with a smaller digit
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        rank[r] = radix_rank(cnt[warp], w0 + r * 32 + lane < have ? (uint32_t)(key[r] >> shift) & mask : kRadix);
    __syncthreads();
    int32_t run = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const int32_t c = cnt[w][t];
        cnt[w][t] = run;
        run += c;
    }
    const int32_t s0 = digit_scan(run, ws);
    start[t] = s0;
    dst[t] = digit0 + rows[(int64_t)t * tiles + blockIdx.x] - s0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (w0 + r * 32 + lane < have) {
            const uint32_t d = (uint32_t)(key[r] >> shift) & mask;
            sk[start[d] + cnt[warp][d] + rank[r]] = key[r];
        }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int j = r * kSortThreads + t;
        if (j < have) {
            const uint64_t k = sk[j];
            out[dst[(uint32_t)(k >> shift) & mask] + j] = k;
        }
    }
}

template <int ITEMS>
mce_status radix_passes(uint64_t *keys, uint64_t *tmp, int64_t n, int lo, int hi, int width, cudaStream_t s) {
    constexpr int TILE = kSortThreads * ITEMS;
    const int32_t tiles = (int32_t)((n + TILE - 1) / TILE);
    DevBuf counts;
    MCE_TRY(counts.alloc(((size_t)kRadix * tiles + kRadix) * sizeof(int32_t), s));
    int32_t *rows = counts.as<int32_t>(), *total = rows + (size_t)kRadix * tiles;
    uint64_t *src = keys, *dst = tmp;
    for (int shift = lo; shift < hi; shift += width) {
        const uint32_t mask = (1u << (hi - shift < width ? hi - shift : width)) - 1u;
        MCE_LAUNCH(k_radix_hist<ITEMS>, tiles, kSortThreads, 0, s, src, n, shift, mask, rows, tiles);
        MCE_LAUNCH(k_radix_rows, kRadix, kSortThreads, 0, s, rows, tiles, total);
        MCE_LAUNCH(k_radix_scatter<ITEMS>, tiles, kSortThreads, 0, s, src, dst, n, shift, mask, rows, tiles, total);
        uint64_t *t = src;
        src = dst;
        dst = t;
    }
    if (src != keys) MCE_CUDA(cudaMemcpyAsync(keys, src, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    return MCE_OK;
}

}  // namespace

mce_status exclusive_scan_i32(const int32_t *in, int32_t *out, int64_t n, cudaStream_t s) {
    return exclusive_scan<int32_t>(in, out, n, s);
}

mce_status exclusive_scan_i64(const int64_t *in, int64_t *out, int64_t n, cudaStream_t s) {
    return exclusive_scan<int64_t>(in, out, n, s);
}

mce_status radix_sort_u64(uint64_t *keys, uint64_t *tmp, int64_t n, int32_t lo, int32_t hi, cudaStream_t s) {
    if (n <= 1 || hi <= lo) return MCE_OK;
    if (n >= (int64_t)1 << 31) {
        g_last_error = "radix_sort_u64: too many keys";
        return MCE_EINVAL;
    }
    const int passes = (hi - lo + 7) / 8;
    const int width = (hi - lo + passes - 1) / passes;   // equal digits: shorter rows of counters
    if (n <= kOneKeys) {
        MCE_CUDA(cudaFuncSetAttribute(k_radix_one, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOneSmem));
        MCE_LAUNCH(k_radix_one, 1, kOneThreads, kOneSmem, s, keys, (int32_t)n, lo, hi, width);
        return MCE_OK;
    }
    // tiles of 4,096 keys once they fill the GPU, else of 1,024
    if (n >= (int64_t)num_sms() * kSortThreads * 16) return radix_passes<16>(keys, tmp, n, lo, hi, width, s);
    return radix_passes<4>(keys, tmp, n, lo, hi, width, s);
}

}  // namespace mce
