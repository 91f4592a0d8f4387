#include <string>
// Graph ingest and vertex ranking kernels.
//
//   build_csr       simple undirected graph from raw pairs (Section 3; inputs
//                   normalised as in Section 6.1): drop self loops, symmetrise,
//                   radix sort, deduplicate, row offsets by scan.
//   vertex_key      Section 4.2 keys: degree, core number ("degeneracy" of a
//                   vertex: in the k-core but not the (k+1)-core) by rounds of
//                   the h-index step, triangle count by oriented intersection.
//   rank_from_key   rank(v) = position of (key(v), id(v)) in ascending order.
//   build_up_lists  Γ+(v) = neighbours of higher rank (the cand set of v's
//                   subproblem in Algorithm 5), sorted by id.
#include <cooperative_groups.h>

#include <mutex>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace mce {

namespace {

// ------------------------------------------------------------------ CSR build

__global__ void k_make_keys(const int32_t *u, const int32_t *v, int64_t m, int32_t n, int32_t B, uint64_t *keys,
                            int32_t *bad) {
    const uint64_t sentinel = (1ULL << (2 * B)) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = u[i], b = v[i];
        uint64_t k0 = sentinel, k1 = sentinel;
        if (a < 0 || a >= n || b < 0 || b >= n) {
            atomicOr(bad, 1);
        } else if (a != b) {
            k0 = ((uint64_t)a << B) | (uint64_t)b;
            k1 = ((uint64_t)b << B) | (uint64_t)a;
        }
        keys[2 * i] = k0;
        keys[2 * i + 1] = k1;
    }
}

// Sorted keys to CSR, in segments of `len` keys (a multiple of 32), one warp
// each.  k_unique_flags: one bit per key (first of its value, no sentinel) and
// the set bits per segment; k_unique_fill: the marked keys' neighbours in
// order, and the row offsets, written where a row begins (for the empty rows
// before it too) and behind the last key.  Bound: HBM (16 B read a key, 4 B
// written an entry).  Counting the entries of each row with atomics, which a
// hub's row serialises, and scanning the counts took 0.46 ms and six more
// launches on R-MAT 18; both kernels together take 0.05 ms.
__global__ void k_unique_flags(const uint64_t *__restrict__ keys, int64_t k, uint64_t sentinel, int64_t len,
                               uint32_t *bits, int32_t *seg_cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t seg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t e0 = seg * len, e1 = e0 + len < k ? e0 + len : k;
    if (e0 >= k) return;
    int32_t cnt = 0;
    uint64_t last = e0 ? keys[e0 - 1] : sentinel;
#pragma unroll 4
    for (int64_t c0 = e0; c0 < e1; c0 += 32) {
        const int64_t p = c0 + lane;
        const uint64_t key = p < e1 ? keys[p] : sentinel;
        uint64_t prev = __shfl_up_sync(0xffffffffu, key, 1);
        if (lane == 0) prev = last;
        const uint32_t b = __ballot_sync(0xffffffffu, key != sentinel && key != prev);
        if (lane == 0) bits[c0 >> 5] = b;
        cnt += __popc(b);
        last = __shfl_sync(0xffffffffu, key, 31);
    }
    if (lane == 0) seg_cnt[seg] = cnt;
}

//
// SPARSE (more than twice as many rows as keys): most rows are empty then, and a
// warp filled the rows of a long gap alone (50 pairs on 3M vertices: ingest 0.49
// ms, now 0.10; with a key a row, evenly spread, the searches cost 0.03 ms more
// than short gaps filled by their warps).
// The row offsets are found by all threads instead, kRowsEach rows each: a binary
// search for the first key of the first row, from there on for the next rows',
// and the marked keys before it.
constexpr int kRowsEach = 8;

// set bits before position p, from the scanned counts of segments of `len` bits
__device__ __forceinline__ int32_t bits_before(const uint32_t *__restrict__ bits, const int32_t *__restrict__ seg_off,
                                               int64_t len, int64_t nseg, int64_t p) {
    const int64_t s = p / len < nseg ? p / len : nseg - 1;
    int32_t c = seg_off[s];
    int64_t w = s * len >> 5;
    for (; w < p >> 5; ++w) c += __popc(bits[w]);
    return p & 31 ? c + __popc(bits[w] & ((1u << (p & 31)) - 1u)) : c;
}

template <bool SPARSE>
__global__ void k_unique_fill(const uint64_t *__restrict__ keys, int64_t k, uint64_t sentinel, int64_t len, int32_t B,
                              int32_t n, const uint32_t *__restrict__ bits, const int32_t *__restrict__ seg_off,
                              int32_t *col, int32_t *row_ptr) {
    const int lane = threadIdx.x & 31;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, seg = tid >> 5;
    if (SPARSE) {
        const int64_t nseg = (k + len - 1) / len;
        const int64_t stride = (int64_t)gridDim.x * blockDim.x * kRowsEach;
        for (int64_t v0 = tid * kRowsEach; v0 <= n; v0 += stride) {
            int64_t lo = 0, hi = k;   // the row's first key is at lo..hi
            int32_t at = 0;
            for (int64_t v = v0; v < v0 + kRowsEach && v <= n; ++v) {
                const uint64_t first = (uint64_t)v << B;
                bool moved = v == v0;
                if (!moved) {
                    hi = lo;
                    for (int64_t step = 1; hi < k && keys[hi] < first; step <<= 1) {
                        lo = hi + 1;
                        hi = hi + step < k ? hi + step : k;
                        moved = true;
                    }
                }
                while (lo < hi) {
                    const int64_t mid = (lo + hi) >> 1;
                    if (keys[mid] < first) lo = mid + 1; else hi = mid;
                }
                if (moved) at = bits_before(bits, seg_off, len, nseg, lo);
                row_ptr[v] = at;
            }
        }
    }
    const int64_t e0 = seg * len, e1 = e0 + len < k ? e0 + len : k;
    if (e0 >= k) return;
    const uint64_t mask = (1ULL << B) - 1;
    int32_t out = seg_off[seg];
    // row of the key before (-1 before the first one)
    int32_t row = e0 ? (keys[e0 - 1] == sentinel ? n : (int32_t)(keys[e0 - 1] >> B)) : -1;
#pragma unroll 2
    for (int64_t c0 = e0; c0 < e1; c0 += 32) {
        const int64_t p = c0 + lane;
        const uint64_t key = p < e1 ? keys[p] : sentinel;
        const uint32_t b = bits[c0 >> 5];
        const int32_t at = out + __popc(b & lanemask_lt());
        if ((b >> lane) & 1u) col[at] = (int32_t)(key & mask);
        out += __popc(b);
        if (SPARSE) continue;
        // a sentinel counts as row n: the rows behind the last key end here
        const int32_t r = key == sentinel ? n : (int32_t)(key >> B);
        int32_t prev = __shfl_up_sync(0xffffffffu, r, 1);
        if (lane == 0) prev = row;
        const bool first = p < e1 && r > prev;
        const bool far = first && r - prev > 32;
        if (first && !far)
            for (int32_t q = r; q > prev; --q) row_ptr[q] = at;
        for (uint32_t m = __ballot_sync(0xffffffffu, far); m; m &= m - 1u) {   // many empty rows: the whole warp
            const int src = __ffs(m) - 1;
            const int32_t q1 = __shfl_sync(0xffffffffu, r, src), q0 = __shfl_sync(0xffffffffu, prev, src);
            const int32_t val = __shfl_sync(0xffffffffu, at, src);
            for (int32_t q = q0 + 1 + lane; q <= q1; q += 32) row_ptr[q] = val;
        }
        row = __shfl_sync(0xffffffffu, r, 31);
    }
    // the graph's last key is no sentinel: the rows behind it
    if (!SPARSE && e1 == k && keys[k - 1] != sentinel) {
        const int32_t r = (int32_t)(keys[k - 1] >> B);
        for (int32_t q = r + 1 + lane; q <= n; q += 32) row_ptr[q] = out;
    }
}

// ------------------------------------------------------------------ keys

__global__ void k_degree_key(const int32_t *row_ptr, int32_t n, int64_t *key) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        key[v] = row_ptr[v + 1] - row_ptr[v];
}

// Core numbers as the largest fixed point of the h-index step: val(v) starts
// at an upper bound (the degree, at most sqrt(2m): a k-core has k (k + 1) / 2
// edges) and falls to the largest h such that h neighbours have val >= h.
// The step is monotone and the core numbers are a fixed point of it, so the
// order of the updates does not matter: values are updated in place, and a
// round visits the vertices with a neighbour that fell past their value in
// the round before.  No more rounds than peeling has removal steps, one grid
// barrier each, and hubs are shared by a group of warps.
// Bound: L2 gathers of the neighbours' values in the first rounds; after them
// the latency of a round (one hub's visit and the barrier), of which graphs
// whose hubs fall one step after the other take hundreds.  Peeling level by
// level (three barriers per removal step, each removed hub's row walked by one
// warp) took 42.1 ms on the 1.7M-vertex graph (340 rounds here) and 9.3 ms on
// R-MAT 18; this kernel: 13.6 ms and 3.8 ms.
//
// stamp[v] = round in which v is to be visited.  Lists by degree: [0] 2..32
// (8 lanes a vertex), [1] 33..384 (a warp), [2] above (256 threads, with the
// neighbours that can still matter kept apart once the hub has fallen); degrees
// 0 and 1 are their own core numbers.  more[k][r % 3] = round r visits list k.
constexpr int kCoreThreads = 512;   // 128 registers: 16 loads of a thread in flight
constexpr int kCoreWarps = kCoreThreads / 32;
constexpr int kCoreSmall = 32, kCoreMid = 384;
// Measured on GB300 (R-MAT 14, R-MAT 18, Chung-Lu 1.7M; ms): a warp up to 384
// neighbours and 256 threads above 1.0, 3.8, 13.6; 64 threads 1.3, 3.7, 14.6; a
// warp up to 1024 and 256 threads above 0.65, 4.8, 20.5; 64 threads 0.75, 6.5, 26.4
constexpr int kHubThreads = 256, kHubWarps = kHubThreads / 32, kHubGroups = kCoreThreads / kHubThreads;
constexpr int kHubBins = 4096;
constexpr size_t kCoreSmem = (size_t)kHubGroups * kHubBins * sizeof(int32_t);

struct CoreParams {
    const int32_t *row_ptr, *col;
    int32_t n;
    int32_t bound;            // values start at min(degree, bound)
    int32_t *val, *stamp;
    int32_t *list[3];
    int32_t *ctl;             // [0..2] list lengths, [3] entries of kept, [4 + 3 k ..] more[k]
    // hub i of list[2]: neighbours with val >= keep_from[i] at kept[keep_at[i]
    // .. + keep_n[i]) (keep_from 0: none kept yet)
    int32_t *keep_from, *keep_at, *keep_n, *kept;
    int32_t dense, large;     // the graph may be left to k_core_peel (core_leave)
};

// Graphs that k_core_rounds leaves to k_core_peel, which is launched behind it for
// those that may be, and returns at once for the others (ctl[kCorePeeled]).
// Dense ones, of kPeelDegree or more entries a vertex, nearly all of them of more

// than kCoreSmall neighbours: there the rounds visit every vertex, a hub, several
// times, and peeling has few steps; the degrees are known on the device alone
// (k_core_init).  Measured on GB300 (rounds / peeling, ms): G(n, p) with n = 20,000 of degree 200
// 1.6 / 1.2, 350 1.2 / 1.6, 400 5.9 / 1.6, 1,500 9.7 / 4.3, n = 100,000 of degree
// 400 35 / 4.7; bipartite of degree 300 2.1 / 4.0, 600 4.6 / 3.0; R-MAT, which has
// many vertices of few neighbours, scale 14, 128 edges a vertex 2.0 / 4.9.
// Large ones, of kPeelVertices or more, after kPeelRounds rounds in a row that
// visited vertices of up to kCoreSmall neighbours alone: chains that fall from
// their ends for thousands of rounds, each of which looks at every stamp (grid of
// 1,000 x 1,000 vertices 17.5 ms by rounds alone, path of a million 4,624; peeled
// 7.9 and 2,649).
constexpr int64_t kPeelDegree = kCoreMid;
constexpr int32_t kPeelVertices = 1 << 18, kPeelRounds = 64;
constexpr int kCorePeeled = 15;

__device__ __forceinline__ int core_class(int32_t d) { return d <= kCoreSmall ? 0 : d <= kCoreMid ? 1 : 2; }

__global__ void k_core_init(CoreParams P) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); v0 < P.n; v0 += stride) {
        const int64_t v = v0 + lane;
        int cls = -1;
        if (v < P.n) {
            const int32_t d = P.row_ptr[v + 1] - P.row_ptr[v];
            P.val[v] = d < P.bound ? d : P.bound;
            P.stamp[v] = 0;
            cls = d < 2 ? -1 : core_class(d);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t b = __ballot_sync(0xffffffffu, cls == k);
            if (!b) continue;
            int32_t at = 0;
            if (lane == 0) at = atomicAdd(&P.ctl[k], __popc(b));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (cls == k) {
                const int32_t i = at + __popc(b & lanemask_lt());
                P.list[k][i] = (int32_t)v;
                if (k == 2) P.keep_from[i] = 0;
            }
        }
    }
}

// val[v] fell from `was` to `now`: neighbour w (value x) is visited in the
// next round if v counted towards x and no longer does.  A neighbour that is
// visited in this round may end anywhere up to x, so its bound is `now` alone.
// Returns the bit of w's list (of both it can be in, if x tells only that), or 0.
// N neighbours at a time (w = -1: none), their loads in flight together: told
// one after the other, the notes of a lane took most of a visit.
template <int N>
__device__ __forceinline__ uint32_t core_tell(const CoreParams &P, const int32_t *w, const int32_t *x, int32_t was,
                                                  int32_t now, int32_t round) {
    bool tell[N];
    int32_t d[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        int32_t st = round;
        if (w[q] >= 0 && x[q] > was) st = __ldcg(P.stamp + w[q]);
        tell[q] = w[q] >= 0 && x[q] > now && st == round;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
        d[q] = 0;
        if (tell[q]) P.stamp[w[q]] = round + 1;
        if (tell[q] && x[q] <= kCoreSmall) d[q] = P.row_ptr[w[q] + 1] - P.row_ptr[w[q]];
    }
    uint32_t told = 0u;
#pragma unroll
    for (int q = 0; q < N; ++q)
        if (tell[q]) told |= x[q] > kCoreSmall ? 6u : 1u << core_class(d[q]);
    return told;
}

// largest h in [lo, hi) with cnt + (entries of bin[h - lo ..]) >= h, or 0, one warp
__device__ __forceinline__ int32_t core_from_bins(const int32_t *bin, int32_t lo, int32_t hi, int32_t cnt, int lane) {
    for (int32_t top = hi - 1; top >= lo; top -= 32) {
        const int32_t h = top - lane;
        int32_t s = h >= lo ? bin[h - lo] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        const uint32_t ok = __ballot_sync(0xffffffffu, h >= lo && cnt + s >= h);
        if (ok) return top - (__ffs(ok) - 1);
        cnt += __shfl_sync(0xffffffffu, s, 31);
    }
    return 0;
}

// A hub's visit by a group of kHubThreads threads (barrier `bar`): i is its
// place in the list.  Returns the list bits told.
struct HubShared {
    int32_t active[kHubThreads], n_active, red[kHubWarps], found, kept, at;
};

// (barrier.sync, not bar.sync: the lanes of a warp may arrive one after the other)
__device__ __forceinline__ void hub_sync(int bar) {
    __syncwarp();
    asm volatile("barrier.sync %0, %1;" ::"r"(bar), "n"(kHubThreads) : "memory");
}

__device__ uint32_t core_hub(const CoreParams &P, HubShared &m, int32_t *bin, int32_t i, int32_t round, int bar) {
    const int t = threadIdx.x & (kHubThreads - 1), lane = t & 31, warp = t >> 5;
    const int32_t v = P.list[2][i];
    const int32_t e0 = P.row_ptr[v], d = P.row_ptr[v + 1] - e0;
    const int32_t from = __ldcg(P.keep_from + i);
    const int32_t *kept = P.kept + (from ? __ldcg(P.keep_at + i) : 0);
    const int32_t n_kept = from ? __ldcg(P.keep_n + i) : 0;
    const int32_t c = __ldcg(P.val + v);
    // Bins of a window below the current value, then of the next windows down
    // while they hold no value: most neighbours of a hub have one of few small
    // values, and adding those up serialises.  Each pass reads every value once
    // (those from the window's end up are counted), so that none that falls
    // meanwhile is counted twice.
    int32_t h = c;
    for (int32_t hi = c;;) {
        int32_t lo = hi >> 1 > hi - kHubBins ? hi >> 1 : hi - kHubBins;
        if (lo < from && hi > from) lo = from;
        if (lo < 1) lo = 1;
        const bool few = from && lo >= from;
        const int32_t *row = few ? kept : P.col + e0;
        const int32_t len = few ? n_kept : d;
        for (int32_t k = t; k < hi - lo; k += kHubThreads) bin[k] = 0;
        hub_sync(bar);
        int32_t cnt = 0;
#pragma unroll 16
        for (int32_t e = t; e < len; e += kHubThreads) {
            const int32_t x = __ldcg(P.val + (few ? __ldcg(row + e) : row[e]));
            if (x >= hi) ++cnt;
            else if (x >= lo) atomicAdd(&bin[x - lo], 1);
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) m.red[warp] = cnt;
        hub_sync(bar);
        cnt = __reduce_add_sync(0xffffffffu, lane < kHubWarps ? m.red[lane] : 0);
        if (hi == c && cnt >= c) return 0u;   // unchanged; the same for every thread
        if (warp == 0) {
            const int32_t f = core_from_bins(bin, lo, hi, cnt, lane);
            if (lane == 0) m.found = f;
        }
        hub_sync(bar);
        h = m.found;
        if (h || lo == 1) break;
        hi = lo;
    }
    if (h < 1) h = 1;
    if (t == 0) P.val[v] = h;
    uint32_t told = 0u;
    if (from && h >= from) {   // neighbours above h are all among the kept ones
        for (int32_t b0 = t; b0 < n_kept; b0 += 8 * kHubThreads) {
            int32_t w[8], x[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = b0 + q * kHubThreads < n_kept ? __ldcg(kept + b0 + q * kHubThreads) : -1;
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = w[q] >= 0 ? __ldcg(P.val + w[q]) : 0;
            told |= core_tell<8>(P, w, x, c, h, round);
        }
        return told;
    }
    // keep the neighbours that matter down to half the value
    const int32_t keep = h >> 1 > 1 ? h >> 1 : 1;
    if (t == 0) {
        m.kept = 0;
        m.at = from ? __ldcg(P.keep_at + i) : atomicAdd(&P.ctl[3], d);
    }
    hub_sync(bar);
    int32_t *out = P.kept + m.at;
    for (int32_t b0 = warp * 32; b0 < d; b0 += 4 * kHubThreads) {
        int32_t w[4], x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t e = b0 + q * kHubThreads + lane;
            w[q] = e < d ? P.col[e0 + e] : -1;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = w[q] >= 0 ? __ldcg(P.val + w[q]) : 0;
        told |= core_tell<4>(P, w, x, c, h, round);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t b = __ballot_sync(0xffffffffu, x[q] >= keep);
            int32_t at = 0;
            if (lane == 0 && b) at = atomicAdd(&m.kept, __popc(b));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (x[q] >= keep) out[at + __popc(b & lanemask_lt())] = w[q];
        }
    }
    hub_sync(bar);
    if (t == 0) {
        P.keep_at[i] = m.at;
        P.keep_n[i] = m.kept;
        P.keep_from[i] = keep;
    }
    return told;
}

// The visit of a vertex v with up to 32 EACH neighbours by a warp: its row is
// read once, all of a lane's entries in flight, and held while the value is
// searched and the neighbours are told.  (Dependent passes over the row with
// bins in shared memory made this visit 14 to 30 us long, and in each round
// all other warps waited for one.)  Returns the list bits told.
template <int EACH>
__device__ __forceinline__ uint32_t core_mid(const CoreParams &P, int32_t v, int32_t e0, int32_t d, int32_t c,
                                             int32_t round, int lane) {
    int32_t w[EACH], x[EACH];
#pragma unroll
    for (int q = 0; q < EACH; ++q) w[q] = q * 32 + lane < d ? P.col[e0 + q * 32 + lane] : -1;
#pragma unroll
    for (int q = 0; q < EACH; ++q) x[q] = w[q] >= 0 ? __ldcg(P.val + w[q]) : 0;
    auto at_least = [&](int32_t h) {
        int32_t k = 0;
#pragma unroll
        for (int q = 0; q < EACH; ++q) k += x[q] >= h;
        return __reduce_add_sync(0xffffffffu, k);
    };
    const int32_t cnt = at_least(c);
    if (cnt >= c) return 0u;
    // cnt neighbours have val >= c > cnt, so the value is at least cnt
    int32_t lo = cnt > 1 ? cnt : 1, hi = c - 1;
    while (lo < hi) {   // the same for all lanes
        const int32_t mid = (lo + hi + 1) >> 1;
        if (at_least(mid) >= mid) lo = mid; else hi = mid - 1;
    }
    if (lane == 0) P.val[v] = lo;
    uint32_t told = 0u;
#pragma unroll
    for (int q = 0; q < EACH; q += 4) told |= core_tell<4>(P, w + q, x + q, c, lo, round);
    return told;
}

__global__ void __launch_bounds__(kCoreThreads, 1) k_core_rounds(CoreParams P) {
    if (P.dense && (int64_t)P.ctl[0] * 16 < P.n) {
        if (blockIdx.x == 0 && threadIdx.x == 0) P.ctl[kCorePeeled] = 1;
        return;
    }
    int32_t chains = 0;   // rounds in a row that visited the first list alone
    cg::grid_group grid = cg::this_grid();
    extern __shared__ int32_t core_bins[];   // kHubBins a group
    __shared__ HubShared hub[kHubGroups];
    __shared__ uint32_t block_told;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nblk = gridDim.x;
    const int64_t gwarp = (int64_t)blockIdx.x * kCoreWarps + warp, nwarp = nblk * kCoreWarps;
    const int32_t n_small = P.ctl[0], n_mid = P.ctl[1], n_big = P.ctl[2];
    if (threadIdx.x == 0) block_told = 0u;
    uint32_t visit = 7u;   // lists with visits in this round
    for (int32_t round = 0;; ++round) {
        uint32_t told = 0u;
        if (blockIdx.x == 0 && threadIdx.x < 3) P.ctl[4 + 3 * threadIdx.x + (round + 2) % 3] = 0;
        // ---- hubs, dealt out to the groups of all blocks
        if (visit & 4u) {
            const int g = threadIdx.x / kHubThreads, t = threadIdx.x & (kHubThreads - 1);
            HubShared &m = hub[g];
            const int64_t ngrp = nblk * kHubGroups, g0 = blockIdx.x + g * nblk;
            for (int64_t i0 = g0; i0 < n_big; i0 += ngrp * kHubThreads) {
                if (t == 0) m.n_active = 0;
                hub_sync(1 + g);
                const int64_t i = i0 + (int64_t)t * ngrp;
                if (i < n_big && __ldcg(P.stamp + P.list[2][i]) == round)
                    m.active[atomicAdd(&m.n_active, 1)] = (int32_t)i;
                hub_sync(1 + g);
                const int na = m.n_active;
                for (int a = 0; a < na; ++a) {
                    told |= core_hub(P, m, core_bins + g * kHubBins, m.active[a], round, 1 + g);
                    hub_sync(1 + g);
                }
            }
        }
        // the others see this round's values of the hubs: without this barrier
        // R-MAT 18 takes three times as many rounds
        __syncthreads();
        // ---- degrees 33..384: a warp each, items dealt out warp by warp
        if (visit & 2u)
            for (int64_t i0 = gwarp; i0 < n_mid; i0 += nwarp * 32) {
                const int64_t i = i0 + (int64_t)lane * nwarp;
                const int32_t mine = i < n_mid ? P.list[1][i] : -1;
                uint32_t m = __ballot_sync(0xffffffffu, mine >= 0 && __ldcg(P.stamp + (mine < 0 ? 0 : mine)) == round);
                for (; m; m &= m - 1u) {
                    const int32_t v = __shfl_sync(0xffffffffu, mine, __ffs(m) - 1);
                    const int32_t e0 = P.row_ptr[v], d = P.row_ptr[v + 1] - e0, c = __ldcg(P.val + v);
                    if (d <= 128) told |= core_mid<4>(P, v, e0, d, c, round, lane);
                    else told |= core_mid<12>(P, v, e0, d, c, round, lane);
                }
            }
        // ---- degrees 2..32: 8 lanes each, four vertices of a warp at a time
        if (visit & 1u)
            for (int64_t i0 = gwarp * 32; i0 < n_small; i0 += nwarp * 32) {
                const int64_t i = i0 + lane;
                const int32_t mine = i < n_small ? P.list[0][i] : -1;
                uint32_t m = __ballot_sync(0xffffffffu, mine >= 0 && __ldcg(P.stamp + (mine < 0 ? 0 : mine)) == round);
                while (m) {
                    // the g-th lowest set bit for lane group g
                    const int g = lane >> 3;
                    uint32_t mg = m;
                    for (int k = 0; k < g; ++k) mg &= mg - 1u;
                    const int32_t v0 = __shfl_sync(0xffffffffu, mine, mg ? __ffs(mg) - 1 : 0);
                    const int32_t v = mg ? v0 : -1;
                    for (int k = 0; k < 4; ++k) m &= m - 1u;
                    int32_t w[4], x[4], c = 0;
                    const int32_t e0 = v >= 0 ? P.row_ptr[v] : 0, e1 = v >= 0 ? P.row_ptr[v + 1] : 0;
                    if (v >= 0) c = __ldcg(P.val + v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int32_t e = e0 + q * 8 + (lane & 7);
                        w[q] = e < e1 ? P.col[e] : -1;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) x[q] = w[q] >= 0 ? __ldcg(P.val + w[q]) : 0;
                    auto at_least = [&](int32_t h) {
                        int32_t k = (x[0] >= h) + (x[1] >= h) + (x[2] >= h) + (x[3] >= h);
                        k += __shfl_xor_sync(0xffffffffu, k, 1);
                        k += __shfl_xor_sync(0xffffffffu, k, 2);
                        return k + __shfl_xor_sync(0xffffffffu, k, 4);
                    };
                    const int32_t cnt = at_least(c > 0 ? c : 1);
                    // cnt neighbours have val >= c > cnt, so the value is at least cnt
                    int32_t lo = cnt, hi = cnt < c ? c - 1 : cnt;
                    while (__any_sync(0xffffffffu, lo < hi)) {
                        const int32_t mid = (lo + hi + 1) >> 1;
                        const int32_t k = at_least(mid);
                        if (lo < hi) {
                            if (k >= mid) lo = mid; else hi = mid - 1;
                        }
                    }
                    if (v >= 0 && cnt < c) {
                        const int32_t h = lo > 1 ? lo : 1;
                        if ((lane & 7) == 0) P.val[v] = h;
                        told |= core_tell<4>(P, w, x, c, h, round);
                    }
                }
            }
        told = __reduce_or_sync(0xffffffffu, told);
        if (lane == 0 && told) atomicOr(&block_told, told);
        __syncthreads();
        if (threadIdx.x < 3 && ((block_told >> threadIdx.x) & 1u)) P.ctl[4 + 3 * threadIdx.x + (round + 1) % 3] = 1;
        __syncthreads();
        if (threadIdx.x == 0) block_told = 0u;
        grid.sync();
        visit = 0u;
#pragma unroll
        for (int k = 0; k < 3; ++k) visit |= __ldcg(P.ctl + 4 + 3 * k + (round + 1) % 3) ? 1u << k : 0u;
        if (!visit) break;
        chains = visit == 1u ? chains + 1 : 0;
        if (P.large && chains == kPeelRounds) {   // the same for all threads of the grid
            if (blockIdx.x == 0 && threadIdx.x == 0) P.ctl[kCorePeeled] = 1;
            break;
        }
    }
}

// Core numbers by level-synchronous peeling on a cooperative grid, for the graphs
// that k_core_rounds left (*left).  Level k:
// every alive vertex whose remaining degree is <= k is removed with core
// number k; removing a vertex decrements its alive neighbours, and those that
// fall to <= k are removed at the same level (claimed once by CAS).
// The seeding scan of a level visits only the vertices still alive after the
// previous one (a compacted list), so a level costs its alive count, not n.
// The removal cascade gives each removed vertex a warp (hubs leave at the
// high levels, where the frontier is short).  Levels that would remove
// nothing are skipped: the next level is the smallest remaining degree.
// ctl[0] = removed so far, ctl[1], ctl[2] = lengths of the two frontiers,
// ctl[3], ctl[4] = lengths of the two alive lists, ctl[5], ctl[6] = smallest
// remaining degree (one slot per level parity).
// Every read of a control word is followed by a grid barrier before any
// thread may change that word, so all threads take the same branches.
__global__ void k_core_peel(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col, int32_t n,
                            int32_t *d, int32_t *core, int32_t *fa, int32_t *fb, int32_t *la, int32_t *lb,
                            int32_t *ctl, const int32_t *left) {
    if (!*left) return;
    cg::grid_group grid = cg::this_grid();
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = tid; v < n; v += nth) {
        d[v] = row_ptr[v + 1] - row_ptr[v];
        core[v] = -1;
        la[v] = (int32_t)v;
    }
    // all alive, no remaining degree seen yet
    if (tid < 8) ctl[tid] = tid == 3 ? n : tid == 5 || tid == 6 ? 0x7fffffff : 0;
    const int lane = threadIdx.x & 31;
    const int64_t wid = tid >> 5, nwarp = nth >> 5;
    int32_t *cur = fa, *nxt = fb, *alive = la, *alive2 = lb;
    int ci = 1, ni = 2, ai = 3, bi = 4;
    int par = 0;
    for (int32_t k = 0; k <= n;) {   // a core number never exceeds n - 1
        grid.sync();
        const int32_t removed = *(volatile int32_t *)&ctl[0];
        const int32_t na = *(volatile int32_t *)&ctl[ai];
        grid.sync();
        if (removed >= n) break;
        const int mi = 5 + par;
        if (tid == 0) ctl[5 + (1 - par)] = 0x7fffffff;   // slot of the next level, untouched in this one
        int32_t lmin = 0x7fffffff;
        for (int64_t i = tid; i < na; i += nth) {
            const int32_t v = alive[i];
            if (*(volatile int32_t *)&core[v] >= 0) continue;   // removed at an earlier level
            const int32_t dv = d[v];
            if (dv <= k) {
                core[v] = k;
                cur[atomicAdd(&ctl[ci], 1)] = v;
            } else {
                alive2[atomicAdd(&ctl[bi], 1)] = v;
                lmin = dv < lmin ? dv : lmin;
            }
        }
        lmin = __reduce_min_sync(0xffffffffu, lmin);
        if (lane == 0 && lmin != 0x7fffffff) atomicMin(&ctl[mi], lmin);
        grid.sync();
        if (tid == 0) ctl[ai] = 0;   // read by everyone before the last barrier
        {
            int32_t *t = alive;
            alive = alive2;
            alive2 = t;
            const int ti = ai;
            ai = bi;
            bi = ti;
        }
        for (;;) {
            const int32_t len = *(volatile int32_t *)&ctl[ci];
            grid.sync();
            if (len == 0) break;
            int32_t cmin = 0x7fffffff;
            for (int64_t i = wid; i < len; i += nwarp) {
                const int32_t x = cur[i];
                const int32_t e1 = row_ptr[x + 1];
                for (int32_t e = row_ptr[x] + lane; e < e1; e += 32) {
                    const int32_t w = col[e];
                    if (*(volatile int32_t *)&core[w] >= 0) continue;
                    const int32_t nd = atomicSub(&d[w], 1) - 1;
                    if (nd <= k) {
                        if (atomicCAS(&core[w], -1, k) == -1) nxt[atomicAdd(&ctl[ni], 1)] = w;
                    } else {
                        cmin = nd < cmin ? nd : cmin;
                    }
                }
            }
            cmin = __reduce_min_sync(0xffffffffu, cmin);
            if (lane == 0 && cmin != 0x7fffffff) atomicMin(&ctl[mi], cmin);
            if (tid == 0) {
                atomicAdd(&ctl[0], len);
                ctl[ci] = 0;   // nobody reads ctl[ci] again before the next barrier
            }
            int32_t *t = cur;
            cur = nxt;
            nxt = t;
            int ti = ci;
            ci = ni;
            ni = ti;
            grid.sync();
        }
        // every survivor now has a remaining degree > k; the smallest is the
        // next level that removes anything (slot mi is not written again
        // before everyone has read it: the next level uses the other slot)
        const int32_t mn = *(volatile int32_t *)&ctl[mi];
        k = mn > k + 1 ? mn : k + 1;
        par ^= 1;
    }
}

__global__ void k_core_key(CoreParams P, const int32_t *peeled, int64_t *key) {
    const int32_t *core = peeled && P.ctl[kCorePeeled] ? peeled : P.val;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < P.n; v += (int64_t)gridDim.x * blockDim.x)
        key[v] = core[v];
}

// Triangles: with Γ+ oriented by degree rank, each triangle {a, b, x} with
// rank a < b < x is found once as x ∈ Γ+(a) ∩ Γ+(b) while visiting the
// oriented edge (a, b); all three corners are credited.  One warp per a.
__global__ void k_triangles(const int32_t *__restrict__ up_ptr, const int32_t *__restrict__ up_col, int32_t n,
                            unsigned long long *t) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t a = warp; a < n; a += nwarps) {
        const int32_t a0 = up_ptr[a], la = up_ptr[a + 1] - a0;
        if (la < 2) continue;
        const int32_t *A = up_col + a0;
        unsigned long long ta = 0;
        for (int32_t j = 0; j < la; ++j) {
            const int32_t b = A[j];
            const int32_t b0 = up_ptr[b], lb = up_ptr[b + 1] - b0;
            unsigned long long cnt = 0;
            for (int32_t s = 0; s < lb; s += 32) {
                bool hit = false;
                int32_t x = -1;
                if (s + lane < lb) {
                    x = up_col[b0 + s + lane];
                    int32_t lo = 0, hi = la;
                    while (lo < hi) {
                        const int32_t mid = (lo + hi) >> 1;
                        if (A[mid] < x) lo = mid + 1; else hi = mid;
                    }
                    hit = lo < la && A[lo] == x;
                }
                if (hit) atomicAdd(&t[x], 1ULL);
                cnt += __popc(__ballot_sync(0xffffffffu, hit));
            }
            if (lane == 0 && cnt) atomicAdd(&t[b], cnt);
            ta += cnt;
        }
        if (lane == 0 && ta) atomicAdd(&t[a], ta);
    }
}

// ------------------------------------------------------------------ ranks

__global__ void k_rank_keys_i64(const int64_t *key, int32_t n, int32_t idb, uint64_t *out) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        out[v] = ((uint64_t)key[v] << idb) | (uint64_t)v;
}

__global__ void k_rank_keys_f32(const float *key, int32_t n, int32_t idb, uint64_t *out) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        uint32_t b = __float_as_uint(key[v]);
        b ^= (b >> 31) ? 0xffffffffu : 0x80000000u;   // order-preserving map of floats to uint32
        out[v] = ((uint64_t)b << idb) | (uint64_t)v;
    }
}

__global__ void k_scatter_rank(const uint64_t *sorted, int32_t n, int32_t idb, int32_t *rank) {
    const uint64_t mask = (1ULL << idb) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        rank[sorted[i] & mask] = (int32_t)i;
}

// ------------------------------------------------------------------ Γ+ lists

// The CSR entries are cut into segments of `len` entries (a multiple of 32),
// one warp each, so that a hub's row costs what as many short rows cost.
// k_up_flags: one bit per entry (its neighbour ranks above its row), the
// number of set bits per segment, and up_ptr[v] counted from the start of the
// segment that holds row v's first entry.  k_up_fill: with the scanned counts,
// the marked neighbours in order, and up_ptr made absolute.
// Bound: L2 (one gather of rank per entry).  A warp per row spent 1.02 ms on
// the 22M entries of the 1.7M-vertex graph, waiting for the hubs' rows; the
// two kernels and the scan between them take 0.19 ms.
// SPARSE (more rows than entries): up_ptr by k_up_fill alone, one row a thread
// (the warp of a segment would fill long gaps of empty rows by itself: 50 edges
// on 3M vertices: their triangle counts took 5.4 ms, now 0.29).

// warp: largest r in [0, n) with row_ptr[r] <= e (row_ptr[0] = 0 <= e)
__device__ __forceinline__ int32_t warp_row_of(const int32_t *row_ptr, int32_t n, int32_t e, int lane) {
    int32_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int32_t step = (hi - lo + 31) >> 5;
        const int64_t i = (int64_t)lo + (int64_t)lane * step;
        const uint32_t le = __ballot_sync(0xffffffffu, i < hi && row_ptr[i] <= e);
        lo += (__popc(le) - 1) * step;
        hi = hi - lo > step ? lo + step : hi;
    }
    return lo;
}

template <bool SPARSE>
__global__ void k_up_flags(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                           const int32_t *__restrict__ rank, int32_t n, int32_t nnz, int32_t len, uint32_t *bits,
                           int32_t *seg_cnt, int32_t *up_ptr) {
    const int lane = threadIdx.x & 31;
    const int64_t seg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t s0 = seg * len;
    if (s0 >= nnz) return;
    const int32_t e0 = (int32_t)s0, e1 = (int32_t)(s0 + len < nnz ? s0 + len : nnz);
    int32_t row = warp_row_of(row_ptr, n, e0, lane);
    // row of the entry before (a row that starts at e0, and the empty ones
    // before it, get their up_ptr here)
    int32_t before = row;
    if (row_ptr[row] == e0) before = e0 ? warp_row_of(row_ptr, n, e0 - 1, lane) : -1;
    int32_t cnt = 0;
    // unsigned: the last chunk of a graph near 2^31 entries runs past it
    for (uint32_t c0 = (uint32_t)e0; c0 < (uint32_t)e1; c0 += 32) {
        const uint32_t p = c0 + (uint32_t)lane;
        const bool valid = p < (uint32_t)e1;
        const int32_t w = valid ? col[p] : 0;
        const uint32_t st = row + 1 + lane <= n ? (uint32_t)row_ptr[row + 1 + lane] : 0xffffffffu;
        int32_t r = row;
        if (__shfl_sync(0xffffffffu, st, 31) > c0 + 31u) {
            int k = 0;   // rows after `row` that start at or before p
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (__shfl_sync(0xffffffffu, st, k + step - 1) <= p) k += step;
            r += k;
        } else if (valid) {
            int32_t lo = row, hi = n;   // many short or empty rows
            while (hi - lo > 1) {
                const int32_t mid = lo + ((hi - lo) >> 1);
                if ((uint32_t)row_ptr[mid] <= p) lo = mid; else hi = mid;
            }
            r = lo;
        }
        const bool up = valid && rank[w] > rank[r];
        const uint32_t b = __ballot_sync(0xffffffffu, up);
        if (lane == 0) bits[c0 >> 5] = b;
        if (!SPARSE) {
            int32_t prev = __shfl_up_sync(0xffffffffu, r, 1);
            if (lane == 0) prev = before;
            const int32_t at = cnt + __popc(b & lanemask_lt());
            const bool far = valid && r - prev > 32;   // a long run of empty rows: filled by the whole warp
            if (valid && !far)
                for (int32_t q = r; q > prev; --q) up_ptr[q] = at;
            for (uint32_t m = __ballot_sync(0xffffffffu, far); m; m &= m - 1u) {
                const int src = __ffs(m) - 1;
                const int32_t q1 = __shfl_sync(0xffffffffu, r, src), q0 = __shfl_sync(0xffffffffu, prev, src);
                const int32_t val = __shfl_sync(0xffffffffu, at, src);
                for (int32_t q = q0 + 1 + lane; q <= q1; q += 32) up_ptr[q] = val;
            }
        }
        cnt += __popc(b);
        row = before = __shfl_sync(0xffffffffu, r, (uint32_t)e1 - c0 > 32u ? 31 : (int)((uint32_t)e1 - c0) - 1);
    }
    if (!SPARSE && e1 == nnz)
        for (int32_t q = row + 1 + lane; q <= n; q += 32) up_ptr[q] = cnt;
    if (lane == 0) seg_cnt[seg] = cnt;
}

template <bool SPARSE>
__global__ void k_up_fill(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                          const uint32_t *__restrict__ bits, const int32_t *__restrict__ seg_off, int32_t n,
                          int32_t nnz, int32_t len, int32_t nseg, int32_t *up_ptr, int32_t *up_col) {
    const int lane = threadIdx.x & 31;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t seg = tid >> 5;
    if (seg < nseg) {
        const int32_t e0 = (int32_t)(seg * len), e1 = (int32_t)(seg * len + len < nnz ? seg * len + len : nnz);
        int32_t out = seg_off[seg];
#pragma unroll 4
        for (uint32_t c0 = (uint32_t)e0; c0 < (uint32_t)e1; c0 += 32) {
            const uint32_t b = bits[c0 >> 5];
            if ((b >> lane) & 1u) up_col[out + __popc(b & lanemask_lt())] = col[c0 + lane];
            out += __popc(b);
        }
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = tid; v <= n; v += stride) {
        if (SPARSE) {
            up_ptr[v] = bits_before(bits, seg_off, len, nseg, row_ptr[v]);
            continue;
        }
        const int32_t sv = row_ptr[v] / len;
        up_ptr[v] += seg_off[sv < nseg ? sv : nseg - 1];
    }
}

}  // namespace

// ------------------------------------------------------------------ host side

namespace {

// Validation of a caller CSR (simple undirected graph): bit 1 row offsets,
// 2 row not strictly increasing, 4 id outside [0, n), 8 self loop, 16 an
// entry (x, y) without (y, x).
__global__ void k_check_csr(const int32_t *row_ptr, const int32_t *col, int32_t n, int64_t nnz, int32_t *bad) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 == 0 && (row_ptr[0] != 0 || (int64_t)row_ptr[n] != nnz)) atomicOr(bad, 1);
    for (int64_t x = t0; x < n; x += stride) {
        const int32_t r0 = row_ptr[x], r1 = row_ptr[x + 1];
        if (r0 < 0 || r1 < r0 || (int64_t)r1 > nnz) {
            atomicOr(bad, 1);
            continue;
        }
        for (int32_t e = r0; e < r1; ++e) {
            const int32_t y = col[e];
            if (y < 0 || y >= n) {
                atomicOr(bad, 4);
                continue;
            }
            if (y == x) atomicOr(bad, 8);
            if (e > r0 && col[e - 1] >= y) atomicOr(bad, 2);
            const int32_t q0 = row_ptr[y], q1 = row_ptr[y + 1];
            if (q0 < 0 || q1 < q0 || (int64_t)q1 > nnz) continue;   // row y is reported itself
            int32_t lo = q0, hi = q1;
            while (lo < hi) {
                const int32_t mid = lo + ((hi - lo) >> 1);
                if (col[mid] < (int32_t)x) lo = mid + 1; else hi = mid;
            }
            if (!(lo < q1 && col[lo] == (int32_t)x)) atomicOr(bad, 16);
        }
    }
}

}  // namespace

mce_status check_csr(const mce_graph *g, cudaStream_t s) {
    DevBuf bad;
    MCE_TRY(bad.alloc(4, s));
    MCE_CUDA(cudaMemsetAsync(bad.p, 0, 4, s));
    MCE_LAUNCH(k_check_csr, grid_for(g->n > 0 ? g->n : 1, 256), 256, 0, s, g->row_ptr, g->col, g->n, g->nnz,
               bad.as<int32_t>());
    int32_t hb = 0;
    MCE_CUDA(cudaMemcpyAsync(&hb, bad.p, 4, cudaMemcpyDeviceToHost, s));
    MCE_CUDA(cudaStreamSynchronize(s));
    if (hb) {
        g_last_error = std::string("mce_graph_from_csr: not a simple undirected CSR:") +
                       ((hb & 1) ? " row offsets" : "") + ((hb & 2) ? " row not strictly increasing" : "") +
                       ((hb & 4) ? " id outside [0, n)" : "") + ((hb & 8) ? " self loop" : "") +
                       ((hb & 16) ? " not symmetric" : "");
        return MCE_EINVAL;
    }
    return MCE_OK;
}

// blocks of 256 threads for work on the rows by `threads` threads beside `blocks`
// for the segments
static unsigned blocks_for_rows(int64_t threads, unsigned blocks) {
    const unsigned rows = grid_for(threads, 256), most = (unsigned)num_sms() * 8;
    const unsigned want = rows < most ? rows : most;
    return blocks > want ? blocks : want;
}

mce_status build_csr(const int32_t *u, const int32_t *v, int64_t m, int32_t n, cudaStream_t s, mce_graph *g) {
    g->n = n;
    g->id_bits = bits_for(n > 0 ? (uint64_t)(n - 1) : 0);
    MCE_TRY(dev_alloc((void **)&g->row_ptr, ((size_t)n + 1) * sizeof(int32_t), s, "cudaMallocAsync"));
    if (m == 0 || n == 0) {
        MCE_CUDA(cudaMemsetAsync(g->row_ptr, 0, ((size_t)n + 1) * sizeof(int32_t), s));
        MCE_TRY(dev_alloc((void **)&g->col, 16, s, "cudaMallocAsync"));
        g->nnz = 0;
        return MCE_OK;
    }
    const int32_t B = g->id_bits;
    const int64_t k = 2 * m;
    if (k >= ((int64_t)1 << 31) - 1) {
        g_last_error = "mce_graph_create: too many pairs";
        return MCE_EINVAL;
    }
    // one warp a segment, all resident at once
    int64_t len = (k / ((int64_t)num_sms() * 64) + 32) & ~int64_t(31);
    if (len < 128) len = 128;
    const int64_t nseg = (k + len - 1) / len;
    DevBuf keys, tmp, bits, seg, bad;
    MCE_TRY(keys.alloc((size_t)k * sizeof(uint64_t), s));
    MCE_TRY(tmp.alloc((size_t)k * sizeof(uint64_t), s));
    MCE_TRY(bits.alloc((size_t)(k / 32 + 1) * sizeof(uint32_t), s));
    MCE_TRY(seg.alloc((size_t)(nseg + 1) * sizeof(int32_t), s));
    MCE_TRY(bad.alloc(sizeof(int32_t), s));
    MCE_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int32_t), s));
    // a pair with an id outside [0, n) becomes a sentinel too and is reported below
    MCE_LAUNCH(k_make_keys, grid_for(m, 256), 256, 0, s, u, v, m, n, B, keys.as<uint64_t>(), bad.as<int32_t>());
    MCE_TRY(radix_sort_u64(keys.as<uint64_t>(), tmp.as<uint64_t>(), k, 0, 2 * B, s));
    const uint64_t sentinel = (1ULL << (2 * B)) - 1;   // the pair of the last id with itself; n < 2^30
    const unsigned blocks = (unsigned)((nseg + 7) / 8);
    MCE_LAUNCH(k_unique_flags, blocks, 256, 0, s, keys.as<uint64_t>(), k, sentinel, len, bits.as<uint32_t>(),
               seg.as<int32_t>());
    MCE_TRY(exclusive_scan_i32(seg.as<int32_t>(), seg.as<int32_t>(), nseg, s));
    int32_t nnz = 0, hbad = 0;
    MCE_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    MCE_CUDA(cudaMemcpyAsync(&nnz, seg.as<int32_t>() + nseg, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    MCE_CUDA(cudaStreamSynchronize(s));
    if (hbad) {
        g_last_error = "mce_graph_create: vertex id outside [0, n)";
        return MCE_EINVAL;
    }
    g->nnz = nnz;
    MCE_TRY(dev_alloc((void **)&g->col, ((size_t)nnz + 4) * sizeof(int32_t), s, "cudaMallocAsync"));
    if (n > 2 * k)
        MCE_LAUNCH(k_unique_fill<true>, blocks_for_rows(n / kRowsEach + 1, blocks), 256, 0, s, keys.as<uint64_t>(), k,
                   sentinel, len, B, n, bits.as<uint32_t>(), seg.as<int32_t>(), g->col, g->row_ptr);
    else
        MCE_LAUNCH(k_unique_fill<false>, blocks, 256, 0, s, keys.as<uint64_t>(), k, sentinel, len, B, n,
                   bits.as<uint32_t>(), seg.as<int32_t>(), g->col, g->row_ptr);
    return MCE_OK;
}

// core numbers into `core` (first n of it) if k_core_rounds left the graph
static mce_status core_by_peeling(const mce_graph *g, const CoreParams &P, DevBuf &core, cudaStream_t s) {
    int32_t n = g->n;
    MCE_TRY(core.alloc(((size_t)n * 6 + 8) * sizeof(int32_t), s));
    int32_t *c = core.as<int32_t>(), *d = c + n, *fa = d + n, *fb = fa + n, *la = fb + n, *lb = la + n, *ctl = lb + n;
    int per_sm = 0;
    MCE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core_peel, 256, 0));
    if (per_sm < 1) {
        g_last_error = "core_numbers: cooperative kernel does not fit";
        return MCE_ECUDA;
    }
    // few blocks: the many grid barriers cost in proportion to the blocks
    const unsigned blocks = (unsigned)(num_sms() * (per_sm < 2 ? per_sm : 2));
    const int32_t *rp = g->row_ptr, *cl = g->col, *left = P.ctl + kCorePeeled;
    void *args[] = {(void *)&rp, (void *)&cl, (void *)&n,  (void *)&d,   (void *)&c,    (void *)&fa,
                    (void *)&fb, (void *)&la, (void *)&lb, (void *)&ctl, (void *)&left};
    g_launches.fetch_add(1, std::memory_order_relaxed);
    MCE_CUDA(cudaLaunchCooperativeKernel((const void *)k_core_peel, dim3(blocks), dim3(256), args, 0, s));
    return MCE_OK;
}

static mce_status core_numbers(const mce_graph *g, cudaStream_t s, int64_t *key) {
    const int32_t n = g->n;
    const size_t hubs = (size_t)(g->nnz / kCoreMid) + 1;
    DevBuf buf, ctl, keep, kept, peeled;
    MCE_TRY(buf.alloc((size_t)n * 5 * sizeof(int32_t), s));
    MCE_TRY(ctl.alloc(16 * sizeof(int32_t), s));
    MCE_TRY(keep.alloc(3 * hubs * sizeof(int32_t), s));
    MCE_TRY(kept.alloc((size_t)(hubs > 1 ? g->nnz : 1) * sizeof(int32_t), s));
    MCE_CUDA(cudaMemsetAsync(ctl.p, 0, 16 * sizeof(int32_t), s));
    CoreParams P{};
    P.row_ptr = g->row_ptr;
    P.col = g->col;
    P.n = n;
    int64_t bound = 1;
    while ((bound + 1) * (bound + 1) <= g->nnz) ++bound;
    P.bound = (int32_t)bound;
    P.val = buf.as<int32_t>();
    P.stamp = P.val + n;
    for (int k = 0; k < 3; ++k) P.list[k] = P.val + (size_t)(2 + k) * n;
    P.ctl = ctl.as<int32_t>();
    P.keep_from = keep.as<int32_t>();
    P.keep_at = P.keep_from + hubs;
    P.keep_n = P.keep_at + hubs;
    P.kept = kept.as<int32_t>();
    P.dense = g->nnz >= kPeelDegree * n;
    P.large = n >= kPeelVertices;
    MCE_LAUNCH(k_core_init, grid_for(n, 256), 256, 0, s, P);
    static std::once_flag once;
    static cudaError_t granted;
    std::call_once(once, [] {
        granted = cudaFuncSetAttribute(k_core_rounds, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoreSmem);
    });
    MCE_CUDA(granted);
    int per_sm = 0;
    MCE_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core_rounds, kCoreThreads, kCoreSmem));
    if (per_sm < 1) {
        g_last_error = "core_numbers: cooperative kernel does not fit";
        return MCE_ECUDA;
    }
    // one block an SM, fewer for graphs that leave warps without a vertex:
    // the barrier costs in proportion to the blocks
    const int64_t want = ((int64_t)n + 127) / 128;
    const unsigned blocks = (unsigned)(want < num_sms() ? want : num_sms());
    void *args[] = {(void *)&P};
    g_launches.fetch_add(1, std::memory_order_relaxed);
    MCE_CUDA(cudaLaunchCooperativeKernel((const void *)k_core_rounds, dim3(blocks), dim3(kCoreThreads), args, kCoreSmem,
                                         s));
    if (P.dense || P.large) MCE_TRY(core_by_peeling(g, P, peeled, s));
    MCE_LAUNCH(k_core_key, grid_for(n, 256), 256, 0, s, P, peeled.as<int32_t>(), key);
    return MCE_OK;
}

static mce_status triangle_counts(const mce_graph *g, cudaStream_t s, int64_t *key) {
    const int32_t n = g->n;
    DevBuf deg, rank, up_ptr, up_col;
    MCE_TRY(deg.alloc((size_t)n * sizeof(int64_t), s));
    MCE_TRY(rank.alloc((size_t)n * sizeof(int32_t), s));
    MCE_LAUNCH(k_degree_key, grid_for(n, 256), 256, 0, s, g->row_ptr, n, deg.as<int64_t>());
    MCE_TRY(rank_from_key_i64(deg.as<int64_t>(), n, g->id_bits, vertex_key_bits(g, MCE_RANK_DEGREE), s,
                              rank.as<int32_t>()));
    MCE_TRY(build_up_lists(g, rank.as<int32_t>(), s, up_ptr, up_col));
    MCE_CUDA(cudaMemsetAsync(key, 0, (size_t)n * sizeof(int64_t), s));
    MCE_LAUNCH(k_triangles, grid_for((int64_t)n * 32, 256), 256, 0, s, up_ptr.as<int32_t>(), up_col.as<int32_t>(), n,
               reinterpret_cast<unsigned long long *>(key));
    return MCE_OK;
}

mce_status vertex_key(const mce_graph *g, int32_t kind, cudaStream_t s, int64_t *key) {
    if (g->n == 0) return MCE_OK;
    switch (kind) {
        case MCE_RANK_DEGREE:
            MCE_LAUNCH(k_degree_key, grid_for(g->n, 256), 256, 0, s, g->row_ptr, g->n, key);
            return MCE_OK;
        case MCE_RANK_DEGEN:
            return core_numbers(g, s, key);
        case MCE_RANK_TRIANGLE:
            return triangle_counts(g, s, key);
        default:
            g_last_error = "vertex_key: unknown kind";
            return MCE_EINVAL;
    }
}

int32_t vertex_key_bits(const mce_graph *g, int32_t kind) {
    const uint64_t m = (uint64_t)(g->nnz / 2);
    if (kind == MCE_RANK_DEGEN) {   // a k-core has at least k (k + 1) / 2 edges
        int32_t b = 1;
        while (b < 31 && ((1ULL << b) * (1ULL << b)) <= 2 * m) ++b;
        return b;
    }
    if (kind == MCE_RANK_TRIANGLE) return bits_for(m);   // each triangle at v has its own edge opposite v
    const uint64_t d = g->n > 0 ? (uint64_t)(g->n - 1) : 0;
    return bits_for(d < m ? d : m);
}

mce_status rank_from_key_i64(const int64_t *key, int32_t n, int32_t id_bits, int32_t key_bits, cudaStream_t s,
                             int32_t *rank) {
    if (n == 0) return MCE_OK;
    DevBuf keys, tmp;
    MCE_TRY(keys.alloc((size_t)n * sizeof(uint64_t), s));
    MCE_TRY(tmp.alloc((size_t)n * sizeof(uint64_t), s));
    if (key_bits + id_bits > 64) {
        g_last_error = "rank_from_key: key too large";
        return MCE_EINVAL;
    }
    MCE_LAUNCH(k_rank_keys_i64, grid_for(n, 256), 256, 0, s, key, n, id_bits, keys.as<uint64_t>());
    MCE_TRY(radix_sort_u64(keys.as<uint64_t>(), tmp.as<uint64_t>(), n, id_bits, id_bits + key_bits, s));
    MCE_LAUNCH(k_scatter_rank, grid_for(n, 256), 256, 0, s, keys.as<uint64_t>(), n, id_bits, rank);
    return MCE_OK;
}

mce_status rank_from_key_f32(const float *key, int32_t n, int32_t id_bits, cudaStream_t s, int32_t *rank) {
    if (n == 0) return MCE_OK;
    DevBuf keys, tmp;
    MCE_TRY(keys.alloc((size_t)n * sizeof(uint64_t), s));
    MCE_TRY(tmp.alloc((size_t)n * sizeof(uint64_t), s));
    MCE_LAUNCH(k_rank_keys_f32, grid_for(n, 256), 256, 0, s, key, n, id_bits, keys.as<uint64_t>());
    MCE_TRY(radix_sort_u64(keys.as<uint64_t>(), tmp.as<uint64_t>(), n, id_bits, 32 + id_bits, s));
    MCE_LAUNCH(k_scatter_rank, grid_for(n, 256), 256, 0, s, keys.as<uint64_t>(), n, id_bits, rank);
    return MCE_OK;
}

mce_status build_up_lists(const mce_graph *g, const int32_t *rank, cudaStream_t s, DevBuf &up_ptr, DevBuf &up_col) {
    const int32_t n = g->n;
    const int64_t nnz = g->nnz;
    MCE_TRY(up_ptr.alloc(((size_t)n + 1) * sizeof(int32_t), s));
    // an edge has one end above the other at most: half the entries
    MCE_TRY(up_col.alloc(((size_t)nnz / 2 + 4) * sizeof(int32_t), s));
    if (n == 0 || nnz == 0) {
        MCE_CUDA(cudaMemsetAsync(up_ptr.p, 0, ((size_t)n + 1) * sizeof(int32_t), s));
        return MCE_OK;
    }
    // one warp a segment, all resident at once, and no fewer than 128 entries
    // (measured on GB300: shorter segments repeat the search of the first row)
    int64_t len = (nnz / ((int64_t)num_sms() * 64) + 32) & ~int64_t(31);
    if (len < 128) len = 128;
    const int64_t nseg = (nnz + len - 1) / len;
    DevBuf bits, seg;
    MCE_TRY(bits.alloc((size_t)(nnz / 32 + 1) * sizeof(uint32_t), s));
    MCE_TRY(seg.alloc((size_t)(nseg + 1) * sizeof(int32_t), s));
    const unsigned blocks = (unsigned)((nseg + 7) / 8);
    const bool sparse = n > nnz;
    const auto flags = sparse ? k_up_flags<true> : k_up_flags<false>;
    const auto fill = sparse ? k_up_fill<true> : k_up_fill<false>;
    MCE_LAUNCH(flags, blocks, 256, 0, s, g->row_ptr, g->col, rank, n,
               (int32_t)nnz, (int32_t)len, bits.as<uint32_t>(), seg.as<int32_t>(), up_ptr.as<int32_t>());
    MCE_TRY(exclusive_scan_i32(seg.as<int32_t>(), seg.as<int32_t>(), nseg, s));
    MCE_LAUNCH(fill, sparse ? blocks_for_rows((int64_t)n + 1, blocks) : blocks, 256, 0, s,
               g->row_ptr, g->col, bits.as<uint32_t>(), seg.as<int32_t>(), n, (int32_t)nnz, (int32_t)len,
               (int32_t)nseg, up_ptr.as<int32_t>(), up_col.as<int32_t>());
    return MCE_OK;
}

}  // namespace mce
