// Subproblem builds ahead of the search (ParMCE, Algorithm 5).
//
// The read-only part of every subproblem (bk.cuh: local ids, bounds, rows A,
// the bound-sorted fini list F0, one bitset over F0 per candidate) is built
// into the launch's build cache by k_build_rows before the search starts:
// vertices with 128 or more neighbours by a block each, heaviest first, the
// others by a warp each.  Local order: Γ+(v) (the candidates, ascending id),
// then the lower-ranked neighbours (ascending id).  Row A[x] marks the
// candidates adjacent to x.  Every candidate y adjacent to x has rank(y) >
// rank(v) > rank(x) when x is lower ranked, so y ∈ Γ+(x); for two candidates
// the edge lies in Γ+ of the lower-ranked one.  Looking up the elements of
// Γ+(x) in C for every local x therefore finds each needed adjacency exactly
// once.
//
// Bound: latency of the lookups, so they are spread over as many warps as an
// SM holds.  A warp flattens the Γ+ lists of 32 local vertices: its lanes take
// 32 consecutive elements of the concatenated lists at a time, and look each
// up in a hash table of C in shared memory.  One lane per list with binary
// searches, inside the search kernel at 16 warps an SM and one warp a hub,
// kept every warp busy for 23.6 ms on the 1.7M-vertex graph, and one hub's
// warp for 73 ms under the degeneracy rank; this kernel: 10.6 ms, hubs included.
#include "bk.cuh"

namespace mce {

namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr int kThreads = 512, kWarps = kThreads / 32;
// A warp builds subproblems of fewer than kWarpW local vertices (rows of 4
// words, in shared memory); the rest take a block.
constexpr int kWarpW = 128;
constexpr int kWarpS = 4;
constexpr int kWarpSlots = 256;
// Γ+ lists more than this many times longer than C (hubs) have the candidates
// searched in them instead of their elements looked up in C
constexpr int kReverse = 8;
constexpr int kFlat = 4;   // elements a lane looks up at a time

struct WarpSmem {
    int32_t key[kWarpSlots];
    uint32_t row[kWarpW * kWarpS];
    int32_t gid[kWarpW];
    int32_t bin[kWarpW + 4];
    uint8_t idx[kWarpSlots];
};

// block builds: hash table of up to kBlockC candidates (binary searches in
// memory above), and as many bins for the sort by bound
constexpr int kBlockC = 2048;
constexpr int kBlockSlots = 2 * kBlockC;
struct BlockSmem {
    int32_t key[kBlockSlots];
    int32_t bin[kBlockC];
    uint16_t idx[kBlockSlots];
};

union BuildSmem {
    WarpSmem w[kWarps];
    BlockSmem b;
};

struct BuildParams {
    const int32_t *row_ptr, *col, *up_ptr, *up_col, *order;
    int32_t n_sub;
    uint32_t *cache;
    const long long *cache_off;
    const int32_t *big;                 // vertices for block builds, heavy ones first
    const unsigned long long *n_big;
    unsigned long long *next;           // next entry of big
    int32_t sm_limit;                   // as BkParams
    unsigned long long *claim, *left, *t_start;   // BUILD_CLAIM, BUILD_LEFT, BUILD_T_START
    uint64_t max_run_ns;
    // ring and control words of the search, set to their start values here
    unsigned long long *qseq, *ctl;
    int64_t qcap;
};

// parts of a built subproblem (the layout of ws_layout_split)
struct Parts {
    uint32_t *head, *A, *Cb;
    int32_t *gid, *bnd, *F0;
    int32_t w, c, wc, S;
};

__device__ __forceinline__ Parts parts_of(uint32_t *base, int32_t w, int32_t c) {
    Parts p;
    p.head = base;
    p.w = w;
    p.c = c;
    p.wc = (c + 31) >> 5;
    p.S = (int32_t)bk_row_stride(p.wc);
    p.gid = reinterpret_cast<int32_t *>(base + 32);
    p.bnd = p.gid + w;
    p.A = base + bk_align4(32 + 2 * (int64_t)w);
    p.F0 = reinterpret_cast<int32_t *>(p.A + (int64_t)w * p.S);
    p.Cb = reinterpret_cast<uint32_t *>(p.F0 + (w - c));
    return p;
}

__device__ __forceinline__ uint32_t slot_of(int32_t y, int shift) { return ((uint32_t)y * 0x9E3779B1u) >> shift; }

// The loops below run until a vote of the whole warp ends them and have no
// other exit.  With loops that each lane left by its own return, some runs lost
// bits of a row (one subproblem in some 10^5; R-MAT 12 under one random rank: 8 %
// of the runs); with these, 640 of 640 runs are right.  Why is open: lanes may
// leave a loop one by one before a shuffle that names all of them, and reading
// shows neither an unordered access nor a vote that some lanes miss.

// table of 2^(32 - shift) slots, at most half full: j[u] = index of y[u], or
// -1 (also for y[u] = -1); the whole warp
template <class I>
__device__ __forceinline__ void find(const int32_t *key, const I *idx, int shift, uint32_t mask,
                                     const int32_t (&y)[kFlat], int (&j)[kFlat]) {
    uint32_t s[kFlat];
    bool open[kFlat], any = false;
#pragma unroll
    for (int u = 0; u < kFlat; ++u) {
        s[u] = slot_of(y[u], shift);
        j[u] = -1;
        open[u] = y[u] >= 0;
        any |= open[u];
    }
    while (__any_sync(FULL, any)) {
        any = false;
        int32_t k[kFlat];
#pragma unroll
        for (int u = 0; u < kFlat; ++u) k[u] = open[u] ? key[s[u]] : -1;
#pragma unroll
        for (int u = 0; u < kFlat; ++u) {
            if (open[u] && k[u] == y[u]) j[u] = idx[s[u]];
            open[u] = open[u] && k[u] >= 0 && k[u] != y[u];
            any |= open[u];
            s[u] = (s[u] + 1) & mask;
        }
    }
}

// y (-1 = none) with index i into the table; the whole warp
template <class I>
__device__ __forceinline__ void insert(int32_t *key, I *idx, int shift, uint32_t mask, int32_t y, int i) {
    uint32_t s = slot_of(y, shift);
    bool open = y >= 0;
    while (__any_sync(FULL, open)) {
        if (open && atomicCAS(&key[s], -1, y) == -1) {
            idx[s] = (I)i;
            open = false;
        }
        s = (s + 1) & mask;
    }
}

// position of y in sorted g[0..n), or -1 (n = 0 for a lane without a search);
// the whole warp
__device__ __forceinline__ int search(const int32_t *g, int n, int32_t y) {
    int lo = 0, hi = n;
    while (__any_sync(FULL, lo < hi)) {
        const int mid = (lo + hi) >> 1;
        const bool less = lo < hi && g[mid] < y;
        if (less) lo = mid + 1;
        else if (lo < hi) hi = mid;
    }
    return lo < n && g[lo] == y ? lo : -1;
}

// For the 32 local vertices whose global ids the lanes hold (gx, -1 = none;
// lane l has local id x0 + l): hit(x, j) for every candidate j in Γ+(x).
// lookup(y, j): candidate indices of the y[u], or -1; cand(j) = global id of candidate j.
template <class Lookup, class Cand, class Hit>
__device__ __forceinline__ void flat_lists(const BuildParams &P, int32_t gx, int x0, int c, int lane, Lookup lookup,
                                           Cand cand, Hit hit) {
    int32_t e0 = 0, d = 0;
    if (gx >= 0) {
        e0 = P.up_ptr[gx];
        d = P.up_ptr[gx + 1] - e0;
    }
    const bool rev = d > kReverse * c + 32;
    const int32_t items = rev ? c : d;
    int32_t end = items;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(FULL, end, o);
        if (lane >= o) end += y;
    }
    const int32_t total = __shfl_sync(FULL, end, 31);
    const uint32_t revs = __ballot_sync(FULL, rev);
    const int32_t from = e0 - (end - items);   // list start minus the items before it
    // kFlat steps at a time: their loads are in flight together
    for (int32_t t0 = 0; t0 < total; t0 += 32 * kFlat) {
        int own[kFlat];
        int32_t at[kFlat], y[kFlat];
#pragma unroll
        for (int u = 0; u < kFlat; ++u) {
            const int32_t t = t0 + 32 * u + lane;
            // owner: the number of lanes whose items end at or before t
            int o = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (__shfl_sync(FULL, end, o + step - 1) <= t) o += step;
            own[u] = o;
            at[u] = __shfl_sync(FULL, from, o) + t;
            y[u] = t < total && !((revs >> o) & 1u) ? P.up_col[at[u]] : -1;
        }
        int j[kFlat];
        lookup(y, j);
#pragma unroll
        for (int u = 0; u < kFlat; ++u) {
            if (revs) {
                const int32_t s0 = __shfl_sync(FULL, e0, own[u]), dd = __shfl_sync(FULL, d, own[u]);
                const bool mine = t0 + 32 * u + lane < total && ((revs >> own[u]) & 1u);
                const int q = mine ? at[u] - s0 : 0;
                if (search(P.up_col + s0, mine ? dd : 0, cand(q)) >= 0) j[u] = q;
            }
            if (j[u] >= 0) hit(x0 + own[u], j[u]);
        }
    }
}

// Cb of one block of 32 F0 positions (lane l's vertex has row `row`, null past
// the end): word pb of candidate q's bitset = the lanes whose row holds q
__device__ __forceinline__ void transpose_rows(const Parts &p, const uint32_t *row, int pb, int Wf0, int lane) {
    for (int k = 0; k < p.wc; ++k) {
        const uint32_t m = row ? row[k] : 0u;
        uint32_t mine = 0u;
        for (uint32_t u = __reduce_or_sync(FULL, m); u; u &= u - 1u) {
            const int b = __ffs(u) - 1;
            const uint32_t w = __ballot_sync(FULL, (m >> b) & 1u);
            if (lane == b) mine = w;
        }
        const int q = (k << 5) + lane;
        if (q < p.c) p.Cb[(int64_t)q * Wf0 + pb] = mine;
    }
}

// exclusive scan of bin[0..n) from the top down, one warp: bin[b] = entries in larger bins
__device__ __forceinline__ void scan_down(int32_t *bin, int n, int lane) {
    int32_t run = 0;
    for (int top = n - 1; top >= 0; top -= 32) {
        const int b = top - lane;
        const int32_t h = b >= 0 ? bin[b] : 0;
        int32_t incl = h;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (b >= 0) bin[b] = run + incl - h;
        run += __shfl_sync(FULL, incl, 31);
    }
}

__device__ void build_by_warp(const BuildParams &P, WarpSmem &m, const Parts &p, int32_t v, int lane) {
    const int32_t r0 = P.row_ptr[v], u0 = P.up_ptr[v];
    const int w = p.w, c = p.c;
    // slots: the power of two from 2c up, at least 32
    const int bits = c <= 16 ? 5 : 33 - __clz(c - 1);
    const int shift = 32 - bits;
    const uint32_t mask = (1u << bits) - 1u;
    for (int s = lane; s <= (int)mask; s += 32) m.key[s] = -1;
    for (int k = lane; k < w; k += 32) *reinterpret_cast<uint4 *>(m.row + k * kWarpS) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    for (int i0 = 0; i0 < c; i0 += 32) {
        const int i = i0 + lane;
        const int32_t y = i < c ? P.up_col[u0 + i] : -1;
        if (i < c) m.gid[i] = y;
        insert(m.key, m.idx, shift, mask, y, i);
    }
    __syncwarp();
    auto lookup = [&](const int32_t (&y)[kFlat], int (&j)[kFlat]) { find(m.key, m.idx, shift, mask, y, j); };
    // the other neighbours rank below v
    int out = c;
    for (int b0 = 0; b0 < w; b0 += 32 * kFlat) {
        int32_t x[kFlat];
        int j[kFlat];
#pragma unroll
        for (int u = 0; u < kFlat; ++u) {
            const int k = b0 + 32 * u + lane;
            x[u] = k < w ? P.col[r0 + k] : -1;
        }
        lookup(x, j);
#pragma unroll
        for (int u = 0; u < kFlat; ++u) {
            const bool low = x[u] >= 0 && j[u] < 0;
            const uint32_t b = __ballot_sync(FULL, low);
            if (low) m.gid[out + __popc(b & lanemask_lt())] = x[u];
            out += __popc(b);
        }
    }
    __syncwarp();
    for (int x0 = 0; x0 < w; x0 += 32) {
        const int32_t gx = x0 + lane < w ? m.gid[x0 + lane] : -1;
        if (gx >= 0) p.gid[x0 + lane] = gx;
        flat_lists(
            P, gx, x0, c, lane, lookup, [&](int j) { return m.gid[j]; },
            [&](int x, int j) {
                atomicOr(&m.row[x * kWarpS + (j >> 5)], 1u << (j & 31));
                if (x < c) atomicOr(&m.row[j * kWarpS + (x >> 5)], 1u << (x & 31));
            });
    }
    for (int b = lane; b < c; b += 32) m.bin[b] = 0;
    __syncwarp();
    // rows out, bounds, and the lower-ranked vertices that touch a candidate by bound
    int f = 0;
    for (int x0 = 0; x0 < w; x0 += 32) {
        const int x = x0 + lane;
        int bnd = 0;
        if (x < w) {
            const uint4 r = *reinterpret_cast<const uint4 *>(m.row + x * kWarpS);
            *reinterpret_cast<uint4 *>(p.A + x * kWarpS) = r;
            bnd = __popc(r.x) + __popc(r.y) + __popc(r.z) + __popc(r.w);
            p.bnd[x] = bnd;
        }
        const bool kept = x >= c && bnd > 0;
        if (kept) atomicAdd(&m.bin[bnd - 1], 1);
        f += __popc(__ballot_sync(FULL, kept));
    }
    __syncwarp();
    if (f) {
        scan_down(m.bin, c, lane);
        __syncwarp();
        // F0 in the table's place, which is not needed any more
        for (int x = c + lane; x < w; x += 32) {
            const uint4 r = *reinterpret_cast<const uint4 *>(m.row + x * kWarpS);
            const int bnd = __popc(r.x) + __popc(r.y) + __popc(r.z) + __popc(r.w);
            if (bnd) {
                const int at = atomicAdd(&m.bin[bnd - 1], 1);
                m.key[at] = x;
                p.F0[at] = x;
            }
        }
        __syncwarp();
        const int Wf0 = (f + 31) >> 5;
        for (int pb = 0; pb < Wf0; ++pb) {
            const int pos = (pb << 5) + lane;
            transpose_rows(p, pos < f ? m.row + m.key[pos] * kWarpS : nullptr, pb, Wf0, lane);
        }
    }
    if (lane == 0) {
        p.head[0] = (uint32_t)w;
        p.head[1] = (uint32_t)f;
    }
    __syncwarp();
}

__device__ void build_by_block(const BuildParams &P, BlockSmem &m, const Parts &p, int32_t v, int32_t *red) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int32_t r0 = P.row_ptr[v], u0 = P.up_ptr[v];
    const int w = p.w, c = p.c;
    const bool table = c <= kBlockC;
    const int bits = c <= 16 ? 5 : 33 - __clz(c - 1);
    const int shift = 32 - bits;
    const uint32_t mask = (1u << bits) - 1u;
    if (table)
        for (int s = t; s <= (int)mask; s += kThreads) m.key[s] = -1;
    __syncthreads();
    const int32_t *cl = P.up_col + u0;
    for (int i0 = warp * 32; i0 < c; i0 += kThreads) {
        const int i = i0 + lane;
        const int32_t y = i < c ? cl[i] : -1;
        if (i < c) p.gid[i] = y;
        if (table) insert(m.key, m.idx, shift, mask, y, i);
    }
    uint4 *rows = reinterpret_cast<uint4 *>(p.A);
    for (int64_t k = t; k < (int64_t)w * (p.S >> 2); k += kThreads) rows[k] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    auto lookup = [&](const int32_t (&y)[kFlat], int (&j)[kFlat]) {
        if (table) {
            find(m.key, m.idx, shift, mask, y, j);
        } else {
#pragma unroll
            for (int u = 0; u < kFlat; ++u) j[u] = search(cl, y[u] >= 0 ? c : 0, y[u]);
        }
    };
    // lower-ranked neighbours, in order
    int out = c;
    for (int b0 = 0; b0 < w; b0 += kThreads) {
        const int32_t x = b0 + t < w ? P.col[r0 + b0 + t] : -1;
        int32_t y[kFlat] = {x, -1, -1, -1};
        int j[kFlat];
        lookup(y, j);
        const bool low = x >= 0 && j[0] < 0;
        const uint32_t b = __ballot_sync(FULL, low);
        if (lane == 0) red[warp] = __popc(b);
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int k = 0; k < kWarps; ++k) {
            const int r = red[k];
            before += k < warp ? r : 0;
            all += r;
        }
        if (low) p.gid[out + before + __popc(b & lanemask_lt())] = x;
        out += all;
        __syncthreads();
    }
    // lists of 32 local vertices a warp at a time, fewer where that leaves warps
    // without any (bipartite graphs of degree 200, nine of sixteen idle: 22.3 ms,
    // now 15.7)
    const int each = w >= kThreads ? 32 : (w + kWarps - 1) / kWarps;
    for (int x0 = warp * each; x0 < w; x0 += kWarps * each)
        flat_lists(
            P, lane < each && x0 + lane < w ? p.gid[x0 + lane] : -1, x0, c, lane, lookup, [&](int j) { return cl[j]; },
            [&](int x, int j) {
                atomicOr(&p.A[(int64_t)x * p.S + (j >> 5)], 1u << (j & 31));
                if (x < c) atomicOr(&p.A[(int64_t)j * p.S + (x >> 5)], 1u << (x & 31));
            });
    // bounds; bins of the sort by bound in shared memory, or where Cb will be
    // (c words at least: it has one for each candidate as soon as w > c)
    int32_t *bin = table ? m.bin : reinterpret_cast<int32_t *>(p.Cb);
    if (w > c)
        for (int b = t; b < c; b += kThreads) bin[b] = 0;
    __syncthreads();
    int kept = 0;
    for (int x = t; x < w; x += kThreads) {
        const uint4 *row = reinterpret_cast<const uint4 *>(p.A + (int64_t)x * p.S);
        int bnd = 0;
        for (int g = 0; g < (p.S >> 2); ++g) {
            const uint4 r = __ldcg(row + g);   // written by atomics of other threads: read through L2
            bnd += __popc(r.x) + __popc(r.y) + __popc(r.z) + __popc(r.w);
        }
        p.bnd[x] = bnd;
        if (x >= c && bnd > 0) {
            ++kept;
            atomicAdd(&bin[bnd - 1], 1);
        }
    }
    kept = __reduce_add_sync(FULL, kept);
    if (lane == 0) red[warp] = kept;
    __syncthreads();
    int f = 0;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) f += red[k];
    if (f) {   // the same for every thread
        if (warp == 0) scan_down(bin, c, lane);
        __syncthreads();
        for (int x = c + t; x < w; x += kThreads) {
            const int bnd = p.bnd[x];   // this thread's own store
            if (bnd) p.F0[atomicAdd(&bin[bnd - 1], 1)] = x;
        }
        __syncthreads();
        const int Wf0 = (f + 31) >> 5;
        for (int pb = warp; pb < Wf0; pb += kWarps) {
            const int pos = (pb << 5) + lane;
            transpose_rows(p, pos < f ? p.A + (int64_t)p.F0[pos] * p.S : nullptr, pb, Wf0, lane);
        }
    }
    if (t == 0) {
        p.head[0] = (uint32_t)w;
        p.head[1] = (uint32_t)f;
    }
    __syncthreads();
}

// LIMITED: with sm_limit (an instance of its own, calls without it make no claims)
template <bool LIMITED> __global__ void __launch_bounds__(kThreads, 2) k_build_rows(BuildParams P) {
    extern __shared__ __align__(16) unsigned char build_smem[];
    BuildSmem &m = *reinterpret_cast<BuildSmem *>(build_smem);
    __shared__ int32_t red[kWarps];
    __shared__ int32_t claim;
    const uint64_t t0 = globaltimer_ns();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tid = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    for (int64_t i = tid; i < P.qcap; i += (int64_t)gridDim.x * kThreads) P.qseq[i] = (unsigned long long)i;
    if (tid < CTL_WORDS && tid != CTL_ABORT) P.ctl[tid] = tid == CTL_PENDING ? (unsigned long long)P.n_sub : 0ULL;
    if (tid == 0) *P.t_start = t0;
    // one thread: the time limit has passed (looked at before each build); the
    // search then finds the abort word set and leaves before it reads a build
    auto late = [&]() {
        if (globaltimer_ns() - t0 <= P.max_run_ns) return false;
        atomicOr(&P.ctl[CTL_ABORT], 2ULL);
        return true;
    };
    // sm_limit (scaling measurements): only the blocks placed on the first SMs
    // build, as in the search.  A block elsewhere leaves, unless all others have
    // left: then nobody else is there to take what remains.
    if (LIMITED) {
        uint32_t smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        if (threadIdx.x == 0) claim = (int32_t)smid < P.sm_limit || atomicAdd(P.left, 1ULL) + 1 == gridDim.x;
        __syncthreads();
        const bool stays = claim != 0;
        __syncthreads();
        if (!stays) return;
    }
    const int32_t n_big = (int32_t)*P.n_big;
    for (;;) {
        if (threadIdx.x == 0) claim = late() ? n_big : (int32_t)atomicAdd(P.next, 1ULL);
        __syncthreads();
        const int32_t i = claim;
        __syncthreads();
        if (i >= n_big) break;
        const int32_t v = P.big[i];
        build_by_block(P, m.b, parts_of(P.cache + P.cache_off[v], P.row_ptr[v + 1] - P.row_ptr[v],
                                        P.up_ptr[v + 1] - P.up_ptr[v]),
                       v, red);
    }
    // ---- warp builds, dealt out evenly; claimed one by one where blocks are missing
    const int64_t nwarp = (int64_t)gridDim.x * kWarps;
    auto claimed = [&]() {
        unsigned long long k = 0;
        if (lane == 0) k = atomicAdd(P.claim, 1ULL);
        return (int64_t)__shfl_sync(FULL, k, 0);
    };
    for (int64_t i = LIMITED ? claimed() : (int64_t)blockIdx.x + (int64_t)warp * gridDim.x; i < P.n_sub;
         i = LIMITED ? claimed() : i + nwarp) {
        const int32_t v = P.order[i];
        const int32_t w = P.row_ptr[v + 1] - P.row_ptr[v];
        const long long off = P.cache_off[v];
        if (w >= kWarpW || off < 0) continue;
        if (__shfl_sync(FULL, lane == 0 && late(), 0)) break;
        build_by_warp(P, m.w[warp], parts_of(P.cache + off, w, P.up_ptr[v + 1] - P.up_ptr[v]), v, lane);
    }
    if (LIMITED) {
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(P.left, 1ULL);
    }
}

// cache_off[v] of every scheduled subproblem: room in the build cache in
// processing order (blocks may swap), -1 once it is full; and the list of
// those that a block builds, in about the same order
__global__ void k_build_offsets(const int32_t *order, int32_t n_sub, const int32_t *row_ptr, const int32_t *up_ptr,
                                int64_t cap, unsigned long long *top, long long *cache_off, int32_t *big,
                                unsigned long long *n_big) {
    __shared__ unsigned long long ws[32], base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t v = i < n_sub ? order[i] : -1;
    unsigned long long sw = 0;
    int32_t w = 0;
    if (v >= 0) {
        w = row_ptr[v + 1] - row_ptr[v];
        sw = (unsigned long long)bk_shared_words(w, up_ptr[v + 1] - up_ptr[v]);
    }
    unsigned long long incl = sw;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long run = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            const unsigned long long x = ws[k];
            ws[k] = run;
            run += x;
        }
        base = atomicAdd(top, run);
    }
    __syncthreads();
    const unsigned long long off = base + ws[warp] + incl - sw;
    const bool fits = v >= 0 && off + sw <= (unsigned long long)cap;
    if (v >= 0) cache_off[v] = fits ? (long long)off : -1;
    const uint32_t b = __ballot_sync(FULL, fits && w >= kWarpW);
    if (b) {
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(n_big, (unsigned long long)__popc(b));
        at = __shfl_sync(FULL, at, 0);
        if ((b >> lane) & 1u) big[at + __popc(b & lanemask_lt())] = v;
    }
}

}  // namespace

mce_status build_prepare() {
    // above the 48 KB default: opted into once, outside any stream capture
    static std::atomic<bool> done{false};
    if (done.load()) return MCE_OK;
    for (auto k : {k_build_rows<false>, k_build_rows<true>})
        MCE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BuildSmem)));
    done.store(true);
    return MCE_OK;
}

mce_status launch_build_layout(const BkParams &P, cudaStream_t s) {
    MCE_LAUNCH(k_build_offsets, (unsigned)((P.n_sub + 255) / 256), 256, 0, s, P.order, P.n_sub, P.row_ptr, P.up_ptr,
               P.cache_words, P.build_ctl + BUILD_TOP, P.cache_off, P.build_big, P.build_ctl + BUILD_BIG);
    return MCE_OK;
}

mce_status launch_build_rows(const BkParams &P, cudaStream_t s) {
    MCE_TRY(build_prepare());
    BuildParams B{};
    B.row_ptr = P.row_ptr;
    B.col = P.col;
    B.up_ptr = P.up_ptr;
    B.up_col = P.up_col;
    B.order = P.order;
    B.n_sub = P.n_sub;
    B.cache = P.cache;
    B.cache_off = P.cache_off;
    B.big = P.build_big;
    B.n_big = P.build_ctl + BUILD_BIG;
    B.next = P.build_ctl + BUILD_NEXT;
    B.sm_limit = P.sm_limit;
    B.claim = P.build_ctl + BUILD_CLAIM;
    B.left = P.build_ctl + BUILD_LEFT;
    B.t_start = P.build_ctl + BUILD_T_START;
    B.max_run_ns = P.max_run_ns;
    B.qseq = P.qseq;
    B.qcap = P.qcap;
    B.ctl = P.ctl;
    const int64_t blocks = ((int64_t)P.n_sub + kWarps - 1) / kWarps, most = (int64_t)num_sms() * 2;
    if (P.sm_limit > 0)   // a full grid, so that the first SMs get their blocks
        MCE_LAUNCH(k_build_rows<true>, (unsigned)most, kThreads, sizeof(BuildSmem), s, B);
    else
        MCE_LAUNCH(k_build_rows<false>, (unsigned)(blocks < most ? blocks : most), kThreads, sizeof(BuildSmem), s, B);
    return MCE_OK;
}

}  // namespace mce
