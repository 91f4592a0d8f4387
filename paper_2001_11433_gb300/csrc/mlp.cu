// Learned cost model for the vertex rank.
//
// Section 4.2 ranks vertices by a cheap estimate of the cost of their
// subproblem, giving costlier subproblems a higher rank so that they keep a
// smaller share of the cliques (the load-balancing idea taken from PECO).
// Here the estimate is learned: an MLP 8 -> H -> H -> 1 (ReLU) over
// per-vertex features predicts log(1 + search-tree nodes) of the vertex's
// subproblem, trained on node counts recorded by the search itself.
//
//   k_features    per-vertex features (eight lanes a vertex, a block a hub)
//   k_mlp_fwd, k_mlp_fwd_bf16   inference, FP32 or BF16 weights and activations
//                 (FP32 sums)
//   k_mlp_grad    forward + backward of the MSE loss over tiles of rows as
//                 register-tiled products; weight gradients summed in registers
//   k_adam        Adam update
#include <cuda_bf16.h>
#include <string.h>

#include <vector>

#include "mce_host.h"

struct mce_model {
    int32_t H = 64;
    int32_t feature_kind = 0;   // MCE_FEATURES_* the model reads
    int64_t np = 0;
    float *w = nullptr;       // parameters, device
    float *m = nullptr;       // Adam first moment
    float *v = nullptr;       // Adam second moment
    float *g = nullptr;       // gradient
    int64_t step = 0;
};

namespace mce {

namespace {

constexpr int kFeat = 8;
constexpr int kMaxH = 64;

struct Off {
    int64_t W1, b1, W2, b2, w3, b3, n;
};

__host__ __device__ inline Off offsets(int H) {
    Off o;
    o.W1 = 0;
    o.b1 = o.W1 + (int64_t)H * kFeat;
    o.W2 = o.b1 + H;
    o.b2 = o.W2 + (int64_t)H * H;
    o.w3 = o.b2 + H;
    o.b3 = o.w3 + H;
    o.n = o.b3 + 1;
    return o;
}

// ------------------------------------------------------------------ features

// Degree statistics of a vertex's neighbours.  A neighbour w ranks higher than
// v by degree when (d(w), w) > (d(v), v).
struct NbrSums {
    float s = 0.f, s2 = 0.f, mx = 0.f, mins = 0.f, dsum = 0.f;
    int hi = 0;
    template <bool LIGHT>
    __device__ __forceinline__ void add(const int32_t *__restrict__ row_ptr, int32_t w, int32_t v, int32_t d) {
        const int32_t dw = row_ptr[w + 1] - row_ptr[w];
        const float x = log1pf((float)dw);
        s += x;
        s2 += x * x;
        mx = fmaxf(mx, x);
        if (LIGHT) {
            mins += (float)min(dw, d);
            dsum += (float)dw;
            hi += (dw > d || (dw == d && w > v)) ? 1 : 0;
        }
    }
    // sum over the lanes that differ in the bits of `from`, `from` / 2, ... 1
    template <bool LIGHT> __device__ __forceinline__ void reduce(int from) {
        for (int o = from; o; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (LIGHT) {
                mins += __shfl_xor_sync(0xffffffffu, mins, o);
                dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
                hi += __shfl_xor_sync(0xffffffffu, hi, o);
            }
        }
    }
};

struct FeatParams {
    const int32_t *row_ptr, *col;
    const int64_t *core, *tri;   // MCE_FEATURES_FULL
    const int32_t *up_ptr;       //
    int32_t n;
    float *feat;
};

// feature k of vertex v from its reduced sums
template <bool LIGHT>
__device__ __forceinline__ float feature(const FeatParams &P, int64_t v, int32_t d, const NbrSums &a, int k) {
    const float mean = d ? a.s / d : 0.f;
    const float var = d ? fmaxf(a.s2 / d - mean * mean, 0.f) : 0.f;
    if (LIGHT) {   // MCE_FEATURES_LIGHT: one pass, degrees only
        switch (k) {
            case 0: return log1pf((float)d);
            case 1: return mean;
            case 2: return sqrtf(var);
            case 3: return a.mx;
            case 4: return log1pf((float)a.hi);
            case 5: return log1pf(a.mins * 0.5f);
            case 6: return d ? (float)a.hi / (float)d : 0.f;
            default: return log1pf(a.dsum);
        }
    }
    switch (k) {
        case 0: return log1pf((float)d);
        case 1: return (float)P.core[v];
        case 2: return log1pf((float)P.tri[v]);
        case 3: return mean;
        case 4: return sqrtf(var);
        case 5: return a.mx;
        case 6: return log1pf((float)(P.up_ptr[v + 1] - P.up_ptr[v]));
        default: return d >= 2 ? (float)(2.0 * (double)P.tri[v] / ((double)d * (d - 1))) : 0.f;
    }
}

// Eight lanes a vertex, one feature a lane at the end; vertices of more than
// kFeatHub neighbours by a block each, before the others: block b of an odd number
// looks for them among b, b + blocks, b + 2 blocks, ..., so that hubs with close
// ids, or ids a power of two apart as in R-MAT graphs, are spread over the blocks.
// Bound: instructions (54 % of their throughput at 400,000 vertices) and the
// latency of two gathers a neighbour through L1 and L2.  A warp per vertex left
// most lanes of short rows idle and took 0.99 ms on the 1.7M-vertex graph, waiting
// for the hubs; a call with this takes 0.29 ms.  (A list of the hubs in memory for
// a second kernel made that 0.36 ms, and a call on a few thousand vertices 9 us
// longer.)
constexpr int kFeatHub = 512;
constexpr int kFeatThreads = 256, kFeatWarps = kFeatThreads / 32;

template <bool LIGHT> __global__ void __launch_bounds__(kFeatThreads) k_features(FeatParams P) {
    __shared__ __align__(8) unsigned char raw[kFeatWarps * sizeof(NbrSums)];
    __shared__ int32_t hubs[kFeatThreads], n_hubs;
    NbrSums *part = reinterpret_cast<NbrSums *>(raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = lane & 7;
    const int64_t looking = gridDim.x - ((gridDim.x & 1u) ? 0 : 1);
    // the same number of rounds for every thread of the block
    for (int64_t v0 = blockIdx.x < looking ? blockIdx.x : P.n; v0 < P.n; v0 += looking * kFeatThreads) {
        if (threadIdx.x == 0) n_hubs = 0;
        __syncthreads();
        const int64_t mine = v0 + threadIdx.x * looking;
        if (mine < P.n && P.row_ptr[mine + 1] - P.row_ptr[mine] > kFeatHub)
            hubs[atomicAdd(&n_hubs, 1)] = (int32_t)mine;
        __syncthreads();
        const int nh = n_hubs;
        for (int h = 0; h < nh; ++h) {
            const int32_t v = hubs[h];
            const int32_t e0 = P.row_ptr[v], d = P.row_ptr[v + 1] - e0;
            NbrSums a;
#pragma unroll 8
            for (int32_t e = threadIdx.x; e < d; e += kFeatThreads) a.add<LIGHT>(P.row_ptr, P.col[e0 + e], v, d);
            __syncwarp();
            a.reduce<LIGHT>(16);
            if (lane == 0) part[warp] = a;
            __syncthreads();
            if (warp == 0) {
                a = lane < kFeatWarps ? part[lane] : NbrSums();
                a.reduce<LIGHT>(kFeatWarps / 2);
                if (lane < kFeat) P.feat[(int64_t)v * kFeat + lane] = feature<LIGHT>(P, v, d, a, lane);
            }
            __syncthreads();
        }
    }
    const int64_t g0 = ((int64_t)blockIdx.x * kFeatThreads + threadIdx.x) >> 3;
    const int64_t stride = ((int64_t)gridDim.x * kFeatThreads) >> 3;
    for (int64_t w0 = g0 - (lane >> 3); w0 < P.n; w0 += stride) {   // the same for the whole warp
        const int64_t v = w0 + (lane >> 3);
        int32_t e0 = 0, d = 0;
        if (v < P.n) {
            e0 = P.row_ptr[v];
            d = P.row_ptr[v + 1] - e0;
        }
        const bool hub = d > kFeatHub;
        NbrSums a;
        if (!hub) {
#pragma unroll 4
            for (int32_t e = k; e < d; e += 8) a.add<LIGHT>(P.row_ptr, P.col[e0 + e], (int32_t)v, d);
        }
        __syncwarp();
        a.reduce<LIGHT>(4);
        if (v < P.n && !hub) P.feat[v * kFeat + k] = feature<LIGHT>(P, v, d, a, k);
    }
}

// ------------------------------------------------------------------ MLP

// FP32 inference, one thread per row.  HC > 0 fixes the hidden width at
// compile time, so that the hidden activations stay in registers and the
// weight rows are read from shared memory four at a time (same operations in
// the same order as the generic path, HC = 0).
template <int HC>
__global__ void k_mlp_fwd(const float *__restrict__ wts, int H_rt, const float *__restrict__ feat, int32_t rows,
                          float *out) {
    extern __shared__ __align__(16) float sw[];
    const int H = HC > 0 ? HC : H_rt;
    const Off o = offsets(H);
    for (int64_t i = threadIdx.x; i < o.n; i += blockDim.x) sw[i] = wts[i];
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x) {
        float x[kFeat];
#pragma unroll
        for (int k = 0; k < kFeat; ++k) x[k] = feat[r * kFeat + k];
        float h1[kMaxH];
        float y = sw[o.b3];
        if constexpr (HC > 0) {
            static_assert(HC % 4 == 0 && HC <= kMaxH, "fixed hidden width");
            // weights are read per row, not held in registers across rows
            asm volatile("" ::: "memory");
#pragma unroll
            for (int j = 0; j < HC; ++j) {
                float a = sw[o.b1 + j];
#pragma unroll
                for (int k = 0; k < kFeat; ++k) a = fmaf(sw[o.W1 + j * kFeat + k], x[k], a);
                h1[j] = fmaxf(a, 0.f);
            }
#pragma unroll 1
            for (int j = 0; j < HC; ++j) {
                float a = sw[o.b2 + j];
                const float4 *wr = reinterpret_cast<const float4 *>(sw + o.W2 + j * HC);
#pragma unroll
                for (int i = 0; i < HC / 4; ++i) {
                    const float4 w = wr[i];
                    a = fmaf(w.x, h1[4 * i], a);
                    a = fmaf(w.y, h1[4 * i + 1], a);
                    a = fmaf(w.z, h1[4 * i + 2], a);
                    a = fmaf(w.w, h1[4 * i + 3], a);
                }
                y = fmaf(sw[o.w3 + j], fmaxf(a, 0.f), y);
            }
        } else {
#pragma unroll 4
            for (int j = 0; j < H; ++j) {
                float a = sw[o.b1 + j];
#pragma unroll
                for (int k = 0; k < kFeat; ++k) a = fmaf(sw[o.W1 + j * kFeat + k], x[k], a);
                h1[j] = fmaxf(a, 0.f);
            }
            for (int j = 0; j < H; ++j) {
                float a = sw[o.b2 + j];
                const float *wr = sw + o.W2 + (int64_t)j * H;
#pragma unroll 8
                for (int i = 0; i < H; ++i) a = fmaf(wr[i], h1[i], a);
                y = fmaf(sw[o.w3 + j], fmaxf(a, 0.f), y);
            }
        }
        out[r] = y;
    }
}

// two floats rounded to BF16, `lo` in the low half
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// D (16 rows x 8 columns) += A (16 x 8) B (8 x 8), BF16 operands, FP32 sums
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(b));
}

// D (16 x 8) += A (16 x 16) B (16 x 8)
__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// BF16 inference (BF16 weights, biases and activations, FP32 sums), hidden
// width H padded with zero weights to HP, a warp per 16 rows at a time.
// Bound: latency (12 warps an SM, as the weights fill their registers; at
// 400,000 rows a quarter of the issue slots, 0.5 TB/s).  Both layers run on warp-level matrix instructions because their
// accumulator fragments, rounded to BF16, are the next layer's operand
// fragments as they stand: the activations never leave registers, where a
// TMEM accumulator would be read back and staged again for an 8-deep and a
// 64-deep product.  All weight fragments stay in registers over the rows.
// One thread per row with the weights broadcast from shared memory took
// 0.49 ms for 1.7M rows at H = 64; this kernel takes 0.10 ms.
template <int HP>
__global__ void __launch_bounds__(128, 3) k_mlp_fwd_bf16(const float *__restrict__ wts, int H,
                                                         const float *__restrict__ feat, int32_t rows, float *out) {
    constexpr int NT = HP / 8, KS = HP / 16;
    __shared__ __align__(16) float sb1[HP], sb2[HP], sw3[HP];
    const Off o = offsets(H);
    auto rounded = [](float w) { return __bfloat162float(__float2bfloat16(w)); };
    for (int i = threadIdx.x; i < HP; i += blockDim.x) {
        sb1[i] = i < H ? rounded(wts[o.b1 + i]) : 0.f;
        sb2[i] = i < H ? rounded(wts[o.b2 + i]) : 0.f;
        sw3[i] = i < H ? rounded(wts[o.w3 + i]) : 0.f;
    }
    __syncthreads();
    const float b3 = rounded(wts[o.b3]);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint32_t f1[NT], f2[NT][KS][2];
    auto w1 = [&](int j, int k) { return j < H ? wts[o.W1 + j * kFeat + k] : 0.f; };
    auto w2 = [&](int j, int k) { return j < H && k < H ? wts[o.W2 + (int64_t)j * H + k] : 0.f; };
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int j = nt * 8 + g;
        f1[nt] = bf16_pair(w1(j, 2 * t), w1(j, 2 * t + 1));
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int k = ks * 16 + q * 8 + 2 * t;
                f2[nt][ks][q] = bf16_pair(w2(j, k), w2(j, k + 1));
            }
    }
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t tiles = ((int64_t)rows + 15) >> 4;
    float x[4];   // row g: features 2t, 2t + 1; row g + 8: the same
    auto load = [&](int64_t tile) {
        const int64_t ra = tile * 16 + g, rb = ra + 8;
        x[0] = ra < rows ? feat[ra * kFeat + 2 * t] : 0.f;
        x[1] = ra < rows ? feat[ra * kFeat + 2 * t + 1] : 0.f;
        x[2] = rb < rows ? feat[rb * kFeat + 2 * t] : 0.f;
        x[3] = rb < rows ? feat[rb * kFeat + 2 * t + 1] : 0.f;
    };
    if (warp < tiles) load(warp);
    for (int64_t tile = warp; tile < tiles; tile += nwarps) {
        const uint32_t a0 = bf16_pair(x[0], x[1]), a1 = bf16_pair(x[2], x[3]);
        if (tile + nwarps < tiles) load(tile + nwarps);   // in flight during this tile
        uint32_t h[KS][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float2 b = *reinterpret_cast<const float2 *>(sb1 + nt * 8 + 2 * t);
            float d[4] = {b.x, b.y, b.x, b.y};
            mma_k8(d, a0, a1, f1[nt]);
            h[nt >> 1][(nt & 1) * 2] = bf16_pair(fmaxf(d[0], 0.f), fmaxf(d[1], 0.f));
            h[nt >> 1][(nt & 1) * 2 + 1] = bf16_pair(fmaxf(d[2], 0.f), fmaxf(d[3], 0.f));
        }
        float ya = 0.f, yb = 0.f;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float2 b = *reinterpret_cast<const float2 *>(sb2 + nt * 8 + 2 * t);
            const float2 w = *reinterpret_cast<const float2 *>(sw3 + nt * 8 + 2 * t);
            float d[4] = {b.x, b.y, b.x, b.y};
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) mma_k16(d, h[ks], f2[nt][ks][0], f2[nt][ks][1]);
            const uint32_t ha = bf16_pair(fmaxf(d[0], 0.f), fmaxf(d[1], 0.f));
            const uint32_t hb = bf16_pair(fmaxf(d[2], 0.f), fmaxf(d[3], 0.f));
            ya = fmaf(w.x, __uint_as_float(ha << 16), ya);
            ya = fmaf(w.y, __uint_as_float(ha & 0xffff0000u), ya);
            yb = fmaf(w.x, __uint_as_float(hb << 16), yb);
            yb = fmaf(w.y, __uint_as_float(hb & 0xffff0000u), yb);
        }
        ya += __shfl_xor_sync(0xffffffffu, ya, 1);
        yb += __shfl_xor_sync(0xffffffffu, yb, 1);
        ya += __shfl_xor_sync(0xffffffffu, ya, 2);
        yb += __shfl_xor_sync(0xffffffffu, yb, 2);
        if (t == 0) {
            const int64_t ra = tile * 16 + g;
            if (ra < rows) out[ra] = ya + b3;
            if (ra + 8 < rows) out[ra + 8] = yb + b3;
        }
    }
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf).
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    return (f32x2)__float_as_uint(lo) | ((f32x2)__float_as_uint(hi) << 32);
}

__device__ __forceinline__ float lo2(f32x2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f32x2 v) { return __uint_as_float((uint32_t)(v >> 32)); }

// Gradient tile: kGradRows rows on kGradRows threads.  Matrices of the tile
// are stored column by column (element [c][row]) with kRowStride floats a
// column: 16-byte aligned columns that start 4 banks apart, so that eight
// lanes reading 16 bytes of eight neighbouring columns hit all banks once.
constexpr int kGradRows = 256;
constexpr int kRowStride = kGradRows + 4;

// Shared memory of k_mlp_grad (floats).  Weights are held as pairs (w, w),
// ready for fma2 against two rows.
template <int HP> struct GradSmem {
    static constexpr int W1d = 0;                               // [8][2 HP]   (w, w) of W1[c][k] at [k][2c]
    static constexpr int W2Td = W1d + kFeat * 2 * HP;           // [HP][2 HP]  W2[c][k] at [k][2c]
    static constexpr int W2d = W2Td + HP * 2 * HP;              // [HP][2 HP]  W2[k][c] at [k][2c]
    static constexpr int b1 = W2d + HP * 2 * HP;
    static constexpr int b2 = b1 + HP;
    static constexpr int w3 = b2 + HP;
    static constexpr int xT = w3 + HP;                          // [8][rows]
    static constexpr int h1T = xT + kFeat * kRowStride;         // [HP][rows]: h1, later dh1
    static constexpr int dT = h1T + HP * kRowStride;            // [HP][rows]: dh2
    static constexpr int part = dT + HP * kRowStride;           // [2][rows]: halves of y
    static constexpr int dy = part + 2 * kGradRows;             // [rows]
    static constexpr int n = dy + kGradRows;
    // resident blocks an SM: what the shared memory leaves room for
    static constexpr int blocks = HP <= 16 ? 4 : HP <= 32 ? 2 : 1;
};

// acc (8 rows as 4 pairs, NC columns) += A^T B over k < K: A[k][row] from
// `a` (this thread's rows), B[k][2c] as (b, b) pairs from `b` (its columns).
template <int NC, int V, int HP>
__device__ __forceinline__ void grad_mm(f32x2 (&acc)[4][NC], const float *a, const float *b, int K) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        f32x2 ar[4], br[NC];
        const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(a + k * kRowStride);
        const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(a + k * kRowStride + kGradRows / 2);
        ar[0] = a0.x;
        ar[1] = a0.y;
        ar[2] = a1.x;
        ar[3] = a1.y;
#pragma unroll
        for (int c = 0; c < NC; c += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(b + k * 2 * HP + 2 * ((c / V) * 8 * V + c % V));
            br[c] = t.x;
            br[c + 1] = t.y;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][c] = fma2(ar[p], br[c], acc[p][c]);
    }
}

// this thread's 8 rows of column c of a tile matrix
__device__ __forceinline__ void grad_put(float *col, const f32x2 (&v)[4]) {
    *reinterpret_cast<ulonglong2 *>(col) = make_ulonglong2(v[0], v[1]);
    *reinterpret_cast<ulonglong2 *>(col + kGradRows / 2) = make_ulonglong2(v[2], v[3]);
}

// Forward + backward over rows idx[r0 .. r0 + cnt) (or r0.. when idx is null),
// loss = (1/N) sum (y - t)^2, hidden width H padded with zero weights to HP.
// Bound: shared-memory reads (71 % of their throughput at 200,000 rows, H = 64)
// for FP32 multiply-adds (28,000 flops a row; 45 % of the instruction slots).
// Persistent blocks, one an SM (two up to HP = 32, four up to 16), take tiles of
// 256 rows; each layer, forward and backward, is a register-tiled product (8 rows
// x HP/8 columns a thread, 32 packed multiply-adds for six 16-byte shared-memory
// loads at HP = 64), and every weight gradient is summed over the block's rows in
// registers and added to memory once.  One
// thread per row with serial dot products (columns of one row in one bank)
// took 6.47 ms for 200,000 rows at H = 64; a call with this kernel takes
// 0.20 ms, 28 TFLOP/s.
template <int HP>
__global__ void __launch_bounds__(kGradRows, GradSmem<HP>::blocks) k_mlp_grad(const float *__restrict__ wts, int H,
                                                           const float *__restrict__ feat,
                                                           const float *__restrict__ label,
                                                           const int32_t *__restrict__ idx, int64_t r0, int64_t cnt,
                                                           float inv_n, float *grad, float *loss) {
    using S = GradSmem<HP>;
    constexpr int NC = HP / 8;             // columns a thread
    constexpr int V = NC < 4 ? NC : 4;     // consecutive ones among them
    constexpr int NJ = HP / 16;            // W2 gradient: NJ x NJ entries a thread
    constexpr int KT = HP / 32 > 0 ? HP / 32 : 1;   // W1 gradient: entries a thread
    extern __shared__ __align__(16) float sm[];
    const Off o = offsets(H);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = t; i < HP * HP; i += kGradRows) {
        const int j = i / HP, k = i % HP;
        const float w = j < H && k < H ? wts[o.W2 + (int64_t)j * H + k] : 0.f;
        *reinterpret_cast<float2 *>(sm + S::W2Td + k * 2 * HP + 2 * j) = make_float2(w, w);
        *reinterpret_cast<float2 *>(sm + S::W2d + j * 2 * HP + 2 * k) = make_float2(w, w);
    }
    for (int i = t; i < HP * kFeat; i += kGradRows) {
        const int j = i / kFeat, k = i % kFeat;
        const float w = j < H ? wts[o.W1 + i] : 0.f;
        *reinterpret_cast<float2 *>(sm + S::W1d + k * 2 * HP + 2 * j) = make_float2(w, w);
    }
    for (int i = t; i < HP; i += kGradRows) {
        sm[S::b1 + i] = i < H ? wts[o.b1 + i] : 0.f;
        sm[S::b2 + i] = i < H ? wts[o.b2 + i] : 0.f;
        sm[S::w3 + i] = i < H ? wts[o.w3 + i] : 0.f;
    }
    const float b3 = wts[o.b3];
    // rows 4 tr .. 4 tr + 3 and the same of the tile's second half; columns
    // (c / V) * 8 V + tc V + c % V
    const int tr = (warp & 3) * 8 + (lane & 7), tc = (warp >> 2) * 4 + (lane >> 3);
    auto column = [&](int c) { return (c / V) * 8 * V + tc * V + c % V; };
    // W2 gradient entries (tj + 16 a, ti + 16 b)
    const int tj = (warp & 1) * 8 + (lane & 7), ti = (warp >> 1) * 4 + (lane >> 3);
    // a warp whose columns, or W2 entries, are all padding has none to add up (for
    // widths of 12 and less)
    const bool cols = (warp >> 2) * 4 * V < H, entries = (warp & 1) * 8 < H && (warp >> 1) * 4 < H;
    f32x2 gW2[NJ][NJ], gW1[KT];
    float gb1[NC], gb2[NC], gw3[NC], gb3 = 0.f, gl = 0.f;
#pragma unroll
    for (int a = 0; a < NJ; ++a)
#pragma unroll
        for (int b = 0; b < NJ; ++b) gW2[a][b] = 0ULL;
#pragma unroll
    for (int a = 0; a < KT; ++a) gW1[a] = 0ULL;
#pragma unroll
    for (int c = 0; c < NC; ++c) gb1[c] = gb2[c] = gw3[c] = 0.f;
    const int64_t tiles = (cnt + kGradRows - 1) / kGradRows;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t rr = tile * kGradRows + t;
        const bool valid = rr < cnt;
        const int64_t row = valid ? (idx ? idx[r0 + rr] : r0 + rr) : 0;
#pragma unroll
        for (int k = 0; k < kFeat; ++k) sm[S::xT + k * kRowStride + t] = valid ? feat[row * kFeat + k] : 0.f;
        __syncthreads();
        f32x2 acc[4][NC];
        // ---- h1 = relu(W1 x + b1)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float b = sm[S::b1 + column(c)];
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][c] = pack2(b, b);
        }
        if (cols) grad_mm<NC, V, HP>(acc, sm + S::xT + tr * 4, sm + S::W1d + 2 * V * tc, kFeat);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            f32x2 v[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) v[p] = pack2(fmaxf(lo2(acc[p][c]), 0.f), fmaxf(hi2(acc[p][c]), 0.f));
            grad_put(sm + S::h1T + column(c) * kRowStride + tr * 4, v);
        }
        __syncthreads();
        // ---- h2 = relu(W2 h1 + b2), kept in registers; y = w3 h2 + b3
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float b = sm[S::b2 + column(c)];
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][c] = pack2(b, b);
        }
        if (cols) grad_mm<NC, V, HP>(acc, sm + S::h1T + tr * 4, sm + S::W2Td + 2 * V * tc, HP <= 16 ? H : HP);
        {
            float y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) y[q] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float w = sm[S::w3 + column(c)];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float a = fmaxf(lo2(acc[p][c]), 0.f), b = fmaxf(hi2(acc[p][c]), 0.f);
                    acc[p][c] = pack2(a, b);
                    y[2 * p] = fmaf(w, a, y[2 * p]);
                    y[2 * p + 1] = fmaf(w, b, y[2 * p + 1]);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                y[q] += __shfl_xor_sync(0xffffffffu, y[q], 8);
                y[q] += __shfl_xor_sync(0xffffffffu, y[q], 16);
            }
            if (lane < 8) {
                float *half = sm + S::part + (warp >> 2) * kGradRows + tr * 4;
                *reinterpret_cast<float4 *>(half) = make_float4(y[0], y[1], y[2], y[3]);
                *reinterpret_cast<float4 *>(half + kGradRows / 2) = make_float4(y[4], y[5], y[6], y[7]);
            }
        }
        __syncthreads();
        {
            const float y = sm[S::part + t] + sm[S::part + kGradRows + t] + b3;
            const float err = valid ? y - label[row] : 0.f;
            const float d = 2.f * err * inv_n;
            gl += err * err * inv_n;
            gb3 += d;
            sm[S::dy + t] = d;
        }
        __syncthreads();
        // ---- dh2 = dy w3 where h2 > 0; gradients of w3 and b2
        {
            const float4 d0 = *reinterpret_cast<const float4 *>(sm + S::dy + tr * 4);
            const float4 d1 = *reinterpret_cast<const float4 *>(sm + S::dy + tr * 4 + kGradRows / 2);
            const float d[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float w = sm[S::w3 + column(c)];
                f32x2 v[4];
                float sw = 0.f, sb = 0.f;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float a = lo2(acc[p][c]), b = hi2(acc[p][c]);
                    sw = fmaf(d[2 * p], a, sw);
                    sw = fmaf(d[2 * p + 1], b, sw);
                    const float da = a > 0.f ? d[2 * p] * w : 0.f, db = b > 0.f ? d[2 * p + 1] * w : 0.f;
                    sb += da;
                    sb += db;
                    v[p] = pack2(da, db);
                }
                gw3[c] += sw;
                gb2[c] += sb;
                grad_put(sm + S::dT + column(c) * kRowStride + tr * 4, v);
            }
        }
        __syncthreads();
        // ---- dh1 = W2^T dh2 where h1 > 0 (kept in registers); gradient of b1
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][c] = 0ULL;
        if (cols) grad_mm<NC, V, HP>(acc, sm + S::dT + tr * 4, sm + S::W2d + 2 * V * tc, HP <= 16 ? H : HP);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float *h = sm + S::h1T + column(c) * kRowStride + tr * 4;
            const float4 h0 = *reinterpret_cast<const float4 *>(h);
            const float4 h1 = *reinterpret_cast<const float4 *>(h + kGradRows / 2);
            const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
            float sb = 0.f;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float a = hv[2 * p] > 0.f ? lo2(acc[p][c]) : 0.f;
                const float b = hv[2 * p + 1] > 0.f ? hi2(acc[p][c]) : 0.f;
                sb += a;
                sb += b;
                acc[p][c] = pack2(a, b);
            }
            gb1[c] += sb;
        }
        // ---- gradient of W2: sum over rows of dh2[j] h1[i], even and odd rows apart
#pragma unroll 2
        for (int r = 0; r < (entries ? kGradRows : 0); r += 4) {
            ulonglong2 dj[NJ], hi[NJ];
#pragma unroll
            for (int a = 0; a < NJ; ++a) {
                dj[a] = *reinterpret_cast<const ulonglong2 *>(sm + S::dT + (tj + 16 * a) * kRowStride + r);
                hi[a] = *reinterpret_cast<const ulonglong2 *>(sm + S::h1T + (ti + 16 * a) * kRowStride + r);
            }
#pragma unroll
            for (int a = 0; a < NJ; ++a)
#pragma unroll
                for (int b = 0; b < NJ; ++b) {
                    gW2[a][b] = fma2(dj[a].x, hi[b].x, gW2[a][b]);
                    gW2[a][b] = fma2(dj[a].y, hi[b].y, gW2[a][b]);
                }
        }
        __syncthreads();   // h1 is read by now: dh1 takes its place
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const f32x2 v[4] = {acc[0][c], acc[1][c], acc[2][c], acc[3][c]};
            grad_put(sm + S::h1T + column(c) * kRowStride + tr * 4, v);
        }
        __syncthreads();
        // ---- gradient of W1: sum over rows of dh1[i] x[k]
        if (t / HP * KT < kFeat) {
            const float *d = sm + S::h1T + (t % HP) * kRowStride, *x = sm + S::xT + (t / HP) * KT * kRowStride;
#pragma unroll 4
            for (int r = 0; r < kGradRows; r += 4) {
                const ulonglong2 dv = *reinterpret_cast<const ulonglong2 *>(d + r);
#pragma unroll
                for (int a = 0; a < KT; ++a) {
                    const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(x + a * kRowStride + r);
                    gW1[a] = fma2(dv.x, xv.x, gW1[a]);
                    gW1[a] = fma2(dv.y, xv.y, gW1[a]);
                }
            }
        }
        __syncthreads();   // x and dh1 are read: the next tile may overwrite them
    }
    // ---- the block's sums to memory
#pragma unroll
    for (int a = 0; a < NJ; ++a)
#pragma unroll
        for (int b = 0; b < NJ; ++b) {
            const int j = tj + 16 * a, i = ti + 16 * b;
            if (j < H && i < H) atomicAdd(&grad[o.W2 + (int64_t)j * H + i], lo2(gW2[a][b]) + hi2(gW2[a][b]));
        }
    if (t / HP * KT < kFeat && t % HP < H)
#pragma unroll
        for (int a = 0; a < KT; ++a)
            atomicAdd(&grad[o.W1 + (int64_t)(t % HP) * kFeat + t / HP * KT + a], lo2(gW1[a]) + hi2(gW1[a]));
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int of = 1; of < 8; of <<= 1) {
            gb1[c] += __shfl_xor_sync(0xffffffffu, gb1[c], of);
            gb2[c] += __shfl_xor_sync(0xffffffffu, gb2[c], of);
            gw3[c] += __shfl_xor_sync(0xffffffffu, gw3[c], of);
        }
        if ((lane & 7) == 0 && column(c) < H) {
            atomicAdd(&grad[o.b1 + column(c)], gb1[c]);
            atomicAdd(&grad[o.b2 + column(c)], gb2[c]);
            atomicAdd(&grad[o.w3 + column(c)], gw3[c]);
        }
    }
    for (int of = 16; of; of >>= 1) {
        gl += __shfl_xor_sync(0xffffffffu, gl, of);
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, of);
    }
    if (lane == 0) {
        if (gl != 0.f) atomicAdd(loss, gl);
        atomicAdd(&grad[o.b3], gb3);
    }
}

__global__ void k_adam(float *w, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// permutation keys: hash of (seed, i) in the high bits, i in the low bits
__global__ void k_perm_keys(int32_t n, uint64_t seed, int32_t idb, uint64_t *keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = ((fmix64(seed ^ ((uint64_t)i * kGolden)) >> idb) << idb) | (uint64_t)i;
}

__global__ void k_keys_to_idx(const uint64_t *keys, int32_t n, int32_t idb, int32_t *idx) {
    const uint64_t mask = (1ULL << idb) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        idx[i] = (int32_t)(keys[i] & mask);
}

}  // namespace

int32_t model_feature_kind(const mce_model *m) { return m ? m->feature_kind : 0; }

mce_status features(const mce_graph *g, int32_t kind, cudaStream_t s, float *feat) {
    const int32_t n = g->n;
    if (n == 0) return MCE_OK;
    FeatParams P{};
    P.row_ptr = g->row_ptr;
    P.col = g->col;
    P.n = n;
    P.feat = feat;
    DevBuf core, tri, deg, drank, up_ptr, up_col;
    if (kind == MCE_FEATURES_LIGHT) {
        MCE_LAUNCH(k_features<true>, grid_for((int64_t)n * 8, kFeatThreads), kFeatThreads, 0, s, P);
        return MCE_OK;
    }
    MCE_TRY(core.alloc((size_t)n * 8, s));
    MCE_TRY(tri.alloc((size_t)n * 8, s));
    MCE_TRY(deg.alloc((size_t)n * 8, s));
    MCE_TRY(drank.alloc((size_t)n * 4, s));
    MCE_TRY(vertex_key(g, MCE_RANK_DEGEN, s, core.as<int64_t>()));
    MCE_TRY(vertex_key(g, MCE_RANK_TRIANGLE, s, tri.as<int64_t>()));
    MCE_TRY(vertex_key(g, MCE_RANK_DEGREE, s, deg.as<int64_t>()));
    MCE_TRY(rank_from_key_i64(deg.as<int64_t>(), n, g->id_bits, vertex_key_bits(g, MCE_RANK_DEGREE), s,
                              drank.as<int32_t>()));
    MCE_TRY(build_up_lists(g, drank.as<int32_t>(), s, up_ptr, up_col));
    P.core = core.as<int64_t>();
    P.tri = tri.as<int64_t>();
    P.up_ptr = up_ptr.as<int32_t>();
    MCE_LAUNCH(k_features<false>, grid_for((int64_t)n * 8, kFeatThreads), kFeatThreads, 0, s, P);
    return MCE_OK;
}

mce_status model_predict(const mce_model *m, const float *feat, int32_t rows, int32_t bf16, cudaStream_t s,
                         float *out) {
    if (rows <= 0) return MCE_OK;
    if (bf16) {
        // persistent warps: the weight fragments are loaded once a warp
        void (*kb)(const float *, int, const float *, int32_t, float *) =
            m->H <= 16 ? k_mlp_fwd_bf16<16> : m->H <= 32 ? k_mlp_fwd_bf16<32> : k_mlp_fwd_bf16<kMaxH>;
        const int64_t blocks = ((int64_t)rows + 63) / 64;
        const int64_t most = (int64_t)num_sms() * 3;
        MCE_LAUNCH(kb, (unsigned)(blocks < most ? blocks : most), 128, 0, s, m->w, m->H, feat, rows, out);
        return MCE_OK;
    }
    const size_t smem = (size_t)offsets(m->H).n * 4;
    // the default width has its own compiled kernel
    void (*kf)(const float *, int, const float *, int32_t, float *) = m->H == kMaxH ? k_mlp_fwd<kMaxH> : k_mlp_fwd<0>;
    MCE_CUDA(cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    MCE_LAUNCH(kf, grid_for(rows, 128), 128, smem, s, m->w, m->H, feat, rows, out);
    return MCE_OK;
}

template <int HP>
static mce_status grad_launch_hp(const mce_model *m, const float *feat, const float *label, const int32_t *idx,
                                 int64_t r0, int64_t cnt, float inv_n, float *loss, cudaStream_t s) {
    const size_t smem = (size_t)GradSmem<HP>::n * 4;
    MCE_CUDA(cudaFuncSetAttribute(k_mlp_grad<HP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int64_t tiles = (cnt + kGradRows - 1) / kGradRows;
    const int64_t most = (int64_t)num_sms() * GradSmem<HP>::blocks;
    const unsigned blocks = (unsigned)(tiles < most ? tiles : most);
    MCE_LAUNCH(k_mlp_grad<HP>, blocks, kGradRows, smem, s, m->w, m->H, feat, label, idx, r0, cnt, inv_n, m->g, loss);
    return MCE_OK;
}

static mce_status grad_launch(const mce_model *m, const float *feat, const float *label, const int32_t *idx,
                              int64_t r0, int64_t cnt, float inv_n, float *loss, cudaStream_t s) {
    if (m->H <= 16) return grad_launch_hp<16>(m, feat, label, idx, r0, cnt, inv_n, loss, s);
    if (m->H <= 32) return grad_launch_hp<32>(m, feat, label, idx, r0, cnt, inv_n, loss, s);
    return grad_launch_hp<kMaxH>(m, feat, label, idx, r0, cnt, inv_n, loss, s);
}

}  // namespace mce

using namespace mce;

extern "C" {

mce_status mce_features(const mce_graph *g, void *stream, float *feat) {
    return mce_features_kind(g, MCE_FEATURES_FULL, stream, feat);
}

mce_status mce_features_kind(const mce_graph *g, int32_t kind, void *stream, float *feat) {
    if (!g || !feat || (kind != MCE_FEATURES_FULL && kind != MCE_FEATURES_LIGHT)) {
        g_last_error = "mce_features_kind: bad arguments";
        return MCE_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    MCE_TRY(features(g, kind, s, feat));
    MCE_CUDA(cudaStreamSynchronize(s));
    return MCE_OK;
}

mce_status mce_model_set_features(mce_model *m, int32_t kind) {
    if (!m || (kind != MCE_FEATURES_FULL && kind != MCE_FEATURES_LIGHT)) {
        g_last_error = "mce_model_set_features: bad arguments";
        return MCE_EINVAL;
    }
    m->feature_kind = kind;
    return MCE_OK;
}

mce_status mce_model_create(int32_t hidden, uint64_t seed, mce_model **out) {
    if (!out || hidden < 1 || hidden > kMaxH) {
        g_last_error = "mce_model_create: hidden must be in [1, 64]";
        return MCE_EINVAL;
    }
    mce_model *m = new mce_model();
    m->H = hidden;
    const Off o = offsets(hidden);
    m->np = o.n;
    std::vector<float> h((size_t)o.n, 0.f);
    // He-style uniform initialisation from a splitmix64 stream
    uint64_t st = seed;
    auto next = [&]() {
        uint64_t z = (st += 0x9E3779B97F4A7C15ULL);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        z ^= z >> 31;
        return (double)(z >> 11) * 0x1.0p-53 * 2.0 - 1.0;
    };
    for (int64_t i = 0; i < (int64_t)hidden * kFeat; ++i) h[o.W1 + i] = (float)(next() * sqrt(6.0 / kFeat));
    for (int64_t i = 0; i < (int64_t)hidden * hidden; ++i) h[o.W2 + i] = (float)(next() * sqrt(6.0 / hidden));
    for (int64_t i = 0; i < hidden; ++i) h[o.w3 + i] = (float)(next() * sqrt(3.0 / hidden));
    for (int64_t i = 0; i < hidden; ++i) {
        h[o.b1 + i] = 0.01f;
        h[o.b2 + i] = 0.01f;
    }
    mce_status st2 = MCE_OK;
    const size_t bytes = (size_t)o.n * 4;
    st2 = cuda_status(cudaMalloc(&m->w, bytes), "model alloc");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMalloc(&m->m, bytes), "model alloc");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMalloc(&m->v, bytes), "model alloc");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMalloc(&m->g, bytes), "model alloc");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMemcpy(m->w, h.data(), bytes, cudaMemcpyHostToDevice), "model init");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMemset(m->m, 0, bytes), "model init");
    if (st2 == MCE_OK) st2 = cuda_status(cudaMemset(m->v, 0, bytes), "model init");
    if (st2 != MCE_OK) {
        mce_model_free(m);
        return st2;
    }
    *out = m;
    return MCE_OK;
}

void mce_model_free(mce_model *m) {
    if (!m) return;
    cudaDeviceSynchronize();
    cudaFree(m->w);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->g);
    delete m;
}

int64_t mce_model_num_params(const mce_model *m) { return m ? m->np : 0; }

mce_status mce_model_get(const mce_model *m, float *host) {
    if (!m || !host) return MCE_EINVAL;
    MCE_CUDA(cudaMemcpy(host, m->w, (size_t)m->np * 4, cudaMemcpyDeviceToHost));
    return MCE_OK;
}

mce_status mce_model_set(mce_model *m, const float *host) {
    if (!m || !host) return MCE_EINVAL;
    MCE_CUDA(cudaMemcpy(m->w, host, (size_t)m->np * 4, cudaMemcpyHostToDevice));
    return MCE_OK;
}

mce_status mce_model_loss_grad(const mce_model *m, const float *feat, const float *label, int32_t rows, void *stream,
                               float *loss, float *host_grad) {
    if (!m || !feat || !label || rows <= 0) return MCE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    DevBuf dl;
    MCE_TRY(dl.alloc(4, s));
    MCE_CUDA(cudaMemsetAsync(dl.p, 0, 4, s));
    MCE_CUDA(cudaMemsetAsync(m->g, 0, (size_t)m->np * 4, s));
    MCE_TRY(grad_launch(m, feat, label, nullptr, 0, rows, 1.f / rows, dl.as<float>(), s));
    if (loss) MCE_CUDA(cudaMemcpyAsync(loss, dl.p, 4, cudaMemcpyDeviceToHost, s));
    if (host_grad) MCE_CUDA(cudaMemcpyAsync(host_grad, m->g, (size_t)m->np * 4, cudaMemcpyDeviceToHost, s));
    MCE_CUDA(cudaStreamSynchronize(s));
    return MCE_OK;
}

mce_status mce_model_train(mce_model *m, const float *feat, const float *label, int32_t rows, int32_t epochs,
                           int32_t batch, float lr, uint64_t seed, void *stream, float *loss_out) {
    if (!m || !feat || !label || rows <= 0 || epochs < 0 || batch <= 0) return MCE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int32_t idb = bits_for((uint64_t)rows);
    DevBuf keys, tmp, idx, dl;
    MCE_TRY(keys.alloc((size_t)rows * 8, s));
    MCE_TRY(tmp.alloc((size_t)rows * 8, s));
    MCE_TRY(idx.alloc((size_t)rows * 4, s));
    MCE_TRY(dl.alloc((size_t)(epochs + 1) * 4, s));
    MCE_CUDA(cudaMemsetAsync(dl.p, 0, (size_t)(epochs + 1) * 4, s));
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int32_t ep = 0; ep < epochs; ++ep) {
        MCE_LAUNCH(k_perm_keys, grid_for(rows, 256), 256, 0, s, rows, seed + (uint64_t)ep * 7919, idb,
                   keys.as<uint64_t>());
        MCE_TRY(radix_sort_u64(keys.as<uint64_t>(), tmp.as<uint64_t>(), rows, idb, 64, s));
        MCE_LAUNCH(k_keys_to_idx, grid_for(rows, 256), 256, 0, s, keys.as<uint64_t>(), rows, idb, idx.as<int32_t>());
        for (int64_t r0 = 0; r0 < rows; r0 += batch) {
            const int64_t cnt = (r0 + batch <= rows) ? batch : rows - r0;
            MCE_CUDA(cudaMemsetAsync(m->g, 0, (size_t)m->np * 4, s));
            // per-batch mean for the gradient; the epoch loss is the mean over rows
            MCE_TRY(grad_launch(m, feat, label, idx.as<int32_t>(), r0, cnt, 1.f / (float)cnt,
                                dl.as<float>() + ep, s));
            m->step++;
            const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
            MCE_LAUNCH(k_adam, grid_for(m->np, 256), 256, 0, s, m->w, m->g, m->m, m->v, m->np, lr, b1, b2, eps, c1,
                       c2);
        }
    }
    std::vector<float> hl((size_t)epochs + 1);
    MCE_CUDA(cudaMemcpyAsync(hl.data(), dl.p, (size_t)(epochs + 1) * 4, cudaMemcpyDeviceToHost, s));
    MCE_CUDA(cudaStreamSynchronize(s));
    if (loss_out && epochs > 0) {
        // each batch added (mean batch loss); divide by the number of batches
        const int64_t nb = (rows + batch - 1) / batch;
        *loss_out = hl[epochs - 1] / (float)nb;
    }
    return MCE_OK;
}

mce_status mce_model_predict(const mce_model *m, const float *feat, int32_t rows, int32_t bf16, void *stream,
                             float *out) {
    if (!m || !feat || !out || rows < 0) return MCE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    MCE_TRY(model_predict(m, feat, rows, bf16, s, out));
    MCE_CUDA(cudaStreamSynchronize(s));
    return MCE_OK;
}

}  // extern "C"
