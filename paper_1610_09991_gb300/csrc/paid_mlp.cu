// Learned refinement proposal: a 5-layer MLP, 32 -> 256 -> 256 -> 256 -> 256 -> 256,
// GELU after the four hidden layers, that maps an integral's parameters
// (sin/cos of qx, qy; one-hot l and m; log10 T; mu; t'; one-hot kind) to a
// 16 x 16 map of predicted log10 cell errors.  It only decides where the
// initial partition is pre-split; the cubature's own error sums still decide
// convergence.  (Not part of the paper: the proposal of the workload
// specification.)
//
// Kernels: the forward pass of all five layers in one launch on the tcgen05
// tensor cores (TMEM accumulators, fused bias / GELU / BF16 epilogues); for
// training, one launch for the loss gradient and the chain of hidden gradients, one
// for every layer's weight and bias gradient (BF16 products on mma.sync m16n8k16),
// and AdamW on FP32 master weights with the BF16 copies of the next step.
//
// Parameter buffer (FP32 master weights), layer l = 0..4 with K_0 = 32,
// K_l = 256 otherwise, N = 256:  W_l [K_l][N] row-major, then b_l [N].
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/paid.h"

namespace {

constexpr int kIn = PAID_MLP_IN, kHid = PAID_MLP_HIDDEN;
constexpr int kLayers = PAID_MLP_LAYERS;
static_assert(PAID_MLP_OUT == PAID_MLP_HIDDEN, "the output layer has the hidden width");

__host__ __device__ inline int layer_k(int l) { return l == 0 ? kIn : kHid; }
__host__ __device__ inline int64_t layer_w_off(int l)
{
    int64_t o = 0;
    for (int i = 0; i < l; ++i) o += int64_t(layer_k(i)) * kHid + kHid;
    return o;
}
__host__ __device__ inline int64_t param_count()
{
    return layer_w_off(kLayers);
}

// ---------------------------------------------------------------------------
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x)
{
    const float cdf = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
    const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
    return cdf + x * pdf;
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// four 8 x 8 BF16 matrices of a fragment, rows as stored or transposed
__device__ __forceinline__ void ldsm(uint32_t* r, const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ void ldsm_t(uint32_t* r, const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
// 16 bytes from global to shared memory, zeros when !in (asynchronous)
__device__ __forceinline__ void cp16(void* dst, const void* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 :: "r"(smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// BF16 copies of a master weight, index i over all parameters: W [K][N] for the
// backward products, and its transpose in the byte order of the forward kernel's
// shared-memory operand (canonical K-major layout of 8-row x 16-byte core matrices:
// element (n, k) of layer l at byte ((n/8) (K/8) + k/8) 128 + (n%8) 16 + (k%8) 2 of
// the layer's block), so that one bulk copy stages a layer.  Returns whether i is a
// bias.
__device__ __forceinline__ bool cast_weight(int64_t i, float value, __nv_bfloat16* __restrict__ w,
                                            __nv_bfloat16* __restrict__ wc)
{
    int64_t o = 0, ob = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int K = layer_k(l);
        const int64_t kn = int64_t(K) * kHid;
        if (i < o + kn + kHid) {
            const int64_t e = i - o;
            if (e >= kn) return true;
            if (w) {
                const int k = int(e / kHid), n = int(e % kHid);
                const __nv_bfloat16 v = __float2bfloat16(value);
                w[ob + e] = v;
                wc[ob + (((n >> 3) * (K >> 3) + (k >> 3)) * 64 + (n & 7) * 8 + (k & 7))] = v;
            }
            return false;
        }
        o += kn + kHid;
        ob += kn;
    }
    return true;
}

__global__ void k_cast_weights(const float* __restrict__ p, int64_t n, __nv_bfloat16* __restrict__ w,
                               __nv_bfloat16* __restrict__ wc)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) cast_weight(i, p[i], w, wc);
}

// ---------------------------------------------------------------------------
// Training, backward.  Bound: latency (a minibatch of 1,024 rows is 1.6 GFLOP, a
// microsecond of the tensor cores); what counts is launches, and that every product
// keeps its order: each output is one chain of m16n8k16 products over its
// contraction in steps of 16, so that a run's weights are reproducible.  One GEMM
// per product with scalar loads, and a thread per column for the bias gradients,
// took 890 us a minibatch of 1,024 rows; these two kernels take 37 (27 and 10).
//
// The gradients with respect to the pre-activations: d_4 = 2 (y - t) / (M 256), then
// d_{l-1} = (d_l W_l^T) gelu'(pre_{l-1}) down the layers, every d_l rounded to BF16.
// A CTA takes 16 rows through all four products; each of its eight warps owns 32 of
// the outputs and stages their rows of W_l for itself, the next layer's while the
// epilogue of this one runs.
constexpr int kBackRows = 16, kBackThreads = 256, kBackPitch = kHid + 8;

struct BackSmem {
    __nv_bfloat16 d[2][kBackRows][kBackPitch];
    __nv_bfloat16 w[kHid][kBackPitch];
    float loss[kBackThreads / 32];
};
static_assert(kBackPitch * sizeof(__nv_bfloat16) % 16 == 0 &&
                  offsetof(BackSmem, w) % 16 == 0,
              "every row is a target of 16-byte copies (back_raw is 16-byte aligned)");

struct BackArgs {
    const __nv_bfloat16* w;                // BF16 W_l [K][256], layers back to back
    const float* pre[kLayers];             // pre-activations [M][256]
    const float* target;                   // [M][256]
    __nv_bfloat16* d[kLayers];             // out: d_l [M][256]
    float* loss;                           // += sum (y - t)^2 scale
    int64_t M;
    float scale;                           // 1 / (M 256)
    int64_t wofs[kLayers];                 // offset of W_l in w
};

__global__ void __launch_bounds__(kBackThreads) k_backward(BackArgs g)
{
    extern __shared__ __align__(16) unsigned char back_raw[];
    BackSmem& S = *reinterpret_cast<BackSmem*>(back_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t m0 = int64_t(blockIdx.x) * kBackRows;
    auto stage = [&](int l) {   // this warp's 32 rows of W_l
        const __nv_bfloat16* src = g.w + g.wofs[l] + int64_t(32 * wid) * kHid + 8 * lane;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) cp16(&S.w[32 * wid + i][8 * lane], src + i * kHid, true);
        cp_commit();
    };
    stage(kLayers - 1);
    float loss = 0.0f;
#pragma unroll 4
    for (int r = 0; r < kBackRows; ++r) {
        const int64_t m = m0 + r;
        __nv_bfloat16 v = __float2bfloat16(0.0f);
        if (m < g.M) {
            const float e = g.pre[kLayers - 1][m * kHid + tid] - g.target[m * kHid + tid];
            v = __float2bfloat16(2.0f * e * g.scale);
            g.d[kLayers - 1][m * kHid + tid] = v;
            loss += e * e * g.scale;
        }
        S.d[0][r][tid] = v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) S.loss[wid] = loss;
    const int r = lane >> 2, c = (lane & 3) * 2;   // the fragment's rows r, r + 8 and columns c, c + 1
    int cur = 0;
    for (int l = kLayers - 1; l > 0; --l) {
        // gelu' of this thread's outputs: rows r and r + 8, columns 32 wid + 8 j + c, + 1
        float2 pre[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t m = m0 + r + 8 * h;
                pre[j][h] = m < g.M ? *reinterpret_cast<const float2*>(
                                          g.pre[l - 1] + m * kHid + 32 * wid + 8 * j + c)
                                    : make_float2(0.0f, 0.0f);
            }
        cp_wait<0>();
        __syncthreads();
        if (l == kLayers - 1 && tid == 0) {
            float sum = 0.0f;
            for (int q = 0; q < kBackThreads / 32; ++q) sum += S.loss[q];
            atomicAdd(g.loss, sum);
        }
        float acc[4][4] = {};
#pragma unroll 4
        for (int k0 = 0; k0 < kHid; k0 += 16) {
            uint32_t a[4], b[2][4];
            ldsm(a, &S.d[cur][lane & 15][k0 + (lane >> 4) * 8]);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                ldsm(b[j], &S.w[32 * wid + 16 * j + (lane >> 4) * 8 + (lane & 7)]
                               [k0 + ((lane >> 3) & 1) * 8]);
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(acc[j], a, &b[j >> 1][2 * (j & 1)]);
        }
        __syncwarp();
        if (l > 1) stage(l - 1);
        cur ^= 1;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t m = m0 + r + 8 * h;
                const int n = 32 * wid + 8 * j + c;
                __nv_bfloat162 v;
                v.x = __float2bfloat16(acc[j][2 * h] * gelu_grad(pre[j][h].x));
                v.y = __float2bfloat16(acc[j][2 * h + 1] * gelu_grad(pre[j][h].y));
                *reinterpret_cast<__nv_bfloat162*>(&S.d[cur][r + 8 * h][n]) = v;
                if (m < g.M) *reinterpret_cast<__nv_bfloat162*>(g.d[l - 1] + m * kHid + n) = v;
            }
    }
}

// Weight and bias gradients of every layer, dW_l[k][n] = sum_m in_l[m][k] d_l[m][n]
// (in_0 = x, in_l = h_{l-1}) in 32 x 32 tiles of four warps, 64 rows a stage, three
// stages in flight; db_l[n] = sum_m d_l[m][n], a thread per column adding the rows in
// order from shared memory (no atomics: training is bitwise reproducible).  With
// splits > 1 the rows are cut into blockIdx.y parts and the tiles added to a zeroed
// gradient.
constexpr int kDwTile = 32, kDwRows = 64, kDwStages = 3, kDwPitch = kDwTile + 8;
constexpr int kDwThreads = 128, kBiasRows = 256;

struct DwArgs {
    const __nv_bfloat16* in[kLayers];
    const __nv_bfloat16* d[kLayers];
    float* grad;
    int M, chunk;                          // rows, rows per split
    int64_t off[kLayers];                  // offset of dW_l in grad
    bool x_aligned;                        // in[0] allows 16-byte loads
};

// the block's shared memory: operand tiles, or the bias gradients' rows.  16-byte
// cp.async and ldmatrix address it, whose rows' start must be a multiple of 16 bytes.
union __align__(16) DwSmem {
    struct { __nv_bfloat16 a[kDwStages][kDwRows][kDwPitch], b[kDwStages][kDwRows][kDwPitch]; } t;
    __nv_bfloat16 bias[2][kBiasRows][kDwTile];
};
static_assert(alignof(DwSmem) >= 16 && kDwPitch * sizeof(__nv_bfloat16) % 16 == 0 &&
                  kDwTile * sizeof(__nv_bfloat16) % 16 == 0,
              "every row is a target of 16-byte copies");

constexpr int dw_tiles(int l) { return (l == 0 ? kIn : kHid) / kDwTile * (kHid / kDwTile); }
constexpr int kDwTiles = dw_tiles(0) + (kLayers - 1) * dw_tiles(1);
constexpr int kBiasTiles = kLayers * (kHid / kDwTile);

__global__ void __launch_bounds__(kDwThreads) k_weight_grad(DwArgs g)
{
    __shared__ DwSmem S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int tile = blockIdx.x;
    if (tile >= kDwTiles) {   // bias gradients
        if (blockIdx.y != 0) return;
        tile -= kDwTiles;
        const int l = tile / (kHid / kDwTile), n0 = tile % (kHid / kDwTile) * kDwTile;
        const __nv_bfloat16* d = g.d[l] + n0;
        auto stage = [&](int i) {
            for (int q = tid; q < kBiasRows * 4; q += kDwThreads) {
                const int m = i * kBiasRows + (q >> 2);
                cp16(&S.bias[i & 1][q >> 2][8 * (q & 3)],
                     d + int64_t(m < g.M ? m : 0) * kHid + 8 * (q & 3), m < g.M);
            }
            cp_commit();
        };
        const int n_stages = (g.M + kBiasRows - 1) / kBiasRows;
        stage(0);
        float s = 0.0f;
        for (int i = 0; i < n_stages; ++i) {
            if (i + 1 < n_stages) { stage(i + 1); cp_wait<1>(); } else { cp_wait<0>(); }
            __syncthreads();
            if (tid < kDwTile) {
                const int rows = min(kBiasRows, g.M - i * kBiasRows);
#pragma unroll 16
                for (int r = 0; r < rows; ++r) s += __bfloat162float(S.bias[i & 1][r][tid]);
            }
            __syncthreads();
        }
        const int K = l == 0 ? kIn : kHid;
        if (tid < kDwTile) g.grad[g.off[l] + int64_t(K) * kHid + n0 + tid] = s;
        return;
    }
    int l = 0;
    if (tile >= dw_tiles(0)) {
        l = 1 + (tile - dw_tiles(0)) / dw_tiles(1);
        tile = (tile - dw_tiles(0)) % dw_tiles(1);
    }
    const int K = l == 0 ? kIn : kHid;
    const int k0 = tile / (kHid / kDwTile) * kDwTile, n0 = tile % (kHid / kDwTile) * kDwTile;
    const __nv_bfloat16 *in = g.in[l] + k0, *d = g.d[l] + n0;
    const bool vec = l > 0 || g.x_aligned;
    const int mbeg = blockIdx.y * g.chunk, mend = min(g.M, mbeg + g.chunk);
    const int n_stages = mend > mbeg ? (mend - mbeg + kDwRows - 1) / kDwRows : 0;
    auto stage = [&](int i) {
        if (i < n_stages) {
            const int m_ = mbeg + i * kDwRows, st = i % kDwStages;
            for (int q = tid; q < kDwRows * 4; q += kDwThreads) {
                const int row = q >> 2, col = 8 * (q & 3), m = m_ + row;
                const bool ok = m < mend;
                const int64_t src = ok ? m : mbeg;
                cp16(&S.t.b[st][row][col], d + src * kHid + col, ok);
                if (vec) {
                    cp16(&S.t.a[st][row][col], in + src * K + col, ok);
                } else {
                    for (int e = 0; e < 8; ++e)
                        S.t.a[st][row][col + e] =
                            ok ? in[src * K + col + e] : __float2bfloat16(0.0f);
                }
            }
        }
        cp_commit();
    };
    const int wm = 16 * (warp >> 1), wn = 16 * (warp & 1);
    float acc[2][4] = {};
    for (int i = 0; i < kDwStages - 1; ++i) stage(i);
    for (int i = 0; i < n_stages; ++i) {
        cp_wait<kDwStages - 2>();
        __syncthreads();
        stage(i + kDwStages - 1);
        const int st = i % kDwStages;
#pragma unroll
        for (int s = 0; s < kDwRows; s += 16) {
            uint32_t a[4], b[4];
            // A (k, m) and B (m, n) both lie with m in the rows: transposed fragments
            ldsm_t(a, &S.t.a[st][s + (lane >> 4) * 8 + (lane & 7)][wm + ((lane >> 3) & 1) * 8]);
            ldsm_t(b, &S.t.b[st][s + ((lane >> 3) & 1) * 8 + (lane & 7)][wn + (lane >> 4) * 8]);
            mma_bf16(acc[0], a, b);
            mma_bf16(acc[1], a, b + 2);
        }
    }
    float* out = g.grad + g.off[l];
    const int r = lane >> 2, c = (lane & 3) * 2;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int k = k0 + wm + r + (h >= 2 ? 8 : 0), n = n0 + wn + 8 * j + c + (h & 1);
            float* o = out + int64_t(k) * kHid + n;
            if (gridDim.y > 1) atomicAdd(o, acc[j][h]);
            else *o = acc[j][h];
        }
}

// AdamW on the FP32 master weights (biases not decayed); with w and wc also the
// BF16 copies of the updated weights for the next forward and backward.
__global__ void k_adamw(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                        float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                        float wd, float c1, float c2, __nv_bfloat16* __restrict__ w,
                        __nv_bfloat16* __restrict__ wc)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool is_bias = cast_weight(i, 0.0f, nullptr, nullptr);
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float upd = (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] -= lr * (upd + (is_bias ? 0.0f : wd * p[i]));
    if (w) cast_weight(i, p[i], w, wc);
}

// Seeded uniform(-a, a) initialisation (a = 1/sqrt(K), biases 0) from a
// counter-based hash (splitmix64) of (seed, index).
__global__ void k_init(float* __restrict__ p, uint64_t seed)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    int64_t o = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int64_t kn = int64_t(layer_k(l)) * kHid;
        if (i >= o && i < o + kn + kHid) {
            if (i >= o + kn) { p[i] = 0.0f; return; }
            uint64_t z = seed + 0x9e3779b97f4a7c15ull * uint64_t(i + 1);
            z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
            z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
            z ^= z >> 31;
            const float u = float(z >> 40) * (1.0f / 16777216.0f);   // [0, 1)
            const float a = rsqrtf(float(layer_k(l)));
            p[i] = (2.0f * u - 1.0f) * a;
            return;
        }
        o += kn + kHid;
    }
}

struct MlpWork {
    __nv_bfloat16 *w, *wc;                 // BF16 weights, in forward-operand order
    float* pre[kLayers];                    // pre-activations (FP32) [M][256]
    __nv_bfloat16* h[kLayers - 1];          // activations (BF16) [M][256]
    __nv_bfloat16* d[kLayers];              // BF16 gradients of the pre-activations [M][256]
    float* grad;                            // FP32 [param_count]
    float* loss;                            // FP32 scalar
};

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

size_t mlp_work_bytes(int64_t M, MlpWork* w, char* base)
{
    size_t o = 0;
    auto take = [&](size_t b) { size_t at = o; o = align256(o + b); return base ? base + at : nullptr; };
    const int64_t nw = param_count() - int64_t(kLayers) * kHid;   // weights only
    char* p;
    const size_t act = sizeof(__nv_bfloat16) * size_t(M) * kHid;
    p = take(sizeof(__nv_bfloat16) * nw); if (w) w->w = (__nv_bfloat16*)p;
    p = take(sizeof(__nv_bfloat16) * nw);   // (kept: the size is part of the interface's sizing)
    p = take(sizeof(__nv_bfloat16) * nw); if (w) w->wc = (__nv_bfloat16*)p;
    for (int l = 0; l < kLayers; ++l) {
        p = take(sizeof(float) * M * kHid); if (w) w->pre[l] = (float*)p;
        p = take(act);
        if (w && l < kLayers - 1) w->h[l] = (__nv_bfloat16*)p;
        if (w && l == kLayers - 1) w->d[0] = (__nv_bfloat16*)p;
    }
    p = take(act); if (w) w->d[4] = (__nv_bfloat16*)p;
    p = take(act); if (w) w->d[3] = (__nv_bfloat16*)p;
    p = take(2 * act);
    if (w) { w->d[2] = (__nv_bfloat16*)p; w->d[1] = (__nv_bfloat16*)(p + act); }
    p = take(sizeof(float) * param_count()); if (w) w->grad = (float*)p;
    p = take(sizeof(float)); if (w) w->loss = (float*)p;
    return o;
}

int64_t wofs(int l)   // offset of W_l in the BF16 weight arrays
{
    int64_t o = 0;
    for (int i = 0; i < l; ++i) o += int64_t(layer_k(i)) * kHid;
    return o;
}

// ---------------------------------------------------------------------------
// Forward pass on the 5th-generation tensor cores (tcgen05): a cluster of C CTAs of
// 256 threads runs all five layers for 128 rows, each CTA 256 / C of every layer's
// outputs.  Per layer one bulk copy (cp.async.bulk, completion on an mbarrier) stages
// the CTA's part of the layer's BF16 weights W_l^T, already in the operand's byte
// order, in shared memory; one thread issues K/16 tcgen05.mma (M = 128, N = 256 / C, K =
// 16, BF16 in, FP32 out) into 256 / C TMEM columns and commits them to a second
// mbarrier; the next layer's weight copy then starts at once and overlaps the
// epilogue, in which the eight warps read the accumulators back with tcgen05.ld (warp
// w: TMEM lanes = rows 32 (w mod 4) ..., half w / 4 of the columns): + bias, GELU, BF16
// into every CTA's shared memory as the next layer's input (two buffers in turn, so
// that one cluster barrier a layer orders them), or FP32 rows of the output after
// the last layer.
//
// Bound: latency.  The epilogue of 128 x 256 outputs on one SM is some 9 us a layer
// and 9 CTAs leave the chip idle for a flow step's 1,152 rows, so the clusters are as
// wide as keeps all CTAs on SMs at once: C = 8 up to 1,920 rows, 4 up to 4,608, 2 up
// to 9,728 (asked of the device); from there one CTA per 128 rows (C = 1), which
// needs the fewest barriers.  1,024 training
// rows: 36 us with C = 8, 69 with C = 1 (serialised, cold caches).
//
// Shared-memory operands use the canonical K-major layout without swizzling:
// 8-row x 16-byte core matrices, core matrix (r/8, k/8) at ((r/8) (K/8) + k/8)
// x 128 bytes, so the descriptor's K step between core matrices (leading byte
// offset) is 128 B and its row-group step (stride byte offset) K/8 x 128 B.
namespace tc {

constexpr int kRows = 128;            // rows per CTA = MMA M = TMEM lanes
constexpr int kThreads = 256;
// instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bit 17,
// M >> 4 at bit 24
constexpr uint32_t idesc(int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t(N) >> 3) << 17) |
           ((uint32_t(kRows) >> 4) << 24);
}
constexpr int kWaitLimit = 1 << 22;   // mbarrier polls before the CTA gives up

template <int C>
struct Smem {
    static constexpr int kBufs = C > 1 ? 2 : 1;
    unsigned char a[kBufs][kRows * kHid * 2];   // input rows, canonical layout
    unsigned char b[kHid / C * kHid * 2];       // this CTA's rows of W_l^T, canonical layout
    unsigned long long bar_mma, bar_w;
    uint32_t tmem;
};
template <int C>
constexpr size_t smem_bytes() { return sizeof(Smem<C>) + 1024; }   // + alignment of the operands

struct Args {
    const float* params;
    const __nv_bfloat16* wc;              // BF16 W_l^T in operand order, layers back to back
    const __nv_bfloat16* x;               // [M][32]
    int M;
    float* out;                           // last layer's pre-activation [M][256]
    float* pre[kLayers - 1];              // hidden pre-activations [M][256], or null
    __nv_bfloat16* h[kLayers - 1];        // hidden activations [M][256], or null
};

__device__ __forceinline__ uint32_t canon(int row, int kg, int KG)
{
    return uint32_t(((row >> 3) * KG + kg) * 128 + (row & 7) * 16);
}
// shared-memory descriptor: start, leading byte offset (K), stride byte offset
// (rows), bits 46-47 = 1 (tcgen05 descriptor version), no swizzle
__device__ __forceinline__ uint64_t desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return uint64_t((saddr >> 4) & 0x3FFFu) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity)
{
    for (int it = 0; it < kWaitLimit; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
// layer l's weights (bytes, 16-byte aligned at both ends) into b, completing on bar
__device__ __forceinline__ void copy_weights(uint32_t sb, const __nv_bfloat16* src, uint32_t bytes,
                                             uint32_t bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 :: "r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(sb), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// every thread of the cluster (C = 1: of the block), with generic-proxy writes of the
// next operand visible to the tensor core
template <int C>
__device__ __forceinline__ void sync_operands()
{
    if (C > 1) {
        asm volatile("fence.proxy.async;" ::: "memory");
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        asm volatile("fence.proxy.async;" ::: "memory");
    } else {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
    }
}
// 16 bytes to the same shared-memory offset of CTA r of the cluster
template <int C>
__device__ __forceinline__ void put16(uint32_t addr, int r, uint4 v)
{
    if (C > 1) {
        uint32_t to;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(addr), "r"(r));
        asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};"
                     :: "r"(to), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
    } else {
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};"
                     :: "r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
    }
}

}  // namespace tc

template <int C>
__global__ void __launch_bounds__(tc::kThreads, 1) k_mlp_forward_tc(tc::Args g)
{
    constexpr int NS = kHid / C;          // outputs of this CTA
    extern __shared__ unsigned char smem_raw[];
    tc::Smem<C>& S = *reinterpret_cast<tc::Smem<C>*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, half = warp >> 2;
    const int m0 = int(blockIdx.x / C) * tc::kRows;
    const int n0 = int(blockIdx.x % C) * NS;   // = the CTA's rank in its cluster times NS
    const uint32_t bar_mma = smem_u32(&S.bar_mma), bar_w = smem_u32(&S.bar_w);
    const uint32_t sb = smem_u32(S.b);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar_mma) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar_w) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&S.tmem)), "r"(uint32_t(NS)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = S.tmem;
    // layer 0's weights in flight while the input rows are staged
    if (tid == 0) tc::copy_weights(sb, g.wc + int64_t(n0) * kIn, uint32_t(kIn * NS * 2), bar_w);
    for (int c = tid; c < tc::kRows * kIn; c += tc::kThreads) {
        const int r = c / kIn, k = c - r * kIn;
        const __nv_bfloat16 v = m0 + r < g.M ? g.x[int64_t(m0 + r) * kIn + k]
                                             : __float2bfloat16(0.0f);
        *reinterpret_cast<__nv_bfloat16*>(S.a[0] + tc::canon(r, k >> 3, kIn / 8) + (k & 7) * 2) = v;
    }
    const int row = quarter * 32 + lane, grow = m0 + row;   // this thread's TMEM lane and row
    // a wait that ran out: the CTA leaves its tensor core alone from there, goes on
    // through its cluster's barriers and gives NaN
    bool ok = true;
    uint32_t phase = 0;            // completions seen on each barrier (one per layer)
    bool copy_pending = true;      // a weight copy issued and not yet waited for
    bool mma_pending = false;      // MMAs committed and not yet waited for
    int64_t wo = 0;                // offset of W_l^T in wc
    for (int l = 0; l < kLayers; ++l) {
        const int K = layer_k(l), KG = K / 8;
        const uint32_t sa = smem_u32(S.a[C > 1 ? l & 1 : 0]);
        const uint32_t sa_next = smem_u32(S.a[C > 1 ? (l + 1) & 1 : 0]);
        tc::sync_operands<C>();
        if (ok) {
            bool here = true;
            if (tid == 0) {
                here = tc::wait_bar(bar_w, phase & 1);       // this layer's weights
                if (here) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int kk = 0; kk < K / 16; ++kk) {
                        const uint64_t ad = tc::desc(sa + kk * 256, 128, KG * 128);
                        const uint64_t bd = tc::desc(sb + kk * 256, 128, KG * 128);
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                     :: "r"(tmem), "l"(ad), "l"(bd), "r"(tc::idesc(NS)), "r"(kk)
                                     : "memory");
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                                 :: "r"(bar_mma) : "memory");
                }
            }
            ok = __syncthreads_and(here);
            if (ok) {
                copy_pending = false;
                mma_pending = true;
                ok = __syncthreads_and(tc::wait_bar(bar_mma, phase & 1));
            }
            if (ok) {
                mma_pending = false;
                ++phase;
                wo += int64_t(K) * kHid;
                // the MMAs are done with b: the next layer's weights stream in during the
                // epilogue
                if (tid == 0 && l + 1 < kLayers)
                    tc::copy_weights(sb, g.wc + wo + int64_t(n0) * kHid, uint32_t(kHid * NS * 2),
                                     bar_w);
                copy_pending = l + 1 < kLayers;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
        }
        // alone, the CTA has no barrier to keep up: it leaves, and the epilogue below
        // needs no test (100,000 rows 300 -> 290 us)
        if (C == 1 && !ok) break;
        const float* bias = g.params + layer_w_off(l) + int64_t(K) * kHid + n0;
        const bool last = l == kLayers - 1;
        for (int c0 = half * (NS / 2); c0 < (half + 1) * (NS / 2); c0 += 16) {
            float y[16];
            __syncwarp();
            if (C == 1 || ok) {
                uint32_t r[16];
                tc::ld16(tmem + (uint32_t(quarter * 32) << 16) + uint32_t(c0), r);
#pragma unroll
                for (int j = 0; j < 16; ++j) y[j] = __uint_as_float(r[j]) + __ldg(bias + c0 + j);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) y[j] = __int_as_float(0x7fc00000);
            }
            const int n = n0 + c0;
            if (last) {
                if (grow < g.M) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        *reinterpret_cast<float4*>(g.out + int64_t(grow) * kHid + n + j) =
                            make_float4(y[j], y[j + 1], y[j + 2], y[j + 3]);
                }
            } else {
                __align__(16) __nv_bfloat16 hb[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) hb[j] = __float2bfloat16(gelu(y[j]));
                const uint4 h0 = *reinterpret_cast<const uint4*>(hb);
                const uint4 h1 = *reinterpret_cast<const uint4*>(hb + 8);
#pragma unroll
                for (int r = 0; r < C; ++r) {
                    tc::put16<C>(sa_next + tc::canon(row, n >> 3, kHid / 8), r, h0);
                    tc::put16<C>(sa_next + tc::canon(row, (n >> 3) + 1, kHid / 8), r, h1);
                }
                if (g.pre[l] && grow < g.M) {
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        *reinterpret_cast<float4*>(g.pre[l] + int64_t(grow) * kHid + n + j) =
                            make_float4(y[j], y[j + 1], y[j + 2], y[j + 3]);
                    *reinterpret_cast<uint4*>(g.h[l] + int64_t(grow) * kHid + n) = h0;
                    *reinterpret_cast<uint4*>(g.h[l] + int64_t(grow) * kHid + n + 8) = h1;
                }
            }
        }
        // every TMEM read done before the next layer's MMAs overwrite the columns
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    if (!ok) {
        // a copy or an MMA that never signalled: wait once more (bounded) so
        // that nothing is in flight when the CTA exits
        if (copy_pending) tc::wait_bar(bar_w, phase & 1);
        if (mma_pending) tc::wait_bar(bar_mma, phase & 1);
        if (C == 1 && grow < g.M)
            for (int c = half * (NS / 2); c < (half + 1) * (NS / 2); ++c)
                g.out[int64_t(grow) * kHid + c] = __int_as_float(0x7fc00000);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem), "r"(uint32_t(NS)) : "memory");
    }
}

// a launch of `clusters` clusters of C CTAs; `cluster` holds its attribute
template <int C>
cudaLaunchConfig_t forward_config(int clusters, cudaLaunchAttribute& cluster)
{
    cluster = cudaLaunchAttribute{};
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = C;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * C);
    cfg.blockDim = dim3(tc::kThreads);
    cfg.dynamicSmemBytes = tc::smem_bytes<C>();
    cfg.attrs = &cluster;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cfg;
}

template <int C>
cudaError_t allow_smem()
{
    return cudaFuncSetAttribute(k_mlp_forward_tc<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(tc::smem_bytes<C>()));
}

template <int C>
cudaError_t launch_forward(const tc::Args& g, cudaStream_t s)
{
    cudaError_t e;
    if ((e = allow_smem<C>()) != cudaSuccess) return e;
    cudaLaunchAttribute cluster;
    cudaLaunchConfig_t cfg = forward_config<C>((g.M + tc::kRows - 1) / tc::kRows, cluster);
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, k_mlp_forward_tc<C>, g);
}

// Clusters of C CTAs that the current device holds at once: a property of the chip
// (how many of its GPCs have room for how many), asked once per device.
template <int C>
int resident_clusters()
{
    static std::atomic<int> known[64];
    int dev = -1, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if ((n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
    cudaLaunchAttribute cluster;
    const cudaLaunchConfig_t cfg = forward_config<C>(1, cluster);
    if (allow_smem<C>() != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_mlp_forward_tc<C>, &cfg) != cudaSuccess) {
        cudaGetLastError();   // no answer: narrower clusters, which need none
        return 0;
    }
    known[dev].store(n, std::memory_order_relaxed);
    return n;
}

// forward of M rows: x [M][32] BF16 -> out [M][256] FP32 (the last layer's
// pre-activation); without out (training) the result goes to w.pre[4] and the
// hidden layers' pre-activations and activations are kept for the backward
cudaError_t forward(const float* params, const __nv_bfloat16* x, int64_t M, float* out,
                    MlpWork& w, cudaStream_t s)
{
    tc::Args g{};
    g.params = params;
    g.wc = w.wc;
    g.x = x;
    g.M = int(M);
    g.out = out ? out : w.pre[kLayers - 1];
    for (int l = 0; l < kLayers - 1; ++l) {
        g.pre[l] = out ? nullptr : w.pre[l];
        g.h[l] = out ? nullptr : w.h[l];
    }
    // The widest clusters that are all resident: one cluster more is a second wave.
    // On GB300 15 of eight, 36 of four and 76 of two fit; 16 blocks take 71 us with
    // eight CTAs each and 49 with four, 38 take 72 with four and 56 with two, 77 take
    // 85 with two and 68 with one.
    const int64_t blocks = (M + tc::kRows - 1) / tc::kRows;
    if (blocks <= resident_clusters<8>()) return launch_forward<8>(g, s);
    if (blocks <= resident_clusters<4>()) return launch_forward<4>(g, s);
    if (blocks <= resident_clusters<2>()) return launch_forward<2>(g, s);
    return launch_forward<1>(g, s);
}

cudaError_t cast_weights(const float* params, MlpWork& w, cudaStream_t s)
{
    const int64_t n = param_count();
    k_cast_weights<<<int((n + 255) / 256), 256, 0, s>>>(params, n, w.w, w.wc);
    return cudaGetLastError();
}

// MSE gradient of M rows into grad, loss added to *loss; the BF16 weights of params
// are in w (cast_weights or k_adamw).
cudaError_t grad_rows(const float* params, const __nv_bfloat16* xb, const float* target, int64_t M,
                      float* grad, float* loss, MlpWork& w, cudaStream_t s)
{
    cudaError_t e;
    if ((e = forward(params, xb, M, nullptr, w, s)) != cudaSuccess) return e;
    BackArgs b{};
    DwArgs g{};
    b.w = w.w;
    b.target = target;
    b.loss = loss;
    b.M = M;
    b.scale = 1.0f / float(M * kHid);
    for (int l = 0; l < kLayers; ++l) {
        b.pre[l] = w.pre[l];
        b.d[l] = w.d[l];
        b.wofs[l] = wofs(l);
        g.in[l] = l == 0 ? xb : w.h[l - 1];
        g.d[l] = w.d[l];
        g.off[l] = layer_w_off(l);
    }
    if ((e = cudaFuncSetAttribute(k_backward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  int(sizeof(BackSmem)))) != cudaSuccess)
        return e;
    k_backward<<<int((M + kBackRows - 1) / kBackRows), kBackThreads, sizeof(BackSmem), s>>>(b);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int splits = int(std::min<int64_t>(64, (M + 1023) / 1024));
    g.grad = grad;
    g.M = int(M);
    // whole steps of 32 rows per part
    g.chunk = int(((M + splits - 1) / splits + 31) / 32 * 32);
    g.x_aligned = reinterpret_cast<uintptr_t>(xb) % 16 == 0;
    const int parts = int((M + g.chunk - 1) / g.chunk);
    if (parts > 1 &&
        (e = cudaMemsetAsync(grad, 0, sizeof(float) * param_count(), s)) != cudaSuccess)
        return e;
    k_weight_grad<<<dim3(kDwTiles + kBiasTiles, parts), kDwThreads, 0, s>>>(g);
    return cudaGetLastError();
}

// rows perm[r0 .. r0 + n) of x and target into xb, tb
__global__ void k_gather_rows(const __nv_bfloat16* __restrict__ x, const float* __restrict__ t,
                              const int32_t* __restrict__ perm, int64_t r0, int64_t n,
                              __nv_bfloat16* __restrict__ xb, float* __restrict__ tb)
{
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n * kHid) return;
    const int64_t r = i / kHid, c = i % kHid;
    const int64_t src = perm[r0 + r];
    tb[i] = t[src * kHid + c];
    if (c < kIn) xb[r * kIn + c] = x[src * kIn + c];
}

// AdamW with bias corrections for step k (counting from 1)
cudaError_t adamw_step(float* params, const float* grad, float* m, float* v, int step, float lr,
                       float weight_decay, const MlpWork* w, cudaStream_t s)
{
    const int64_t n = param_count();
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, float(step)), c2 = 1.0f - powf(b2, float(step));
    k_adamw<<<int((n + 255) / 256), 256, 0, s>>>(params, grad, m, v, n, lr, b1, b2, 1e-8f,
                                                 weight_decay, c1, c2, w ? w->w : nullptr,
                                                 w ? w->wc : nullptr);
    return cudaGetLastError();
}

// Workspace of paid_proposal_train: the permutation, one minibatch of inputs
// and targets, the per-step losses of an epoch, the gradient and the forward /
// backward buffers of one minibatch.
struct TrainWork {
    int32_t* perm;
    __nv_bfloat16* xb;
    float* tb;
    float* losses;
    float* grad;
    char* mlp;
};

size_t train_work_bytes(int64_t M, int64_t batch, TrainWork* t, char* base)
{
    size_t o = 0;
    auto take = [&](size_t b) { size_t at = o; o = align256(o + b); return base ? base + at : nullptr; };
    const int64_t steps = (M + batch - 1) / batch;
    char* p;
    p = take(sizeof(int32_t) * M); if (t) t->perm = (int32_t*)p;
    p = take(sizeof(__nv_bfloat16) * batch * kIn); if (t) t->xb = (__nv_bfloat16*)p;
    p = take(sizeof(float) * batch * kHid); if (t) t->tb = (float*)p;
    p = take(sizeof(float) * steps); if (t) t->losses = (float*)p;
    p = take(sizeof(float) * param_count()); if (t) t->grad = (float*)p;
    p = take(mlp_work_bytes(batch, nullptr, nullptr)); if (t) t->mlp = p;
    return o;
}

// splitmix64 (Steele, Lea and Flood), the seeded source of the minibatch order
uint64_t splitmix64(uint64_t& z)
{
    uint64_t r = (z += 0x9e3779b97f4a7c15ull);
    r = (r ^ (r >> 30)) * 0xbf58476d1ce4e5b9ull;
    r = (r ^ (r >> 27)) * 0x94d049bb133111ebull;
    return r ^ (r >> 31);
}

constexpr char kMagic[8] = {'P', 'A', 'I', 'D', 'M', 'L', 'P', '1'};

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

}  // namespace

extern "C" {

int paid_mlp_param_count(int64_t* n)
{
    if (!n) return PAID_ERR_ARG;
    *n = param_count();
    return PAID_OK;
}

int paid_mlp_workspace_size(int64_t M, size_t* bytes)
{
    if (!bytes || M < 0) return PAID_ERR_ARG;
    *bytes = mlp_work_bytes(M, nullptr, nullptr);
    return PAID_OK;
}

int paid_mlp_init(float* params, uint64_t seed, void* stream)
{
    if (!params) return PAID_ERR_ARG;
    const int64_t n = param_count();
    k_init<<<int((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(params, seed);
    return cudaGetLastError() == cudaSuccess ? PAID_OK : PAID_ERR_CUDA;
}

int paid_mlp_forward(const float* params, const uint16_t* x, int64_t M, float* out, void* workspace,
                     size_t ws_bytes, void* stream)
{
    if (!params || (M > 0 && (!x || !out)) || M < 0) return PAID_ERR_ARG;
    if (M == 0) return PAID_OK;
    // the forward kernel stores output rows as 16-byte vectors and stages
    // weights with bulk copies from the workspace (16-byte aligned blocks)
    if (!aligned(out, 16) || !aligned(workspace, 256)) return PAID_ERR_ARG;
    if (M > int64_t(0x7fffffff)) return PAID_ERR_ARG;
    if (!workspace || ws_bytes < mlp_work_bytes(M, nullptr, nullptr)) return PAID_ERR_OOM;
    MlpWork w;
    mlp_work_bytes(M, &w, static_cast<char*>(workspace));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return cast_weights(params, w, s) == cudaSuccess &&
                   forward(params, reinterpret_cast<const __nv_bfloat16*>(x), M, out, w, s) ==
                       cudaSuccess
               ? PAID_OK : PAID_ERR_CUDA;
}

int paid_mlp_grad(const float* params, const uint16_t* x, const float* target, int64_t M,
                  float* grad, float* loss, void* workspace, size_t ws_bytes, void* stream)
{
    if (!params || !x || !target || !grad || !loss || M <= 0) return PAID_ERR_ARG;
    if (M > int64_t(0x7fffffff)) return PAID_ERR_ARG;
    if (!aligned(workspace, 256)) return PAID_ERR_ARG;
    if (!workspace || ws_bytes < mlp_work_bytes(M, nullptr, nullptr)) return PAID_ERR_OOM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    MlpWork w;
    mlp_work_bytes(M, &w, static_cast<char*>(workspace));
    return cast_weights(params, w, s) == cudaSuccess &&
                   cudaMemsetAsync(loss, 0, sizeof(float), s) == cudaSuccess &&
                   grad_rows(params, reinterpret_cast<const __nv_bfloat16*>(x), target, M, grad,
                             loss, w, s) == cudaSuccess
               ? PAID_OK : PAID_ERR_CUDA;
}

int paid_mlp_adamw(float* params, const float* grad, float* m, float* v, int step, float lr,
                   float weight_decay, void* stream)
{
    if (!params || !grad || !m || !v || step < 1) return PAID_ERR_ARG;
    return adamw_step(params, grad, m, v, step, lr, weight_decay, nullptr,
                      static_cast<cudaStream_t>(stream)) == cudaSuccess ? PAID_OK : PAID_ERR_CUDA;
}

int paid_proposal_train_workspace_size(int64_t M, int64_t batch, size_t* bytes)
{
    if (!bytes || M <= 0 || batch <= 0 || M > int64_t(0x7fffffff)) return PAID_ERR_ARG;
    *bytes = train_work_bytes(M, std::min(M, batch), nullptr, nullptr);
    return PAID_OK;
}

int paid_proposal_train(float* params, float* m, float* v, const uint16_t* x, const float* target,
                        int64_t M, int epochs, int64_t batch, float lr, float weight_decay,
                        uint64_t seed, int* step, float* epoch_loss, void* workspace,
                        size_t ws_bytes, void* stream)
{
    if (!params || !m || !v || !x || !target || !step || *step < 0 || M <= 0 || epochs < 0 ||
        batch <= 0 || M > int64_t(0x7fffffff) || !(lr >= 0.0f) || !(weight_decay >= 0.0f))
        return PAID_ERR_ARG;
    batch = std::min(M, batch);
    if (!aligned(workspace, 256)) return PAID_ERR_ARG;
    if (!workspace || ws_bytes < train_work_bytes(M, batch, nullptr, nullptr)) return PAID_ERR_OOM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    TrainWork t;
    train_work_bytes(M, batch, &t, static_cast<char*>(workspace));
    MlpWork w;
    mlp_work_bytes(batch, &w, t.mlp);
    const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(x);
    const int64_t steps = (M + batch - 1) / batch;
    const int64_t total = steps * int64_t(epochs);
    std::vector<int32_t> perm(static_cast<size_t>(M));
    std::vector<float> losses(static_cast<size_t>(steps));
    uint64_t z = seed;
    int64_t k = 0;
    if (total > 0 && cast_weights(params, w, s) != cudaSuccess) return PAID_ERR_CUDA;
    for (int ep = 0; ep < epochs; ++ep) {
        // a fresh Fisher-Yates order of the rows for every epoch
        for (int64_t i = 0; i < M; ++i) perm[size_t(i)] = int32_t(i);
        for (int64_t i = M - 1; i > 0; --i) {
            const int64_t j = int64_t(splitmix64(z) % uint64_t(i + 1));
            std::swap(perm[size_t(i)], perm[size_t(j)]);
        }
        // the host order is copied before this call returns control (pageable
        // source), so the vector may be refilled for the next epoch
        if (cudaMemcpyAsync(t.perm, perm.data(), sizeof(int32_t) * M, cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
            cudaMemsetAsync(t.losses, 0, sizeof(float) * steps, s) != cudaSuccess)
            return PAID_ERR_CUDA;
        for (int64_t b = 0; b < steps; ++b, ++k) {
            const int64_t r0 = b * batch, n = std::min(batch, M - r0);
            k_gather_rows<<<int((n * kHid + 255) / 256), 256, 0, s>>>(xb, target, t.perm, r0, n,
                                                                     t.xb, t.tb);
            // cosine decay of the learning rate over all steps of the call
            const float a = lr * 0.5f * (1.0f + cosf(3.14159265358979f * float(k) /
                                                     float(std::max<int64_t>(1, total))));
            if (grad_rows(params, t.xb, t.tb, n, t.grad, t.losses + b, w, s) != cudaSuccess ||
                adamw_step(params, t.grad, m, v, *step + 1, a, weight_decay, &w, s) != cudaSuccess)
                return PAID_ERR_CUDA;
            ++*step;
        }
        if (epoch_loss) {
            if (cudaMemcpyAsync(losses.data(), t.losses, sizeof(float) * steps,
                                cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                return PAID_ERR_CUDA;
            double sum = 0.0;
            for (float l : losses) sum += l;
            epoch_loss[ep] = float(sum / double(steps));
        }
    }
    return cudaGetLastError() == cudaSuccess ? PAID_OK : PAID_ERR_CUDA;
}

int paid_proposal_save(const float* params, const char* path, void* stream)
{
    if (!params || !path) return PAID_ERR_ARG;
    const int64_t n = param_count();
    std::vector<float> h(static_cast<size_t>(n));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(h.data(), params, sizeof(float) * n, cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return PAID_ERR_CUDA;
    FILE* f = std::fopen(path, "wb");
    if (!f) return PAID_ERR_ARG;
    const bool ok = std::fwrite(kMagic, 1, 8, f) == 8 && std::fwrite(&n, sizeof(n), 1, f) == 1 &&
                    std::fwrite(h.data(), sizeof(float), size_t(n), f) == size_t(n);
    return (std::fclose(f) == 0 && ok) ? PAID_OK : PAID_ERR_ARG;
}

int paid_proposal_load(float* params, const char* path, void* stream)
{
    if (!params || !path) return PAID_ERR_ARG;
    FILE* f = std::fopen(path, "rb");
    if (!f) return PAID_ERR_ARG;
    char magic[8] = {};
    int64_t n = 0;
    const int64_t want = param_count();
    std::vector<float> h(static_cast<size_t>(want));
    const bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMagic, 8) == 0 &&
                    std::fread(&n, sizeof(n), 1, f) == 1 && n == want &&
                    std::fread(h.data(), sizeof(float), size_t(n), f) == size_t(n) &&
                    std::fgetc(f) == EOF;
    std::fclose(f);
    if (!ok) return PAID_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the host copy lives on this call's stack: wait for the upload
    if (cudaMemcpyAsync(params, h.data(), sizeof(float) * n, cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return PAID_ERR_CUDA;
    return PAID_OK;
}

}  // extern "C"
