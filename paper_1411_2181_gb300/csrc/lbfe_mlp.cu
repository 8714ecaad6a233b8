// lbfe_mlp.cu -- the Ca_cr proposal network (lbfe_mlp.h):
// 6 -> 128 -> 128 -> 128 -> 128 -> 4, GELU.
//
//   k_net    forward, loss and data gradients of R rows per block: rows are
//            independent until the weight gradients, so one launch takes them
//            through all layers and back with every weight in shared memory;
//   k_wgrad  weight and bias gradients, 32 x 32 outputs per block, the batch
//            split over blocks and summed in a fixed order (deterministic);
//   k_adamw  the optimiser (in an epoch the last part of k_wgrad instead).
//
// The contractions are small (a 256-row step is 0.08 GFLOP, about 1 us of
// FP32 units) and activations and gradients are FP32, so they run on the
// CUDA cores.  Bound by latency: launches, and the chain of nine dependent
// layers.  Measured, with the host's part: an epoch of 1792 rows in batches of
// 256 took 3.82 ms layer by layer (fifteen launches of 2 to 16 blocks a batch,
// the weight gradient one serial sum over the batch per thread), 1.02 ms with
// these kernels and 0.48 ms as one call (lbfe_mlp_epoch: two launches a batch,
// no synchronisation between batches); gradient of 256 rows 22 us.  A forward
// pass of 341 rows from and to host arrays 179 -> 97 us (kernel 8 us).
#include <cmath>
#include <cstring>
#include <new>

#include "../../include/lbfe_mlp.h"
#include "lbfe_internal.cuh"

namespace lbfe {
// Whether [p, p + bytes) lies in one allocation of device dev (lbfe_capi.cu).
bool device_range(const void *p, size_t bytes, int dev);
}  // namespace lbfe

namespace {

constexpr int kLayers = 5;
// width of layer boundary l: 6, 128, 128, 128, 128, 4
__host__ __device__ constexpr int dim(int l) { return l == 0 ? 6 : (l == kLayers ? 4 : 128); }
constexpr int kHidden = 128;
constexpr int kNetThreads = 512;
constexpr int kTile = 32;       // weight-gradient tile
constexpr int kMaxSplit = 16;   // most parts of the batch in the weight gradients
constexpr int kSplitRows = 64;  // rows of a part staged at a time
constexpr int kMaxBatch = 65536;

__host__ __device__ constexpr size_t layer_offset(int l) {
    size_t o = 0;
    for (int k = 0; k < l; ++k) o += (size_t)dim(k) * dim(k + 1) + dim(k + 1);
    return o;
}
constexpr size_t kParams = layer_offset(kLayers);

// ---------------------------------------------------------------- k_net
// Shared memory of a block: the three 128 x 128 layers row by row (Wt[in][out],
// rows padded by 16 bytes: the forward reads along a row, the backward 16
// bytes of each of 32 rows, both without bank conflicts), the small layers and
// the biases in FP32, and the rows' activations [k][R].
template <typename W, int R>
struct NetSmem {
    static constexpr int ROW = kHidden * (int)sizeof(W) + 16;      // bytes of a padded row
    static constexpr int BIG = 0;                                  // [3][128] rows
    static constexpr int SMALL = 3 * kHidden * ROW;                // floats below
    static constexpr int W0 = 0, B0 = W0 + 6 * kHidden, B = B0 + kHidden, W4 = B + 3 * kHidden,
                         B4 = W4 + 4 * kHidden, X = B4 + 4, ACT = X + 8 * R, GRAD = ACT + kHidden * R,
                         RED = GRAD + 4 * kHidden * R, END = RED + 8 * kHidden * R;
    static constexpr size_t BYTES = SMALL + sizeof(float) * END;
    static_assert(BYTES <= 227 * 1024, "shared memory of a block");
    static_assert(SMALL % 16 == 0 && (ACT * 4) % 16 == 0 && (RED * 4) % 16 == 0, "16-byte rows");
};

template <typename W> struct WVec;
template <> struct WVec<__nv_bfloat16> {
    static __device__ __forceinline__ float2 pair(const char *p) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
    }
    static constexpr int N = 8;      // weights in 16 bytes
    static __device__ __forceinline__ void vec(const char *p, float w[N]) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w[2 * j] = __uint_as_float(u[j] << 16);
            w[2 * j + 1] = __uint_as_float(u[j] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ float one(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
};
template <> struct WVec<float> {
    static __device__ __forceinline__ float2 pair(const char *p) { return *reinterpret_cast<const float2 *>(p); }
    static constexpr int N = 4;
    static __device__ __forceinline__ void vec(const char *p, float w[N]) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
    static __device__ __forceinline__ float one(const float *p) { return *p; }
};

template <int R>
__device__ __forceinline__ void load_rows(const float *p, float a[R]) {
    if constexpr (R == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        a[0] = v.x;
        a[1] = v.y;
    }
#pragma unroll
    for (int q = 0; q < R / 4; ++q) {
        const float4 v = reinterpret_cast<const float4 *>(p)[q];
        a[4 * q] = v.x; a[4 * q + 1] = v.y; a[4 * q + 2] = v.z; a[4 * q + 3] = v.w;
    }
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Rows [r0, r0 + R) of the batch through the network; with GRAD also the loss
// (one FP64 partial per block) and dL/dZ of every layer.  A[l] and dZ[l] are
// [B][128] (l = 0..3), dY [B][4].
struct NetArgs {
    const void *w;                   // parameters in the kernel's weight type
    const float *x, *t, *mask;
    float *y, *A[4], *dZ[4], *dY;
    double *partial;
    int B;
};

template <typename W, int R, bool GRAD>
__global__ void __launch_bounds__(kNetThreads) k_net(const __grid_constant__ NetArgs N) {
    using Sm = NetSmem<W, R>;
    extern __shared__ __align__(16) char net_smem[];
    float *sf = reinterpret_cast<float *>(net_smem + Sm::SMALL);
    const W *w = (const W *)N.w;
    const int t = threadIdx.x, r0 = blockIdx.x * R, rows = min(R, N.B - r0);
    // every weight starts its way into shared memory, one group per layer
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const char *src = (const char *)(w + layer_offset(l + 1));
        constexpr int CH = kHidden * (int)sizeof(W) / 16;           // 16-byte chunks of a row
        for (int q = t; q < kHidden * CH; q += kNetThreads) {
            const int row = q / CH, c = q - row * CH;
            cp_async16(net_smem + Sm::BIG + (l * kHidden + row) * Sm::ROW + 16 * c, src + 16 * (size_t)q);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int q = t; q < 7 * kHidden; q += kNetThreads) sf[Sm::W0 + q] = WVec<W>::one(w + q);   // W0, then b0
    if (t < 3 * kHidden)
        sf[Sm::B + t] = WVec<W>::one(w + layer_offset(t / kHidden + 1) + kHidden * kHidden + (t & (kHidden - 1)));
    for (int q = t; q < 4 * kHidden + 4; q += kNetThreads) sf[Sm::W4 + q] = WVec<W>::one(w + layer_offset(4) + q);
    if (t < 6 * R) {
        const int r = t / 6, i = t - 6 * r;
        sf[Sm::X + i * R + r] = r < rows ? N.x[(size_t)(r0 + r) * 6 + i] : 0.f;
    }
    __syncthreads();
    float *act = sf + Sm::ACT, *red = sf + Sm::RED;
    // hidden output o of row r from its sum z: activation, its derivative, store
    auto finish = [&](int l, int o, int r, float z) {
        const float cdf = 0.5f * (1.0f + erff(z * 0.70710678118654752f));
        const float a = z * cdf;
        act[o * R + r] = a;
        if (GRAD) {
            sf[Sm::GRAD + (l * kHidden + o) * R + r] = cdf + z * 0.39894228040143268f * expf(-0.5f * z * z);
            if (r < rows) N.A[l][(size_t)(r0 + r) * kHidden + o] = a;
        }
    };
    {
        const int o = t & (kHidden - 1);
        for (int r = t >> 7; r < R; r += kNetThreads / kHidden) {
            float z = sf[Sm::B0 + o];
#pragma unroll
            for (int i = 0; i < 6; ++i) z += sf[Sm::X + i * R + r] * sf[Sm::W0 + i * kHidden + o];
            finish(0, o, r, z);
        }
    }
#pragma unroll
    for (int l = 1; l < 4; ++l) {
        if (l == 1) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (l == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // outputs 2 op and 2 op + 1, inputs [16 g, 16 g + 16) of all rows
        const int op = t & 63, g = t >> 6;
        const char *wp = net_smem + Sm::BIG + ((l - 1) * kHidden + 16 * g) * Sm::ROW + op * 2 * (int)sizeof(W);
        float s0[R], s1[R];
#pragma unroll
        for (int r = 0; r < R; ++r) s0[r] = s1[r] = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float2 v = WVec<W>::pair(wp + k * Sm::ROW);
            float a[R];
            load_rows<R>(act + (16 * g + k) * R, a);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                s0[r] += a[r] * v.x;
                s1[r] += a[r] * v.y;
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            *reinterpret_cast<float2 *>(red + (g * R + r) * kHidden + 2 * op) = make_float2(s0[r], s1[r]);
        __syncthreads();
        const int o = t & (kHidden - 1);
        for (int r = t >> 7; r < R; r += kNetThreads / kHidden) {
            float z = sf[Sm::B + (l - 1) * kHidden + o];
#pragma unroll
            for (int q = 0; q < 8; ++q) z += red[(q * R + r) * kHidden + o];
            finish(l, o, r, z);
        }
    }
    __syncthreads();
    // output layer: a warp per (row, output)
    float *y = red;                  // [R][4]
    for (int q = t >> 5; q < 4 * R; q += kNetThreads / 32) {
        const int r = q >> 2, o = q & 3, lane = t & 31;
        float s = 0.f;
#pragma unroll
        for (int k = lane; k < kHidden; k += 32) s += act[k * R + r] * sf[Sm::W4 + k * 4 + o];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        s += sf[Sm::B4 + o];
        if (lane == 0) {
            y[q] = s;
            if (N.y && r < rows) N.y[(size_t)(r0 + r) * 4 + o] = s;
        }
    }
    if (!GRAD) return;
    __syncthreads();
    float *dy = red + 4 * R;         // [R][4]
    double *ls = reinterpret_cast<double *>(red + 8 * R);           // [R]
    if (t < R) {
        double loss = 0.0;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        if (t < rows) {
            const float *yr = y + 4 * t, *tr = N.t + 4 * (size_t)(r0 + t);
            const float mk = N.mask ? N.mask[r0 + t] : 1.f;
            const float e0 = yr[0] - tr[0], e1 = yr[1] - tr[1], e3 = yr[3] - tr[3], z = yr[2];
            // binary cross-entropy of sigmoid(z) with target t[2], stable form
            const float bce = fmaxf(z, 0.f) - z * tr[2] + log1pf(expf(-fabsf(z)));
            const float sig = 1.f / (1.f + expf(-z));
            loss = (double)(mk * (e0 * e0 + e1 * e1 + e3 * e3) + bce);
            const float sc = 1.f / (float)N.B;
            d[0] = 2.f * mk * e0 * sc;
            d[1] = 2.f * mk * e1 * sc;
            d[2] = (sig - tr[2]) * sc;
            d[3] = 2.f * mk * e3 * sc;
            *reinterpret_cast<float4 *>(N.dY + 4 * (size_t)(r0 + t)) = make_float4(d[0], d[1], d[2], d[3]);
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) dy[4 * t + o] = d[o];
        ls[t] = loss;
    }
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int r = 0; r < R; ++r) s += ls[r];
        N.partial[blockIdx.x] = s;
    }
    // dZ of the last hidden layer, then down; dz [o][R] in act
    {
        const int i = t & (kHidden - 1);
        for (int r = t >> 7; r < R; r += kNetThreads / kHidden) {
            float s = 0.f;
#pragma unroll
            for (int o = 0; o < 4; ++o) s += dy[4 * r + o] * sf[Sm::W4 + 4 * i + o];
            s *= sf[Sm::GRAD + (3 * kHidden + i) * R + r];
            act[i * R + r] = s;
            if (r < rows) N.dZ[3][(size_t)(r0 + r) * kHidden + i] = s;
        }
    }
#pragma unroll
    for (int l = 3; l >= 1; --l) {
        __syncthreads();
        // input i of all rows from outputs [32 g, 32 g + 32)
        const int i = t & (kHidden - 1), g = t >> 7;
        const char *wp = net_smem + Sm::BIG + ((l - 1) * kHidden + i) * Sm::ROW + 32 * g * (int)sizeof(W);
        float s[R];
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = 0.f;
        constexpr int V = WVec<W>::N;
#pragma unroll
        for (int q = 0; q < 32 / V; ++q) {
            float v[V];
            WVec<W>::vec(wp + 16 * q, v);
#pragma unroll
            for (int j = 0; j < V; ++j) {
                float a[R];
                load_rows<R>(act + (32 * g + V * q + j) * R, a);
#pragma unroll
                for (int r = 0; r < R; ++r) s[r] += a[r] * v[j];
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) red[(g * R + r) * kHidden + i] = s[r];
        __syncthreads();
        for (int r = t >> 7; r < R; r += kNetThreads / kHidden) {
            float d = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) d += red[(q * R + r) * kHidden + i];
            d *= sf[Sm::GRAD + ((l - 1) * kHidden + i) * R + r];
            act[i * R + r] = d;
            if (r < rows) N.dZ[l - 1][(size_t)(r0 + r) * kHidden + i] = d;
        }
    }
}

// One layer of a forward pass with FP32 weights, sixteen rows per block: out =
// A W + b, with the activation where asked for.  k_net takes FP32 weights two
// rows a block, because little shared memory is left beside them, and every
// block brings all 197 KB of them in: 4.8 us a wave of blocks however many follow.
// Beyond fifteen waves five launches of this kernel, which reads its weights
// through the caches once for sixteen rows, are faster (fp32_layers).
constexpr int kLayerRows = 16;
__global__ void __launch_bounds__(kHidden)
k_layer(const float *__restrict__ A, int in, const float *__restrict__ w, int out, float *__restrict__ Z, bool act, int B) {
    __shared__ float tile[kLayerRows][kHidden];
    const int r0 = blockIdx.x * kLayerRows, o = threadIdx.x;
    for (int k = threadIdx.x; k < kLayerRows * in; k += kHidden) {
        const int r = k / in, i = k - r * in;
        tile[r][i] = r0 + r < B ? A[(size_t)(r0 + r) * in + i] : 0.f;
    }
    __syncthreads();
    if (o >= out) return;
    float acc[kLayerRows];
    const float bias = w[in * out + o];
#pragma unroll
    for (int r = 0; r < kLayerRows; ++r) acc[r] = bias;
    for (int i = 0; i < in; ++i) {
        const float v = w[i * out + o];
#pragma unroll
        for (int r = 0; r < kLayerRows; ++r) acc[r] += tile[r][i] * v;
    }
#pragma unroll
    for (int r = 0; r < kLayerRows; ++r) {
        if (r0 + r >= B) break;
        const float z = acc[r];
        Z[(size_t)(r0 + r) * out + o] = act ? z * (0.5f * (1.0f + erff(z * 0.70710678118654752f))) : z;
    }
}

// One AdamW step of parameter k; bc1, bc2: 1 - beta^t.
struct AdamArgs {
    float *w, *m, *v;                // w null: no step
    __nv_bfloat16 *w16;
    float lr, b1, b2, eps, wd, bc1, bc2;
};
__device__ __forceinline__ void adam_step(const AdamArgs &P, size_t k, float gk) {
    const float mk = P.b1 * P.m[k] + (1.f - P.b1) * gk;
    const float vk = P.b2 * P.v[k] + (1.f - P.b2) * gk * gk;
    P.m[k] = mk;
    P.v[k] = vk;
    const float upd = (mk / P.bc1) / (sqrtf(vk / P.bc2) + P.eps) + P.wd * P.w[k];
    const float wn = P.w[k] - P.lr * upd;
    P.w[k] = wn;
    P.w16[k] = __float2bfloat16_rn(wn);
}

// ---------------------------------------------------------------- k_wgrad
// Tile (i0, o0) of dW_l[i][o] = sum_b A_{l-1}[b][i] dZ_l[b][o] over the rows of
// part blockIdx.y, and, in the tiles with i0 = 0, of db_l[o] = sum_b dZ_l[b][o].
// With several parts each leaves its sums in part[], and the last part of a
// tile to finish adds them in the order of the parts.  In an epoch it also takes
// the optimiser's step (no kernel after this one reads the old weights).
constexpr int kTiles = 4 + 3 * 16 + 4;

struct WgradArgs {
    const float *x, *A[4], *dZ[4], *dY;
    float *g, *part;                 // gradient vector; [splits][kParams] partial sums
    unsigned *done;                  // [kTiles] finished parts, zero between launches
    const double *partial;           // k_net's loss partials, and where block 0 leaves their sum
    double *loss;
    AdamArgs adam;
    int B, rows, loss_blocks;        // rows of a part
};

__global__ void __launch_bounds__(256) k_wgrad(const __grid_constant__ WgradArgs G) {
    __shared__ __align__(16) float sa[kSplitRows][kTile], sd[kSplitRows][kTile];
    __shared__ bool s_last;
    const int t = threadIdx.x, tile = blockIdx.x, splits = gridDim.y;
    int l, i0, o0;
    if (tile < 4) { l = 0; i0 = 0; o0 = 32 * tile; }
    else if (tile < 52) { l = 1 + (tile - 4) / 16; i0 = 32 * ((tile - 4) / 4 % 4); o0 = 32 * ((tile - 4) & 3); }
    else { l = 4; i0 = 32 * (tile - 52); o0 = 0; }
    const int in = dim(l), out = dim(l + 1);
    const float *A = l == 0 ? G.x : G.A[l - 1];
    const float *D = l == 4 ? G.dY : G.dZ[l];
    const int ti = (t >> 4) * 2, to = (t & 15) * 2;
    float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, bsum = 0.f;
    const int b0 = blockIdx.y * G.rows, b1 = min(G.B, b0 + G.rows);
    for (int bb = b0; bb < b1; bb += kSplitRows) {
        const int n = min(kSplitRows, b1 - bb);
#pragma unroll
        for (int q = t; q < kSplitRows * kTile; q += 256) {
            const int r = q / kTile, c = q % kTile;
            sa[r][c] = r < n && i0 + c < in ? A[(size_t)(bb + r) * in + i0 + c] : 0.f;
            sd[r][c] = r < n && o0 + c < out ? D[(size_t)(bb + r) * out + o0 + c] : 0.f;
        }
        __syncthreads();
#pragma unroll 16
        for (int r = 0; r < kSplitRows; ++r) {
            const float2 a = *reinterpret_cast<const float2 *>(&sa[r][ti]);
            const float2 d = *reinterpret_cast<const float2 *>(&sd[r][to]);
            acc[0][0] += a.x * d.x; acc[0][1] += a.x * d.y;
            acc[1][0] += a.y * d.x; acc[1][1] += a.y * d.y;
        }
        if (i0 == 0 && t < kTile) {
#pragma unroll 16
            for (int r = 0; r < kSplitRows; ++r) bsum += sd[r][t];
        }
        __syncthreads();
    }
    const size_t base = layer_offset(l);
    float *dst = G.part + (size_t)blockIdx.y * kParams + base;
    auto finish = [&](int k, float v) {
        G.g[base + k] = v;
        if (G.adam.w) adam_step(G.adam, base + k, v);
    };
    auto each = [&](auto &&fn) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (i0 + ti + a < in && o0 + to + c < out) fn((i0 + ti + a) * out + o0 + to + c, acc[a][c]);
        if (i0 == 0 && t < kTile && o0 + t < out) fn(in * out + o0 + t, bsum);
    };
    if (splits == 1) {
        each([&](int k, float v) { finish(k, v); });
    } else {
        each([&](int k, float v) { dst[k] = v; });
        __threadfence();
        __syncthreads();
        if (t == 0) {
            s_last = atomicAdd(G.done + tile, 1u) == (unsigned)splits - 1;
            if (s_last) G.done[tile] = 0u;
            __threadfence();
        }
        __syncthreads();
        if (s_last)
            each([&](int k, float) {
                float v[kMaxSplit];
#pragma unroll
                for (int s = 0; s < kMaxSplit; ++s)
                    v[s] = s < splits ? __ldcg(G.part + (size_t)s * kParams + base + k) : 0.f;
                float sum = 0.f;
#pragma unroll
                for (int s = 0; s < kMaxSplit; ++s) sum += v[s];
                finish(k, sum);
            });
    }
    if (tile == 0 && blockIdx.y == 0) {
        // the loss: partials in a fixed order, strided sums then a tree
        __shared__ double red[256];
        double s = 0.0;
        for (int q = t; q < G.loss_blocks; q += 256) s += G.partial[q];
        red[t] = s;
        __syncthreads();
        for (int d = 128; d > 0; d >>= 1) {
            if (t < d) red[t] += red[t + d];
            __syncthreads();
        }
        if (t == 0) G.loss[0] = red[0];
    }
}

__global__ void k_adamw(size_t n, const __grid_constant__ AdamArgs P, const float *__restrict__ g) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) adam_step(P, k, g[k]);
}

__global__ void k_to_bf16(size_t n, const float *__restrict__ w, __nv_bfloat16 *__restrict__ w16) {
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) w16[k] = __float2bfloat16_rn(w[k]);
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

struct MlpLayout {
    size_t w32, w16, m, v, g, done, A[kLayers - 1], dZ[kLayers - 1], dY, partial, losses, part, total;
};

constexpr int kFp32Rows = 2, kSmallRows = 4, kLargeRows = 16;   // rows of a k_net block

constexpr int kEpochLosses = 1024;   // batches of an epoch between two readings of their losses

MlpLayout mlp_plan(int B) {
    MlpLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align256(off + bytes); return o; };
    L.w32 = take(sizeof(float) * kParams);
    L.w16 = take(sizeof(__nv_bfloat16) * kParams);
    L.m = take(sizeof(float) * kParams);
    L.v = take(sizeof(float) * kParams);
    L.g = take(sizeof(float) * kParams);
    L.done = take(sizeof(unsigned) * kTiles);
    for (int l = 0; l < kLayers - 1; ++l) L.A[l] = take(sizeof(float) * (size_t)B * kHidden);
    for (int l = 0; l < kLayers - 1; ++l) L.dZ[l] = take(sizeof(float) * (size_t)B * kHidden);
    L.dY = take(sizeof(float) * (size_t)B * 4);
    L.partial = take(sizeof(double) * (size_t)((B + kFp32Rows - 1) / kFp32Rows));
    L.losses = take(sizeof(double) * kEpochLosses);
    L.part = take(sizeof(float) * kParams * kMaxSplit);
    L.total = off;
    return L;
}

}  // namespace

struct lbfe_mlp {
    int max_batch = 0, use16 = 1, steps = 0, device = -1;
    cudaStream_t stream = nullptr;
    char *base = nullptr;
    MlpLayout L;
    float *p32() const { return (float *)(base + L.w32); }
    __nv_bfloat16 *p16() const { return (__nv_bfloat16 *)(base + L.w16); }
    float *f(size_t off) const { return (float *)(base + off); }
};

namespace {

template <typename W, int R, bool GRAD>
cudaError_t net_launch(const NetArgs &N, cudaStream_t st) {
    // per device and cheap: every call states the shared memory it needs
    const cudaError_t e = cudaFuncSetAttribute(k_net<W, R, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)NetSmem<W, R>::BYTES);
    if (e != cudaSuccess) return e;
    k_net<W, R, GRAD><<<(N.B + R - 1) / R, kNetThreads, NetSmem<W, R>::BYTES, st>>>(N);
    return cudaGetLastError();
}

// Rows of a k_net block.  Four fill the GPU from small batches on (a row's
// time through the layers is latency); above four waves of such blocks the
// weights' way into shared memory counts, and sixteen rows share it.  FP32
// weights leave room for the activations of two rows.
int net_rows(const lbfe_mlp *m, int B) {
    if (!m->use16) return kFp32Rows;
    return B > 4 * 152 * kSmallRows ? kLargeRows : kSmallRows;
}

template <bool GRAD>
cudaError_t net(lbfe_mlp *m, const float *x, const float *t, const float *mask, int B, float *y) {
    NetArgs N{};
    N.w = m->use16 ? (const void *)m->p16() : (const void *)m->p32();
    N.x = x;
    N.t = t;
    N.mask = mask;
    N.y = y;
    for (int l = 0; l < kLayers - 1; ++l) {
        N.A[l] = m->f(m->L.A[l]);
        N.dZ[l] = m->f(m->L.dZ[l]);
    }
    N.dY = m->f(m->L.dY);
    N.partial = (double *)(m->base + m->L.partial);
    N.B = B;
    if (!m->use16) return net_launch<float, kFp32Rows, GRAD>(N, m->stream);
    return net_rows(m, B) == kLargeRows ? net_launch<__nv_bfloat16, kLargeRows, GRAD>(N, m->stream)
                                        : net_launch<__nv_bfloat16, kSmallRows, GRAD>(N, m->stream);
}

// Whether a forward pass goes layer by layer (k_layer).  Measured, us, k_net /
// layers: 4560 rows 78 / 70, 8192 rows 134 / 82, 65536 rows 1010 / 380.
bool fp32_layers(const lbfe_mlp *m, int B) { return !m->use16 && B > 15 * 152 * kFp32Rows; }

cudaError_t forward(lbfe_mlp *m, const float *x, int B, float *y) {
    if (!fp32_layers(m, B)) return net<false>(m, x, nullptr, nullptr, B, y);
    const float *a = x;
    for (int l = 0; l < kLayers; ++l) {
        float *z = l < kLayers - 1 ? m->f(m->L.A[l]) : y;
        k_layer<<<(B + kLayerRows - 1) / kLayerRows, kHidden, 0, m->stream>>>(a, dim(l), m->p32() + layer_offset(l),
                                                                             dim(l + 1), z, l < kLayers - 1, B);
        a = z;
    }
    return cudaGetLastError();
}

// Gradient of a batch, its loss sum (FP64) into *loss, and the optimiser's step
// where adam asks for one.
cudaError_t loss_grad(lbfe_mlp *m, const float *x_dev, const float *t_dev, const float *mask_dev, int B, double *loss,
                      const AdamArgs &adam) {
    cudaError_t e = net<true>(m, x_dev, t_dev, mask_dev, B, nullptr);
    if (e != cudaSuccess) return e;
    WgradArgs G{};
    G.x = x_dev;
    for (int l = 0; l < kLayers - 1; ++l) {
        G.A[l] = m->f(m->L.A[l]);
        G.dZ[l] = m->f(m->L.dZ[l]);
    }
    G.dY = m->f(m->L.dY);
    G.g = m->f(m->L.g);
    G.part = m->f(m->L.part);
    G.done = (unsigned *)(m->base + m->L.done);
    G.partial = (const double *)(m->base + m->L.partial);
    G.loss = loss;
    G.adam = adam;
    G.B = B;
    // parts of at least 64 rows (one staging round), at most 16 of them
    int splits = (B + kSplitRows - 1) / kSplitRows;
    if (splits > kMaxSplit) splits = kMaxSplit;
    G.rows = ((B + splits - 1) / splits + kSplitRows - 1) / kSplitRows * kSplitRows;
    splits = (B + G.rows - 1) / G.rows;
    const int R = net_rows(m, B);
    G.loss_blocks = (B + R - 1) / R;
    k_wgrad<<<dim3(kTiles, splits), 256, 0, m->stream>>>(G);
    return cudaGetLastError();
}

AdamArgs adam_args(lbfe_mlp *m, float lr, float beta1, float beta2, float eps, float weight_decay) {
    m->steps += 1;
    AdamArgs P{};
    P.w = m->p32();
    P.w16 = m->p16();
    P.m = m->f(m->L.m);
    P.v = m->f(m->L.v);
    P.lr = lr;
    P.b1 = beta1;
    P.b2 = beta2;
    P.eps = eps;
    P.wd = weight_decay;
    P.bc1 = 1.f - powf(beta1, (float)m->steps);
    P.bc2 = 1.f - powf(beta2, (float)m->steps);
    return P;
}

bool adam_valid(float lr, float beta1, float beta2, float eps) {
    return lr >= 0.f && beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f && beta2 < 1.f && eps > 0.f;
}

}  // namespace

extern "C" {

size_t lbfe_mlp_param_count(void) { return kParams; }

lbfe_status lbfe_mlp_required_bytes(int max_batch, size_t *bytes) {
    if (max_batch < 1 || max_batch > kMaxBatch || !bytes) return LBFE_ERR_BAD_PARAM;
    *bytes = mlp_plan(max_batch).total;
    return LBFE_OK;
}

lbfe_status lbfe_mlp_create(lbfe_mlp **mp, int max_batch, int weights_bf16, void *device_block, size_t bytes,
                            void *stream) {
    if (!mp) return LBFE_ERR_BAD_PARAM;
    *mp = nullptr;
    size_t need = 0;
    lbfe_status s = lbfe_mlp_required_bytes(max_batch, &need);
    if (s != LBFE_OK) return s;
    if (!device_block || ((uintptr_t)device_block % 256) != 0) return LBFE_ERR_BAD_PARAM;
    if (bytes < need) return LBFE_ERR_NO_MEMORY;
    lbfe_mlp *m = new (std::nothrow) lbfe_mlp;
    if (!m) return LBFE_ERR_NO_MEMORY;
    m->max_batch = max_batch;
    m->use16 = weights_bf16 ? 1 : 0;
    m->stream = (cudaStream_t)stream;
    m->base = (char *)device_block;
    m->L = mlp_plan(max_batch);
    cudaError_t e = cudaGetDevice(&m->device);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->base, 0, m->L.A[0], m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        delete m;
        return LBFE_ERR_CUDA;
    }
    *mp = m;
    return LBFE_OK;
}

lbfe_status lbfe_mlp_set_params(lbfe_mlp *m, const float *host_params) {
    if (!m || !host_params) return LBFE_ERR_BAD_PARAM;
    cudaError_t e = cudaMemcpyAsync(m->p32(), host_params, sizeof(float) * kParams, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->f(m->L.m), 0, sizeof(float) * kParams, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->f(m->L.v), 0, sizeof(float) * kParams, m->stream);
    if (e == cudaSuccess) {
        k_to_bf16<<<(unsigned)((kParams + 255) / 256), 256, 0, m->stream>>>(kParams, m->p32(), m->p16());
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    m->steps = 0;
    return e == cudaSuccess ? LBFE_OK : LBFE_ERR_CUDA;
}

lbfe_status lbfe_mlp_get_params(lbfe_mlp *m, float *host_params) {
    if (!m || !host_params) return LBFE_ERR_BAD_PARAM;
    cudaError_t e = cudaMemcpyAsync(host_params, m->p32(), sizeof(float) * kParams, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? LBFE_OK : LBFE_ERR_CUDA;
}

lbfe_status lbfe_mlp_forward(lbfe_mlp *m, const float *x_dev, int batch, float *y_dev) {
    if (!m || !x_dev || !y_dev || batch < 1 || batch > m->max_batch) return LBFE_ERR_BAD_PARAM;
    // The blocks write their rows of y while others still read x.  Where y overlaps x, or
    // does not lie in one allocation of the network's device, the result goes through the
    // workspace (the loss gradient's dY) and a copy, which refuses what is no such buffer.
    const size_t bytes = sizeof(float) * 4 * (size_t)batch;
    const uintptr_t x0 = (uintptr_t)x_dev, y0 = (uintptr_t)y_dev;
    const bool apart = y0 + bytes <= x0 || x0 + sizeof(float) * 6 * (size_t)batch <= y0;
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return LBFE_ERR_CUDA;
    const bool direct = apart && device == m->device && lbfe::device_range(y_dev, bytes, device);
    float *y = direct ? y_dev : m->f(m->L.dY);
    cudaError_t e = forward(m, x_dev, batch, y);
    if (e == cudaSuccess && !direct) e = cudaMemcpyAsync(y_dev, y, bytes, cudaMemcpyDeviceToDevice, m->stream);
    return e == cudaSuccess ? LBFE_OK : LBFE_ERR_CUDA;
}

lbfe_status lbfe_mlp_loss_grad(lbfe_mlp *m, const float *x_dev, const float *t_dev, const float *mask_dev, int batch,
                               float *loss_host) {
    if (!m || !x_dev || !t_dev || batch < 1 || batch > m->max_batch) return LBFE_ERR_BAD_PARAM;
    cudaError_t e = loss_grad(m, x_dev, t_dev, mask_dev, batch, (double *)(m->base + m->L.losses), AdamArgs{});
    if (e != cudaSuccess) return LBFE_ERR_CUDA;
    if (loss_host) {
        double sum = 0.0;
        e = cudaMemcpyAsync(&sum, m->base + m->L.losses, sizeof sum, cudaMemcpyDeviceToHost, m->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
        if (e != cudaSuccess) return LBFE_ERR_CUDA;
        *loss_host = (float)(sum / batch);
    }
    return LBFE_OK;
}

lbfe_status lbfe_mlp_get_grads(lbfe_mlp *m, float *host_grads) {
    if (!m || !host_grads) return LBFE_ERR_BAD_PARAM;
    cudaError_t e = cudaMemcpyAsync(host_grads, m->f(m->L.g), sizeof(float) * kParams, cudaMemcpyDeviceToHost,
                                    m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? LBFE_OK : LBFE_ERR_CUDA;
}

lbfe_status lbfe_mlp_adamw(lbfe_mlp *m, float lr, float beta1, float beta2, float eps, float weight_decay) {
    if (!m || !adam_valid(lr, beta1, beta2, eps)) return LBFE_ERR_BAD_PARAM;
    k_adamw<<<(unsigned)((kParams + 255) / 256), 256, 0, m->stream>>>(
        kParams, adam_args(m, lr, beta1, beta2, eps, weight_decay), m->f(m->L.g));
    return cudaGetLastError() == cudaSuccess ? LBFE_OK : LBFE_ERR_CUDA;
}

lbfe_status lbfe_mlp_epoch(lbfe_mlp *m, const float *x_dev, const float *t_dev, const float *mask_dev, int rows,
                           int batch, float lr, float beta1, float beta2, float eps, float weight_decay,
                           double *loss_sum_host) {
    if (!m || !x_dev || !t_dev || rows < 1 || batch < 1 || batch > m->max_batch || !adam_valid(lr, beta1, beta2, eps))
        return LBFE_ERR_BAD_PARAM;
    double *losses = (double *)(m->base + m->L.losses), host[kEpochLosses];
    double total = 0.0;
    long long first = 0;             // row of losses[0]
    int n = 0;                       // batches since
    auto read = [&]() {
        if (!loss_sum_host || n == 0) return cudaSuccess;
        cudaError_t e = cudaMemcpyAsync(host, losses, sizeof(double) * n, cudaMemcpyDeviceToHost, m->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
        if (e != cudaSuccess) return e;
        for (int k = 0; k < n; ++k, first += batch) {
            const int B = (int)(rows - first < batch ? rows - first : batch);
            total += (double)(float)(host[k] / B) * B;
        }
        n = 0;
        return cudaSuccess;
    };
    for (long long s = 0; s < rows; s += batch) {
        const int B = (int)(rows - s < batch ? rows - s : batch);
        cudaError_t e = loss_grad(m, x_dev + 6 * s, t_dev + 4 * s, mask_dev ? mask_dev + s : nullptr, B, losses + n,
                                  adam_args(m, lr, beta1, beta2, eps, weight_decay));
        if (e == cudaSuccess && ++n == kEpochLosses) {
            e = read();
            n = 0;
        }
        if (e != cudaSuccess) return LBFE_ERR_CUDA;
    }
    if (read() != cudaSuccess) return LBFE_ERR_CUDA;
    if (loss_sum_host) *loss_sum_host = total;
    return LBFE_OK;
}

lbfe_status lbfe_mlp_destroy(lbfe_mlp *m) {
    if (!m) return LBFE_ERR_BAD_PARAM;
    cudaStreamSynchronize(m->stream);
    delete m;
    return LBFE_OK;
}

}  // extern "C"
