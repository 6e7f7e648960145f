// The VLM's LLM prefill (App. A, Tab. "Model architecture parameters of pi series VLA models",
// Sec. 4.3): Gemma-shaped blocks over the prefix tokens, writing each layer's rotated keys and
// values straight into the action expert's KV store.
//
// The Q/K/V, output, gate/up and down projections are plain GEMMs with batch * prefix rows (816
// per request) on this file's tcgen05 GEMM (bf16 operands by bulk tensor copies, fp32
// accumulation in TMEM, see k_pf_gemm); the residual stream stays fp32 and the two residual
// projections accumulate into it in place. Attention (all heads stacked as query rows, since the
// single KV head is shared) runs on the expert's tcgen05 attention kernel with every key visible;
// for head dims or store strides that kernel does not take, it falls back to per-request GEMMs:
// the scores q K^T, a row softmax, V transposed, and the probabilities times V. This file's other
// kernels do the rest: RMSNorm to a bf16 operand, rotary coding of q and k from a table built
// once in double precision (with k and v scattered into the store), and GeGLU.

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <new>
#include <type_traits>
#include <vector>

#include "jpi_prefill.h"
#include "../ptx.h"
#include "../attn_t5_kernel.cuh"

namespace {

thread_local char g_err[1024] = "";

jpi_status pfail(jpi_status s, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return s;
}

#define PF_CUDA(expr)                                                                              \
    do {                                                                                           \
        cudaError_t e_ = (expr);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return pfail(JPI_ERR_CUDA, "%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e_),     \
                         __FILE__, __LINE__);                                                      \
    } while (0)

#define PF_TRY(expr)                         \
    do {                                     \
        jpi_status s_ = (expr);              \
        if (s_ != JPI_OK) return s_;         \
    } while (0)

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

__device__ __forceinline__ float gelu_tanh_f(float y) {
    // 0.5 y (1 + tanh(sqrt(2/pi) (y + 0.044715 y^3))), the tanh form of GELU.
    return 0.5f * y * (1.f + tanhf(0.7978845608028654f * (y + 0.044715f * y * y * y)));
}

__global__ void k_pf_cast(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16_rn(src[i]);
}

// h = x (fp32 or bf16 embeddings) as the fp32 residual stream.
__global__ void k_pf_load_x(const void* __restrict__ x, int x_fp32, float* __restrict__ h, long long n) {
    jpi::ptx::grid_dep_launch();   // the next kernel waits for this one's results
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        h[i] = x_fp32 ? static_cast<const float*>(x)[i] : __bfloat162float(static_cast<const __nv_bfloat16*>(x)[i]);
}

// Row kernels of W floats (W a multiple of 4): one block of RB threads per row (grid-stride over
// rows), a row of up to RB x RB_CAP float4 held in registers with every load in flight, the sum
// of squares reduced over the block.
constexpr int RB = 128;
constexpr int RB_CAP = 8;   // 4096 floats per row
__device__ __forceinline__ float block_sum_rb(float v, float* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < RB / 32; ++i) t += red[i];
    __syncthreads();   // red is reused by the next row
    return t;
}
// y[4 i .. 4 i + 3] of row r = v * rinv * (1 + w). An fp32 y is the caller's and may be only
// element-aligned.
template <typename TO>
__device__ __forceinline__ void store_normed4(TO* y, const float* w, long long r, int W, int i, float4 v, float rinv) {
    const float4 g = reinterpret_cast<const float4*>(w)[i];
    const float a0 = v.x * rinv * (1.f + g.x), a1 = v.y * rinv * (1.f + g.y);
    const float a2 = v.z * rinv * (1.f + g.z), a3 = v.w * rinv * (1.f + g.w);
    if constexpr (sizeof(TO) == 2) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(a0, a1), hi = __floats2bfloat162_rn(a2, a3);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t*>(&lo);
        u.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(y + r * W + 4 * i) = u;
    } else if ((reinterpret_cast<uintptr_t>(y) & 15) == 0) {
        *reinterpret_cast<float4*>(y + r * W + 4 * i) = make_float4(a0, a1, a2, a3);
    } else {
        y += r * W + 4 * i;
        y[0] = a0;
        y[1] = a1;
        y[2] = a2;
        y[3] = a3;
    }
}
__device__ __forceinline__ float sq4(float4 v) {
    return (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
}

// y = h / sqrt(mean(h^2) + eps) * (1 + w), row by row.
template <typename TO>
__global__ void __launch_bounds__(RB) k_pf_rmsnorm(const float* __restrict__ h, const float* __restrict__ w,
                                                   TO* __restrict__ y, long long rows, int W, float eps) {
    __shared__ float red[RB / 32];
    const int t = threadIdx.x, n4 = W >> 2;
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
        const float4* hr = reinterpret_cast<const float4*>(h + r * W);
        if (n4 <= RB * RB_CAP) {
            float4 v[RB_CAP];
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                v[k] = i < n4 ? hr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) s += sq4(v[k]);
            const float rinv = 1.f / sqrtf(block_sum_rb(s, red) / (float)W + eps);
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                if (i < n4) store_normed4(y, w, r, W, i, v[k], rinv);
            }
        } else {
            float s = 0.f;
            for (int i = t; i < n4; i += RB) s += sq4(hr[i]);
            const float rinv = 1.f / sqrtf(block_sum_rb(s, red) / (float)W + eps);
            for (int i = t; i < n4; i += RB) store_normed4(y, w, r, W, i, hr[i], rinv);
        }
    }
}

// From the projections qkv [B P][(H + 2) D] (fp32): rotated queries q [B P][H][D] (bf16), and the
// rotated keys and the values of request b, row p into kd / vd + b stride + p D (bf16). One block
// per token row (grid-stride), its threads over the (section, rotary pair) slots of the row;
// rope[p][j] = (cos, sin) of p base^(-2j/D).
__global__ void k_pf_rope_scatter(const float* __restrict__ qkv, const float2* __restrict__ rope,
                                  __nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ kd,
                                  __nv_bfloat16* __restrict__ vd, long long stride, int B, int P, int H,
                                  int D) {
    const int half = D / 2, secs = H + 2, slots = secs * half;
    constexpr int RS_BATCH = 8;   // slots of a thread whose loads are in flight together
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    for (long long r = blockIdx.x; r < (long long)B * P; r += gridDim.x) {   // r = b P + p
        const int p = (int)(r % P), b = (int)(r / P);
        const float* row = qkv + r * (long long)secs * D;
        for (int t0 = threadIdx.x; t0 < slots; t0 += RS_BATCH * blockDim.x) {
            float x1[RS_BATCH], x2[RS_BATCH];
            float2 cs[RS_BATCH];
#pragma unroll
            for (int u = 0; u < RS_BATCH; ++u) {
                const int t = t0 + u * blockDim.x;
                x1[u] = x2[u] = 0.f;
                cs[u] = make_float2(1.f, 0.f);
                if (t < slots) {
                    const int s = t / half, j = t - s * half;
                    const float* src = row + s * D;
                    x1[u] = src[j];
                    x2[u] = src[j + half];
                    if (s <= H) cs[u] = rope[(size_t)p * half + j];
                }
            }
#pragma unroll
            for (int u = 0; u < RS_BATCH; ++u) {
                const int t = t0 + u * blockDim.x;
                if (t >= slots) break;
                const int s = t / half, j = t - s * half;
                float y1 = x1[u], y2 = x2[u];
                if (s <= H) {
                    y1 = x1[u] * cs[u].x - x2[u] * cs[u].y;
                    y2 = x2[u] * cs[u].x + x1[u] * cs[u].y;
                }
                __nv_bfloat16* dst;
                if (s < H) dst = q + (r * H + s) * (long long)D;
                else dst = (s == H ? kd : vd) + b * stride + (long long)p * D;
                dst[j] = __float2bfloat16_rn(y1);
                dst[j + half] = __float2bfloat16_rn(y2);
            }
        }
    }
}

// probs[r][0 .. n) = softmax(s[r][0 .. n)) as bf16 (rows of stride ld); one warp per row. Rows of
// up to SM_CAP values per lane are read once into registers (all loads in flight together);
// longer rows take three strided passes.
constexpr int SM_CAP = 32;   // 1024 keys
__global__ void __launch_bounds__(256) k_pf_softmax(const float* __restrict__ s, __nv_bfloat16* __restrict__ p,
                                                    long long rows, int n, int ld) {
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows; r += nwarps) {
        const float* sr = s + r * ld;
        __nv_bfloat16* pr = p + r * ld;
        if (n <= 32 * SM_CAP) {
            float v[SM_CAP];
            float mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < SM_CAP; ++k) {
                const int j = lane + 32 * k;
                v[k] = j < n ? sr[j] : -INFINITY;
            }
#pragma unroll
            for (int k = 0; k < SM_CAP; ++k) mx = fmaxf(mx, v[k]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float den = 0.f;
#pragma unroll
            for (int k = 0; k < SM_CAP; ++k) {
                v[k] = lane + 32 * k < n ? expf(v[k] - mx) : 0.f;
                den += v[k];
            }
            const float inv = 1.f / warp_sum(den);
#pragma unroll
            for (int k = 0; k < SM_CAP; ++k) {
                const int j = lane + 32 * k;
                if (j < n) pr[j] = __float2bfloat16_rn(v[k] * inv);
            }
        } else {
            float mx = -INFINITY;
            for (int j = lane; j < n; j += 32) mx = fmaxf(mx, sr[j]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            float den = 0.f;
            for (int j = lane; j < n; j += 32) den += expf(sr[j] - mx);
            const float inv = 1.f / warp_sum(den);
            for (int j = lane; j < n; j += 32) pr[j] = __float2bfloat16_rn(expf(sr[j] - mx) * inv);
        }
    }
}

// Stream-K pieces of tile t (nkb k-blocks each) over T units and G CTAs: first CTA and count.
__host__ __device__ __forceinline__ int pg_cta_of(long long x, long long T, int G) {
    return (int)(((x + 1) * G - 1) / T);
}
__host__ __device__ __forceinline__ int pg_pieces(int t, int nkb, long long T, int G) {
    return pg_cta_of((long long)(t + 1) * nkb - 1, T, G) - pg_cta_of((long long)t * nkb, T, G) + 1;
}

// After a stream-K product: h += (piece 0 + piece 1 + ...) of each 128 x 256 tile in order (pieces
// [rows][W] fp32, `pstride` elements apart; ntm row tiles, nkb k-blocks a tile dealt to G CTAs), then,
// when w is set, the next RMSNorm y = h / sqrt(mean(h^2) + eps) * (1 + w) as k_pf_rmsnorm computes it.
template <typename TO>
__global__ void __launch_bounds__(RB) k_pf_residual_norm(float* __restrict__ h, const float* __restrict__ parts,
                                                         long long pstride, int ntm, int nkb, long long T, int G,
                                                         const float* __restrict__ w, TO* __restrict__ y, long long rows,
                                                         int W, float eps) {
    __shared__ float red[RB / 32];
    const int t = threadIdx.x, n4 = W >> 2;
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
        float4* hr = reinterpret_cast<float4*>(h + r * W);
        const int tm = (int)(r >> 7);
        // Pieces of the tile that holds float4 i of this row (256 columns are 64 float4).
        auto pieces = [&](int i) { return pg_pieces((i >> 6) * ntm + tm, nkb, T, G); };
        auto part = [&](int q) { return reinterpret_cast<const float4*>(parts + (size_t)q * pstride + r * W); };
        if (n4 <= RB * RB_CAP) {
            // Passes over the row held in registers: piece 0, each further piece, then h.
            float4 v[RB_CAP];
            int np[RB_CAP], most = 0;
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                np[k] = i < n4 ? pieces(i) : 0;
                most = max(most, np[k]);
                v[k] = i < n4 ? part(0)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            for (int q = 1; q < most; ++q) {
#pragma unroll
                for (int k = 0; k < RB_CAP; ++k) {
                    if (q < np[k]) {
                        const float4 e = part(q)[t + RB * k];
                        v[k] = make_float4(v[k].x + e.x, v[k].y + e.y, v[k].z + e.z, v[k].w + e.w);
                    }
                }
            }
            // The residual row: every load before the stores that update it.
            float4 o[RB_CAP];
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                o[k] = i < n4 ? hr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                if (i < n4) {
                    v[k] = make_float4(o[k].x + v[k].x, o[k].y + v[k].y, o[k].z + v[k].z, o[k].w + v[k].w);
                    hr[i] = v[k];
                }
            }
            if (!w) continue;
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) s += sq4(v[k]);
            const float rinv = 1.f / sqrtf(block_sum_rb(s, red) / (float)W + eps);
#pragma unroll
            for (int k = 0; k < RB_CAP; ++k) {
                const int i = t + RB * k;
                if (i < n4) store_normed4(y, w, r, W, i, v[k], rinv);
            }
        } else {
            float s = 0.f;
            for (int i = t; i < n4; i += RB) {
                float4 d = part(0)[i];
                const int np = pieces(i);
                for (int q = 1; q < np; ++q) {
                    const float4 e = part(q)[i];
                    d = make_float4(d.x + e.x, d.y + e.y, d.z + e.z, d.w + e.w);
                }
                const float4 o = hr[i];
                const float4 v = make_float4(o.x + d.x, o.y + d.y, o.z + d.z, o.w + d.w);
                hr[i] = v;
                s += sq4(v);
            }
            if (!w) continue;
            const float rinv = 1.f / sqrtf(block_sum_rb(s, red) / (float)W + eps);
            for (int i = t; i < n4; i += RB) store_normed4(y, w, r, W, i, hr[i], rinv);
        }
    }
}

// Gate (off = 0) or up (off = 128) rows [F][W] fp32 -> bf16 rows of the packed gate/up matrix,
// where 256-row tile t holds gate rows 128 t..128 t + 127, then the up rows of the same features.
__global__ void k_pf_cast_gu(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, int F, int W, int off) {
    const long long n = (long long)F * W;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int f = (int)(i / W), c = (int)(i - (long long)f * W);
        const long long row = (long long)(f >> 7) * 256 + off + (f & 127);
        dst[row * W + c] = __float2bfloat16_rn(src[i]);
    }
}

int grid_for(long long threads, int block = 256, int cap = 16384) {
    long long g = (threads + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

struct LayerW {
    __nv_bfloat16 *wqkv = nullptr, *wo = nullptr, *wgu = nullptr, *wd = nullptr;
    float *attn_norm = nullptr, *mlp_norm = nullptr;
};

// ---------------------------------------------------------------------------------------------
// The products: Y[m][n] = alpha sum_k X[m][k] W[n][k] (+ Y[m][n]), X [M][K] and W [N][K] row-major
// bf16, Y fp32 or bf16, fp32 accumulation. One output tile = 128 rows of X (the MMA's M) x 256
// rows of W (its N) over the whole K range, in TMEM as [X row = lane][W row = column]: each k-block
// brings 48 KB into the SM for 2 M multiply-adds (a 128 x 128 tile brings 32 KB for 1 M), and only the
// token dimension, 816 rows at Gemma-2B sizes, is padded. Persistent: one CTA per SM walks the tiles
// u = blockIdx.x, + gridDim.x, ... with the X tile fastest, so the CTAs that run together share one W
// tile through L2 and every W tile is read from HBM once (W is the large operand: 134 MB for
// gate/up, X 3.3 MB):
//   warp 0  one thread streams (X block, W block) pairs of 64 K-columns by bulk tensor copies
//           (128-byte swizzle; rows and columns past the tensors' extents arrive as zeros) into a
//           ring of PG_STAGES stages (W blocks of the first stages before the dependency wait);
//   warp 1  one thread issues the tcgen05.mma chain (M = 128, N = 256, K = 16 each) into one of two
//           TMEM accumulators and releases each stage through tcgen05.commit;
//   warps 2-9  one TMEM lane (X row m) per thread, two groups of four warps with half of the columns
//           each. Every warp passes its 32 rows through 4 KB of shared memory of its own, 128 bytes of
//           a row at a time (16-byte chunks XOR-swizzled by the row), and writes 128-byte pieces of four
//           rows per instruction (a row per thread, each store would touch 32 lines). The QKV form applies
//           the rotary coding there and scatters q, k and v.
// Stream-K (args.stream): a product with fewer tiles than SMs deals its (tile, k-block) units out
// evenly, CTA c taking [c T / G, (c + 1) T / G); each piece of a tile goes to its own partial buffer
// (piece p of a tile: the p-th CTA that touches it), and the consumer adds a tile's pieces in order.
// Every wait is bounded; a timeout records a device error in the handle's word and the CTA returns.

constexpr int PG_TM = 128;                                      // X rows per tile (MMA M)
constexpr int PG_TN = 256;                                      // W rows per tile (MMA N)
constexpr int PG_KBLK = 64;
constexpr int PG_STAGES = 4;
constexpr int PG_XBYTES = PG_TM * PG_KBLK * 2;                  // 16 KB
constexpr int PG_WBYTES = PG_TN * PG_KBLK * 2;                  // 32 KB
constexpr int PG_STAGE_BYTES = PG_XBYTES + PG_WBYTES;
constexpr int PG_EPI = 256;                                     // epilogue threads: two groups of four warps
constexpr int PG_THREADS = 64 + PG_EPI;
constexpr uint64_t PG_WAIT_NS = 200ull * 1000 * 1000;
constexpr int PG_STAGING = 32 * 128;                            // one epilogue warp: 32 rows of 128 bytes
constexpr size_t PG_SMEM = 1024 + (size_t)PG_STAGES * PG_STAGE_BYTES + 8 * PG_STAGING + 128;

enum PfDeviceError { PF_DEV_OK = 0, PF_DEV_TIMEOUT_LOAD = 1, PF_DEV_TIMEOUT_MMA = 2 };

struct PfGemmArgs {
    int M, N, K;          // K: columns the maps cover (a multiple of 64 is not required)
    float alpha;
    int accumulate;       // Y += ... (fp32 Y only)
    int out_bf16;
    void* Y;              // 16-byte aligned rows
    long long ldy;        // elements
    // Stream-K: piece p of a tile writes Y + p * ysplit (fp32, never accumulating).
    int stream;
    long long ysplit;
    // GeGLU: W tile t holds gate rows 128 t.. then the up rows of the same features; Y is bf16
    // z [M][ldy] = gelu_tanh(alpha gate) * (alpha up) for the nz features.
    int geglu, nz;
    int w_const;          // W is a weight matrix (not an output of an earlier kernel)
    // QKV (D = 128 or 256): columns are H query heads, the key head and the values, D each; rotated
    // queries to q [M][H][D], rotated keys and the values of row m = b P + p to kd / vd + b kv_stride +
    // p D. rope[p][j] = (cos, sin) of pair j.
    int qkv, H, D, P;
    const float2* rope;
    __nv_bfloat16 *q, *kd, *vd;
    long long kv_stride;
    int v_pairs;          // vd takes 4-byte stores
    int* err;
};

__global__ void __launch_bounds__(PG_THREADS, 1) k_pf_gemm(const __grid_constant__ CUtensorMap wmap,
                                                         const __grid_constant__ CUtensorMap xmap,
                                                         const __grid_constant__ PfGemmArgs a) {
    namespace ptx = jpi::ptx;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stages = smem;                                  // [stage][X 16 KB | W 32 KB]
    uint8_t* staging = smem + (size_t)PG_STAGES * PG_STAGE_BYTES;   // [8 warps][32 rows][128 B]
    uint64_t* full = (uint64_t*)(staging + 8 * PG_STAGING);
    uint64_t* empty = full + PG_STAGES;
    uint64_t* accf = empty + PG_STAGES;
    uint64_t* acce = accf + 2;
    uint32_t* tmem_slot = (uint32_t*)(acce + 2);
    int* flag = (int*)(tmem_slot + 1);

    const int tid = threadIdx.x, warp = ptx::warp_index(), lane = tid & 31;
    const int nkb = (a.K + PG_KBLK - 1) / PG_KBLK;
    const int ntn = (a.N + PG_TN - 1) / PG_TN, ntm = (a.M + PG_TM - 1) / PG_TM;
    const int tiles = ntn * ntm;
    // Segment j of this CTA: a tile (X tile fastest) and k-blocks [kb_lo, kb_hi) of it.
    const long long T = (long long)tiles * nkb;
    const long long x0 = a.stream ? blockIdx.x * T / gridDim.x : 0, x1 = a.stream ? (blockIdx.x + 1) * T / gridDim.x : 0;
    const int first = a.stream ? (int)(x0 / nkb) : (int)blockIdx.x, dstep = a.stream ? 1 : (int)gridDim.x;
    const int nseg = a.stream ? (x1 > x0 ? (int)((x1 - 1) / nkb) - first + 1 : 0)
                              : (first < tiles ? (tiles - first + dstep - 1) / dstep : 0);
    auto segment = [&](int j, int& tm, int& tn, int& piece, int& kb_lo, int& kb_hi) {
        const int u = first + j * dstep;
        tm = u % ntm;
        tn = u / ntm;
        piece = 0;
        kb_lo = 0;
        kb_hi = nkb;
        if (a.stream) {
            const long long base = (long long)u * nkb;
            kb_lo = x0 > base ? (int)(x0 - base) : 0;
            kb_hi = x1 < base + nkb ? (int)(x1 - base) : nkb;
            piece = (int)blockIdx.x - pg_cta_of(base, T, gridDim.x);
        }
    };

    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, 2 * PG_TN);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2 * PG_STAGES; ++i) ptx::mbar_init(&full[i], 1);
        ptx::mbar_init(&accf[0], 1);
        ptx::mbar_init(&accf[1], 1);
        ptx::mbar_init(&acce[0], PG_EPI);
        ptx::mbar_init(&acce[1], PG_EPI);
        ptx::fence_mbar_init();
        *flag = 0;
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (ptx::elect_one()) {
            int it = 0, issued = 0;
            bool ok = true;
            auto load_w = [&](int tn, int kb, int s) {
                ptx::mbar_expect_tx(&full[s], (uint32_t)PG_STAGE_BYTES);
                ptx::tma_load_2d_plain(stages + (size_t)s * PG_STAGE_BYTES + PG_XBYTES, &wmap, &full[s], kb * PG_KBLK,
                                       tn * PG_TN);
            };
            auto load_x = [&](int tm, int kb, int s) {
                ptx::tma_load_2d_plain(stages + (size_t)s * PG_STAGE_BYTES, &xmap, &full[s], kb * PG_KBLK, tm * PG_TM);
            };
            // The weights depend on nothing upstream: the first segment's first stages.
            int npre = 0;
            if (a.w_const && nseg > 0) {
                int tm, tn, piece, kb_lo, kb_hi;
                segment(0, tm, tn, piece, kb_lo, kb_hi);
                npre = min(PG_STAGES, kb_hi - kb_lo);
                issued = npre;
                for (int i = 0; i < npre; ++i) load_w(tn, kb_lo + i, i);
            }
            ptx::prefetch_tmap(&xmap);
            ptx::grid_dep_wait();
            for (int j = 0; j < nseg && ok; ++j) {
                int tm, tn, piece, kb_lo, kb_hi;
                segment(j, tm, tn, piece, kb_lo, kb_hi);
                for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                    const int s = it % PG_STAGES, n = it / PG_STAGES;
                    if (it >= PG_STAGES && !ptx::mbar_wait_bounded(&empty[s], (n - 1) & 1, PG_WAIT_NS)) {
                        *flag = PF_DEV_TIMEOUT_LOAD;
                        ok = false;
                        break;
                    }
                    if (it >= npre) load_w(tn, kb, s);
                    load_x(tm, kb, s);
                    issued = max(issued, it + 1);
                }
            }
            if (!ptx::ring_drain(full, PG_STAGES, issued, PG_WAIT_NS)) *flag = PF_DEV_TIMEOUT_LOAD;
        }
    } else if (warp == 1) {
        if (ptx::elect_one()) {
            constexpr uint32_t IDESC = ptx::idesc_bf16_f32(PG_TM, PG_TN);
            const uint32_t base = ptx::smem_u32(stages);
            bool good = true;
            int it = 0;
            for (int j = 0; j < nseg; ++j) {
                const int buf = j & 1;
                if (j >= 2 && !ptx::mbar_wait_bounded(&acce[buf], ((j - 2) >> 1) & 1, PG_WAIT_NS)) good = false;
                ptx::tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * PG_TN);
                int tm, tn, piece, kb_lo, kb_hi;
                segment(j, tm, tn, piece, kb_lo, kb_hi);
                for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                    const int s = it % PG_STAGES, n = it / PG_STAGES;
                    if (good && !ptx::mbar_wait_bounded(&full[s], n & 1, PG_WAIT_NS)) good = false;
                    ptx::tc_fence_after();
                    if (good) {
                        const uint64_t x = ptx::desc_sw128(base + (uint32_t)(s * PG_STAGE_BYTES)), w = ptx::desc_add(x, PG_XBYTES);
#pragma unroll
                        for (int kk = 0; kk < PG_KBLK / 16; ++kk)
                            ptx::mma_bf16(acc, ptx::desc_add(x, kk * 32), ptx::desc_add(w, kk * 32), IDESC,
                                          (kb != kb_lo) || (kk != 0));
                    }
                    ptx::mma_commit(&empty[s]);
                }
                // Committed even after a timeout so that the epilogue wakes up.
                ptx::mma_commit(&accf[buf]);
            }
            if (!good) *flag = PF_DEV_TIMEOUT_MMA;
        }
    } else {
        // One TMEM lane (X row of the tile) per thread; group g of four warps takes half of the columns.
        const int qd = warp & 3, g = (warp - 2) >> 2;
        uint8_t* stg = staging + (warp - 2) * PG_STAGING;
        // Through the staging, lane l handles 16-byte chunk l mod 8 of rows 4 i + l / 8 of the warp's 32.
        const int sr = lane >> 3, sc = lane & 7;
        auto own_chunk = [&](int c) { return (uint4*)(stg + lane * 128 + ((c ^ (lane & 7)) << 4)); };
        auto row_chunk = [&](int r, int c) { return (const uint4*)(stg + r * 128 + ((c ^ (r & 7)) << 4)); };
        auto pack2 = [](float lo, float hi) {
            const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
            return *reinterpret_cast<const uint32_t*>(&v);
        };
        ptx::grid_dep_wait();   // outputs may still be read by the previous kernel
        for (int j = 0; j < nseg; ++j) {
            const int buf = j & 1;
            int tm, tn, piece, kb_lo, kb_hi;
            segment(j, tm, tn, piece, kb_lo, kb_hi);
            if (!ptx::mbar_wait_bounded(&accf[buf], (j >> 1) & 1, PG_WAIT_NS)) *flag = PF_DEV_TIMEOUT_MMA;
            const bool ok = __all_sync(0xffffffffu, *flag == 0);
            ptx::tc_fence_after();
            // The last accumulator is complete: the next kernel's CTAs may come in.
            if (j + 1 == nseg) ptx::grid_dep_launch();
            const uint32_t acc = tmem + (uint32_t)(buf * PG_TN) + ((uint32_t)(qd * 32) << 16);
            const int m0 = tm * PG_TM + qd * 32;   // the warp's first row
            // Stream-K: this piece of the tile has its own partial buffer.
            void* Y = a.stream ? (void*)(static_cast<float*>(a.Y) + (size_t)piece * a.ysplit) : a.Y;
            if (a.qkv) {
                // Steps of 16 rotary pairs: columns c1.. and c1 + D / 2.. of one head section.
                const int half = a.D >> 1;
                int pos[8];
                size_t kvo[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int m = min(m0 + 4 * i + sr, a.M - 1), b = m / a.P;
                    pos[i] = m - b * a.P;
                    kvo[i] = (size_t)b * a.kv_stride + (size_t)pos[i] * a.D;
                }
#pragma unroll 1
                for (int s = g * (PG_TN / 64); s < (g + 1) * (PG_TN / 64); ++s) {
                    const int sl = 16 * s / half, j0 = 16 * s - sl * half;   // section of the tile, first pair
                    const int sec = tn * (PG_TN / a.D) + sl, c1 = sl * a.D + j0;
                    const bool rot = sec <= a.H, in = sec < a.H + 2;
                    float4 cs[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        cs[i] = rot ? __ldg((const float4*)(a.rope + (size_t)pos[i] * half + j0) + sc)
                                    : make_float4(1.f, 0.f, 1.f, 0.f);
                    uint32_t r1[16], r2[16];
                    ptx::tmem_ld_x16(acc + (uint32_t)c1, r1);
                    ptx::tmem_ld_x16(acc + (uint32_t)(c1 + half), r2);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 8; ++c) *own_chunk(c) = make_uint4(r1[2 * c], r1[2 * c + 1], r2[2 * c], r2[2 * c + 1]);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint4 v = *row_chunk(4 * i + sr, sc);
                        const float ua = __uint_as_float(v.x), ub = __uint_as_float(v.y);
                        const float va = __uint_as_float(v.z), vb = __uint_as_float(v.w);
                        if (!ok || !in || m0 + 4 * i + sr >= a.M) continue;
                        __nv_bfloat16* d = (sec < a.H ? a.q + ((size_t)(m0 + 4 * i + sr) * a.H + sec) * a.D : (sec == a.H ? a.kd : a.vd) + kvo[i]) +
                                           j0 + 2 * sc;
                        const uint32_t w0 = pack2(ua * cs[i].x - va * cs[i].y, ub * cs[i].z - vb * cs[i].w);
                        const uint32_t w1 = pack2(va * cs[i].x + ua * cs[i].y, vb * cs[i].z + ub * cs[i].w);
                        if (sec > a.H && !a.v_pairs) {
                            unsigned short* e = reinterpret_cast<unsigned short*>(d);
                            e[0] = (unsigned short)w0;
                            e[1] = (unsigned short)(w0 >> 16);
                            e[half] = (unsigned short)w1;
                            e[half + 1] = (unsigned short)(w1 >> 16);
                        } else {
                            *(uint32_t*)d = w0;
                            *(uint32_t*)(d + half) = w1;
                        }
                    }
                    __syncwarp();
                }
            } else if (a.geglu || a.out_bf16) {
                // 64 bf16 outputs of a row per pass (GeGLU: gate columns c.. and up columns 128 + c..).
                const int nc = a.geglu ? PG_TN / 2 : PG_TN, nlim = a.geglu ? a.nz : a.N;
                for (int c0 = g * nc / 2; c0 < (g + 1) * nc / 2; c0 += 64) {
                    const int n0 = tn * nc + c0;
                    if (n0 >= nlim) break;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t r[16], r2[16];
                        ptx::tmem_ld_x16(acc + (uint32_t)(c0 + 16 * q), r);
                        if (a.geglu) ptx::tmem_ld_x16(acc + (uint32_t)(PG_TN / 2 + c0 + 16 * q), r2);
                        ptx::tmem_ld_wait();
                        uint32_t o[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            float v0 = a.alpha * __uint_as_float(r[2 * i]), v1 = a.alpha * __uint_as_float(r[2 * i + 1]);
                            if (a.geglu) {
                                v0 = gelu_tanh_f(v0) * (a.alpha * __uint_as_float(r2[2 * i]));
                                v1 = gelu_tanh_f(v1) * (a.alpha * __uint_as_float(r2[2 * i + 1]));
                            }
                            o[i] = pack2(v0, v1);
                        }
                        *own_chunk(2 * q) = make_uint4(o[0], o[1], o[2], o[3]);
                        *own_chunk(2 * q + 1) = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                    __syncwarp();
                    const int n = n0 + 8 * sc;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int m = m0 + 4 * i + sr;
                        const uint4 v = *row_chunk(4 * i + sr, sc);
                        if (!ok || m >= a.M) continue;
                        __nv_bfloat16* y = static_cast<__nv_bfloat16*>(Y) + (size_t)m * a.ldy + n;
                        if (n + 8 <= nlim) {
                            *(uint4*)y = v;
                        } else {
                            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                if (n + e < nlim)
                                    reinterpret_cast<unsigned short*>(y)[e] = (unsigned short)(w[e / 2] >> (16 * (e & 1)));
                        }
                    }
                    __syncwarp();
                }
            } else {
                // 32 fp32 outputs of a row per pass.
                const bool accum = a.accumulate && !a.stream;
                for (int c0 = g * PG_TN / 2; c0 < (g + 1) * PG_TN / 2; c0 += 32) {
                    const int n0 = tn * PG_TN + c0;
                    if (n0 >= a.N) break;
                    const int n = n0 + 4 * sc;
                    float4 old[8];   // before the accumulator is read: the loads overlap it
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int m = m0 + 4 * i + sr;
                        old[i] = accum && m < a.M && n + 4 <= a.N
                                     ? *(const float4*)(static_cast<const float*>(Y) + (size_t)m * a.ldy + n)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    uint32_t r[2][16];
                    ptx::tmem_ld_x16(acc + (uint32_t)c0, r[0]);
                    ptx::tmem_ld_x16(acc + (uint32_t)(c0 + 16), r[1]);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *own_chunk(c) = make_uint4(r[c >> 2][4 * (c & 3)], r[c >> 2][4 * (c & 3) + 1],
                                                   r[c >> 2][4 * (c & 3) + 2], r[c >> 2][4 * (c & 3) + 3]);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int m = m0 + 4 * i + sr;
                        const uint4 u = *row_chunk(4 * i + sr, sc);
                        if (!ok || m >= a.M) continue;
                        const float4 v = make_float4(old[i].x + a.alpha * __uint_as_float(u.x),
                                                     old[i].y + a.alpha * __uint_as_float(u.y),
                                                     old[i].z + a.alpha * __uint_as_float(u.z),
                                                     old[i].w + a.alpha * __uint_as_float(u.w));
                        float* y = static_cast<float*>(Y) + (size_t)m * a.ldy + n;
                        if (n + 4 <= a.N) {
                            *(float4*)y = v;
                        } else {
                            const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (n + e < a.N) y[e] = accum ? y[e] + w[e] : w[e];
                        }
                    }
                    __syncwarp();
                }
            }
            ptx::tc_fence_before();
            ptx::mbar_arrive(&acce[buf]);
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (tid == 0 && *flag != 0) atomicCAS(a.err, 0, *flag);   // after every role's last word on it
    if (warp == 1) ptx::tmem_dealloc(tmem, 2 * PG_TN);
}

// vt[d][p] = v[p][d] for one request (p < P), so that P V runs as a product of K-major operands.
__global__ void k_pf_transpose(const __nv_bfloat16* __restrict__ v, __nv_bfloat16* __restrict__ vt, int P, int D,
                               int ldt) {
    __shared__ __nv_bfloat16 t[32][33];
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const int p0 = blockIdx.x * 32, d0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int p = p0 + i, d = d0 + threadIdx.x;
        if (p < P && d < D) t[i][threadIdx.x] = v[(size_t)p * D + d];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int d = d0 + i, p = p0 + threadIdx.x;
        if (p < P && d < D) vt[(size_t)d * ldt + p] = t[threadIdx.x][i];
    }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

}  // namespace

struct jpi_prefill_handle {
    jpi_prefill_config cfg;
    int L = 0, W = 0, H = 0, D = 0, F = 0, QKV = 0, Bm = 0, Pm = 0, Pp = 0;
    std::vector<void*> allocs;
    size_t bytes = 0;
    std::vector<LayerW> layers;
    float* final_norm = nullptr;
    float2* rope = nullptr;          // [Pm][D / 2]
    float* h = nullptr;              // [Bm Pm][W] residual stream
    __nv_bfloat16* xn = nullptr;     // [Bm Pm][W] GEMM operand: normed h
    float* qkv = nullptr;            // [Bm Pm][(H + 2) D] (head dims without the fused epilogue)
    __nv_bfloat16* q = nullptr;      // [Bm Pm][H][D]
    __nv_bfloat16* o = nullptr;      // [Bm Pm][H D]
    __nv_bfloat16* z = nullptr;      // [Bm Pm][F] GeGLU output (the gate/up product's epilogue)
    float* part = nullptr;           // pieces of a stream-K residual product
    long long part_elems = 0;        // floats `part` holds
    int Fp = 0;                      // F rounded up to 128: gate/up tiles of 128 features
    float* sc = nullptr;             // [H Pm][Pp] scores of one request
    __nv_bfloat16* pr = nullptr;     // [H Pm][Pp] probabilities of one request
    __nv_bfloat16* vt = nullptr;     // [D][Pp] one request's values, transposed
    int* dev_err = nullptr;          // device error word of the GEMM's bounded waits
    int num_sms = 0;
    int t5_clusters[5] = {};         // row blocks whose s-CTA clusters of the attention are co-resident
    void *t5_ws = nullptr, *t5_wml = nullptr;   // its key-split workspace: partial outputs, (m, l)
    bool qkv_fused() const { return D == 128 || D == 256; }
};

namespace {

template <typename T>
jpi_status pf_alloc(jpi_prefill_handle* h, T** p, size_t count) {
    void* q = nullptr;
    const size_t bytes = count * sizeof(T);
    const cudaError_t e = cudaMalloc(&q, bytes ? bytes : 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return pfail(JPI_ERR_OOM, "cudaMalloc(%zu bytes) failed: %s", bytes, cudaGetErrorString(e));
    }
    h->allocs.push_back(q);
    h->bytes += bytes;
    *p = static_cast<T*>(q);
    return JPI_OK;
}

void release(jpi_prefill_handle* h) {
    for (void* p : h->allocs) cudaFree(p);
    h->allocs.clear();
}

// 2D bf16 tensor map over a row-major [rows][cols] matrix of leading dimension ld (elements),
// 128-byte swizzle, boxes of 64 columns x box_rows rows; reads past the extents return zeros.
jpi_status make_map(const void* base, long long rows, long long cols, long long ld, int box_rows, CUtensorMap* map) {
    auto enc = get_encode();
    if (!enc) return pfail(JPI_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable from the driver");
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld * 2) % 16)
        return pfail(JPI_ERR_INVALID_ARG, "a GEMM operand is not 16-byte aligned (address or row stride)");
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)PG_KBLK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return pfail(JPI_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return JPI_OK;
}

// Launch with programmatic dependent launch: the kernel waits for its predecessor (griddepcontrol)
// before it touches what that reads or writes, and starts its weight copies before. A failed launch
// leaves its error for the cudaGetLastError check that follows.
template <typename... KArgs, typename... Args>
void pdl(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*k)(KArgs...), Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, k, args...);
}

// Y [M][N] (leading dimension ldy; fp32, or bf16 when y_bf16) = alpha X [M][K] W[N][K]^T, plus Y
// when accumulating. X and W are bf16 with leading dimensions ldx and ldw; w_const: W is a weight
// matrix. `more` sets the fields of the other forms (GeGLU, QKV, stream-K); grid > 0 fixes the CTAs.
template <typename F>
jpi_status row_gemm(jpi_prefill_handle* h, cudaStream_t st, const __nv_bfloat16* X, long long ldx,
                    const __nv_bfloat16* Wm, long long ldw, bool w_const, void* Y, bool y_bf16, long long ldy, int M,
                    int N, int K, float alpha, bool accumulate, int grid, F&& more) {
    CUtensorMap wmap, xmap;
    if (reinterpret_cast<uintptr_t>(Y) % 16 || ldy % (y_bf16 ? 8 : 4))   // never: widths are multiples of 8
        return pfail(JPI_ERR_UNSUPPORTED, "a product's output rows are not 16-byte aligned");
    PF_TRY(make_map(Wm, N, K, ldw, PG_TN, &wmap));
    PF_TRY(make_map(X, M, K, ldx, PG_TM, &xmap));
    PfGemmArgs a = {};
    a.M = M;
    a.N = N;
    a.K = K;
    a.alpha = alpha;
    a.accumulate = accumulate ? 1 : 0;
    a.out_bf16 = y_bf16 ? 1 : 0;
    a.Y = Y;
    a.ldy = ldy;
    a.w_const = w_const ? 1 : 0;
    a.err = h->dev_err;
    more(a);
    if (grid <= 0) {
        const long long tiles = (long long)((N + PG_TN - 1) / PG_TN) * ((M + PG_TM - 1) / PG_TM);
        grid = (int)(tiles < h->num_sms ? tiles : h->num_sms);
    }
    pdl(st, dim3(grid), dim3(PG_THREADS), PG_SMEM, k_pf_gemm, wmap, xmap, a);
    PF_CUDA(cudaGetLastError());
    return JPI_OK;
}
jpi_status row_gemm(jpi_prefill_handle* h, cudaStream_t st, const __nv_bfloat16* X, long long ldx,
                    const __nv_bfloat16* Wm, long long ldw, bool w_const, void* Y, bool y_bf16, long long ldy, int M,
                    int N, int K, float alpha, bool accumulate) {
    return row_gemm(h, st, X, ldx, Wm, ldw, w_const, Y, y_bf16, ldy, M, N, K, alpha, accumulate, 0, [](PfGemmArgs&) {});
}

// CTAs a residual product [M][N] over K is dealt out to (stream-K), or 0: whole tiles, accumulated in
// place. Up to 4/5 of a wave of tiles, at most 8 CTAs a tile and at least 8 k-blocks a CTA. A CTA that
// cuts across tiles writes a piece for each, worth about PG_PIECE_KB k-blocks, so the choice is between
// every SM (each CTA two pieces) and the whole number of CTAs per tile that fits (one piece): at
// Gemma-2B sizes and 816 tokens (56 tiles) down (256 k-blocks a tile) takes 152 CTAs of 94.3 k-blocks,
// O (32) 112 of 16. Measured, whole tiles, every SM, whole CTAs per tile, us a layer: 8 tiles 167, 98, 98; 56: 230,
// 191, 191 (as chosen 188); 96: 305, 294, 306; 112: 334, 335, 337 (331); 128: 374, 386, 376; at width 1024 28
// tiles 88, 81, 77; 72: 123, 125, 122; 112: 173, 188, 173 (180).
constexpr int PG_PIECE_KB = 8;
int stream_grid(int num_sms, int M, int N, int K) {
    const long long tiles = (long long)((N + PG_TN - 1) / PG_TN) * ((M + PG_TM - 1) / PG_TM);
    const int nkb = (K + PG_KBLK - 1) / PG_KBLK;
    if (tiles * 5 > num_sms * 4ll) return 0;
    const long long most = std::min<long long>(std::min<long long>(num_sms, 8 * tiles), tiles * nkb / 8);
    const long long whole = most / tiles * tiles;
    if (whole <= 0) return 0;
    const long long kb_most = (tiles * nkb + most - 1) / most + 2 * PG_PIECE_KB;
    const long long kb_whole = (nkb + whole / tiles - 1) / (whole / tiles) + PG_PIECE_KB;
    const long long g = kb_most < kb_whole ? most : whole;
    return g > tiles ? (int)g : 0;
}
// Most pieces a tile of such a product has.
int stream_pieces(int grid, int M, int N) {
    const int tiles = ((N + PG_TN - 1) / PG_TN) * ((M + PG_TM - 1) / PG_TM);
    return (grid + tiles - 1) / tiles + 1;
}

// Attention of the requests of one layer on the tcgen05 attention kernel: the queries h->q
// [B P H][D] against this layer's keys and values kd / vd (request b at row b * kv_rows, P rows
// each), every key visible, into h->o. Used for head dims 128 and 256 when the request stride is
// a whole number of rows; the maps' row extents end at the last request's last key, so no copy
// reads past what the caller owns (the kernel masks the zero-filled rows past P).
template <int D>
jpi_status attention_t5(jpi_prefill_handle* h, cudaStream_t st, const __nv_bfloat16* kd, const __nv_bfloat16* vd,
                        int batch, int P, long long kv_rows) {
    CUtensorMap qmap, kmap, vmap;
    const long long nrows = (long long)P * h->H;
    const long long krows = (long long)(batch - 1) * kv_rows + P;
    PF_TRY(make_map(h->q, (long long)batch * nrows, D, D, jpi::T5_ROWS, &qmap));
    PF_TRY(make_map(kd, krows, D, D, jpi::T5_KEYS, &kmap));
    PF_TRY(make_map(vd, krows, D, D, jpi::T5_KEYS, &vmap));
    jpi::T5Args a;
    a.S = P;
    a.nctx = 0;
    a.H = h->H;
    a.P = 0;
    a.kv_rows = (int)kv_rows;
    a.maxB = batch;
    a.layer = 0;
    a.scale_log2 = 1.4426950408889634f / sqrtf((float)D);
    a.o = h->o;
    a.err = h->dev_err;
    // Key splits (a cluster of 4 or 2 CTAs per row block) while they are co-resident: 51 row blocks
    // at 816 tokens and 8 heads leave two thirds of the SMs idle unsplit.
    const int rblocks = (int)((nrows + jpi::T5_ROWS - 1) / jpi::T5_ROWS), nb = (P + jpi::T5_KEYS - 1) / jpi::T5_KEYS;
    int splits = 1;
    for (int s = 4; s >= 2 && splits == 1; s /= 2)
        if (h->t5_ws && nb >= s && (long long)rblocks * batch <= h->t5_clusters[s]) splits = s;
    a.ws = reinterpret_cast<float4*>(h->t5_ws);
    a.wml = reinterpret_cast<float2*>(h->t5_wml);
    const dim3 grid((unsigned)rblocks, (unsigned)batch, (unsigned)splits);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(jpi::T5_THREADS);
    cfg.dynamicSmemBytes = jpi::T5Smem<D>::BYTES;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 1;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = (unsigned)splits;
    cfg.attrs = at;
    cfg.numAttrs = splits > 1 ? 2 : 1;
    (void)cudaLaunchKernelEx(&cfg, jpi::k_attn_t5<D>, qmap, kmap, vmap, a);
    PF_CUDA(cudaGetLastError());
    return JPI_OK;
}

jpi_status check_config(const jpi_prefill_config* c) {
    if (c->n_layers < 1 || c->n_heads < 1 || c->max_batch < 1 || c->max_prefix < 1)
        return pfail(JPI_ERR_INVALID_ARG, "n_layers, n_heads, max_batch and max_prefix must be >= 1");
    if (c->width < 8 || c->width % 8 || c->mlp_dim < 8 || c->mlp_dim % 8)
        return pfail(JPI_ERR_UNSUPPORTED, "width and mlp_dim must be multiples of 8");
    if (c->head_dim < 8 || c->head_dim % 8 || c->head_dim > 512)
        return pfail(JPI_ERR_UNSUPPORTED, "head_dim must be a multiple of 8 and at most 512");
    if ((long long)c->max_batch * c->max_prefix > (1ll << 24) || c->max_prefix > 65536)
        return pfail(JPI_ERR_UNSUPPORTED, "max_batch * max_prefix or max_prefix too large");
    if (!(c->rms_eps >= 0.f) || !(c->rope_base >= 0.f))
        return pfail(JPI_ERR_INVALID_ARG, "rms_eps and rope_base must be >= 0");
    return JPI_OK;
}

// fp32 tensor (host or device) -> bf16 at dst.
jpi_status put_bf16(jpi_prefill_handle* h, bool dev, float* staging, __nv_bfloat16* dst, const float* src,
                    size_t n, const char* name, int layer) {
    if (!src) return pfail(JPI_ERR_INVALID_ARG, "weight %s of layer %d is NULL", name, layer);
    const float* s = src;
    if (!dev) {
        PF_CUDA(cudaMemcpy(staging, src, n * sizeof(float), cudaMemcpyHostToDevice));
        s = staging;
    }
    k_pf_cast<<<grid_for((long long)n), 256>>>(s, dst, (long long)n);
    PF_CUDA(cudaGetLastError());
    // The staging buffer is reused by the next tensor; finish this conversion first.
    PF_CUDA(cudaStreamSynchronize(nullptr));
    return JPI_OK;
}

// Gate (off 0) or up (off 128) rows [F][W] (host or device fp32) into the packed gate/up matrix.
jpi_status put_gu(jpi_prefill_handle* h, bool dev, float* staging, __nv_bfloat16* dst, const float* src, int off,
                  const char* name, int layer) {
    if (!src) return pfail(JPI_ERR_INVALID_ARG, "weight %s of layer %d is NULL", name, layer);
    const size_t n = (size_t)h->F * h->W;
    const float* s = src;
    if (!dev) {
        PF_CUDA(cudaMemcpy(staging, src, n * sizeof(float), cudaMemcpyHostToDevice));
        s = staging;
    }
    k_pf_cast_gu<<<grid_for((long long)n), 256>>>(s, dst, h->F, h->W, off);
    PF_CUDA(cudaGetLastError());
    PF_CUDA(cudaStreamSynchronize(nullptr));
    return JPI_OK;
}

jpi_status put_f32(jpi_prefill_handle* h, bool dev, float** dst, const float* src, size_t n, const char* name,
                   int layer) {
    if (!src) return pfail(JPI_ERR_INVALID_ARG, "weight %s of layer %d is NULL", name, layer);
    PF_TRY(pf_alloc(h, dst, n));
    PF_CUDA(cudaMemcpy(*dst, src, n * sizeof(float), dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice));
    return JPI_OK;
}

jpi_status setup(jpi_prefill_handle* h, const jpi_prefill_config* c, const jpi_prefill_weights* w) {
    h->cfg = *c;
    h->L = c->n_layers;
    h->W = c->width;
    h->H = c->n_heads;
    h->D = c->head_dim;
    h->F = c->mlp_dim;
    h->QKV = (h->H + 2) * h->D;
    h->Bm = c->max_batch;
    h->Pm = c->max_prefix;
    h->Pp = (h->Pm + 7) / 8 * 8;
    const size_t W = (size_t)h->W, D = (size_t)h->D, F = (size_t)h->F, HD = (size_t)h->H * D;
    const size_t Mm = (size_t)h->Bm * h->Pm;
    h->Fp = (h->F + 127) / 128 * 128;
    const size_t Fp = (size_t)h->Fp;
    const bool dev = w->on_device != 0;
    if (!w->attn_norm || !w->wq || !w->wk || !w->wv || !w->wo || !w->mlp_norm || !w->w_gate || !w->w_up ||
        !w->w_down || !w->final_norm)
        return pfail(JPI_ERR_INVALID_ARG, "a weight array is NULL");

    int device = 0;
    PF_CUDA(cudaGetDevice(&device));
    PF_CUDA(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, device));
    PF_CUDA(cudaFuncSetAttribute(k_pf_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM));
    PF_CUDA(cudaFuncSetAttribute(jpi::k_attn_t5<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 jpi::T5Smem<128>::BYTES));
    PF_CUDA(cudaFuncSetAttribute(jpi::k_attn_t5<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 jpi::T5Smem<256>::BYTES));
    if (h->qkv_fused()) {
        // Attention key splits: clusters that fit at once, and a workspace slot per CTA.
        for (int s = 2; s <= 4; s *= 2) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(h->num_sms / s), 1, (unsigned)s);
            cfg.blockDim = dim3(jpi::T5_THREADS);
            cfg.dynamicSmemBytes = D == 256 ? jpi::T5Smem<256>::BYTES : jpi::T5Smem<128>::BYTES;
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 1;
            at.val.clusterDim.y = 1;
            at.val.clusterDim.z = (unsigned)s;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int n = 0;
            const cudaError_t e = D == 256 ? cudaOccupancyMaxActiveClusters(&n, jpi::k_attn_t5<256>, &cfg)
                                           : cudaOccupancyMaxActiveClusters(&n, jpi::k_attn_t5<128>, &cfg);
            if (e != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            h->t5_clusters[s] = std::min(n, h->num_sms / s);
        }
        uint8_t* ws = nullptr;
        const size_t part = (size_t)h->num_sms * (D / 4) * jpi::T5_ROWS * sizeof(float4);
        PF_TRY(pf_alloc(h, &ws, part + (size_t)h->num_sms * jpi::T5_ROWS * sizeof(float2)));
        h->t5_ws = ws;
        h->t5_wml = ws + part;
    }
    PF_TRY(pf_alloc(h, &h->dev_err, 1));
    PF_CUDA(cudaMemset(h->dev_err, 0, sizeof(int)));
    float* staging = nullptr;
    if (!dev) PF_TRY(pf_alloc(h, &staging, std::max({F, HD, D}) * W));   // the largest tensor put_bf16 / put_gu take
    h->layers.resize((size_t)h->L);
    for (int l = 0; l < h->L; ++l) {
        LayerW& lw = h->layers[(size_t)l];
        PF_TRY(pf_alloc(h, &lw.wqkv, (HD + 2 * D) * W));
        PF_TRY(put_bf16(h, dev, staging, lw.wqkv, w->wq[l], HD * W, "wq", l));
        PF_TRY(put_bf16(h, dev, staging, lw.wqkv + HD * W, w->wk[l], D * W, "wk", l));
        PF_TRY(put_bf16(h, dev, staging, lw.wqkv + (HD + D) * W, w->wv[l], D * W, "wv", l));
        PF_TRY(pf_alloc(h, &lw.wo, W * HD));
        PF_TRY(put_bf16(h, dev, staging, lw.wo, w->wo[l], W * HD, "wo", l));
        PF_TRY(pf_alloc(h, &lw.wgu, 2 * Fp * W));
        PF_CUDA(cudaMemset(lw.wgu, 0, 2 * Fp * W * sizeof(__nv_bfloat16)));   // rows of features past F
        PF_TRY(put_gu(h, dev, staging, lw.wgu, w->w_gate[l], 0, "w_gate", l));
        PF_TRY(put_gu(h, dev, staging, lw.wgu, w->w_up[l], 128, "w_up", l));
        PF_TRY(pf_alloc(h, &lw.wd, W * F));
        PF_TRY(put_bf16(h, dev, staging, lw.wd, w->w_down[l], W * F, "w_down", l));
        PF_TRY(put_f32(h, dev, &lw.attn_norm, w->attn_norm[l], W, "attn_norm", l));
        PF_TRY(put_f32(h, dev, &lw.mlp_norm, w->mlp_norm[l], W, "mlp_norm", l));
    }
    PF_TRY(put_f32(h, dev, &h->final_norm, w->final_norm, W, "final_norm", -1));

    // Rotary table, in double precision on the host: angle p base^(-2j/D) for p < Pm, j < D/2.
    std::vector<float2> tab((size_t)h->Pm * (D / 2));
    for (int p = 0; p < h->Pm; ++p)
        for (size_t j = 0; j < D / 2; ++j) {
            float2 cs = make_float2(1.f, 0.f);
            if (c->rope_base > 0.f) {
                const double ang = (double)p * std::pow((double)c->rope_base, -2.0 * (double)j / (double)D);
                cs = make_float2((float)std::cos(ang), (float)std::sin(ang));
            }
            tab[(size_t)p * (D / 2) + j] = cs;
        }
    PF_TRY(pf_alloc(h, &h->rope, tab.size()));
    PF_CUDA(cudaMemcpy(h->rope, tab.data(), tab.size() * sizeof(float2), cudaMemcpyHostToDevice));

    PF_TRY(pf_alloc(h, &h->h, Mm * W));
    PF_TRY(pf_alloc(h, &h->xn, Mm * W));
    PF_TRY(pf_alloc(h, &h->z, Mm * F));
    // Pieces of the residual products (O and down) that are dealt out by stream-K: the most any token
    // count up to the maximum needs (pieces x 128-row tiles).
    for (long long m = 1; m <= (long long)((Mm + PG_TM - 1) / PG_TM); ++m)
        for (int K : {h->H * h->D, h->F}) {
            const int M = (int)std::min<long long>(m * PG_TM, (long long)Mm), g = stream_grid(h->num_sms, M, h->W, K);
            if (g > 0) h->part_elems = std::max(h->part_elems, (long long)stream_pieces(g, M, h->W) * M * h->W);
        }
    if (h->part_elems > 0) PF_TRY(pf_alloc(h, &h->part, (size_t)h->part_elems));
    // Head dims 128 and 256 rotate and scatter in the product's epilogue; others through fp32.
    if (!h->qkv_fused()) PF_TRY(pf_alloc(h, &h->qkv, Mm * (size_t)h->QKV));
    PF_TRY(pf_alloc(h, &h->q, Mm * HD));
    PF_TRY(pf_alloc(h, &h->o, Mm * HD));
    PF_TRY(pf_alloc(h, &h->sc, (size_t)h->H * h->Pm * h->Pp));
    PF_TRY(pf_alloc(h, &h->pr, (size_t)h->H * h->Pm * h->Pp));
    PF_TRY(pf_alloc(h, &h->vt, D * (size_t)h->Pp));
    return JPI_OK;
}

}  // namespace

extern "C" {

JPI_API const char* jpi_prefill_last_error(void) { return g_err; }

JPI_API jpi_status jpi_prefill_create(const jpi_prefill_config* cfg, const jpi_prefill_weights* w,
                                      jpi_prefill_handle** out) {
    g_err[0] = '\0';
    if (!out) return pfail(JPI_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!cfg || !w) return pfail(JPI_ERR_INVALID_ARG, "config or weights is NULL");
    PF_TRY(check_config(cfg));
    jpi_prefill_handle* h = new (std::nothrow) jpi_prefill_handle();
    if (!h) return pfail(JPI_ERR_OOM, "host allocation failed");
    const jpi_status s = setup(h, cfg, w);
    if (s != JPI_OK) {
        cudaStreamSynchronize(nullptr);
        cudaGetLastError();
        release(h);
        delete h;
        return s;
    }
    *out = h;
    return JPI_OK;
}

JPI_API jpi_status jpi_prefill_destroy(jpi_prefill_handle* h) {
    g_err[0] = '\0';
    if (!h) return JPI_OK;
    release(h);
    delete h;
    return JPI_OK;
}

JPI_API jpi_status jpi_prefill_run(jpi_prefill_handle* h, const void* x, int x_is_fp32, int batch, int prefix_len,
                                   void* const* k_layers, void* const* v_layers, long long request_stride,
                                   float* out_final, void* stream) {
    g_err[0] = '\0';
    if (!h) return pfail(JPI_ERR_INVALID_ARG, "handle is NULL");
    if (!x || !k_layers || !v_layers) return pfail(JPI_ERR_INVALID_ARG, "NULL input or KV destination array");
    if (batch < 1 || prefix_len < 1) return pfail(JPI_ERR_INVALID_ARG, "batch and prefix_len must be >= 1");
    if (batch > h->Bm || prefix_len > h->Pm)
        return pfail(JPI_ERR_SHAPE, "batch %d / prefix_len %d exceed the maxima %d / %d", batch, prefix_len, h->Bm,
                     h->Pm);
    if (request_stride < (long long)prefix_len * h->D || request_stride % 8)
        return pfail(JPI_ERR_INVALID_ARG, "request_stride must be >= prefix_len * head_dim and a multiple of 8");
    for (int l = 0; l < h->L; ++l)
        if (!k_layers[l] || !v_layers[l]) return pfail(JPI_ERR_INVALID_ARG, "KV destination of layer %d is NULL", l);
    // Whether the attention runs on the tcgen05 attention kernel (scores and probabilities never leave the
    // SM), else per request through the GEMM: scores, softmax, V^T, probabilities times V. Keys are read by
    // bulk tensor copies either way, values only by the former.
    const bool t5 = h->qkv_fused() && request_stride % h->D == 0 && request_stride / h->D <= INT32_MAX;
    for (int l = 0; l < h->L; ++l) {
        const uintptr_t ka = reinterpret_cast<uintptr_t>(k_layers[l]), va = reinterpret_cast<uintptr_t>(v_layers[l]);
        if ((ka & 15) || (va & (t5 ? 15 : 1)))
            return pfail(JPI_ERR_INVALID_ARG, "K or V destination of layer %d is not aligned (K 16 bytes, V %d)", l, t5 ? 16 : 2);
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int W = h->W, D = h->D, H = h->H, F = h->F, P = prefix_len, Pp = (P + 7) / 8 * 8;
    const long long M = (long long)batch * P;
    const float eps = h->cfg.rms_eps, scale = 1.f / sqrtf((float)D);

    k_pf_load_x<<<grid_for(M * W), 256, 0, st>>>(x, x_is_fp32, h->h, M * W);
    PF_CUDA(cudaGetLastError());
    // A residual product (O or down): dealt out by stream-K with its pieces added by the row kernel
    // that also writes the next norm, or whole tiles accumulated into h and the norm alone after it.
    // norm null: no norm follows.
    const dim3 rows_grid(grid_for(M, 1, 16384));
    auto residual = [&](const __nv_bfloat16* X, int K, const __nv_bfloat16* Wm, const float* norm, auto* y) -> jpi_status {
        using TO = std::remove_reference_t<decltype(*y)>;
        const int g = stream_grid(h->num_sms, (int)M, W, K);
        if (g > 0) {
            const long long pstride = M * W;   // elements between the pieces
            PF_TRY(row_gemm(h, st, X, K, Wm, K, true, h->part, false, W, (int)M, W, K, 1.f, false, g, [&](PfGemmArgs& a) {
                a.stream = 1;
                a.ysplit = pstride;
            }));
            const int ntm = (int)((M + PG_TM - 1) / PG_TM), nkb = (K + PG_KBLK - 1) / PG_KBLK;
            const long long T = (long long)((W + PG_TN - 1) / PG_TN) * ntm * nkb;
            pdl(st, rows_grid, dim3(RB), 0, k_pf_residual_norm<TO>, h->h, (const float*)h->part, pstride, ntm, nkb, T, g,
                norm, y, M, W, eps);
        } else {
            PF_TRY(row_gemm(h, st, X, K, Wm, K, true, h->h, false, W, (int)M, W, K, 1.f, true));
            if (norm) pdl(st, rows_grid, dim3(RB), 0, k_pf_rmsnorm<TO>, (const float*)h->h, norm, y, M, W, eps);
        }
        PF_CUDA(cudaGetLastError());
        return JPI_OK;
    };
    pdl(st, rows_grid, dim3(RB), 0, k_pf_rmsnorm<__nv_bfloat16>, (const float*)h->h, (const float*)h->layers[0].attn_norm,
        h->xn, M, W, eps);
    PF_CUDA(cudaGetLastError());
    for (int l = 0; l < h->L; ++l) {
        const LayerW& lw = h->layers[(size_t)l];
        __nv_bfloat16* kd = static_cast<__nv_bfloat16*>(k_layers[l]);
        __nv_bfloat16* vd = static_cast<__nv_bfloat16*>(v_layers[l]);
        // Attention sublayer: projections, rotary coding, scatter into q and the caller's KV store.
        if (h->qkv_fused()) {
            PF_TRY(row_gemm(h, st, h->xn, W, lw.wqkv, W, true, h->q, true, H * D, (int)M, h->QKV, W, 1.f, false, 0,
                            [&](PfGemmArgs& a) {
                                a.qkv = 1;
                                a.H = H;
                                a.D = D;
                                a.P = P;
                                a.rope = h->rope;
                                a.q = h->q;
                                a.kd = kd;
                                a.vd = vd;
                                a.kv_stride = request_stride;
                                a.v_pairs = reinterpret_cast<uintptr_t>(vd) % 4 == 0 ? 1 : 0;
                            }));
        } else {
            PF_TRY(row_gemm(h, st, h->xn, W, lw.wqkv, W, true, h->qkv, false, h->QKV, (int)M, h->QKV, W, 1.f, false));
            pdl(st, rows_grid, dim3(256), 0, k_pf_rope_scatter, (const float*)h->qkv, (const float2*)h->rope, h->q, kd, vd,
                request_stride, batch, P, H, D);
            PF_CUDA(cudaGetLastError());
        }
        if (t5) {
            PF_TRY(D == 256 ? attention_t5<256>(h, st, kd, vd, batch, P, request_stride / D)
                            : attention_t5<128>(h, st, kd, vd, batch, P, request_stride / D));
        }
        for (int b = 0; b < batch && !t5; ++b) {
            const __nv_bfloat16* qb = h->q + (size_t)b * P * H * D;     // [(P H)][D]
            const __nv_bfloat16* kb = kd + (size_t)b * request_stride;  // [P][D]
            const __nv_bfloat16* vb = vd + (size_t)b * request_stride;  // [P][D]
            __nv_bfloat16* ob = h->o + (size_t)b * P * H * D;           // [(P H)][D] = [P][H D]
            PF_TRY(row_gemm(h, st, qb, D, kb, D, false, h->sc, false, Pp, P * H, P, D, scale, false));
            pdl(st, dim3(grid_for((long long)P * H * 32)), dim3(256), 0, k_pf_softmax, (const float*)h->sc, h->pr,
                (long long)P * H, P, Pp);
            PF_CUDA(cudaGetLastError());
            pdl(st, dim3((P + 31) / 32, (D + 31) / 32), dim3(32, 8), 0, k_pf_transpose, vb, h->vt, P, D, Pp);
            PF_CUDA(cudaGetLastError());
            PF_TRY(row_gemm(h, st, h->pr, Pp, h->vt, Pp, false, ob, true, D, P * H, D, P, 1.f, false));
        }
        PF_TRY(residual(h->o, H * D, lw.wo, lw.mlp_norm, h->xn));
        // MLP sublayer: gate/up with GeGLU in its epilogue (z bf16), then down into the residual.
        PF_TRY(row_gemm(h, st, h->xn, W, lw.wgu, W, true, h->z, true, F, (int)M, 2 * h->Fp, W, 1.f, false, 0,
                        [&](PfGemmArgs& a) {
                            a.geglu = 1;
                            a.nz = F;
                        }));
        if (l + 1 < h->L) PF_TRY(residual(h->z, F, lw.wd, h->layers[(size_t)l + 1].attn_norm, h->xn));
        else PF_TRY(residual(h->z, F, lw.wd, out_final ? h->final_norm : nullptr, out_final));
    }
    return JPI_OK;
}

JPI_API jpi_status jpi_prefill_device_status(jpi_prefill_handle* h) {
    g_err[0] = '\0';
    if (!h) return pfail(JPI_ERR_INVALID_ARG, "handle is NULL");
    PF_CUDA(cudaDeviceSynchronize());
    int err = 0;
    PF_CUDA(cudaMemcpy(&err, h->dev_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (err != PF_DEV_OK) {
        PF_CUDA(cudaMemset(h->dev_err, 0, sizeof(int)));
        return pfail(JPI_ERR_DEVICE_TIMEOUT, "device-side error code %d (a bounded wait in a product gave up)", err);
    }
    return JPI_OK;
}

JPI_API jpi_status jpi_prefill_memory_usage(const jpi_prefill_handle* h, long long* bytes) {
    g_err[0] = '\0';
    if (!h || !bytes) return pfail(JPI_ERR_INVALID_ARG, "handle or bytes is NULL");
    *bytes = (long long)h->bytes;
    return JPI_OK;
}

}  // extern "C"
