// CUDA-core kernels: time conditioning, token embedding, the fp32 verification path of every
// layer op, the final norm + action-out projection + Euler update, and KV-store conversion.
//
// Every reduction here runs in a fixed order (fixed per-thread strides, then a fixed shuffle
// tree), so results are bitwise reproducible run to run.

#include "jpi_internal.h"
#include "tc_path.h"
#include "ptx.h"

#include <cmath>
#include <type_traits>

namespace jpi {
namespace {

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
    return __bfloat162float(*p);
}
template <typename T> __device__ __forceinline__ T cvt(float v);
template <> __device__ __forceinline__ float cvt<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}

// v rounded to T's precision, as fp32.
template <typename T> __device__ __forceinline__ float ldf_round(float v);
template <> __device__ __forceinline__ float ldf_round<float>(float v) { return v; }
template <> __device__ __forceinline__ float ldf_round<__nv_bfloat16>(float v) {
    return __bfloat162float(__float2bfloat16_rn(v));
}

__device__ __forceinline__ float swishf(float z) { return z / (1.f + expf(-z)); }

// GELU, tanh form (Gemma's MLP activation).
__device__ __forceinline__ float gelu_tanhf(float y) {
    const float k0 = 0.7978845608028654f;   // sqrt(2 / pi)
    return 0.5f * y * (1.f + tanhf(k0 * (y + 0.044715f * y * y * y)));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over a block of up to 1024 threads (blockDim a multiple of 32), fixed order.
__device__ float block_sum(float v, float* scratch /* >= 32 floats */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    float t = lane < nw ? scratch[lane] : 0.f;
    t = warp_sum(t);
    return t;
}

// Four consecutive elements (k a multiple of 4, rows 4-element aligned), or with VEC false four
// elements 32 apart per lane (any K), zero past K; rows_k says which k they are.
template <bool VEC> __device__ __forceinline__ int rows_k(int k0, int lane, int e) {
    return VEC ? k0 + 4 * lane + e : k0 + lane + 32 * e;
}
template <bool VEC>
__device__ __forceinline__ float4 rows_load(const float* p, int k0, int lane, int K) {
    if (VEC) {
        const int k = k0 + 4 * lane;
        return k < K ? *reinterpret_cast<const float4*>(p + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = rows_k<false>(k0, lane, e);
        v[e] = k < K ? p[k] : 0.f;
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}
template <bool VEC>
__device__ __forceinline__ float4 rows_load(const __nv_bfloat16* p, int k0, int lane, int K) {
    if (VEC) {
        const int k = k0 + 4 * lane;
        if (k >= K) return make_float4(0.f, 0.f, 0.f, 0.f);
        const uint2 u = *reinterpret_cast<const uint2*>(p + k);
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                           __uint_as_float(u.y & 0xFFFF0000u));
    }
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = rows_k<false>(k0, lane, e);
        v[e] = k < K ? __bfloat162float(p[k]) : 0.f;
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------------------------------------
// Time conditioning: flow time enters the expert only through a sinusoidal embedding followed
// by a two-layer swish MLP; the per-layer modulation vectors are a linear map of the result.
// All of it depends on t alone, so it is evaluated once per call for every step time.

// Grid (steps, ceil(half / 32)): one frequency i of one step time per thread, a warp per block (fp64
// sin/cos are slow on this GPU, two lanes' worth a clock: spread over the SMs they run side by side).
// The periods are tabulated at create.
constexpr int TE_THREADS = 32;
__global__ void k_time_embed(float* temb, const double* __restrict__ period, int nsteps, int dt, double t_override) {
    ptx::grid_dep_launch();   // the next kernel waits for this one's results before reading them
    const int k = blockIdx.x;
    const double t = t_override >= 0.0 ? t_override : (double)k / (double)nsteps;
    const int half = dt / 2, i = blockIdx.y * TE_THREADS + threadIdx.x;
    if (i >= half) return;
    const double theta = 2.0 * 3.14159265358979323846 * t / period[i];
    double s, c;
    sincos(theta, &s, &c);
    temb[(size_t)k * dt + i] = (float)s;
    temb[(size_t)k * dt + half + i] = (float)c;
}

// Y[n][r] = act(sum_k W[r][k] X[n][k] + b[r]) for n < N <= GV_N, r < R: one warp per output row,
// its first GV_U x 128 weights in registers before the dependency wait, X in shared memory (read as
// 16-byte chunks, four consecutive k per lane). Launches of the time MLP are short chains; weight loads of 2
// bytes issued after the inputs are staged make 1024 rows x 1024 bf16 weights an 11 us one.
// The modulation vectors (no swish) are read by kernels before their own dependency wait: that
// launch does not release its dependent early.
constexpr int GV_N = 16, GV_U = 8;
template <typename TW, bool SWISH, bool VEC>
__global__ void __launch_bounds__(256) k_gemv_multi(const TW* __restrict__ Wm, const float* __restrict__ bias,
                                                    const float* __restrict__ X, float* __restrict__ Y, int R, int K,
                                                    int N) {
    extern __shared__ __align__(16) float xs[];   // [N][K]
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    float4 w4[GV_U];
    auto load = [&](int r, int kb) {
#pragma unroll
        for (int u = 0; u < GV_U; ++u)
            w4[u] = r < R ? rows_load<VEC>(Wm + (size_t)r * K, kb + 128 * u, lane, K) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    load(warp, 0);
    ptx::grid_dep_wait();
    if (SWISH) ptx::grid_dep_launch();
    // Eight loads of each thread in flight before their stores.
    if (VEC) {
        const int n4 = N * K / 4;
        for (int i0 = threadIdx.x; i0 < n4; i0 += 8 * blockDim.x) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * blockDim.x;
                v[u] = i < n4 ? reinterpret_cast<const float4*>(X)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * blockDim.x;
                if (i < n4) reinterpret_cast<float4*>(xs)[i] = v[u];
            }
        }
    } else {
        for (int i = threadIdx.x; i < N * K; i += blockDim.x) xs[i] = X[i];
    }
    __syncthreads();
    for (int r = warp; r < R; r += nwarps) {
        float acc[GV_N];
#pragma unroll
        for (int j = 0; j < GV_N; ++j) acc[j] = 0.f;
        for (int kb = 0; kb < K; kb += 128 * GV_U) {
            if (kb > 0 || r != warp) load(r, kb);
#pragma unroll
            for (int u = 0; u < GV_U; ++u) {
                if (kb + 128 * u >= K) break;
#pragma unroll
                for (int j = 0; j < GV_N; ++j)
                    if (j < N) {
                        const float4 x4 = rows_load<VEC>(xs + (size_t)j * K, kb + 128 * u, lane, K);
                        acc[j] = fmaf(w4[u].x, x4.x, acc[j]);
                        acc[j] = fmaf(w4[u].y, x4.y, acc[j]);
                        acc[j] = fmaf(w4[u].z, x4.z, acc[j]);
                        acc[j] = fmaf(w4[u].w, x4.w, acc[j]);
                    }
            }
        }
        const float br = bias[r];
#pragma unroll
        for (int j = 0; j < GV_N; ++j)
            if (j < N) {
                const float y = warp_sum(acc[j]) + br;
                if (lane == 0) Y[(size_t)j * R + r] = SWISH ? swishf(y) : y;
            }
    }
}

// Y[n][r] = sum_k W[r][k] X[n][k] + b[r] for all n < NG step times at once: the stacked
// modulation matrix (6 L + 2) W rows is streamed from HBM exactly once per call. Each thread
// owns MOD_RT consecutive rows; per 16-wide K slab it loads 32 bytes of every row (full
// sectors) and reads each X value as a shared-memory broadcast, so the inner loop is FMAs.
constexpr int MOD_RT = 4;

template <typename TW> struct Slab;                 // 16 consecutive weights of one row
template <> struct Slab<__nv_bfloat16> {
    uint4 v[2];
    __device__ __forceinline__ void load(const __nv_bfloat16* p) {
        v[0] = __ldg((const uint4*)p);
        v[1] = __ldg((const uint4*)p + 1);
    }
    __device__ __forceinline__ float get(int i) const {
        const uint32_t u = (&v[0].x)[i >> 1];
        return __uint_as_float((i & 1) ? (u & 0xFFFF0000u) : (u << 16));
    }
};
template <> struct Slab<float> {
    float4 v[4];
    __device__ __forceinline__ void load(const float* p) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __ldg((const float4*)p + i);
    }
    __device__ __forceinline__ float get(int i) const { return (&v[0].x)[i]; }
};

template <typename TW, int NG>
__global__ void __launch_bounds__(256) k_mod_gemv(const TW* __restrict__ Wm, const float* __restrict__ bias,
                                                   const float* __restrict__ X, float* __restrict__ Y,
                                                   int R, int K) {
    extern __shared__ float xs[];                     // [NG][K]
    for (int i = threadIdx.x; i < NG * K; i += blockDim.x) xs[i] = X[i];
    __syncthreads();
    const int r0 = (blockIdx.x * blockDim.x + threadIdx.x) * MOD_RT;
    if (r0 >= R) return;
    float acc[MOD_RT][NG];
#pragma unroll
    for (int rr = 0; rr < MOD_RT; ++rr)
#pragma unroll
        for (int n = 0; n < NG; ++n) acc[rr][n] = 0.f;
    const TW* rowp[MOD_RT];
#pragma unroll
    for (int rr = 0; rr < MOD_RT; ++rr) rowp[rr] = Wm + (size_t)min(r0 + rr, R - 1) * K;
    Slab<TW> cur[MOD_RT], nxt[MOD_RT];
#pragma unroll
    for (int rr = 0; rr < MOD_RT; ++rr) cur[rr].load(rowp[rr]);
    for (int k0 = 0; k0 < K; k0 += 16) {
        if (k0 + 16 < K) {
#pragma unroll
            for (int rr = 0; rr < MOD_RT; ++rr) nxt[rr].load(rowp[rr] + k0 + 16);
        }
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            float w[MOD_RT];
#pragma unroll
            for (int rr = 0; rr < MOD_RT; ++rr) w[rr] = cur[rr].get(kk);
#pragma unroll
            for (int n = 0; n < NG; ++n) {
                const float xv = xs[n * K + k0 + kk];
#pragma unroll
                for (int rr = 0; rr < MOD_RT; ++rr) acc[rr][n] = fmaf(w[rr], xv, acc[rr][n]);
            }
        }
#pragma unroll
        for (int rr = 0; rr < MOD_RT; ++rr) cur[rr] = nxt[rr];
    }
#pragma unroll
    for (int n = 0; n < NG; ++n)
#pragma unroll
        for (int rr = 0; rr < MOD_RT; ++rr)
            if (r0 + rr < R) Y[(size_t)n * R + r0 + rr] = acc[rr][n] + bias[r0 + rr];
}

// ---------------------------------------------------------------------------------------------
// Token embedding: row 0 of each request is the state token, rows 1..nctx-1 the correction
// items (context tokens, taken as given), then the C action tokens.
// Block = 512 features (four per thread, a warp per 128-feature slice) of up to tpb tokens that share
// one input matrix: blockIdx.y counts groups of action tokens first, then groups of state and context
// tokens. A thread keeps its features' weights in registers for all of the block's tokens and reads
// the tokens' inputs from shared memory as broadcasts. What bounds it: with a token per block, the
// weight rows (a line per feature) were fetched again for every token (382 us at 3264 tokens x 1024
// features); with a feature per thread, the instructions around each token's 32 products (31 us).
// The outputs alone are 20 MB, 3 us.
// For the tensor-core path it also writes the operand of the first layer's norm-fed projection
// (xs = bf16((1 + sigma) * h) at row xs_row(m), and beta in the last row of every 64-row tile) and
// each token's sum of squares over the 128 features (ss[slice][m]).
struct EmbedArgs {
    float* hres;
    __nv_bfloat16* xs;   // null without the tensor-core path (as is ss)
    const float *sigma, *beta;
    float* ss;
    int ss_ld;
    const float *state, *x, *Ws, *bs, *Wa, *ba, *corr;
    int nctx, B, S, C, W, Sd, A;
    int tpb, action_groups;   // tokens per block; groups of action tokens
};
constexpr int EMB_MAX_TPB = 16;
constexpr int EMB_K = 32;     // inputs per token kept in registers / shared memory

__device__ __forceinline__ uint2 pack_bf16x4(float a, float b, float c, float d) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

__global__ void __launch_bounds__(128) k_embed(const EmbedArgs a) {
    __shared__ __align__(16) float in_s[EMB_MAX_TPB][EMB_K];
    const int tid = threadIdx.x, lane = tid & 31;
    const bool act = (int)blockIdx.y < a.action_groups;
    // Tokens [j0, j0 + nt) of this block's kind: action token j = (request j / C, action j mod C),
    // else context token j = (request j / nctx, row j mod nctx).
    const int per = act ? a.C : a.nctx;
    const int j0 = (act ? blockIdx.y : blockIdx.y - a.action_groups) * a.tpb;
    const int nt = min(a.tpb, a.B * per - j0);
    const int K = act ? a.A : a.Sd;
    const int Kr = min(K, EMB_K);
    const float* Wm = act ? a.Wa : a.Ws;
    const int n = (blockIdx.x * 128 + tid) * 4;   // first of four features (W is a multiple of 32)
    const bool live = n < a.W;
    // The weights depend on nothing upstream. Products past K multiply zeros.
    float4 wv[EMB_K];   // input k of the four features (the matrices are stored [K][W])
    float4 bv = make_float4(0.f, 0.f, 0.f, 0.f), sg = bv, bt = bv;
#pragma unroll
    for (int k = 0; k < EMB_K; ++k)
        wv[k] = k < K && live ? __ldg(reinterpret_cast<const float4*>(Wm + (size_t)k * a.W + n)) : bv;
    if (live) {
        bv = *reinterpret_cast<const float4*>((act ? a.ba : a.bs) + n);
    }
    // Launched with programmatic dependent launch: x comes from the previous step's final kernel;
    // the next kernel may start its weight prefetch at once.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (live && a.xs) {
        sg = *reinterpret_cast<const float4*>(a.sigma + n);
        bt = *reinterpret_cast<const float4*>(a.beta + n);
    }
    // Inputs of token j: its action row, or its request's state (context rows past 0 have none).
    auto input = [&](int j) { return act ? a.x + (size_t)j * a.A : a.state + (size_t)(j / a.nctx) * a.Sd; };
    for (int i = tid; i < nt * EMB_K; i += 128) {
        const int tt = i / EMB_K, k = i % EMB_K;
        in_s[tt][k] = k < Kr ? input(j0 + tt)[k] : 0.f;
    }
    __syncthreads();
    int b = j0 / per, i = j0 - b * per;   // request and row within its kind, advanced token by token
    for (int tt = 0; tt < nt; ++tt) {
        const int m = b * a.S + (act ? a.nctx : 0) + i;
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (live) {
            if (!act && i > 0) {
                const float4 c = *reinterpret_cast<const float4*>(a.corr + ((size_t)b * (a.nctx - 1) + (i - 1)) * a.W + n);
                v[0] = c.x;
                v[1] = c.y;
                v[2] = c.z;
                v[3] = c.w;
            } else {
                const float4* iv = reinterpret_cast<const float4*>(in_s[tt]);
                auto add = [&](const float4& w, float x) {
                    v[0] = fmaf(w.x, x, v[0]);
                    v[1] = fmaf(w.y, x, v[1]);
                    v[2] = fmaf(w.z, x, v[2]);
                    v[3] = fmaf(w.w, x, v[3]);
                };
#pragma unroll
                for (int k = 0; k < EMB_K; k += 4) {
                    const float4 x4 = iv[k / 4];
                    add(wv[k], x4.x);
                    add(wv[k + 1], x4.y);
                    add(wv[k + 2], x4.z);
                    add(wv[k + 3], x4.w);
                }
                if (K > EMB_K) {
                    const float* in = input(j0 + tt);
                    for (int k = EMB_K; k < K; ++k)
                        add(__ldg(reinterpret_cast<const float4*>(Wm + (size_t)k * a.W + n)), in[k]);
                }
                v[0] += bv.x;
                v[1] += bv.y;
                v[2] += bv.z;
                v[3] += bv.w;
            }
            *reinterpret_cast<float4*>(a.hres + (size_t)m * a.W + n) = make_float4(v[0], v[1], v[2], v[3]);
            if (a.xs)
                *reinterpret_cast<uint2*>(a.xs + (size_t)xs_row(m) * a.W + n) =
                    pack_bf16x4((1.f + sg.x) * v[0], (1.f + sg.y) * v[1], (1.f + sg.z) * v[2], (1.f + sg.w) * v[3]);
        }
        if (a.ss) {   // W is a multiple of 128 then: a warp is one slice
            const float t = warp_sum(fmaf(v[0], v[0], v[1] * v[1]) + fmaf(v[2], v[2], v[3] * v[3]));
            if (lane == 0 && live) a.ss[(size_t)(n >> 7) * a.ss_ld + m] = t;
        }
        if (++i == per) {
            i = 0;
            ++b;
        }
    }
    if (a.xs && live) {
        // Tile z's beta row: block y takes tiles y tpb .. (the blocks' token slots cover the tiles).
        const int z0 = blockIdx.y * a.tpb, z1 = min(z0 + a.tpb, xs_tiles(a.B * a.S));
        for (int z = z0; z < z1; ++z)
            *reinterpret_cast<uint2*>(a.xs + ((size_t)z * 64 + 63) * a.W + n) = pack_bf16x4(bt.x, bt.y, bt.z, bt.w);
    }
}

// ---------------------------------------------------------------------------------------------
// The layer ops on CUDA cores (the fp32 verification mode, and bf16 dims the tensor-core kernels do
// not tile): five launches per layer, each product with the passes around it fused in.
//   RK_QKV    adaptive RMSNorm of h, product, rotary coding, scatter into q and the KV store's tail
//   RK_GEGLU  adaptive RMSNorm of h, gate and up products, z = gelu_tanh(gate) * up
//   RK_RESID  product, gated residual h += gamma * y
// A warp owns ROWS_M token rows x 4 weight rows ("slots") over one of KS ranges of K; a lane takes
// four consecutive k of every 128 for all 16 x 4 outputs (20 loads of 16 bytes per 256 FMAs in fp32),
// so no operand passes through shared memory and every load of a k step is in flight at once. The
// 64 sums are then reduced over the lanes by a reduce-scatter (lane L ends with row L / 2, slots
// 2 (L mod 2) and + 1) and over the KS warps in order. A small batch (9 tokens) is bound by latency,
// not by its operations: a 64 x 64 tile per block walked K alone, 4-16 blocks on the GPU, at 26 us
// (K = 256) to 100 us (K = 1024) per product.
// Slots: QKV (j, j + D/2) of two rotary pairs, GeGLU (gate, up) of two features, else 4 features.
enum { RK_QKV = 0, RK_RESID = 1, RK_GEGLU = 2 };
constexpr int ROWS_M = 16;
constexpr int ROWS_WARPS = 4;

struct RowsArgs {
    const void* X;              // RESID: [M][K] input (T)
    const float* h;             // norm kinds: residual stream [M][K]
    const float *sigma, *beta;  // norm kinds
    const void *W1, *W2;        // [N][K]; GeGLU: gate and up
    int M, N, K;                // N: output features (QKV: (H + 2) D)
    float eps;
    float* hres;                // RESID: [M][N] updated in place
    const float* gamma;
    void* z;                    // GeGLU: [M][N]
    void *q, *kst, *vst;        // QKV
    const float2* rope;
    int S, H, D, P, kv_rows;
};

template <typename T, int KIND, bool VEC, int KS>
__global__ void __launch_bounds__(32 * ROWS_WARPS) k_rows_gemm(const RowsArgs a) {
    constexpr bool NORM = KIND != RK_RESID;
    constexpr int CW = ROWS_WARPS / KS;   // slot groups per block
    __shared__ float rinv_s[ROWS_M];
    __shared__ float2 red[ROWS_WARPS][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ks = warp % KS, cw = warp / KS;
    const int g = blockIdx.x * CW + cw;              // slot group
    const int m0 = blockIdx.y * ROWS_M;
    const int hd = KIND == RK_QKV ? a.D >> 1 : 0;
    // Slot s of group g: feature (row of W) and matrix.
    auto feature = [&](int s) {
        if (KIND == RK_QKV) {
            const int pair = 2 * g + (s >> 1), sec = pair / hd;
            return sec * a.D + (pair - sec * hd) + (s & 1) * hd;
        }
        if (KIND == RK_GEGLU) return 2 * g + (s >> 1);
        return 4 * g + s;
    };
    const T* wr[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int f = min(feature(s), a.N - 1);   // clamped; result unused
        wr[s] = static_cast<const T*>(KIND == RK_GEGLU && (s & 1) ? a.W2 : a.W1) + (size_t)f * a.K;
    }
    // K range of this warp in steps of 128.
    const int nst = (a.K + 127) / 128;
    const int st_lo = ks * nst / KS, st_hi = (ks + 1) * nst / KS;
    // The first step's weights depend on nothing upstream.
    float4 w4[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) w4[s] = rows_load<VEC>(wr[s], st_lo * 128, lane, a.K);
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    if (NORM) {
        // 1 / rms of the block's rows: warp w takes rows w, w + 4, ..
        float s4[ROWS_M / ROWS_WARPS];
#pragma unroll
        for (int i = 0; i < ROWS_M / ROWS_WARPS; ++i) {
            const int m = m0 + warp + ROWS_WARPS * i;
            const float* hr = a.h + (size_t)m * a.K;
            float s = 0.f;
            if (m < a.M)
                for (int k0 = 0; k0 < a.K; k0 += 128) {
                    const float4 v = rows_load<VEC>(hr, k0, lane, a.K);
                    s = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, s))));
                }
            s4[i] = s;
        }
#pragma unroll
        for (int i = 0; i < ROWS_M / ROWS_WARPS; ++i) {
            const float s = warp_sum(s4[i]);
            if (lane == 0) rinv_s[warp + ROWS_WARPS * i] = rsqrtf(s / (float)a.K + a.eps);
        }
        __syncthreads();
    }
    float acc[ROWS_M][4];
#pragma unroll
    for (int r = 0; r < ROWS_M; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[r][s] = 0.f;
    for (int st = st_lo; st < st_hi; ++st) {
        const int k0 = st * 128;
        float4 sg = make_float4(0.f, 0.f, 0.f, 0.f), bt = sg;
        if (NORM) {
            sg = rows_load<VEC>(a.sigma, k0, lane, a.K);
            bt = rows_load<VEC>(a.beta, k0, lane, a.K);
        }
        float4 wn[4];   // next step's weights
#pragma unroll
        for (int s = 0; s < 4; ++s)
            wn[s] = st + 1 < st_hi ? rows_load<VEC>(wr[s], k0 + 128, lane, a.K) : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool in = VEC ? k0 + 4 * lane < a.K : true;
#pragma unroll
        for (int r0 = 0; r0 < ROWS_M; r0 += 8) {
            if (m0 + r0 >= a.M) break;
            float4 x4[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int m = m0 + r0 + r;
                x4[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m < a.M) {
                    if (NORM) x4[r] = rows_load<VEC>(a.h + (size_t)m * a.K, k0, lane, a.K);
                    else x4[r] = rows_load<VEC>(static_cast<const T*>(a.X) + (size_t)m * a.K, k0, lane, a.K);
                }
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                float4 x = x4[r];
                if (NORM && in) {
                    const float ri = rinv_s[r0 + r];
                    x.x = ldf_round<T>(x.x * ri * (1.f + sg.x) + bt.x);
                    x.y = ldf_round<T>(x.y * ri * (1.f + sg.y) + bt.y);
                    x.z = ldf_round<T>(x.z * ri * (1.f + sg.z) + bt.z);
                    x.w = ldf_round<T>(x.w * ri * (1.f + sg.w) + bt.w);
                }
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    float t = acc[r0 + r][s];
                    t = fmaf(x.x, w4[s].x, t);
                    t = fmaf(x.y, w4[s].y, t);
                    t = fmaf(x.z, w4[s].z, t);
                    t = fmaf(x.w, w4[s].w, t);
                    acc[r0 + r][s] = t;
                }
            }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) w4[s] = wn[s];
    }
    // Reduce-scatter over the lanes: value v = 4 row + slot ends in lane v / 2.
    float pv[4 * ROWS_M];
#pragma unroll
    for (int r = 0; r < ROWS_M; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s) pv[4 * r + s] = acc[r][s];
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
        const bool hi = (lane & sh) != 0;
#pragma unroll
        for (int i = 0; i < 2 * sh; ++i) {
            const float send = hi ? pv[i] : pv[i + 2 * sh];
            const float keep = hi ? pv[i + 2 * sh] : pv[i];
            pv[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
        }
    }
    float y0 = pv[0], y1 = pv[1];
    if (KS > 1) {
        red[warp][lane] = make_float2(y0, y1);
        __syncthreads();
        if (ks != 0) return;
#pragma unroll
        for (int i = 1; i < KS; ++i) {
            const float2 v = red[warp + i][lane];
            y0 += v.x;
            y1 += v.y;
        }
    }
    const int m = m0 + (lane >> 1), sp = 2 * (lane & 1);   // row, first slot of the lane's two
    if (m >= a.M) return;
    const int f = feature(sp);
    if (f >= a.N) return;
    if (KIND == RK_RESID) {
        float* hp = a.hres + (size_t)m * a.N + f;
        hp[0] += a.gamma[f] * y0;
        if (f + 1 < a.N) hp[1] += a.gamma[f + 1] * y1;
    } else if (KIND == RK_GEGLU) {
        static_cast<T*>(a.z)[(size_t)m * a.N + f] = cvt<T>(gelu_tanhf(y0) * y1);
    } else {
        // Rotary pair (d, d + D/2) of head section sec at position P + i (rotate-half).
        const int sec = f / a.D, d = f - sec * a.D;
        const int b = m / a.S, pos = a.P + (m - b * a.S);
        if (a.rope && sec <= a.H) {
            const float2 cs = a.rope[(size_t)pos * hd + d];
            const float r0 = y0 * cs.x - y1 * cs.y, r1 = y1 * cs.x + y0 * cs.y;
            y0 = r0;
            y1 = r1;
        }
        T* dst = sec < a.H ? static_cast<T*>(a.q) + ((size_t)m * a.H + sec) * a.D
                           : static_cast<T*>(sec == a.H ? a.kst : a.vst) + ((size_t)b * a.kv_rows + pos) * a.D;
        dst[d] = cvt<T>(y0);
        dst[d + hd] = cvt<T>(y1);
    }
}

// ---------------------------------------------------------------------------------------------
// Adaptive RMSNorm of one token row: u = h / sqrt(mean(h^2) + eps) * (1 + sigma) + beta.
template <typename TA>
__global__ void k_rms_mod(const float* __restrict__ hres, const float* __restrict__ sigma,
                          const float* __restrict__ beta, TA* __restrict__ out, int W, int ldo,
                          float eps) {
    __shared__ float scratch[32];
    const int m = blockIdx.x;
    const float* hr = hres + (size_t)m * W;
    float ss = 0.f;
    for (int k = threadIdx.x; k < W; k += blockDim.x) ss = fmaf(hr[k], hr[k], ss);
    ss = block_sum(ss, scratch);
    const float rinv = rsqrtf(ss / (float)W + eps);
    for (int k = threadIdx.x; k < W; k += blockDim.x)
        out[(size_t)m * ldo + k] = cvt<TA>(hr[k] * rinv * (1.f + sigma[k]) + beta[k]);
}

// ---------------------------------------------------------------------------------------------
// Products of many tokens (see rows_fit below): Y[m][n] = sum_k X[m][k] W[n][k] with three epilogues:
//   STORE  Y[m][n] = y
//   RESID  Y[m][n] += gamma[n] * y            (gated residual update of h)
//   GEGLU  Z[m][n] = gelu_tanh(y_gate) * y_up (second weight matrix W2 = up)
enum { EPI_STORE = 0, EPI_RESID = 1, EPI_GEGLU = 2 };

constexpr int GB_M = 64, GB_N = 64, GB_K = 16;

template <typename TA, typename TW, int EPI>
__global__ void __launch_bounds__(256) k_gemm_simt(
    const TA* __restrict__ X, int ldx, const TW* __restrict__ W1, const TW* __restrict__ W2,
    int M, int N, int K, float* __restrict__ Y, int ldy, const float* __restrict__ gamma,
    TA* __restrict__ Z, int ldz) {
    __shared__ float xs[GB_K][GB_M + 4];
    __shared__ float ws[GB_K][GB_N + 4];
    __shared__ float us[(EPI == EPI_GEGLU) ? GB_K : 1][GB_N + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * GB_M, n0 = blockIdx.x * GB_N;
    float acc[4][4] = {}, acc2[4][4] = {};
    for (int k0 = 0; k0 < K; k0 += GB_K) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int idx = tid + e * 256;          // 0..1023 over a 64 x 16 tile
            const int r = idx >> 4, kk = idx & 15;
            const int gm = m0 + r, gn = n0 + r, gk = k0 + kk;
            xs[kk][r] = (gm < M && gk < K) ? ldf(X + (size_t)gm * ldx + gk) : 0.f;
            ws[kk][r] = (gn < N && gk < K) ? ldf(W1 + (size_t)gn * K + gk) : 0.f;
            if (EPI == EPI_GEGLU)
                us[kk][r] = (gn < N && gk < K) ? ldf(W2 + (size_t)gn * K + gk) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GB_K; ++kk) {
            float a[4], bw[4], bu[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = xs[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bw[j] = ws[kk][tx * 4 + j];
            if (EPI == EPI_GEGLU) {
#pragma unroll
                for (int j = 0; j < 4; ++j) bu[j] = us[kk][tx * 4 + j];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = fmaf(a[i], bw[j], acc[i][j]);
                    if (EPI == EPI_GEGLU) acc2[i][j] = fmaf(a[i], bu[j], acc2[i][j]);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n >= N) continue;
            if (EPI == EPI_STORE) {
                Y[(size_t)m * ldy + n] = acc[i][j];
            } else if (EPI == EPI_RESID) {
                Y[(size_t)m * ldy + n] += gamma[n] * acc[i][j];
            } else {
                Z[(size_t)m * ldz + n] = cvt<TA>(gelu_tanhf(acc[i][j]) * acc2[i][j]);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Rotary encoding of the suffix q and k at positions P + i (rotate-half pairs (d, d + D/2)),
// then q to the query buffer and k, v into the KV store's suffix tail of this layer.
template <typename TQ, typename TKV>
__global__ void k_qkv_post(const float* __restrict__ qkv, TQ* __restrict__ q,
                           TKV* __restrict__ kst, TKV* __restrict__ vst,
                           const float2* __restrict__ rope, int S, int H, int D, int P,
                           int kv_rows) {
    const int m = blockIdx.x;
    const int b = m / S, i = m % S, pos = P + i;
    const int hd = D / 2, QKVd = (H + 2) * D;
    const float* row = qkv + (size_t)m * QKVd;
    for (int idx = threadIdx.x; idx < (H + 1) * hd; idx += blockDim.x) {
        const int hh = idx / hd, d = idx % hd;       // hh == H is the key head
        const float x1 = row[hh * D + d], x2 = row[hh * D + d + hd];
        float c = 1.f, s = 0.f;
        if (rope) { const float2 cs = rope[(size_t)pos * hd + d]; c = cs.x; s = cs.y; }
        const float y1 = x1 * c - x2 * s, y2 = x2 * c + x1 * s;
        if (hh < H) {
            q[(size_t)m * H * D + hh * D + d] = cvt<TQ>(y1);
            q[(size_t)m * H * D + hh * D + d + hd] = cvt<TQ>(y2);
        } else {
            kst[((size_t)b * kv_rows + pos) * D + d] = cvt<TKV>(y1);
            kst[((size_t)b * kv_rows + pos) * D + d + hd] = cvt<TKV>(y2);
        }
    }
    for (int d = threadIdx.x; d < D; d += blockDim.x)
        vst[((size_t)b * kv_rows + pos) * D + d] = cvt<TKV>(row[(H + 1) * D + d]);
}

// ---------------------------------------------------------------------------------------------
// Attention of one suffix token and HB of its query heads over [prefix ; suffix] keys of the single
// KV head. The state and context rows (i < nctx) see the prefix and each other; action rows see all.
// Warp w takes keys 4 w .. 4 w + 3, then + 32, ..: four keys' rows in flight at a time, the D products
// spread over the lanes (d = lane + 32 j, j < ND), one online softmax per head and warp; the eight
// warps' (max, sum, output) are combined in warp order through shared memory. HB = 4 reads each key
// once for four heads; HB = 1 spreads a small batch over four times the blocks (the launcher has the
// line). Bound by the loads of the keys, 32 in flight a block: 408 tokens x 8 heads x 867 keys (D = 256) 280 us.
constexpr int AR_WARPS = 8;

template <typename T, int HB, int ND>
__global__ void __launch_bounds__(32 * AR_WARPS) k_attn_rows(const T* __restrict__ q, const T* kst, const T* vst,
                                                             T* __restrict__ o, int S, int H, int D, int P,
                                                             int kv_rows, int nctx, float scale) {
    __shared__ float om[AR_WARPS][HB][32 * ND];
    __shared__ float2 ml[AR_WARPS][HB];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int hg = H / HB;
    const int m = blockIdx.x / hg, h0 = (blockIdx.x % hg) * HB;
    const int b = m / S, i = m - b * S;
    const int nvis = i < nctx ? P + nctx : P + S;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    float qf[HB][ND], acc[HB][ND];
    // Running maximum and sum: HB = 4: of head lane / 8, in every lane; HB = 1: of the one head.
    float mx = -INFINITY, l = 0.f;
#pragma unroll
    for (int hh = 0; hh < HB; ++hh) {
#pragma unroll
        for (int j = 0; j < ND; ++j) {
            const int d = lane + 32 * j;
            acc[hh][j] = 0.f;
            qf[hh][j] = d < D ? ldf(q + ((size_t)m * H + h0 + hh) * D + d) : 0.f;
        }
    }
    const T* kb = kst + (size_t)b * kv_rows * D;
    const T* vb = vst + (size_t)b * kv_rows * D;
    for (int key0 = 4 * warp; key0 < nvis; key0 += 4 * AR_WARPS) {
        float kv[4][ND], vv[4][ND];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const size_t row = (size_t)min(key0 + u, nvis - 1) * D;
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                const int d = lane + 32 * j;
                kv[u][j] = d < D ? ldf(kb + row + d) : 0.f;
                vv[u][j] = d < D ? ldf(vb + row + d) : 0.f;
            }
        }
        float s[4 * HB];   // head hh, key u at 4 hh + u: this lane's share of the dot product
#pragma unroll
        for (int hh = 0; hh < HB; ++hh)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float t = 0.f;
#pragma unroll
                for (int j = 0; j < ND; ++j) t = fmaf(qf[hh][j], kv[u][j], t);
                s[4 * hh + u] = t;
            }
        float p[4 * HB], corr[HB];   // probabilities and rescale factors, in every lane
        if constexpr (HB == 4) {
            // Reduce-scatter over the lanes: lane L ends with value L / 2 (head L / 8, key L / 2 mod
            // 4), takes one exponential for it, and the 16 + 4 results are shuffled back.
#pragma unroll
            for (int sh = 16; sh > 1; sh >>= 1) {
                const bool hi = (lane & sh) != 0;
#pragma unroll
                for (int v = 0; v < sh / 2; ++v) {
                    const float send = hi ? s[v] : s[v + sh / 2];
                    const float keep = hi ? s[v + sh / 2] : s[v];
                    s[v] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
                }
            }
            float sv = s[0] + __shfl_xor_sync(0xffffffffu, s[0], 1);
            sv = key0 + ((lane >> 1) & 3) < nvis ? sv * scale : -INFINITY;
            float nm = fmaxf(sv, __shfl_xor_sync(0xffffffffu, sv, 2));
            nm = fmaxf(nm, __shfl_xor_sync(0xffffffffu, nm, 4));
            nm = fmaxf(nm, mx);   // key0 is visible
            const float c = mx == -INFINITY ? 0.f : expf(mx - nm);
            const float e = sv == -INFINITY ? 0.f : expf(sv - nm);
            float es = e + __shfl_xor_sync(0xffffffffu, e, 2);
            es += __shfl_xor_sync(0xffffffffu, es, 4);
            l = l * c + es;
            mx = nm;
#pragma unroll
            for (int v = 0; v < 16; ++v) p[v] = __shfl_sync(0xffffffffu, e, 2 * v);
#pragma unroll
            for (int hh = 0; hh < HB; ++hh) corr[hh] = __shfl_sync(0xffffffffu, c, 8 * hh);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = key0 + u < nvis ? warp_sum(s[u]) * scale : -INFINITY;
            const float nm = fmaxf(fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])), mx);   // key0 is visible
            corr[0] = mx == -INFINITY ? 0.f : expf(mx - nm);
#pragma unroll
            for (int u = 0; u < 4; ++u) p[u] = s[u] == -INFINITY ? 0.f : expf(s[u] - nm);
            l = l * corr[0] + ((p[0] + p[1]) + (p[2] + p[3]));
            mx = nm;
        }
#pragma unroll
        for (int hh = 0; hh < HB; ++hh)
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                float t = acc[hh][j] * corr[hh];
#pragma unroll
                for (int u = 0; u < 4; ++u) t = fmaf(p[4 * hh + u], vv[u][j], t);
                acc[hh][j] = t;
            }
    }
    if (lane % (32 / HB) == 0) ml[warp][lane / (32 / HB)] = make_float2(mx, l);
#pragma unroll
    for (int hh = 0; hh < HB; ++hh)
#pragma unroll
        for (int j = 0; j < ND; ++j) om[warp][hh][lane + 32 * j] = acc[hh][j];
    __syncthreads();
    for (int idx = tid; idx < HB * D; idx += 32 * AR_WARPS) {
        const int hh = idx / D, d = idx - hh * D;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < AR_WARPS; ++w) M = fmaxf(M, ml[w][hh].x);
        float num = 0.f, den = 0.f;
#pragma unroll
        for (int w = 0; w < AR_WARPS; ++w) {
            const float c = ml[w][hh].x == -INFINITY ? 0.f : expf(ml[w][hh].x - M);
            num = fmaf(c, om[w][hh][d], num);
            den = fmaf(c, ml[w][hh].y, den);
        }
        o[((size_t)m * H + h0 + hh) * D + d] = cvt<T>(num / den);
    }
}

// ---------------------------------------------------------------------------------------------
// Final adaptive RMSNorm of an action row, velocity v = u W_out^T + b_out, Euler update
// x <- x + delta v (or, for a single forward, v itself).
// One CTA of FIN_THREADS per FR action rows. The rows' values give the norms and the normalised rows
// go to shared memory; then a warp takes four outputs of all FR rows, a lane four consecutive columns
// of every 128 (FR + 4 16-byte loads per 16 FR products), and the sums are reduced over the lanes.
// With one row per CTA, each CTA reads all of W_out (128 KB at 32 x 1024) from L2: 32 us for 3200
// rows; FR = 1 stays for few rows, where the CTAs run side by side and the chain is shortest.
// A row's sums do not depend on FR: its squares are added as 256 strided partials in the tree of one
// CTA per row (FR = 1), whichever warp owns the row, and its products in the same lanes and order.
constexpr int FIN_THREADS = 256;
constexpr int FIN_CAP = 16;   // W <= 4096
constexpr size_t FIN_SMEM_MAX = 100 * 1024;   // rows of one CTA (two CTAs per SM)
struct FinalArgs {
    const float *hres, *sigma, *beta, *Wout, *bout;
    float *x, *vout;
    int rows, S, nctx, C, W, A;   // rows: action rows of all requests
    float eps, delta;
};

// Sums v over the lanes (reduce-scatter, partners 16, 8, .., 1 lanes apart): lane L is left with the
// totals of values L NV / 32 .. in v[0 .. max(NV / 32, 1)) (for NV < 32, 32 / NV lanes share one).
template <int NV>
__device__ __forceinline__ void lane_reduce(float (&v)[NV], int lane) {
    int n = NV;
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool hi = (lane & sh) != 0;
#pragma unroll
            for (int i = 0; i < NV / 2; ++i) {
                if (i >= n) break;
                const float send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], sh);
        }
    }
}

// Outputs of the FR normalised rows us [FR][W] of the CTA (rows bj0 ..). w0: the first PRE steps of
// the warp's first four rows of W_out.
template <int FR, int PRE>
__device__ __forceinline__ void final_outputs(const FinalArgs& a, const float* us, int bj0, float4 (&w0)[PRE][4]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o0 = 4 * warp; o0 < a.A; o0 += 4 * (FIN_THREADS / 32)) {
        float v[4 * FR];   // row r, output o0 + s at 4 r + s
#pragma unroll
        for (int i = 0; i < 4 * FR; ++i) v[i] = 0.f;
        auto step = [&](int k0, const float4 (&w4)[4]) {
#pragma unroll
            for (int r = 0; r < FR; ++r) {
                const int k = k0 + 4 * lane;
                const float4 u4 = k < a.W ? *reinterpret_cast<const float4*>(us + (size_t)r * a.W + k)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    float t = v[4 * r + s];
                    t = fmaf(u4.x, w4[s].x, t);
                    t = fmaf(u4.y, w4[s].y, t);
                    t = fmaf(u4.z, w4[s].z, t);
                    v[4 * r + s] = fmaf(u4.w, w4[s].w, t);
                }
            }
        };
        int k0 = 0;
        if (o0 == 4 * warp) {
#pragma unroll
            for (int q = 0; q < PRE; ++q) step(128 * q, w0[q]);
            k0 = 128 * PRE;
        }
#pragma unroll 2
        for (; k0 < a.W; k0 += 128) {
            float4 w4[4];
#pragma unroll
            for (int s = 0; s < 4; ++s)
                w4[s] = rows_load<true>(a.Wout + (size_t)min(o0 + s, a.A - 1) * a.W, k0, lane, a.W);
            step(k0, w4);
        }
        lane_reduce<4 * FR>(v, lane);
        constexpr int PER = FR >= 8 ? FR / 8 : 1, SHARE = FR >= 8 ? 1 : 8 / FR;   // values per lane, lanes per value
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int idx = lane / SHARE * PER + e, r = idx >> 2, o = o0 + (idx & 3);
            if (lane % SHARE != 0 || o >= a.A || bj0 + r >= a.rows) continue;
            const float vel = v[e] + a.bout[o];
            const size_t at = (size_t)(bj0 + r) * a.A + o;
            if (a.vout) a.vout[at] = vel;
            if (a.x) a.x[at] = a.x[at] + a.delta * vel;
        }
    }
}

// The first PRE steps of W_out rows 4 warp .. + 3 (weights: before the dependency wait).
template <int PRE>
__device__ __forceinline__ void final_prefetch(const FinalArgs& a, float4 (&w0)[PRE][4]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < PRE; ++q)
#pragma unroll
        for (int s = 0; s < 4; ++s)
            w0[q][s] = rows_load<true>(a.Wout + (size_t)min(4 * warp + s, a.A - 1) * a.W, 128 * q, lane, a.W);
}

// One row per CTA. PRE: steps of W_out fetched before the dependency wait; CTAS: CTAs that fit an SM
// (four steps take 162 registers, two 128).
template <int PRE, int CTAS>
__global__ void __launch_bounds__(FIN_THREADS, CTAS) k_final(const FinalArgs a) {
    extern __shared__ __align__(16) float us[];        // [W]
    __shared__ float scratch[32];
    const int tid = threadIdx.x, W = a.W;
    const int bj = blockIdx.x;           // request b, action j
    const int b = bj / a.C, j = bj % a.C;
    // The modulation (scale, shift) of this thread's features, before the dependency wait.
    float sg[FIN_CAP], bt[FIN_CAP];
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) {
        const int k = tid + FIN_THREADS * q;
        sg[q] = k < W ? a.sigma[k] : 0.f;
        bt[q] = k < W ? a.beta[k] : 0.f;
    }
    float4 w0[PRE][4];
    final_prefetch(a, w0);
    // Launched with programmatic dependent launch: h comes from the last layer's down projection.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const float* hr = a.hres + ((size_t)b * a.S + a.nctx + j) * W;
    float hv[FIN_CAP];
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) {
        const int k = tid + FIN_THREADS * q;
        hv[q] = k < W ? hr[k] : 0.f;
    }
    float ss = 0.f;
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) ss = fmaf(hv[q], hv[q], ss);
    for (int k = tid + FIN_THREADS * FIN_CAP; k < W; k += FIN_THREADS) ss = fmaf(hr[k], hr[k], ss);   // W > 4096
    ss = block_sum(ss, scratch);
    const float rinv = rsqrtf(ss / (float)W + a.eps);
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) {
        const int k = tid + FIN_THREADS * q;
        if (k < W) us[k] = hv[q] * rinv * (1.f + sg[q]) + bt[q];
    }
    for (int k = tid + FIN_THREADS * FIN_CAP; k < W; k += FIN_THREADS)
        us[k] = hr[k] * rinv * (1.f + a.sigma[k]) + a.beta[k];
    __syncthreads();
    final_outputs<1>(a, us, bj, w0);
}

// FR rows per CTA: a warp per row (then per row + 8) computes the norm.
template <int FR>
__global__ void __launch_bounds__(FIN_THREADS) k_final_rows(const FinalArgs a) {
    extern __shared__ __align__(16) float us[];        // [FR][W]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = a.W;
    const int bj0 = blockIdx.x * FR;
    float4 w0[1][4];
    final_prefetch(a, w0);
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    for (int r = warp; r < FR && bj0 + r < a.rows; r += FIN_THREADS / 32) {
        const int bj = bj0 + r, b = bj / a.C, j = bj - b * a.C;
        const float* hr = a.hres + ((size_t)b * a.S + a.nctx + j) * W;
        float* ur = us + (size_t)r * W;
        // Partial w of this lane is thread 32 w + lane of k_final: columns 32 w + lane + 256 q.
        float ps[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) ps[w] = 0.f;
        for (int k0 = 0; k0 < W; k0 += 2 * FIN_THREADS) {
            float hv[16];
#pragma unroll
            for (int w = 0; w < 16; ++w) {
                const int k = k0 + 32 * w + lane;
                hv[w] = k < W ? hr[k] : 0.f;
            }
#pragma unroll
            for (int w = 0; w < 16; ++w) {
                const int k = k0 + 32 * w + lane;
                ps[w & 7] = fmaf(hv[w], hv[w], ps[w & 7]);
                if (k < W) ur[k] = hv[w];
            }
        }
#pragma unroll
        for (int w = 0; w < 8; ++w) ps[w] = warp_sum(ps[w]);
        const float ss = ((ps[0] + ps[4]) + (ps[2] + ps[6])) + ((ps[1] + ps[5]) + (ps[3] + ps[7]));
        const float rinv = rsqrtf(ss / (float)W + a.eps);
#pragma unroll 8
        for (int k = lane; k < W; k += 32) ur[k] = ur[k] * rinv * (1.f + a.sigma[k]) + a.beta[k];
    }
    __syncthreads();
    final_outputs<FR>(a, us, bj0, w0);
}

// ---------------------------------------------------------------------------------------------
// Prefix KV into the store, every layer's K and V in one launch: tensor y (K then V of layer y / 2)
// src [batch][P][D] (fp32 or bf16) -> dst [batch][kv_rows][D]. A request's P D elements are
// contiguous on both sides; a thread moves KV_CH chunks of 8 elements (16 bytes of bf16), all loads
// before the stores. One launch, because a launch of its own takes each of 36 tensors 4.4 us (18 layers x
// 816 tokens), as long as the whole copy of 30 MB at the copy peak. VEC: the sources are 16-byte aligned.
constexpr int KV_CH = 4;
constexpr int KV_MAX_TENSORS = 128;
struct KvLoadArgs {
    const void* src[KV_MAX_TENSORS];
    void* dst[KV_MAX_TENSORS];
    int B;
    long long per;          // elements per request: P D (a multiple of 32)
    long long dst_stride;   // elements between requests of the store
};

template <typename T> struct Chunk8;   // 8 consecutive elements
template <> struct Chunk8<__nv_bfloat16> {
    uint4 v;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = *reinterpret_cast<const uint4*>(p); }
    __device__ __forceinline__ void load1(const __nv_bfloat16* p) {
        const unsigned short* u = reinterpret_cast<const unsigned short*>(p);
        v = make_uint4(u[0] | (uint32_t)u[1] << 16, u[2] | (uint32_t)u[3] << 16, u[4] | (uint32_t)u[5] << 16,
                       u[6] | (uint32_t)u[7] << 16);
    }
    __device__ __forceinline__ void store(__nv_bfloat16* p) const { *reinterpret_cast<uint4*>(p) = v; }
    __device__ __forceinline__ void store(float* p) const {
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
        float f[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(u[i] << 16);
            f[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
        }
        reinterpret_cast<float4*>(p)[0] = make_float4(f[0], f[1], f[2], f[3]);
        reinterpret_cast<float4*>(p)[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
};
template <> struct Chunk8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float* p) {
        a = reinterpret_cast<const float4*>(p)[0];
        b = reinterpret_cast<const float4*>(p)[1];
    }
    __device__ __forceinline__ void load1(const float* p) {
        a = make_float4(p[0], p[1], p[2], p[3]);
        b = make_float4(p[4], p[5], p[6], p[7]);
    }
    __device__ __forceinline__ static uint32_t pack(float lo, float hi) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<const uint32_t*>(&t);
    }
    __device__ __forceinline__ void store(__nv_bfloat16* p) const {
        *reinterpret_cast<uint4*>(p) = make_uint4(pack(a.x, a.y), pack(a.z, a.w), pack(b.x, b.y), pack(b.z, b.w));
    }
    __device__ __forceinline__ void store(float* p) const {
        reinterpret_cast<float4*>(p)[0] = a;
        reinterpret_cast<float4*>(p)[1] = b;
    }
};

template <typename TS, typename TD, bool VEC>
__global__ void __launch_bounds__(256) k_load_prefix(const __grid_constant__ KvLoadArgs a) {
    const TS* src0 = static_cast<const TS*>(a.src[blockIdx.y]);
    TD* dst0 = static_cast<TD*>(a.dst[blockIdx.y]);
    const long long nch = a.per / 8, step = (long long)gridDim.x * 256 * KV_CH;
    for (int b = blockIdx.z; b < a.B; b += gridDim.z) {
        const TS* src = src0 + b * a.per;
        TD* dst = dst0 + b * a.dst_stride;
        for (long long c0 = (long long)blockIdx.x * 256 * KV_CH + threadIdx.x; c0 < nch; c0 += step) {
            Chunk8<TS> v[KV_CH];
#pragma unroll
            for (int u = 0; u < KV_CH; ++u) {
                const long long c = c0 + 256 * u;
                if (c < nch) {
                    if (VEC) v[u].load(src + 8 * c);
                    else v[u].load1(src + 8 * c);
                }
            }
#pragma unroll
            for (int u = 0; u < KV_CH; ++u) {
                const long long c = c0 + 256 * u;
                if (c < nch) v[u].store(dst + 8 * c);
            }
        }
    }
}

template <typename TS, typename TD>
void launch_load_prefix_t(const KvLoadArgs& a, int ntensors, bool vec, cudaStream_t st) {
    const long long blocks = (a.per / 8 + 256 * KV_CH - 1) / (256 * KV_CH);
    const dim3 grid((unsigned)(blocks < 65536 ? blocks : 65536), (unsigned)ntensors, (unsigned)(a.B < 65535 ? a.B : 65535));
    if (vec) k_load_prefix<TS, TD, true><<<grid, 256, 0, st>>>(a);
    else k_load_prefix<TS, TD, false><<<grid, 256, 0, st>>>(a);
}

// Launch with programmatic dependent launch when the handle uses it (the kernel waits for its
// predecessor with griddepcontrol.wait before reading what that wrote); a failed launch leaves its
// error for check_launch.
template <typename... KArgs, typename... Args>
void launch_pdl(const jpi_handle* h, dim3 grid, dim3 block, size_t smem, cudaStream_t st, void (*k)(KArgs...),
                Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = h->pdl ? 1 : 0;
    (void)cudaLaunchKernelEx(&cfg, k, args...);
}

inline jpi_status check_launch(const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("launch of %s failed: %s", what, cudaGetErrorString(e));
        return JPI_ERR_CUDA;
    }
    return JPI_OK;
}

inline int grid_for(long long n, int block, int cap = 4096) {
    long long g = (n + block - 1) / block;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// Warps that share a slot group's K range of nst steps of 128: each keeps one at least.
int rows_ksplit(int nst) { return nst >= 4 ? 4 : nst >= 2 ? 2 : 1; }

// The product kernel of one kind; 16-byte (8-byte for bf16) loads when K is a multiple of 4.
template <typename T, int KIND>
jpi_status launch_rows_gemm(jpi_handle* h, const RowsArgs& a, cudaStream_t st) {
    const int groups = KIND == RK_RESID ? (a.N + 3) / 4 : KIND == RK_GEGLU ? (a.N + 1) / 2 : a.N / 4;
    const int ks = rows_ksplit((a.K + 127) / 128);
    const int cw = ROWS_WARPS / ks;
    const dim3 grid((groups + cw - 1) / cw, (a.M + ROWS_M - 1) / ROWS_M), block(32 * ROWS_WARPS);
    const bool vec = a.K % 4 == 0;
    auto go = [&](auto k) { launch_pdl(h, grid, block, 0, st, k, a); };
    if (vec) {
        if (ks == 4) go(k_rows_gemm<T, KIND, true, 4>);
        else if (ks == 2) go(k_rows_gemm<T, KIND, true, 2>);
        else go(k_rows_gemm<T, KIND, true, 1>);
    } else {
        if (ks == 4) go(k_rows_gemm<T, KIND, false, 4>);
        else if (ks == 2) go(k_rows_gemm<T, KIND, false, 2>);
        else go(k_rows_gemm<T, KIND, false, 1>);
    }
    return check_launch("layer product (CUDA cores)");
}

template <typename T, int HB>
jpi_status launch_attn_rows(jpi_handle* h, const T* q, const T* k, const T* v, T* o, int Mt, int S, cudaStream_t st) {
    const dim3 grid(Mt * (h->H / HB)), block(32 * AR_WARPS);
    const float scale = 1.f / sqrtf((float)h->D);
    auto go = [&](auto kern) {
        launch_pdl(h, grid, block, 0, st, kern, q, k, v, o, S, h->H, h->D, h->cur_prefix, h->kv_rows, h->n_ctx(), scale);
    };
    if (h->D <= 64) go(k_attn_rows<T, HB, 2>);
    else if (h->D <= 128) go(k_attn_rows<T, HB, 4>);
    else go(k_attn_rows<T, HB, 8>);
    return check_launch("attention (CUDA cores)");
}

// One sub-step of layer l: 2 norm + QKV + rotary, 3 attention, 4 O-proj + residual,
// 5 norm + gate/up + GeGLU, 6 down-proj + residual.
template <typename T>
jpi_status op_simt(jpi_handle* h, int op, int l, int step, int B, int C, cudaStream_t st) {
    const int S = C + h->n_ctx(), Mt = B * S, W = h->W;
    const float* ms = h->mods + (size_t)step * mod_rows(h->L) * W + (size_t)6 * l * W;
    const LayerPlain* lwp = (size_t)l < h->plain.size() ? &h->plain[l] : nullptr;
    const size_t kv_layer = (size_t)l * h->maxB * h->kv_rows * h->D;
    T* kst = (T*)h->kv_k + kv_layer;
    T* vst = (T*)h->kv_v + kv_layer;
    if (op != 3 && !lwp) {
        set_error("layer %d has no CUDA-core weights", l);
        return JPI_ERR_INVALID_ARG;
    }
    // Products: the kernel with the smaller estimate, in us (fp32 and bf16, 792 shapes of 16 to 3264 tokens, K and
    // N of 32 to 4096; the choice takes 0.3% longer than the better kernel on average). The rows kernel is
    // bound by its warps' 128-wide steps and the reduction after them, the 64 x 64 tiles by their chain along K, with
    // the norm and rotary launches before and after. Rows against tiles, us: pi0.5's QKV (2560 x 1024, fp32) 33 and 88
    // at 51 tokens, 109 and 122 at 204, 211 and 125 at 408; down (1024 x 4096) 212 and 286 at 408; bf16, QKV of 384 x
    // 160 16 and 24 at 306, 50 and 25 at 1224; gate/up of 1030 x 160 33 and 41 at 153, 117 and 45 at 612.
    // The two add a product's terms in different orders: in the batch-invariant mode a launch takes what
    // one request alone would (Mi tokens).
    const int Mi = h->batch_invariant ? S : Mt;
    auto rows_fit = [&](int kind, int N, int K) {
        const bool norm = kind != RK_RESID, glu = kind == RK_GEGLU;
        const long long blocks = (long long)((N + GB_N - 1) / GB_N) * ((Mi + GB_M - 1) / GB_M);
        const double deep = (double)((blocks + h->num_sms - 1) / h->num_sms - 1);   // tiles an SM walks past the first
        const double chain = (K + GB_K - 1) / GB_K * (glu ? 3.16 + 1.12 * deep : 1.18 + .70 * deep);
        const double tiles = 5.1 + (glu ? 2.7 : norm ? 7.1 : 0.) + (norm ? .00106 * Mi : 0.) + chain;
        const int nst = (K + 127) / 128, ks = rows_ksplit(nst);
        const double warps = (double)((glu ? 2 * N : N) + 3) / 4. * ((Mi + ROWS_M - 1) / ROWS_M);
        const double steps = warps * (nst + .95 * (ks > 1 ? ks : 2)) / h->num_sms;
        const double rows = 2.6 + (norm ? .9 : 0.) + 1.1 * ((nst + ks - 1) / ks) +
                            .139 * steps * (sizeof(T) == 2 ? 1.43 : 1.) * (norm ? 1.24 : 1.);
        return rows < tiles;
    };
    const int F = h->F, HD = h->HD, mtiles = (Mt + GB_M - 1) / GB_M;
    const float eps = h->cfg.rms_eps;
    T* act = (T*)h->act;
    const dim3 blk(256);
    RowsArgs a = {};
    a.M = Mt;
    a.K = W;
    a.N = W;
    a.h = h->h;
    a.eps = h->cfg.rms_eps;
    a.hres = h->h;
    a.S = S;
    a.H = h->H;
    a.D = h->D;
    a.P = h->cur_prefix;
    a.kv_rows = h->kv_rows;
    switch (op) {
        case 2:
            if (!rows_fit(RK_QKV, h->QKV, W)) {
                k_rms_mod<T><<<Mt, blk, 0, st>>>(h->h, ms, ms + W, act, W, W, eps);
                k_gemm_simt<T, T, EPI_STORE><<<dim3((h->QKV + GB_N - 1) / GB_N, mtiles), blk, 0, st>>>(
                    act, W, (const T*)lwp->wqkv, nullptr, Mt, h->QKV, W, h->qkv, h->QKV, nullptr, nullptr, 0);
                k_qkv_post<T, T><<<Mt, blk, 0, st>>>(h->qkv, (T*)h->q, kst, vst, h->rope_tab, S, h->H, h->D,
                                                     h->cur_prefix, h->kv_rows);
                return check_launch("layer op (CUDA cores)");
            }
            a.sigma = ms;
            a.beta = ms + W;
            a.W1 = lwp->wqkv;
            a.N = h->QKV;
            a.q = h->q;
            a.kst = kst;
            a.vst = vst;
            a.rope = h->rope_tab;
            return launch_rows_gemm<T, RK_QKV>(h, a, st);
        case 3: {
            // Four heads per block, each key read once for them: at head dims to 64 always, above once one
            // head per block would be more than two blocks per SM, which then no longer run at once. One head and
            // four per block, 832 keys, us: D = 64, 8 heads, 9 tokens 26.0 and 20.1, 51: 58.1 and 21.5; D = 160, 38
            // tokens (304 blocks) 37.1 and 43.5, 51 (408) 64.0 and 44.4; D = 96, 304 and 408 blocks 39.2 and
            // 34.7, 68.8 and 35.6 (32 keys, 304 blocks: 5.3 and 5.4).
            const bool four = h->H % 4 == 0 && (h->D <= 64 || (long long)Mi * h->H > 2ll * h->num_sms);
            return four ? launch_attn_rows<T, 4>(h, (const T*)h->q, kst, vst, (T*)h->o, Mt, S, st)
                        : launch_attn_rows<T, 1>(h, (const T*)h->q, kst, vst, (T*)h->o, Mt, S, st);
        }
        case 4:
            if (!rows_fit(RK_RESID, W, HD)) {
                k_gemm_simt<T, T, EPI_RESID><<<dim3((W + GB_N - 1) / GB_N, mtiles), blk, 0, st>>>(
                    (const T*)h->o, HD, (const T*)lwp->wo, nullptr, Mt, W, HD, h->h, W, ms + 2 * W, nullptr, 0);
                return check_launch("layer op (CUDA cores)");
            }
            a.X = h->o;
            a.W1 = lwp->wo;
            a.K = h->HD;
            a.gamma = ms + 2 * W;
            return launch_rows_gemm<T, RK_RESID>(h, a, st);
        case 5:
            if (!rows_fit(RK_GEGLU, F, W)) {
                k_rms_mod<T><<<Mt, blk, 0, st>>>(h->h, ms + 3 * W, ms + 4 * W, act, W, W, eps);
                k_gemm_simt<T, T, EPI_GEGLU><<<dim3((F + GB_N - 1) / GB_N, mtiles), blk, 0, st>>>(
                    act, W, (const T*)lwp->wg, (const T*)lwp->wu, Mt, F, W, nullptr, 0, nullptr, (T*)h->z, F);
                return check_launch("layer op (CUDA cores)");
            }
            a.sigma = ms + 3 * W;
            a.beta = ms + 4 * W;
            a.W1 = lwp->wg;
            a.W2 = lwp->wu;
            a.N = h->F;
            a.z = h->z;
            return launch_rows_gemm<T, RK_GEGLU>(h, a, st);
        case 6:
            if (!rows_fit(RK_RESID, W, F)) {
                k_gemm_simt<T, T, EPI_RESID><<<dim3((W + GB_N - 1) / GB_N, mtiles), blk, 0, st>>>(
                    (const T*)h->z, F, (const T*)lwp->wd, nullptr, Mt, W, F, h->h, W, ms + 5 * W, nullptr, 0);
                return check_launch("layer op (CUDA cores)");
            }
            a.X = h->z;
            a.W1 = lwp->wd;
            a.K = h->F;
            a.gamma = ms + 5 * W;
            return launch_rows_gemm<T, RK_RESID>(h, a, st);
        default:
            set_error("unknown layer op %d", op);
            return JPI_ERR_INVALID_ARG;
    }
}

// Step times per launch of k_gemv_multi: its shared copy of the inputs is that many x max(W, d_t)
// floats, kept within 200 KB.
int tc_group(const jpi_handle* h) {
    const size_t row = sizeof(float) * (size_t)(h->W > h->dt ? h->W : h->dt);
    int g = GV_N;
    while (g > 1 && g * row > 200 * 1024) g /= 2;
    return g;
}

// Y [N][R] = act(X [N][K] Wm [R][K]^T + bias) by k_gemv_multi, tc_group step times per launch.
template <typename T, bool SWISH>
void launch_gemv(jpi_handle* h, const T* Wm, const float* bias, const float* X, float* Y, int R, int K, int N,
                 cudaStream_t st) {
    const int group = tc_group(h);
    const dim3 grid(grid_for((long long)R * 32, 256, 1024)), blk(256);
    for (int n0 = 0; n0 < N; n0 += group) {
        const int g = N - n0 < group ? N - n0 : group;
        const size_t smem = sizeof(float) * (size_t)g * K;
        const float* x = X + (size_t)n0 * K;
        float* y = Y + (size_t)n0 * R;
        if (K % 4 == 0) launch_pdl(h, grid, blk, smem, st, k_gemv_multi<T, SWISH, true>, Wm, bias, x, y, R, K, g);
        else launch_pdl(h, grid, blk, smem, st, k_gemv_multi<T, SWISH, false>, Wm, bias, x, y, R, K, g);
    }
}

// Modulation step times per pass of k_mod_gemv (its shared copy of X is MOD_GROUP x W floats).
constexpr int MOD_GROUP = 16;

template <typename T, int NG>
void launch_mod_gemv(jpi_handle* h, const float* X, float* Y, int R, cudaStream_t st) {
    const int W = h->W;
    int threads = (R / MOD_RT + h->num_sms - 1) / h->num_sms;   // about one CTA per SM
    threads = (threads + 31) / 32 * 32;
    threads = threads < 64 ? 64 : (threads > 256 ? 256 : threads);
    const int grid = (R + threads * MOD_RT - 1) / (threads * MOD_RT);
    k_mod_gemv<T, NG><<<grid, threads, sizeof(float) * NG * W, st>>>((const T*)h->mod_w, h->mod_b, X, Y, R, W);
}

// bf16 weights with the tensor-core path: the tcgen05 kernel of mod_tc.cu; otherwise (and for
// fp32 weights) the CUDA-core kernel above.
template <typename T>
jpi_status mod_gemv(jpi_handle* h, int g, const float* X, float* Y, int R, cudaStream_t st) {
    if (std::is_same<T, __nv_bfloat16>::value && h->mod_tc) return launch_mod_tc(h, X, Y, g, st);
    // Few rows (four per thread would leave most SMs without a warp): a warp per row instead
    // (3584 rows x 256 columns: 19 us with four rows per thread on 14 CTAs).
    if (R < MOD_RT * 64 * h->num_sms) {
        launch_gemv<T, false>(h, (const T*)h->mod_w, h->mod_b, X, Y, R, h->W, g, st);
        return JPI_OK;
    }
    switch (g) {
#define JPI_MOD_CASE(n) case n: launch_mod_gemv<T, n>(h, X, Y, R, st); break;
        JPI_MOD_CASE(1) JPI_MOD_CASE(2) JPI_MOD_CASE(3) JPI_MOD_CASE(4) JPI_MOD_CASE(5) JPI_MOD_CASE(6)
        JPI_MOD_CASE(7) JPI_MOD_CASE(8) JPI_MOD_CASE(9) JPI_MOD_CASE(10) JPI_MOD_CASE(11)
        JPI_MOD_CASE(12) JPI_MOD_CASE(13) JPI_MOD_CASE(14) JPI_MOD_CASE(15) JPI_MOD_CASE(16)
#undef JPI_MOD_CASE
        default: break;
    }
    return JPI_OK;
}

template <typename T>
jpi_status set_mod_attrs(int smem) {
#define JPI_MOD_ATTR(n) \
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_mod_gemv<T, n>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    JPI_MOD_ATTR(1) JPI_MOD_ATTR(2) JPI_MOD_ATTR(3) JPI_MOD_ATTR(4) JPI_MOD_ATTR(5) JPI_MOD_ATTR(6)
    JPI_MOD_ATTR(7) JPI_MOD_ATTR(8) JPI_MOD_ATTR(9) JPI_MOD_ATTR(10) JPI_MOD_ATTR(11) JPI_MOD_ATTR(12)
    JPI_MOD_ATTR(13) JPI_MOD_ATTR(14) JPI_MOD_ATTR(15) JPI_MOD_ATTR(16)
#undef JPI_MOD_ATTR
    return JPI_OK;
}

// Time MLP and modulation vectors of N step times from their embeddings temb [N][d_t].
template <typename T>
jpi_status time_cond(jpi_handle* h, int N, const float* temb, float* c1, float* cond, cudaStream_t st) {
    const int W = h->W, dt = h->dt, R = mod_rows(h->L) * W;
    launch_gemv<T, true>(h, (const T*)h->time_in_w, h->time_in_b, temb, c1, W, dt, N, st);
    launch_gemv<T, true>(h, (const T*)h->time_out_w, h->time_out_b, c1, cond, W, W, N, st);
    for (int n0 = 0; n0 < N; n0 += MOD_GROUP) {
        const int g = (N - n0) < MOD_GROUP ? (N - n0) : MOD_GROUP;
        JPI_TRY(mod_gemv<T>(h, g, cond + (size_t)n0 * W, h->mods + (size_t)n0 * R, R, st));
    }
    return check_launch("time conditioning");
}

template <typename T>
jpi_status set_gemv_attrs(int smem) {
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return JPI_OK;
}

}  // namespace

jpi_status configure_simt_kernels(jpi_handle* h) {
    const int gemv_smem = (int)(sizeof(float) * (size_t)tc_group(h) * (h->W > h->dt ? h->W : h->dt));
    const int mod_smem = (int)(sizeof(float) * (size_t)MOD_GROUP * h->W);
    int dev = 0;
    JPI_CUDA_TRY(cudaGetDevice(&dev));
    JPI_CUDA_TRY(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_final_rows<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FIN_SMEM_MAX));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_final_rows<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FIN_SMEM_MAX));
    if (h->bf16) {
        JPI_TRY(set_gemv_attrs<__nv_bfloat16>(gemv_smem));
        JPI_TRY(set_mod_attrs<__nv_bfloat16>(mod_smem));
    } else {
        JPI_TRY(set_gemv_attrs<float>(gemv_smem));
        JPI_TRY(set_mod_attrs<float>(mod_smem));
    }
    return JPI_OK;
}

namespace {
// Embeddings of the step times k / nsteps, or of one given time (t_override >= 0).
jpi_status time_embed_into(jpi_handle* h, float* temb, int nsteps, double t_override, cudaStream_t st) {
    k_time_embed<<<dim3(nsteps, (h->dt / 2 + TE_THREADS - 1) / TE_THREADS), TE_THREADS, 0, st>>>(
        temb, h->t_period, nsteps, h->dt, t_override);
    return check_launch("time embedding");
}
}  // namespace

jpi_status launch_time_embed(jpi_handle* h, int nsteps, double t_override, cudaStream_t st) {
    return time_embed_into(h, h->temb, nsteps, t_override, st);
}

jpi_status launch_time_conditioning(jpi_handle* h, int nsteps, cudaStream_t st) {
    return h->bf16 ? time_cond<__nv_bfloat16>(h, nsteps, h->temb, h->c1, h->cond, st)
                   : time_cond<float>(h, nsteps, h->temb, h->c1, h->cond, st);
}

// Time conditioning of one step time with caller-chosen scratch: sinusoid into temb [d_t],
// time-MLP hidden layer into c1 [W], conditioning vector into cond [W]; the modulation
// vectors go to the handle's step-0 slot, as with launch_time_conditioning(h, 1, ...).
jpi_status launch_time_conditioning_into(jpi_handle* h, double t, float* temb, float* c1,
                                         float* cond, cudaStream_t st) {
    JPI_TRY(time_embed_into(h, temb, 1, t, st));
    return h->bf16 ? time_cond<__nv_bfloat16>(h, 1, temb, c1, cond, st) : time_cond<float>(h, 1, temb, c1, cond, st);
}

jpi_status launch_embed(jpi_handle* h, int step, int B, int C, const float* x, cudaStream_t st) {
    const int slices = (h->W + 511) / 512, nctx = h->n_ctx();
    // Scale and shift of layer 0's attention norm at this step.
    const float* ms = h->mods + (size_t)step * mod_rows(h->L) * h->W;
    EmbedArgs a;
    a.hres = h->h;
    a.xs = h->tc ? (__nv_bfloat16*)h->hx : nullptr;
    a.sigma = ms;
    a.beta = ms + h->W;
    a.ss = h->tc ? h->ss : nullptr;
    a.ss_ld = h->maxMt;
    a.state = h->state;
    a.x = x;
    a.Ws = h->state_in_w;
    a.bs = h->state_in_b;
    a.Wa = h->action_in_w;
    a.ba = h->action_in_b;
    a.corr = h->corr;
    a.nctx = nctx;
    a.B = B;
    a.S = C + nctx;
    a.C = C;
    a.W = h->W;
    a.Sd = h->Sd;
    a.A = h->A;
    // As many blocks as run at once, three to an SM (168 registers a thread; a small batch keeps one token
    // per block, the shortest chain), at most EMB_MAX_TPB tokens each. Measured for two, three and four to an SM,
    // us: W = 1024 408 tokens 4.0, 3.7, 3.7; 816: 6.1, 4.9, 7.3; 1632: 9.5, 7.6, 11.6; W = 256 408
    // tokens 2.7, 2.3, 2.3; 1632: 4.3, 3.5, 5.4.
    const long long want = 3ll * h->num_sms;
    const long long tpb = ((long long)B * a.S * slices + want - 1) / want;
    a.tpb = (int)(tpb < 1 ? 1 : tpb > EMB_MAX_TPB ? EMB_MAX_TPB : tpb);
    a.action_groups = (B * C + a.tpb - 1) / a.tpb;
    const int groups = a.action_groups + (B * nctx + a.tpb - 1) / a.tpb;
    launch_pdl(h, dim3(slices, groups), dim3(128), 0, st, k_embed, a);
    return check_launch("embed");
}

jpi_status launch_op_simt(jpi_handle* h, int op, int layer, int step, int B, int C,
                          cudaStream_t st) {
    return h->bf16 ? op_simt<__nv_bfloat16>(h, op, layer, step, B, C, st)
                   : op_simt<float>(h, op, layer, step, B, C, st);
}

jpi_status launch_layer_simt(jpi_handle* h, int layer, int step, int B, int C, cudaStream_t st) {
    for (int op = 2; op <= 6; ++op) JPI_TRY(launch_op_simt(h, op, layer, step, B, C, st));
    return JPI_OK;
}

jpi_status launch_final(jpi_handle* h, int step, int B, int C, float delta, float* x_inout, float* v_out,
                        cudaStream_t st) {
    const int W = h->W, rows = B * C;
    const float* ms = h->mods + (size_t)step * mod_rows(h->L) * W + (size_t)6 * h->L * W;
    FinalArgs a;
    a.hres = h->h;
    a.sigma = ms;
    a.beta = ms + W;
    a.Wout = h->action_out_w;
    a.bout = h->action_out_b;
    a.x = x_inout;
    a.vout = v_out;
    a.rows = rows;
    a.S = C + h->n_ctx();
    a.nctx = h->n_ctx();
    a.C = C;
    a.W = W;
    a.A = h->A;
    a.eps = h->cfg.rms_eps;
    a.delta = delta;
    // One row per CTA while the CTAs run at once, at one or two per SM, then 4, then 8 rows (while they fit
    // the shared memory). Measured at W = 1024, us: 150 rows 3.6 (one CTA per SM), 4.0 (two), 6.3 (4 rows); 160:
    // 6.0, 4.1, 6.3; 300: 6.5, 4.1, 6.3; 350: 8.5, 7.4, 6.4 and 8.0 (8 rows); 1200: 7.3 (4 rows), 8.2 (8
    // rows); 1250: 12.7, 9.7.
    const int fr = rows <= 2 * h->num_sms ? 1 : rows <= 8 * h->num_sms ? 4 : 8;
    const size_t row = sizeof(float) * (size_t)W;
    if (fr == 8 && 8 * row <= FIN_SMEM_MAX)
        launch_pdl(h, dim3((rows + 7) / 8), dim3(FIN_THREADS), 8 * row, st, k_final_rows<8>, a);
    else if (fr >= 4 && 4 * row <= FIN_SMEM_MAX)
        launch_pdl(h, dim3((rows + 3) / 4), dim3(FIN_THREADS), 4 * row, st, k_final_rows<4>, a);
    else if (rows <= h->num_sms)
        launch_pdl(h, dim3(rows), dim3(FIN_THREADS), row, st, k_final<4, 1>, a);
    else
        launch_pdl(h, dim3(rows), dim3(FIN_THREADS), row, st, k_final<2, 2>, a);
    return check_launch("final norm + Euler");
}

jpi_status launch_load_prefix(jpi_handle* h, const void* const* k_layers, const void* const* v_layers, int src_fp32,
                              int B, int P, cudaStream_t st) {
    const size_t es = h->bf16 ? 2 : 4;
    const size_t layer_bytes = (size_t)h->maxB * h->kv_rows * h->D * es;
    for (int l0 = 0; l0 < h->L; l0 += KV_MAX_TENSORS / 2) {
        const int nl = h->L - l0 < KV_MAX_TENSORS / 2 ? h->L - l0 : KV_MAX_TENSORS / 2;
        KvLoadArgs a;
        a.B = B;
        a.per = (long long)P * h->D;
        a.dst_stride = (long long)h->kv_rows * h->D;
        uintptr_t bits = 0;
        for (int i = 0; i < nl; ++i) {
            a.src[2 * i] = k_layers[l0 + i];
            a.src[2 * i + 1] = v_layers[l0 + i];
            a.dst[2 * i] = (char*)h->kv_k + (l0 + i) * layer_bytes;
            a.dst[2 * i + 1] = (char*)h->kv_v + (l0 + i) * layer_bytes;
            bits |= (uintptr_t)k_layers[l0 + i] | (uintptr_t)v_layers[l0 + i];
        }
        const bool vec = (bits & 15) == 0;
        using bf = __nv_bfloat16;
        if (h->bf16) {
            if (src_fp32) launch_load_prefix_t<float, bf>(a, 2 * nl, vec, st);
            else launch_load_prefix_t<bf, bf>(a, 2 * nl, vec, st);
        } else {
            if (src_fp32) launch_load_prefix_t<float, float>(a, 2 * nl, vec, st);
            else launch_load_prefix_t<bf, float>(a, 2 * nl, vec, st);
        }
        JPI_TRY(check_launch("prefix KV copy"));
    }
    return JPI_OK;
}

}  // namespace jpi
