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

// ---------------------------------------------------------------------------------------------
// Time conditioning: flow time enters the expert only through a sinusoidal embedding followed
// by a two-layer swish MLP; the per-layer modulation vectors are a linear map of the result.
// All of it depends on t alone, so it is evaluated once per call for every step time.

// Grid (steps, ceil(half / blockDim)): one frequency i of one step time per thread (the fp64
// pow/sin/cos are slow on this GPU; spread over the grid they run side by side).
__global__ void k_time_embed(float* temb, int nsteps, int dt, double pmin, double pmax,
                             double t_override) {
    const int k = blockIdx.x;
    const double t = t_override >= 0.0 ? t_override : (double)k / (double)nsteps;
    const int half = dt / 2;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < half; i += gridDim.y * blockDim.x) {
        const double frac = (double)i / (double)(half - 1);
        const double period = pmin * pow(pmax / pmin, frac);
        const double theta = 2.0 * 3.14159265358979323846 * t / period;
        temb[(size_t)k * dt + i] = (float)sin(theta);
        temb[(size_t)k * dt + half + i] = (float)cos(theta);
    }
}

// Y[n][r] = act(sum_k W[r][k] X[n][k] + b[r]) for n < N (<= 8 per pass), r < R.
// One warp per output row; X lives in shared memory.
template <typename TW, bool SWISH>
__global__ void k_gemv_multi(const TW* __restrict__ Wm, const float* __restrict__ bias,
                             const float* __restrict__ X, float* __restrict__ Y, int R, int K,
                             int N) {
    extern __shared__ float xs[];
    // Eight loads of each thread in flight before their stores (one at a time, every store would
    // hold the next load back for a full round trip).
    for (int i0 = threadIdx.x; i0 < N * K; i0 += 8 * blockDim.x) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * blockDim.x;
            v[u] = i < N * K ? X[i] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < N * K) xs[i] = v[u];
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = warp; r < R; r += nwarps) {
        const TW* wr = Wm + (size_t)r * K;
        for (int n0 = 0; n0 < N; n0 += 8) {
            float acc[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = 0.f;
            // Eight weights of the row loaded together, then their products in k order.
            for (int k0 = lane; k0 < K; k0 += 32 * 8) {
                float wv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = k0 + 32 * u;
                    wv[u] = k < K ? ldf(wr + k) : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = k0 + 32 * u;
                    if (k < K) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (n0 + j < N) acc[j] = fmaf(wv[u], xs[(n0 + j) * K + k], acc[j]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float s = warp_sum(acc[j]);
                if (lane == 0 && n0 + j < N) {
                    const float y = s + bias[r];
                    Y[(size_t)(n0 + j) * R + r] = SWISH ? swishf(y) : y;
                }
            }
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
// Block = 128 features of up to TPB tokens that share one input matrix: blockIdx.y counts groups of
// action tokens first, then groups of state and context tokens. A thread keeps its feature's weight
// row in registers for all of them (its 128 bytes are a line of their own, so with one token per
// block every token fetched 16 KB of weights per 128 features again: 382 us at 3264 tokens x 1024
// features, bound by those reads; the outputs alone are 20 MB, 3 us) and reads the tokens' inputs
// from shared memory as broadcasts. The sums keep the order of one token at a time.
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

__global__ void __launch_bounds__(128) k_embed(const EmbedArgs a) {
    __shared__ __align__(16) float in_s[EMB_MAX_TPB][EMB_K];
    __shared__ float part[EMB_MAX_TPB][4];
    const int tid = threadIdx.x;
    const bool act = (int)blockIdx.y < a.action_groups;
    // Tokens [j0, j0 + nt) of this block's kind: action token j = (request j / C, action j mod C),
    // else context token j = (request j / nctx, row j mod nctx).
    const int per = act ? a.C : a.nctx;
    const int j0 = (act ? blockIdx.y : blockIdx.y - a.action_groups) * a.tpb;
    const int nt = min(a.tpb, a.B * per - j0);
    const int K = act ? a.A : a.Sd;
    const int Kr = min(K, EMB_K);
    const float* Wm = act ? a.Wa : a.Ws;
    const int n = blockIdx.x * 128 + tid;
    const bool live = n < a.W;
    // Everything but x (the previous step's actions) is ready before the dependency wait.
    float wv[EMB_K];
    float bv = 0.f, sg = 0.f, bt = 0.f;
    if (live) {
        const float* wr = Wm + (size_t)n * K;
        if (K % 4 == 0) {
#pragma unroll
            for (int k = 0; k < EMB_K; k += 4) {
                const float4 w4 = k < K ? __ldg(reinterpret_cast<const float4*>(wr + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
                wv[k] = w4.x;
                wv[k + 1] = w4.y;
                wv[k + 2] = w4.z;
                wv[k + 3] = w4.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < EMB_K; ++k) wv[k] = k < K ? wr[k] : 0.f;
        }
        bv = (act ? a.ba : a.bs)[n];
        if (a.xs) {
            sg = a.sigma[n];
            bt = a.beta[n];
        }
    }
    // Launched with programmatic dependent launch: x comes from the previous step's final kernel;
    // the next kernel may start its weight prefetch at once.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    // Inputs of token j: its action row, or its request's state (context rows past 0 have none).
    auto input = [&](int j) { return act ? a.x + (size_t)j * a.A : a.state + (size_t)(j / a.nctx) * a.Sd; };
    for (int i = tid; i < nt * EMB_K; i += 128) {
        const int tt = i / EMB_K, k = i % EMB_K;
        in_s[tt][k] = k < Kr ? input(j0 + tt)[k] : 0.f;
    }
    __syncthreads();
    for (int tt = 0; tt < nt; ++tt) {
        const int j = j0 + tt;
        const int b = j / per, i = (act ? a.nctx : 0) + j - b * per;   // request, row in its suffix
        const int m = b * a.S + i;
        float v = 0.f;
        if (live) {
            if (!act && i > 0) {
                v = a.corr[((size_t)b * (a.nctx - 1) + (i - 1)) * a.W + n];
            } else {
                float acc = 0.f;
                const float4* iv = reinterpret_cast<const float4*>(in_s[tt]);
#pragma unroll
                for (int k = 0; k < EMB_K; k += 4) {
                    const float4 x4 = iv[k / 4];
                    if (k < K) acc = fmaf(wv[k], x4.x, acc);
                    if (k + 1 < K) acc = fmaf(wv[k + 1], x4.y, acc);
                    if (k + 2 < K) acc = fmaf(wv[k + 2], x4.z, acc);
                    if (k + 3 < K) acc = fmaf(wv[k + 3], x4.w, acc);
                }
                const float* in = input(j);
                for (int k = EMB_K; k < K; ++k) acc = fmaf(Wm[(size_t)n * K + k], in[k], acc);
                v = acc + bv;
            }
            a.hres[(size_t)m * a.W + n] = v;
            if (a.xs) a.xs[(size_t)xs_row(m) * a.W + n] = __float2bfloat16_rn((1.f + sg) * v);
        }
        if (a.ss) {
            const float t = warp_sum(v * v);
            if ((tid & 31) == 0) part[tt][tid >> 5] = t;
        }
    }
    if (a.xs && live) {
        // Tile z's beta row: block y takes tiles y tpb .. (the blocks' token slots cover the tiles).
        const int z0 = blockIdx.y * a.tpb, z1 = min(z0 + a.tpb, xs_tiles(a.B * a.S));
        for (int z = z0; z < z1; ++z) a.xs[((size_t)z * 64 + 63) * a.W + n] = __float2bfloat16_rn(bt);
    }
    if (a.ss) {
        __syncthreads();
        if (tid < nt) {
            const int j = j0 + tid, b = j / per, i = (act ? a.nctx : 0) + j - b * per;
            a.ss[(size_t)blockIdx.x * a.ss_ld + b * a.S + i] =
                (part[tid][0] + part[tid][2]) + (part[tid][1] + part[tid][3]);
        }
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

// Four consecutive elements (k a multiple of 4, rows 4-element aligned), or with VEC false four
// elements 32 apart per lane (any K), zero past K. kidx(lane) says which k they are.
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
// Products with many tokens (see rows_fit below): Y[m][n] = sum_k X[m][k] W[n][k] with three epilogues:
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
// once for four heads; HB = 1 spreads a small batch over four times the blocks. Measured against a
// block per token with a warp per head and the keys staged 32 at a time: a 9-token request
// 29 -> 6 us; 408 tokens x 8 heads x 867 keys (D = 256) 456 -> 278 us.
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
// One CTA of FIN_THREADS per action row. The row's values (FIN_CAP per thread at most, all loads
// in flight together) give the norm; the normalised row goes to shared memory; then thread t
// takes output a0 + t / 8 over the 16-byte column chunks t mod 8, t mod 8 + 8, .. (a group of 8
// threads reads 128 contiguous bytes per step) and the group adds its 8 partial sums.
constexpr int FIN_THREADS = 256;
constexpr int FIN_CAP = 16;   // W <= 4096
__global__ void __launch_bounds__(FIN_THREADS) k_final(const float* __restrict__ hres, const float* __restrict__ sigma,
                        const float* __restrict__ beta, const float* __restrict__ Wout,
                        const float* __restrict__ bout, float* __restrict__ x,
                        float* __restrict__ vout, float* __restrict__ outcopy, int S, int nctx, int C,
                        int W, int A, float eps, float delta) {
    extern __shared__ float us[];        // [W]
    __shared__ float scratch[32];
    const int tid = threadIdx.x;
    const int bj = blockIdx.x;           // request b, action j
    const int b = bj / C, j = bj % C;
    // The modulation (scale, shift) of this thread's features, before the dependency wait.
    float sg[FIN_CAP], bt[FIN_CAP];
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) {
        const int k = tid + FIN_THREADS * q;
        sg[q] = k < W ? sigma[k] : 0.f;
        bt[q] = k < W ? beta[k] : 0.f;
    }
    // Launched with programmatic dependent launch: h comes from the last layer's down projection.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const float* hr = hres + ((size_t)b * S + nctx + j) * W;
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
    const float rinv = rsqrtf(ss / (float)W + eps);
#pragma unroll
    for (int q = 0; q < FIN_CAP; ++q) {
        const int k = tid + FIN_THREADS * q;
        if (k < W) us[k] = hv[q] * rinv * (1.f + sg[q]) + bt[q];
    }
    for (int k = tid + FIN_THREADS * FIN_CAP; k < W; k += FIN_THREADS)
        us[k] = hr[k] * rinv * (1.f + sigma[k]) + beta[k];
    __syncthreads();
    const int ks = tid & 7;
    const int n4 = W >> 2;   // W is a multiple of 32 (checked at create)
    const float4* us4 = reinterpret_cast<const float4*>(us);
    for (int a0 = 0; a0 < A; a0 += FIN_THREADS / 8) {
        const int a = a0 + (tid >> 3);
        float acc = 0.f;
        if (a < A) {
            const float4* wr = reinterpret_cast<const float4*>(Wout + (size_t)a * W);
#pragma unroll 8
            for (int c = ks; c < n4; c += 8) {
                const float4 w4 = __ldg(wr + c), u4 = us4[c];
                acc = fmaf(u4.x, w4.x, fmaf(u4.y, w4.y, fmaf(u4.z, w4.z, fmaf(u4.w, w4.w, acc))));
            }
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        acc += __shfl_xor_sync(0xffffffffu, acc, 4);
        if (ks == 0 && a < A) {
            const float v = acc + bout[a];
            const size_t idx = (size_t)bj * A + a;
            if (vout) vout[idx] = v;
            if (x) {
                const float xn = x[idx] + delta * v;
                x[idx] = xn;
                if (outcopy) outcopy[idx] = xn;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Prefix KV into the store, every layer's K and V in one launch: tensor y (K then V of layer y / 2)
// src [batch][P][D] (fp32 or bf16) -> dst [batch][kv_rows][D]. A request's P D elements are
// contiguous on both sides; a thread moves KV_CH chunks of 8 elements (16 bytes of bf16), all loads
// before the stores. Bound by launches before (one kernel of 2-byte accesses per tensor: 36 launches
// of 4.4 us each for 15 MB at 18 layers x 816 tokens); the copy alone is 30 MB of traffic, 4.4 us at
// the copy peak. VEC: the sources are 16-byte aligned.
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

// The product kernel of one kind: KS warps share a slot group's K range while each keeps a step of
// 128; 16-byte (8-byte for bf16) loads when K is a multiple of 4.
template <typename T, int KIND>
jpi_status launch_rows_gemm(jpi_handle* h, const RowsArgs& a, cudaStream_t st) {
    const int groups = KIND == RK_RESID ? (a.N + 3) / 4 : KIND == RK_GEGLU ? (a.N + 1) / 2 : a.N / 4;
    const int nst = (a.K + 127) / 128, ks = nst >= 4 ? 4 : nst >= 2 ? 2 : 1;
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
    // Products: 16-token rows kernel while 64 x 64 tiles of the output would leave the GPU about
    // one tile per SM or less, else those tiles, with the norm and rotary passes of their own.
    // Measured, rows against tiles (fp32, us): QKV (2560 x 1024) 33 / 88 at 51 tokens, 109 / 122 at
    // 204 (160 tiles), 211 / 125 at 408 (280); gate/up (4096 x 1024) 164 / 215 at 102 (128), 312 / 246
    // at 204 (256); down (1024 x 4096) 212 / 286 at 408 (112), 842 / 623 at 1632 (416).
    auto rows_fit = [&](int N) {
        return (long long)((N + GB_N - 1) / GB_N) * ((Mt + GB_M - 1) / GB_M) * 4 <= 5ll * h->num_sms;
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
            if (!rows_fit(h->QKV)) {
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
            // Four heads per block once one head per block would be more than four blocks per SM.
            const bool four = h->H % 4 == 0 && (long long)Mt * h->H > 4ll * h->num_sms;
            return four ? launch_attn_rows<T, 4>(h, (const T*)h->q, kst, vst, (T*)h->o, Mt, S, st)
                        : launch_attn_rows<T, 1>(h, (const T*)h->q, kst, vst, (T*)h->o, Mt, S, st);
        }
        case 4:
            if (!rows_fit(W)) {
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
            if (!rows_fit(F)) {
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
            if (!rows_fit(W)) {
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

// Step times are processed in groups of at most 8 so the shared-memory copy of the inputs
// stays at 8 x max(W, d_t) floats whatever the step count.
constexpr int TC_GROUP = 8;

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
    // Few rows (four per thread would leave most SMs without a warp): a warp per row instead, eight
    // step times a launch (3584 rows x 256 columns: 19 us with four rows per thread on 14 CTAs).
    if (R < MOD_RT * 64 * h->num_sms) {
        for (int n0 = 0; n0 < g; n0 += TC_GROUP) {
            const int ng = g - n0 < TC_GROUP ? g - n0 : TC_GROUP;
            k_gemv_multi<T, false><<<grid_for((long long)R * 32, 256, 1024), 256, sizeof(float) * ng * h->W, st>>>(
                (const T*)h->mod_w, h->mod_b, X + (size_t)n0 * h->W, Y + (size_t)n0 * R, R, h->W, ng);
        }
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

template <typename T>
jpi_status time_cond(jpi_handle* h, int N, cudaStream_t st) {
    const int W = h->W, dt = h->dt;
    const int R = mod_rows(h->L) * W;
    const dim3 blk(256);
    for (int n0 = 0; n0 < N; n0 += TC_GROUP) {
        const int g = (N - n0) < TC_GROUP ? (N - n0) : TC_GROUP;
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * g * dt, st>>>(
            (const T*)h->time_in_w, h->time_in_b, h->temb + (size_t)n0 * dt, h->c1 + (size_t)n0 * W, W, dt, g);
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * g * W, st>>>(
            (const T*)h->time_out_w, h->time_out_b, h->c1 + (size_t)n0 * W, h->cond + (size_t)n0 * W, W, W, g);
    }
    for (int n0 = 0; n0 < N; n0 += MOD_GROUP) {
        const int g = (N - n0) < MOD_GROUP ? (N - n0) : MOD_GROUP;
        JPI_TRY(mod_gemv<T>(h, g, h->cond + (size_t)n0 * W, h->mods + (size_t)n0 * R, R, st));
    }
    return check_launch("time conditioning");
}

}  // namespace

jpi_status configure_simt_kernels(jpi_handle* h) {
    const int gemv_smem = (int)(sizeof(float) * (size_t)TC_GROUP * (h->W > h->dt ? h->W : h->dt));
    const int mod_smem = (int)(sizeof(float) * (size_t)MOD_GROUP * h->W);
    int dev = 0;
    JPI_CUDA_TRY(cudaGetDevice(&dev));
    JPI_CUDA_TRY(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev));
    if (h->bf16) {
        using T = __nv_bfloat16;
        JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem));
        JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem));
        JPI_TRY(set_mod_attrs<T>(mod_smem));
    } else {
        using T = float;
        JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem));
        JPI_CUDA_TRY(cudaFuncSetAttribute(k_gemv_multi<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemv_smem));
        JPI_TRY(set_mod_attrs<float>(mod_smem));
    }
    return JPI_OK;
}

jpi_status launch_time_embed(jpi_handle* h, int nsteps, double t_override, cudaStream_t st) {
    k_time_embed<<<dim3(nsteps, (h->dt / 2 + 127) / 128), 128, 0, st>>>(h->temb, nsteps, h->dt, h->cfg.t_min_period,
                                                                      h->cfg.t_max_period, t_override);
    return check_launch("time embedding");
}

jpi_status launch_time_conditioning(jpi_handle* h, int nsteps, cudaStream_t st) {
    return h->bf16 ? time_cond<__nv_bfloat16>(h, nsteps, st) : time_cond<float>(h, nsteps, st);
}

// Time conditioning of one step time with caller-chosen scratch: sinusoid into temb [d_t],
// time-MLP hidden layer into c1 [W], conditioning vector into cond [W]; the modulation
// vectors go to the handle's step-0 slot, as with launch_time_conditioning(h, 1, ...).
jpi_status launch_time_conditioning_into(jpi_handle* h, double t, float* temb, float* c1,
                                         float* cond, cudaStream_t st) {
    const int W = h->W, dt = h->dt;
    const int R = mod_rows(h->L) * W;
    k_time_embed<<<dim3(1, (dt / 2 + 127) / 128), 128, 0, st>>>(temb, 1, dt, h->cfg.t_min_period, h->cfg.t_max_period, t);
    const dim3 blk(256);
    if (h->bf16) {
        using T = __nv_bfloat16;
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * dt, st>>>(
            (const T*)h->time_in_w, h->time_in_b, temb, c1, W, dt, 1);
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * W, st>>>(
            (const T*)h->time_out_w, h->time_out_b, c1, cond, W, W, 1);
        JPI_TRY(mod_gemv<T>(h, 1, cond, h->mods, R, st));
    } else {
        using T = float;
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * dt, st>>>(
            (const T*)h->time_in_w, h->time_in_b, temb, c1, W, dt, 1);
        k_gemv_multi<T, true><<<grid_for((long long)W * 32, 256, 1024), blk, sizeof(float) * W, st>>>(
            (const T*)h->time_out_w, h->time_out_b, c1, cond, W, W, 1);
        JPI_TRY(mod_gemv<T>(h, 1, cond, h->mods, R, st));
    }
    return check_launch("time conditioning (caller scratch)");
}

jpi_status launch_embed(jpi_handle* h, int step, int B, int C, const float* x, cudaStream_t st) {
    const int slices = (h->W + 127) / 128, nctx = h->n_ctx();
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
    // About eight blocks per SM (a small batch keeps one token per block, the shortest chain), at
    // most EMB_MAX_TPB tokens each.
    const long long want = 8ll * h->num_sms;
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

jpi_status launch_final(jpi_handle* h, int step, int B, int C, float delta, float* x_inout,
                        float* v_out, float* out_copy, cudaStream_t st) {
    const int W = h->W;
    const float* ms = h->mods + (size_t)step * mod_rows(h->L) * W + (size_t)6 * h->L * W;
    launch_pdl(h, dim3(B * C), dim3(FIN_THREADS), sizeof(float) * W, st, k_final, (const float*)h->h, ms, ms + W,
               (const float*)h->action_out_w, (const float*)h->action_out_b, x_inout, v_out, out_copy,
               C + h->n_ctx(), h->n_ctx(), C, W, h->A, h->cfg.rms_eps, delta);
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
