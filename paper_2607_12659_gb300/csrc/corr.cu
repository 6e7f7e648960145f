// The future correction module and its Q-Former state compressor on the GPU (Sec. 4.1, App. B
// and its figure, Eq. 2, App. C Alg. 1).
//
// Every token count here is small (T' = 4 compressed tokens, at most 64 committed actions per
// request), so apart from the compressor's pass over the VLM tokens the module is a chain of
// matrix-vector products that stream its ~44M weights once per call: at batch 1 that is HBM
// work (88 MB in bf16), not a dense contraction, and it runs on CUDA cores with every weight
// row read once by one warp (16-byte loads) and the few activation rows served from L1.
//
// The compressor's cross-attention is reassociated. Its queries come from the learned query
// tokens through the query self-attention alone, so they are fixed by the weights; with
// q_hi the scaled query of head h, item i, and W_k,h / W_v,h the head's rows of the key and
// value projections:
//   score_hij = q_hi . (W_k,h v_j + b_k,h) = (W_k,h^T q_hi) . v_j + const_hi,
//   out_hi    = sum_j p_hij (W_v,h v_j + b_v,h) = W_v,h (sum_j p_hij v_j) + b_v,h   (sum_j p = 1).
// The key bias only shifts every score of a query alike, which softmax cancels. So create time
// computes a_hi = W_k,h^T q_hi once ([H T'][d_vlm]); a call scores the raw VLM tokens against
// them, takes the softmax-weighted sum of the raw tokens, and applies W_v,h to that sum: about
// 2 H T' T d_vlm * 2 FLOPs per request instead of the 4 T d_vlm d of projecting every token.

#include "jpi_internal.h"
#include "ptx.h"

#include "jpi_corr.h"

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <new>
#include <utility>

namespace {

constexpr int CORR_MAX_M = 64;          // n_heads * n_items: rows of the reassociated queries
constexpr int LIN_ROWS = 8;             // activation rows one warp carries per weight-row pass

jpi_status cfail(jpi_status s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    jpi::set_error("%s", buf);
    return s;
}

__device__ __forceinline__ float gelu_tanh_f(float y) {
    // 0.5 y (1 + tanh(sqrt(2/pi) (y + 0.044715 y^3))), the tanh form of GELU.
    return 0.5f * y * (1.f + tanhf(0.7978845608028654f * (y + 0.044715f * y * y * y)));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float load1(const float* p) { return __ldg(p); }
__device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(p[0]); }

// y[r][o] = act(sum_i x(r, o)[i] w[o][i] + bias[o]) + res[r][o] for r < rows, o < out.
// x(r, o) is row r of x (stride ldx), or in head-select mode row
// ((r / hs_items) * hs_heads + o / hs_dh) * hs_items + r % hs_items: the reassociated
// cross-attention keeps one weighted token sum per (request, head, item).
// One warp per output feature at a time; LIN_ROWS rows per pass over the weight row. y must not
// overlap x; it may be res (each element is read and written by the same lane).
struct LinArgs {
    const float* x;
    int ldx;
    const void* w;
    const float* bias;
    const float* res;
    int ldr;
    float* y;
    int ldy;
    int rows, in, out, gelu;
    int hs_items, hs_heads, hs_dh;   // head-select mode when hs_items > 0
    // Forms of the streamed product only (k_corr_linear_pipe):
    int res_mod;             // > 0: residual row r mod res_mod (a table shared by the requests)
    const float* x2;         // columns join.. of row r come from row r / x2_div of x2 (null: none)
    int join, x2_div, ldx2;
    int seg_out, seg_rows;   // features below seg_out: rows 0 .. seg_rows - 1 of seg_x into seg_y instead
    const float* seg_x;
    int seg_ldx;
    float* seg_y;
    int seg_ldy;
    const float *ln_g, *ln_b;   // LayerNorm of every input row (width `in`) before the product
    float ln_eps;
    int att_heads_dh;        // attention form: head dim; x holds q, k at + d and v at + 2 d (d = in)
    float att_scale;
    // Confidence of the heads: CTAs past lin_ctas (one per request of conf_items rows) compute
    // conf[b] = conf_w . mean of the request's normalised rows + conf_b.
    int lin_ctas, conf_items;
    const float *conf_w, *conf_b;
    float* conf;
};

template <typename TW, bool VEC>
__global__ void __launch_bounds__(256) k_corr_linear(const LinArgs a) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const TW* W = static_cast<const TW*>(a.w);
    for (int o = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); o < a.out; o += nwarps) {
        const TW* wr = W + (size_t)o * a.in;
        const float bo = a.bias ? a.bias[o] : 0.f;
        for (int r0 = 0; r0 < a.rows; r0 += LIN_ROWS) {
            const float* xr[LIN_ROWS];
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) {
                const int r = r0 + k < a.rows ? r0 + k : a.rows - 1;   // clamped; result unused
                long long row = r;
                if (a.hs_items > 0)
                    row = ((long long)(r / a.hs_items) * a.hs_heads + o / a.hs_dh) * a.hs_items + r % a.hs_items;
                xr[k] = a.x + row * a.ldx;
            }
            float acc[LIN_ROWS];
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) acc[k] = 0.f;
            if (VEC) {
                // Unrolled so that several 4-wide weight loads of the row are in flight at once.
#pragma unroll 4
                for (int i = lane * 4; i < a.in; i += 128) {
                    const float4 w4 = load4(wr + i);
#pragma unroll
                    for (int k = 0; k < LIN_ROWS; ++k) {
                        const float4 x4 = *reinterpret_cast<const float4*>(xr[k] + i);
                        acc[k] = fmaf(w4.x, x4.x, fmaf(w4.y, x4.y, fmaf(w4.z, x4.z, fmaf(w4.w, x4.w, acc[k]))));
                    }
                }
            } else {
                for (int i = lane; i < a.in; i += 32) {
                    const float w1 = load1(wr + i);
#pragma unroll
                    for (int k = 0; k < LIN_ROWS; ++k) acc[k] = fmaf(w1, xr[k][i], acc[k]);
                }
            }
            float mine = 0.f;   // lane k keeps row r0 + k
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) {
                const float v = warp_sum(acc[k]);
                if (lane == k) mine = v;
            }
            const int r = r0 + lane;
            if (lane < LIN_ROWS && r < a.rows) {
                float v = mine + bo;
                if (a.gelu) v = gelu_tanh_f(v);
                if (a.res) v += a.res[(size_t)r * a.ldr + o];
                a.y[(size_t)r * a.ldy + o] = v;
            }
        }
    }
}

// The same product for bf16 weights with 16-byte aligned rows and 16-byte aligned activation rows
// (in a multiple of 8 KS, ldx of 4): a lane streams 16-byte weight chunks, LIN_CH of them in
// flight, and the KS consecutive warps of a block share an output feature, each over in / KS
// inputs, their sums added in warp order through shared memory (deterministic). Blocks of
// 8 / KS output features walk the outputs grid-stride.
constexpr int LIN_CH = 8;
template <int KS>
__global__ void __launch_bounds__(256) k_corr_linear16(const LinArgs a) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ float part[8][LIN_ROWS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slice = warp % KS, og = warp / KS;
    constexpr int OPB = 8 / KS;
    const int kper = a.in / KS, k0 = slice * kper;
    const __nv_bfloat16* W = static_cast<const __nv_bfloat16*>(a.w);
    const int ngroups = (a.out + OPB - 1) / OPB;
    for (int gi = blockIdx.x; gi < ngroups; gi += gridDim.x) {
        const int o = gi * OPB + og;
        const bool live = o < a.out;
        const int oc = live ? o : a.out - 1;   // clamped; result unused
        const __nv_bfloat16* wr = W + (size_t)oc * a.in + k0;
        const float bo = (a.bias && live) ? a.bias[oc] : 0.f;
        for (int r0 = 0; r0 < a.rows; r0 += LIN_ROWS) {
            const float* xr[LIN_ROWS];
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) {
                const int r = r0 + k < a.rows ? r0 + k : a.rows - 1;   // clamped; result unused
                long long row = r;
                if (a.hs_items > 0)
                    row = ((long long)(r / a.hs_items) * a.hs_heads + oc / a.hs_dh) * a.hs_items + r % a.hs_items;
                xr[k] = a.x + row * a.ldx + k0;
            }
            float acc[LIN_ROWS];
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) acc[k] = 0.f;
            for (int base = 0; base < kper; base += 256 * LIN_CH) {
                uint4 wv[LIN_CH];
#pragma unroll
                for (int j = 0; j < LIN_CH; ++j) {
                    const int i = base + 256 * j + 8 * lane;
                    wv[j] = i < kper ? __ldg(reinterpret_cast<const uint4*>(wr + i)) : make_uint4(0u, 0u, 0u, 0u);
                }
#pragma unroll
                for (int j = 0; j < LIN_CH; ++j) {
                    const int i = base + 256 * j + 8 * lane;
                    if (i < kper) {
                        const uint32_t u[4] = {wv[j].x, wv[j].y, wv[j].z, wv[j].w};
                        float w[8];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u[q]));
                            w[2 * q] = f.x;
                            w[2 * q + 1] = f.y;
                        }
#pragma unroll
                        for (int k = 0; k < LIN_ROWS; ++k) {
                            const float4 x0 = *reinterpret_cast<const float4*>(xr[k] + i);
                            const float4 x1 = *reinterpret_cast<const float4*>(xr[k] + i + 4);
                            float t = acc[k];
                            t = fmaf(w[0], x0.x, t);
                            t = fmaf(w[1], x0.y, t);
                            t = fmaf(w[2], x0.z, t);
                            t = fmaf(w[3], x0.w, t);
                            t = fmaf(w[4], x1.x, t);
                            t = fmaf(w[5], x1.y, t);
                            t = fmaf(w[6], x1.z, t);
                            t = fmaf(w[7], x1.w, t);
                            acc[k] = t;
                        }
                    }
                }
            }
            float mine = 0.f;   // lane k keeps row r0 + k
#pragma unroll
            for (int k = 0; k < LIN_ROWS; ++k) {
                const float v = warp_sum(acc[k]);
                if (lane == k) mine = v;
            }
            if (KS > 1) {
                if (lane < LIN_ROWS) part[warp][lane] = mine;
                __syncthreads();
                if (slice == 0 && lane < LIN_ROWS) {
                    float t = part[warp][lane];
#pragma unroll
                    for (int sl = 1; sl < KS; ++sl) t += part[warp + sl][lane];
                    mine = t;
                }
                __syncthreads();   // part is reused by the next row group
            }
            const int r = r0 + lane;
            if (slice == 0 && live && lane < LIN_ROWS && r < a.rows) {
                float v = mine + bo;
                if (a.gelu) v = gelu_tanh_f(v);
                if (a.res) v += a.res[(size_t)r * a.ldr + o];
                a.y[(size_t)r * a.ldy + o] = v;
            }
        }
    }
}

// The same product streamed through shared memory, for bf16 weights (16-byte aligned, in a
// multiple of 8 and at most LP_MAX_IN), 16-byte aligned activation rows (ldx a multiple of 4) and
// no head-select: a persistent CTA walks groups of LP_ROWS consecutive output features; their
// weight rows (contiguous) arrive by per-thread 16-byte cp.async copies into a ring of NST
// stages, the first ones issued before the dependency wait (weights do not depend on the previous
// kernel). Thread t takes the 8-column chunks t, t + 256, ... of the inputs for all LP_ROWS
// features of a group, so each chunk of LP_XR activation rows it loads serves all of them: as
// many activation bytes as weight bytes (one warp per feature reads LIN_ROWS activation chunks per
// weight chunk, and those L1 reads bound it); the per-feature sums are reduced over the block in a fixed order. No waits that can spin: the copies are waited with
// cp.async.wait_group.
//
// Forms that take a neighbouring kernel in, because at a handful of rows every launch of the chain
// costs 4-5 us whatever it computes:
//   LP_LN    LayerNorm of the input rows (in <= 2048, at most LP_LN_ROWS rows): every CTA computes the
//            rows' mean and variance first (a warp per row, two passes over registers), then
//            normalises each chunk as it loads it;
//   LP_ATTN  multi-head attention among four tokens (rows r0 .. r0 + 3 are one request's): the thread's
//            chunk of the attention output is computed in registers from its chunk of q, k and v, the
//            scores summed over the head's lanes by shuffles;
// and, in every form, a residual table indexed by row mod n, an input joined from two sources, a first
// segment of features with rows of its own, and the confidence head on CTAs of its own.
constexpr int LP_ROWS = 8;
constexpr int LP_XR = 4;          // activation rows per pass
constexpr int LP_MAX_IN = 4096;
constexpr int LP_LN_ROWS = 32;
enum { LP_PLAIN = 0, LP_LN = 1, LP_ATTN = 2 };
__host__ __device__ constexpr int lp_stages(int in) {
    return in <= 2048 ? 4 : 3;
}

// Mean and 1 / sqrt(biased variance + eps) of rows r0, r0 + step, .. (< rows) of x (width d <= 2048, a
// multiple of 4, 16-byte aligned rows), one warp per row, into mr[r - base].
__device__ __forceinline__ void lp_row_stats(const float* x, int ldx, int r0, int step, int rows, int d, float eps,
                                             float2* mr, int base) {
    const int lane = threadIdx.x & 31, d4 = d >> 2;
    for (int r = r0; r < rows; r += step) {
        const float4* xr = reinterpret_cast<const float4*>(x + (size_t)r * ldx);
        float4 v[16];
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int i = lane + 32 * k;
            v[k] = i < d4 ? xr[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) s += (v[k].x + v[k].y) + (v[k].z + v[k].w);
        const float mean = warp_sum(s) / (float)d;
        float var = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (lane + 32 * k >= d4) break;
            const float t0 = v[k].x - mean, t1 = v[k].y - mean, t2 = v[k].z - mean, t3 = v[k].w - mean;
            var = fmaf(t0, t0, fmaf(t1, t1, fmaf(t2, t2, fmaf(t3, t3, var))));
        }
        const float rstd = 1.f / sqrtf(warp_sum(var) / (float)d + eps);
        if (lane == 0) mr[r - base] = make_float2(mean, rstd);
    }
}

__device__ __forceinline__ void lp_load8(const float* p, float (&x)[8]) {
    const float4 x0 = *reinterpret_cast<const float4*>(p), x1 = *reinterpret_cast<const float4*>(p + 4);
    x[0] = x0.x; x[1] = x0.y; x[2] = x0.z; x[3] = x0.w;
    x[4] = x1.x; x[5] = x1.y; x[6] = x1.z; x[7] = x1.w;
}

// Columns 8 c .. 8 c + 7 of the attention output of four tokens, c this thread's chunk: base points at
// the chunk of the first token's query, rows ldx apart, keys d and values 2 d further on. The dh / 8
// lanes of a head (a power of two within a warp) sum its scores; every lane of the warp takes part.
__device__ __forceinline__ void attn4_chunk(const float* base, int ldx, int d, int dh, float scale, float (&x)[4][8]) {
    float q[4][8], k[4][8], v[4][8], s[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        lp_load8(base + (size_t)i * ldx, q[i]);
        lp_load8(base + (size_t)i * ldx + d, k[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) lp_load8(base + (size_t)i * ldx + 2 * d, v[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float t = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) t = fmaf(q[i][e], k[j][e], t);
            s[i][j] = t;
        }
    for (int sh = dh / 16; sh > 0; sh >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s[i][j] += __shfl_xor_sync(0xffffffffu, s[i][j], sh);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float mx = -INFINITY, den = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            s[i][j] *= scale;
            mx = fmaxf(mx, s[i][j]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            s[i][j] = expf(s[i][j] - mx);
            den += s[i][j];
        }
        const float inv = 1.f / den;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float t = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) t = fmaf(s[i][j], v[j][e], t);
            x[i][e] = t * inv;
        }
    }
}

// The same attention as a launch of its own (one CTA per request; o [4 B][d]): bit for bit what the
// LP_ATTN form computes, for batches where computing it in every CTA of the product takes longer.
__global__ void __launch_bounds__(256) k_corr_attn4(const float* __restrict__ qkv, float* __restrict__ o, int d, int dh,
                                                    float scale) {
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const int nch = d / 8, c = (int)threadIdx.x < nch ? threadIdx.x : 0;
    float x[4][8];
    attn4_chunk(qkv + (size_t)blockIdx.x * 4 * 3 * d + 8 * c, 3 * d, d, dh, scale, x);
    if ((int)threadIdx.x >= nch) return;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float4* y = reinterpret_cast<float4*>(o + ((size_t)blockIdx.x * 4 + i) * d + 8 * c);
        y[0] = make_float4(x[i][0], x[i][1], x[i][2], x[i][3]);
        y[1] = make_float4(x[i][4], x[i][5], x[i][6], x[i][7]);
    }
}

// SPLIT = 2 (in <= 1024, more than four rows): the two halves of the block take four of a group's
// features each over all chunks, and a pass takes eight rows; otherwise threads past in / 8 chunks would
// idle, and every four rows cost a reduction over the block. The sums are the same either way.
template <int NST, int MODE, int SPLIT>
__global__ void __launch_bounds__(256) k_corr_linear_pipe(const __grid_constant__ LinArgs a) {
    constexpr int XR = LP_XR * SPLIT, FPT = LP_ROWS / SPLIT;   // rows per pass, features per thread
    constexpr int CT = 256 / SPLIT;                            // threads that share a feature's chunks
    static_assert(MODE != LP_ATTN || SPLIT == 1, "the attention form takes four rows");
    extern __shared__ __align__(128) uint8_t lp_smem[];
    __shared__ float red[8][32];
    __shared__ float2 mr[LP_LN_ROWS];   // LayerNorm: (mean, 1 / std) of each row
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int in = a.in, nch = in / 8;
    const int ct = tid % CT, f0 = tid / CT * FPT;   // first chunk, first feature of a group
    if (MODE == LP_LN && a.conf && (int)blockIdx.x >= a.lin_ctas) {
        // The confidence of request b: features tid, tid + 256, .. of the mean normalised row.
        jpi::ptx::grid_dep_wait();
        jpi::ptx::grid_dep_launch();
        const int b = blockIdx.x - a.lin_ctas, n = a.conf_items;
        lp_row_stats(a.x, a.ldx, b * n + warp, 8, (b + 1) * n, in, a.ln_eps, mr, b * n);
        __syncthreads();
        float s = 0.f;
        for (int c = tid; c < in; c += 256) {
            float m = 0.f;
            for (int i = 0; i < n; ++i)
                m += (a.x[(size_t)(b * n + i) * a.ldx + c] - mr[i].x) * mr[i].y * a.ln_g[c] + a.ln_b[c];
            s = fmaf(a.conf_w[c], m / (float)n, s);
        }
        s = warp_sum(s);
        if (lane == 0) red[0][warp] = s;
        __syncthreads();
        if (tid == 0) {
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) v += red[0][w];
            a.conf[b] = v + a.conf_b[0];
        }
        return;
    }
    const int sbytes = LP_ROWS * in * 2;
    const int ngroups = (a.out + LP_ROWS - 1) / LP_ROWS;
    const int nctas = a.lin_ctas;
    const uint8_t* W = static_cast<const uint8_t*>(a.w);
    // Group k of this CTA: blockIdx.x + k nctas; its rows into stage k mod NST (one commit
    // group per k, empty past the last group, so the group count stays uniform).
    auto issue = [&](int k) {
        const int g = blockIdx.x + k * nctas;
        if (g < ngroups) {
            const int rows = min(LP_ROWS, a.out - g * LP_ROWS);
            const int chunks = rows * nch;
            const uint8_t* src = W + (size_t)g * LP_ROWS * in * 2;
            const uint32_t dst = jpi::ptx::smem_u32(lp_smem + (size_t)(k % NST) * sbytes);
            for (int c = tid; c < chunks; c += 256) jpi::ptx::cp_async_16(dst + 16 * c, src + 16 * (size_t)c, true);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int k = 0; k < NST - 1; ++k) issue(k);
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    if (MODE == LP_LN) {
        lp_row_stats(a.x, a.ldx, warp, 8, a.rows, in, a.ln_eps, mr, 0);
        __syncthreads();
    }
    for (int k = 0; blockIdx.x + k * nctas < ngroups; ++k) {
        issue(k + NST - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(NST - 1) : "memory");
        __syncthreads();   // stage k mod NST holds group k for every thread
        const int o0 = (blockIdx.x + k * nctas) * LP_ROWS;
        const int nout = min(LP_ROWS, a.out - o0);
        const uint4* wst = reinterpret_cast<const uint4*>(lp_smem + (size_t)(k % NST) * sbytes);
        // Rows, input and output of this group's segment (seg_out is a multiple of LP_ROWS). The
        // segment's input rows are rows of x: their statistics are found by the address.
        const bool seg = o0 < a.seg_out;
        const int rows = seg ? a.seg_rows : a.rows, ldx = seg ? a.seg_ldx : a.ldx, ldy = seg ? a.seg_ldy : a.ldy;
        const float* xb = seg ? a.seg_x : a.x;
        float* yb = seg ? a.seg_y : a.y;
        for (int r0 = 0; r0 < rows; r0 += XR) {
            const int nr = min(XR, rows - r0);
            // The bias and residual of this thread's output (thread o XR + q writes feature
            // o0 + o of row r0 + q), fetched before the products so their latency hides there.
            float bias_v = 0.f, res_v = 0.f;
            if (tid < LP_ROWS * XR) {
                const int o = tid / XR, q = tid % XR;
                if (o < nout && q < nr) {
                    if (a.bias) bias_v = a.bias[o0 + o];
                    const int rr = a.res_mod > 0 ? (r0 + q) % a.res_mod : r0 + q;
                    if (a.res) res_v = a.res[(size_t)rr * a.ldr + o0 + o];
                }
            }
            float acc[FPT][XR];
#pragma unroll
            for (int o = 0; o < FPT; ++o)
#pragma unroll
                for (int q = 0; q < XR; ++q) acc[o][q] = 0.f;
            // Chunk c (8 columns) of rows r0 .. against this thread's weight rows of the group.
            auto product = [&](int c, const float (&x)[XR][8]) {
#pragma unroll
                for (int o = 0; o < FPT; ++o) {
                    if (f0 + o >= nout) break;
                    const uint4 wv = wst[(size_t)(f0 + o) * nch + c];
                    const uint32_t u[4] = {wv.x, wv.y, wv.z, wv.w};
                    float w[8];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u[e]));
                        w[2 * e] = f.x;
                        w[2 * e + 1] = f.y;
                    }
#pragma unroll
                    for (int q = 0; q < XR; ++q) {
                        float t = acc[o][q];
#pragma unroll
                        for (int e = 0; e < 8; ++e) t = fmaf(w[e], x[q][e], t);
                        acc[o][q] = t;
                    }
                }
            };
            if constexpr (MODE == LP_ATTN) {
                // One chunk per thread (in <= 2048).
                const int c = tid < nch ? tid : 0;
                float x[LP_XR][8];
                attn4_chunk(xb + (size_t)r0 * ldx + 8 * c, ldx, in, a.att_heads_dh, a.att_scale, x);
                if (tid < nch) product(tid, x);
            } else {
                for (int c = ct; c < nch; c += CT) {
                    float x[XR][8];
                    float gv[8], bv[8];
                    if (MODE == LP_LN) {
                        lp_load8(a.ln_g + 8 * c, gv);
                        lp_load8(a.ln_b + 8 * c, bv);
                    }
                    const bool second = a.x2 && 8 * c >= a.join;
                    const float* xc = xb + (size_t)r0 * ldx + 8 * c;
#pragma unroll
                    for (int q = 0; q < XR; ++q) {
                        if (q < nr) {
                            lp_load8(second ? a.x2 + (size_t)((r0 + q) / a.x2_div) * a.ldx2 + (8 * c - a.join)
                                            : xc + (size_t)q * ldx, x[q]);
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) x[q][e] = 0.f;
                        }
                    }
                    if (MODE == LP_LN) {
#pragma unroll
                        for (int q = 0; q < XR; ++q) {
                            if (q >= nr) break;
                            // Row of x this is (a segment's rows are a subset of them).
                            const float2 st = mr[seg ? (int)((a.seg_x - a.x + (size_t)(r0 + q) * ldx) / a.ldx) : r0 + q];
#pragma unroll
                            for (int e = 0; e < 8; ++e) x[q][e] = (x[q][e] - st.x) * st.y * gv[e] + bv[e];
                        }
                    }
                    product(c, x);
                }
            }
            // (feature o, row q) sums: over the warp's lanes, then over the 8 warps in order. The
            // warp sum is a reduce-scatter: at offset 16, 8, .., 1 each lane keeps the half of its
            // pairs whose bit matches its own and adds its partner's partial of them (the same
            // pairwise sums as a butterfly per pair, 31 shuffles instead of 160); lane p ends
            // with pair p = o XR + q of its half's features.
            static_assert(FPT * XR == 32, "one pair per lane");
            float pv[32];
#pragma unroll
            for (int o = 0; o < FPT; ++o)
#pragma unroll
                for (int q = 0; q < XR; ++q) pv[o * XR + q] = acc[o][q];
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) {
                const bool hi = (lane & sh) != 0;
#pragma unroll
                for (int i = 0; i < sh; ++i) {
                    const float send = hi ? pv[i] : pv[i + sh];
                    const float keep = hi ? pv[i + sh] : pv[i];
                    pv[i] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
                }
            }
            red[warp][lane] = pv[0];
            __syncthreads();
            if (tid < LP_ROWS * XR) {
                // Thread o XR + q: lane tid mod 32 of the warps of half tid / 32, in warp order.
                const int o = tid / XR, q = tid % XR;
                float v = 0.f;
#pragma unroll
                for (int w8 = 0; w8 < 8 / SPLIT; ++w8) v += red[(tid >> 5) * (8 / SPLIT) + w8][lane];
                const int of = o0 + o, r = r0 + q;
                if (o < nout && q < nr) {
                    v += bias_v;
                    if (a.gelu) v = gelu_tanh_f(v);
                    if (a.res) v += res_v;
                    yb[(size_t)r * ldy + of] = v;
                }
            }
            __syncthreads();   // red is reused by the next pass
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // nothing lands after exit
}

// LayerNorm of `rows` rows of width d: one warp per row (grid-stride over rows), three passes
// (mean, biased variance, output). VEC: every row and vector 16-byte aligned, d a multiple of 4,
// so the passes move float4s.
template <bool VEC>
__global__ void __launch_bounds__(256) k_corr_layernorm(const float* __restrict__ x, int ldx,
                                                        const float* __restrict__ g,
                                                        const float* __restrict__ b,
                                                        float* __restrict__ y, int ldy, int rows,
                                                        int d, float eps) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const int lane = threadIdx.x & 31, nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int r = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); r < rows; r += nwarps) {
        const float* xr = x + (size_t)r * ldx;
        float* yr = y + (size_t)r * ldy;
        if (VEC) {
            const int d4 = d >> 2;
            const float4* x4 = reinterpret_cast<const float4*>(xr);
            float s = 0.f;
#pragma unroll 8
            for (int i = lane; i < d4; i += 32) {
                const float4 v = x4[i];
                s += (v.x + v.y) + (v.z + v.w);
            }
            const float mean = warp_sum(s) / (float)d;
            float var = 0.f;
#pragma unroll 4
            for (int i = lane; i < d4; i += 32) {
                const float4 v = x4[i];
                const float t0 = v.x - mean, t1 = v.y - mean, t2 = v.z - mean, t3 = v.w - mean;
                var = fmaf(t0, t0, fmaf(t1, t1, fmaf(t2, t2, fmaf(t3, t3, var))));
            }
            const float rstd = 1.f / sqrtf(warp_sum(var) / (float)d + eps);
            float4* y4 = reinterpret_cast<float4*>(yr);
            const float4* g4 = reinterpret_cast<const float4*>(g);
            const float4* b4 = reinterpret_cast<const float4*>(b);
#pragma unroll 4
            for (int i = lane; i < d4; i += 32) {
                const float4 v = x4[i], gg = g4[i], bb = b4[i];
                y4[i] = make_float4((v.x - mean) * rstd * gg.x + bb.x, (v.y - mean) * rstd * gg.y + bb.y,
                                    (v.z - mean) * rstd * gg.z + bb.z, (v.w - mean) * rstd * gg.w + bb.w);
            }
        } else {
            float s = 0.f;
            for (int i = lane; i < d; i += 32) s += xr[i];
            const float mean = warp_sum(s) / (float)d;
            float var = 0.f;
            for (int i = lane; i < d; i += 32) {
                const float t = xr[i] - mean;
                var = fmaf(t, t, var);
            }
            const float rstd = 1.f / sqrtf(warp_sum(var) / (float)d + eps);
            for (int i = lane; i < d; i += 32) yr[i] = (xr[i] - mean) * rstd * g[i] + b[i];
        }
    }
}

// Multi-head attention over few keys: query row (b, i) of head h against key rows (b, j),
// j < nk, every key visible. One warp per (b, h, i); head_dim <= 256, nk <= 64.
struct AttnSmallArgs {
    const float* q;
    int ldq;
    const float* k;
    int ldk;
    const float* v;
    int ldv;
    float* o;
    int ldo;
    int B, nq, nk, H, Dh;
    float scale;
};

__global__ void __launch_bounds__(256) k_corr_attn(const AttnSmallArgs a) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ float sp[8][JPI_CORR_MAX_DELTA];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gw = blockIdx.x * 8 + wib;
    if (gw >= a.B * a.H * a.nq) return;   // whole warps leave; no block barrier follows
    const int i = gw % a.nq, h = (gw / a.nq) % a.H, b = gw / (a.nq * a.H);
    const float* qr = a.q + (size_t)(b * a.nq + i) * a.ldq + h * a.Dh;
    float qf[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int d = lane + 32 * t;
        qf[t] = d < a.Dh ? qr[d] : 0.f;
    }
    // Keys (and below, values) four rows at a time: their loads are in flight together.
    float mx = -INFINITY;
    for (int j0 = 0; j0 < a.nk; j0 += 4) {
        float kv[4][8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u < a.nk ? j0 + u : j0;
            const float* kr = a.k + (size_t)(b * a.nk + j) * a.ldk + h * a.Dh;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int d = lane + 32 * t;
                kv[u][t] = d < a.Dh ? kr[d] : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            if (j >= a.nk) break;
            float s = 0.f;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int d = lane + 32 * t;
                if (d < a.Dh) s = fmaf(qf[t], kv[u][t], s);
            }
            s = warp_sum(s) * a.scale;
            if (lane == 0) sp[wib][j] = s;
            mx = fmaxf(mx, s);
        }
    }
    __syncwarp();
    float den = 0.f;
    for (int j = lane; j < a.nk; j += 32) {
        const float e = expf(sp[wib][j] - mx);
        sp[wib][j] = e;
        den += e;
    }
    den = warp_sum(den);
    __syncwarp();
    float of[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) of[t] = 0.f;
    for (int j0 = 0; j0 < a.nk; j0 += 4) {
        float vv[4][8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u < a.nk ? j0 + u : j0;
            const float* vr = a.v + (size_t)(b * a.nk + j) * a.ldv + h * a.Dh;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int d = lane + 32 * t;
                vv[u][t] = d < a.Dh ? vr[d] : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u;
            if (j >= a.nk) break;
            const float p = sp[wib][j];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int d = lane + 32 * t;
                if (d < a.Dh) of[t] = fmaf(p, vv[u][t], of[t]);
            }
        }
    }
    const float inv = 1.f / den;
    float* orow = a.o + (size_t)(b * a.nq + i) * a.ldo + h * a.Dh;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int d = lane + 32 * t;
        if (d < a.Dh) orow[d] = of[t] * inv;
    }
}

// Create time: a[h T' + i][c] = scale * sum_e qc[i][h Dh + e] wk[h Dh + e][c] (the cross-
// attention's scaled queries mapped into VLM space). Grid (ceil(dv / 256), H).
template <typename TW>
__global__ void __launch_bounds__(256) k_corr_qk(const float* __restrict__ qc, const TW* __restrict__ wk,
                                                 float* __restrict__ qk, int T, int Dh, int d, int dv,
                                                 float scale) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ float qs[JPI_MAX_CORRECTION][256];
    const int h = blockIdx.y, c = blockIdx.x * 256 + threadIdx.x;
    for (int idx = threadIdx.x; idx < T * Dh; idx += 256)
        qs[idx / Dh][idx % Dh] = qc[(size_t)(idx / Dh) * d + h * Dh + idx % Dh];
    __syncthreads();
    if (c >= dv) return;
    float acc[JPI_MAX_CORRECTION];
#pragma unroll
    for (int i = 0; i < JPI_MAX_CORRECTION; ++i) acc[i] = 0.f;
    for (int e = 0; e < Dh; ++e) {
        const float w = to_f(wk[(size_t)(h * Dh + e) * dv + c]);
#pragma unroll
        for (int i = 0; i < JPI_MAX_CORRECTION; ++i)
            if (i < T) acc[i] = fmaf(qs[i][e], w, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < JPI_MAX_CORRECTION; ++i)
        if (i < T) qk[((size_t)h * T + i) * dv + c] = acc[i] * scale;
}

// Partial scores over one chunk of the VLM features: part[b][kc][m][j] = sum over c in chunk kc
// (CORR_KCHUNK features) of qk[m][c] hv[b][j][c], m < M, j < T. Grid (ceil(T / 32), chunks, B):
// 32 tokens per CTA; the chunk's query rows and token rows are staged in shared memory (fp32) with
// all their loads in flight together, then thread (mg, jg) = (tid / 16, tid mod 16) computes the
// register tile of rows mg, mg + 16, .. (< M) x tokens jg, jg + 16 from 16-byte loads of both
// operands (four features at a time, summed in feature order). Splitting the feature sum over
// CTAs keeps the whole GPU busy at batch 1 (26 token tiles alone would not); the chunks are added
// in order by k_corr_softmax_sum.
constexpr int CORR_KCHUNK = 256;
constexpr int CORR_KPAD = CORR_KCHUNK + 4;   // 16-byte rows; 8 consecutive rows hit distinct banks
constexpr size_t CORR_SCORES_SMEM = (size_t)(CORR_MAX_M + 32) * CORR_KPAD * sizeof(float);

// VEC: dv a multiple of 4 and hv aligned to four elements, so the staging moves four features
// per load; every thread's staging loads are issued before any of its stores (one at a time, each
// store would hold the next load back for a full L2 round trip).
// RM: query rows per thread, 8 RM >= M.
template <typename THV, bool VEC, int RM>
__global__ void __launch_bounds__(256) k_corr_scores(const float* __restrict__ qk, const THV* __restrict__ hv,
                                                     float* __restrict__ part, int M, int T, int dv) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    extern __shared__ float4 sm_scores4[];
    float* as = reinterpret_cast<float*>(sm_scores4);   // [M][CORR_KPAD]
    float* bs = as + CORR_MAX_M * CORR_KPAD;            // [32][CORR_KPAD]
    const int b = blockIdx.z, kc = blockIdx.y, j0 = blockIdx.x * 32;
    const int c0 = kc * CORR_KCHUNK, cn = min(CORR_KCHUNK, dv - c0);
    const THV* hb = hv + (size_t)b * T * dv;
    if (VEC) {
        // Thread t takes feature quad t mod 64 of rows t / 64, t / 64 + 4, ..: CORR_MAX_M / 4 query
        // rows and 8 token rows at most.
        const int k4 = threadIdx.x & 63, r0 = threadIdx.x >> 6, kk = 4 * k4;
        const bool kin = kk < cn;
        float4 qa[2 * RM], hb4[8];
#pragma unroll
        for (int i = 0; i < 2 * RM; ++i) {
            const int m = r0 + 4 * i;
            qa[i] = (m < M && kin) ? *reinterpret_cast<const float4*>(qk + (size_t)m * dv + c0 + kk)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = j0 + r0 + 4 * i;
            hb4[i] = (j < T && kin) ? load4(hb + (size_t)j * dv + c0 + kk) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 2 * RM; ++i) *reinterpret_cast<float4*>(as + (r0 + 4 * i) * CORR_KPAD + kk) = qa[i];
#pragma unroll
        for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(bs + (r0 + 4 * i) * CORR_KPAD + kk) = hb4[i];
    } else {
        for (int idx = threadIdx.x; idx < 8 * RM * CORR_KCHUNK; idx += 256) {
            const int m = idx / CORR_KCHUNK, kk = idx % CORR_KCHUNK;
            as[m * CORR_KPAD + kk] = m < M && kk < cn ? qk[(size_t)m * dv + c0 + kk] : 0.f;
        }
        for (int idx = threadIdx.x; idx < 32 * CORR_KCHUNK; idx += 256) {
            const int t = idx / CORR_KCHUNK, kk = idx % CORR_KCHUNK, j = j0 + t;
            bs[t * CORR_KPAD + kk] = (j < T && kk < cn) ? to_f(hb[(size_t)j * dv + c0 + kk]) : 0.f;
        }
    }
    __syncthreads();
    // Thread (kg, mg, jg) takes features 64 kg .. of the chunk, query rows mg + 8 r and tokens jg + 8 u:
    // per four features 8 + RM 16-byte loads for 16 RM products (RM = 4 for M <= 32, else 8).
    const int kg = threadIdx.x >> 6, mg = (threadIdx.x >> 3) & 7, jg = threadIdx.x & 7;
    float acc[RM][4];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[r][u] = 0.f;
    const float* ap = as + mg * CORR_KPAD + 64 * kg;
    const float* bp = bs + jg * CORR_KPAD + 64 * kg;
#pragma unroll 4
    for (int k = 0; k < 64; k += 4) {
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const float4*>(bp + 8 * u * CORR_KPAD + k);
#pragma unroll
        for (int r = 0; r < RM; ++r) {
            const float4 q = *reinterpret_cast<const float4*>(ap + 8 * r * CORR_KPAD + k);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                acc[r][u] = fmaf(q.w, x[u].w, fmaf(q.z, x[u].z, fmaf(q.y, x[u].y, fmaf(q.x, x[u].x, acc[r][u]))));
        }
    }
    // The four feature groups' sums in order, through shared memory (over the staged operands).
    __syncthreads();
    float* sums = as;   // [4][8 RM rows][33]
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) sums[(kg * 8 * RM + mg + 8 * r) * 33 + jg + 8 * u] = acc[r][u];
    __syncthreads();
    for (int idx = threadIdx.x; idx < M * 32; idx += 256) {
        const int m = idx >> 5, u = idx & 31, j = j0 + u;
        float v = 0.f;
#pragma unroll
        for (int g = 0; g < 4; ++g) v += sums[(g * 8 * RM + m) * 33 + u];
        if (j < T) part[(((size_t)b * gridDim.y + kc) * M + m) * T + j] = v;
    }
}

// Block-wide reductions over 256 threads (8 warps), through `red` [8] in shared memory.
__device__ __forceinline__ float block_max256(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) r = fmaxf(r, red[w]);
    __syncthreads();
    return r;
}
__device__ __forceinline__ float block_sum256(float v, float* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) r += red[w];   // fixed order
    __syncthreads();
    return r;
}

// Row r = b M + m of the scores (one CTA of 256 threads per row): the nkc feature chunks added in
// order, then the softmax over its n tokens, written to s[r][.].
__global__ void __launch_bounds__(256) k_corr_softmax_sum(const float* __restrict__ part, float* __restrict__ s,
                                                          int M, int n, int nkc) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ float red[8];
    const int r = blockIdx.x, b = r / M, m = r - b * M;
    const float* p0 = part + ((size_t)b * nkc * M + m) * n;
    float* row = s + (size_t)r * n;
    float mx = -INFINITY;
    for (int j = threadIdx.x; j < n; j += 256) {
        float v = 0.f;
        for (int kc = 0; kc < nkc; ++kc) v += p0[(size_t)kc * M * n + j];
        row[j] = v;
        mx = fmaxf(mx, v);
    }
    mx = block_max256(mx, red);
    float den = 0.f;
    for (int j = threadIdx.x; j < n; j += 256) {
        const float e = expf(row[j] - mx);
        row[j] = e;
        den += e;
    }
    const float inv = 1.f / block_sum256(den, red);
    for (int j = threadIdx.x; j < n; j += 256) row[j] *= inv;
}

// Partial weighted sums over one chunk of CORR_TCHUNK tokens: part[b][tc][m][c] = sum over j in
// chunk tc of p[b][m][j] hv[b][j][c]. Grid (ceil(dv / 256), chunks, B): thread (cg, mg) =
// (tid mod 128, tid / 128) takes columns 2 cg, 2 cg + 1 of the CTA's 256 and rows mg RH .. + RH - 1
// (RH = 16 for M <= 32, else 32), token after token in order; the chunk's probabilities sit in
// shared memory transposed ([token][row], read as 16-byte broadcasts) and each token's two values
// come in one load, CORR_TB tokens' loads in flight together: two L2 round trips a chunk, on 208 CTAs at one
// request of 816 tokens. The token chunks are added in order by k_corr_wsum_reduce.
constexpr int CORR_TCHUNK = 32;
constexpr int CORR_TB = 16;     // tokens whose values a thread has in flight
constexpr int CORR_PTS = CORR_MAX_M + 4;   // row stride of the transposed probabilities

template <typename THV>
__device__ __forceinline__ float2 load2(const THV* p);
template <>
__device__ __forceinline__ float2 load2<float>(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
template <>
__device__ __forceinline__ float2 load2<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint32_t u = __ldg(reinterpret_cast<const unsigned int*>(p));
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
}

// PAIR: dv even and hv aligned to two elements, so a thread's two columns load together; else
// each value on its own (and a last odd column alone).
// At most 128 registers: with the loads of 16 tokens in flight the compiler takes 154 at RH = 32 and a second
// CTA no longer fits an SM (compress, us, unbounded and bounded: 1 request x 816 tokens 53 and 48, 8 x 1500
// 359 and 256, 32 x 1500 1440 and 963).
template <typename THV, int RH, bool PAIR>
__global__ void __launch_bounds__(256, 2) k_corr_wsum(const float* __restrict__ p, const THV* __restrict__ hv,
                                                   float* __restrict__ part, int M, int T, int dv) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ __align__(16) float pt[CORR_TCHUNK][CORR_PTS];
    const int b = blockIdx.z, tc = blockIdx.y;
    const int j0 = tc * CORR_TCHUNK, jn = min(CORR_TCHUNK, T - j0);
    {
        // Thread t loads token t mod 32 of rows t / 32, t / 32 + 8, .. (coalesced along the
        // tokens, all loads before the transposed stores); rows past M are zero.
        const int jj = threadIdx.x & 31, r0 = threadIdx.x >> 5;
        float pv[CORR_MAX_M / 8];
#pragma unroll
        for (int i = 0; i < CORR_MAX_M / 8; ++i) {
            const int r = r0 + 8 * i;
            pv[i] = (jj < jn && r < M) ? p[((size_t)b * M + r) * T + j0 + jj] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < CORR_MAX_M / 8; ++i) pt[jj][r0 + 8 * i] = pv[i];
    }
    __syncthreads();
    const int cg = threadIdx.x & 127, mg = threadIdx.x >> 7;
    const int c = blockIdx.x * 256 + 2 * cg;
    if (c >= dv) return;
    const int m0 = mg * RH;
    float acc[RH][2];
#pragma unroll
    for (int i = 0; i < RH; ++i) acc[i][0] = acc[i][1] = 0.f;
    const THV* hb = hv + ((size_t)b * T + j0) * dv + c;
    for (int jb = 0; jb < jn; jb += CORR_TB) {
        float2 hvv[CORR_TB];
#pragma unroll
        for (int u = 0; u < CORR_TB; ++u) {
            hvv[u] = make_float2(0.f, 0.f);
            if (jb + u < jn) {
                const THV* hp = hb + (size_t)(jb + u) * dv;
                if (PAIR) hvv[u] = load2(hp);
                else hvv[u] = make_float2(load1(hp), c + 1 < dv ? load1(hp + 1) : 0.f);
            }
        }
#pragma unroll
        for (int u = 0; u < CORR_TB; ++u) {
            const float4* prow = reinterpret_cast<const float4*>(&pt[jb + u][m0]);
#pragma unroll
            for (int i4 = 0; i4 < RH / 4; ++i4) {
                const float4 pw = prow[i4];
                const float w4[4] = {pw.x, pw.y, pw.z, pw.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[4 * i4 + e][0] = fmaf(w4[e], hvv[u].x, acc[4 * i4 + e][0]);
                    acc[4 * i4 + e][1] = fmaf(w4[e], hvv[u].y, acc[4 * i4 + e][1]);
                }
            }
        }
    }
    float* out = part + ((size_t)b * gridDim.y + tc) * M * dv + c;
#pragma unroll
    for (int i = 0; i < RH; ++i) {
        const int m = m0 + i;
        if (m >= M) continue;
        if (PAIR) {
            *reinterpret_cast<float2*>(out + (size_t)m * dv) = make_float2(acc[i][0], acc[i][1]);
        } else {
            out[(size_t)m * dv] = acc[i][0];
            if (c + 1 < dv) out[(size_t)m * dv + 1] = acc[i][1];
        }
    }
}

// g[b][m][c] = the ntc token-chunk partials added in order.
__global__ void k_corr_wsum_reduce(const float* __restrict__ part, float* __restrict__ g, int B, int M, int dv,
                                   int ntc) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const long long total = (long long)B * M * dv;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long b = idx / ((long long)M * dv), rest = idx - b * M * dv;
        const float* p0 = part + (size_t)b * ntc * M * dv + rest;
        float v = 0.f;
        for (int tc = 0; tc < ntc; ++tc) v += p0[(size_t)tc * M * dv];
        g[idx] = v;
    }
}

// y[(b n + k)][c] += pos[k][c] for b < B, k < n, c < d.
__global__ void k_corr_add_pos(float* __restrict__ y, const float* __restrict__ pos, int B, int n, int d) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const long long total = (long long)B * n * d;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(idx % d);
        const int k = (int)((idx / d) % n);
        y[idx] += pos[(size_t)k * d + c];
    }
}

// xj[(b T' + i)][0 .. d) = state[b][i][.], xj[(b T' + i)][d .. 2d) = summary[b][.].
__global__ void k_corr_join(const float* __restrict__ state, const float* __restrict__ summary,
                            float* __restrict__ xj, int B, int T, int d) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const long long total = (long long)B * T * 2 * d;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(idx % (2 * d));
        const long long r = idx / (2 * d);   // b T' + i
        const int b = (int)(r / T);
        xj[idx] = c < d ? state[r * d + c] : summary[(size_t)b * d + (c - d)];
    }
}

// conf[b] = w . mean_i u[b T' + i] + bias; one CTA of 256 threads per request.
__global__ void __launch_bounds__(256) k_corr_confidence(const float* __restrict__ u, const float* __restrict__ w,
                                                         const float* __restrict__ bias, float* __restrict__ conf,
                                                         int T, int d) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    __shared__ float red[8];
    const int b = blockIdx.x;
    float s = 0.f;
    for (int c = threadIdx.x; c < d; c += 256) {
        float m = 0.f;
        for (int i = 0; i < T; ++i) m += u[((size_t)b * T + i) * d + c];
        s = fmaf(w[c], m / (float)T, s);
    }
    s = block_sum256(s, red);
    if (threadIdx.x == 0) conf[b] = s + bias[0];
}

__global__ void k_corr_cast(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16_rn(src[i]);
}

// dst[r n + i] = src[i] for r < reps, i < n. src may be the start of dst: the first n elements are
// rewritten with their own values.
__global__ void k_corr_repeat(const float* src, float* dst, long long n, int reps) {
    // Launched with programmatic dependent launch: wait for the previous kernel's results, then
    // let the next kernel's CTAs be scheduled (they wait in turn).
    jpi::ptx::grid_dep_wait();
    jpi::ptx::grid_dep_launch();
    const long long total = n * reps;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x)
        dst[i] = src[i % n];
}

int grid_for(long long threads, int block = 256, int cap = 8192) {
    long long g = (threads + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

// Device copy of one block: q/k/v rows packed as [wq; wk; wv] ([3d][d]) with [bq; bk; bv].
struct BlockDev {
    float *ln1_w = nullptr, *ln1_b = nullptr;
    void* wqkv = nullptr;
    float* bqkv = nullptr;
    void* wo = nullptr;
    float* bo = nullptr;
    float *ln2_w = nullptr, *ln2_b = nullptr;
    void* w1 = nullptr;
    float* b1 = nullptr;
    void* w2 = nullptr;
    float* b2 = nullptr;
};

}  // namespace

struct jpi_corr_handle {
    jpi_corr_config cfg;
    bool bf16 = true;
    int num_sms = 0;   // persistent CTAs of the streamed products
    int d = 0, H = 0, Dh = 0, F = 0, dv = 0, Ti = 0, A = 0, Dm = 0, J = 0, B = 0, Tm = 0, M = 0;
    std::vector<void*> allocs;
    size_t bytes = 0;
    float* staging = nullptr;   // fp32 device staging for host weights
    size_t staging_elems = 0;

    // Weights.
    float* qf_query = nullptr;   // [T'][d]
    BlockDev qf_sa;
    float *qf_ln2_w = nullptr, *qf_ln2_b = nullptr;
    void *qf_ca_wq = nullptr, *qf_ca_wk = nullptr, *qf_ca_wv = nullptr, *qf_ca_wo = nullptr;
    float *qf_ca_bq = nullptr, *qf_ca_bv = nullptr, *qf_ca_bo = nullptr;
    float *qf_ln3_w = nullptr, *qf_ln3_b = nullptr, *qf_lnf_w = nullptr, *qf_lnf_b = nullptr;
    void *qf_w1 = nullptr, *qf_w2 = nullptr;
    float *qf_b1 = nullptr, *qf_b2 = nullptr;
    void *act_w1 = nullptr, *act_w2 = nullptr;
    float *act_b1 = nullptr, *act_b2 = nullptr, *act_pos = nullptr;
    BlockDev ab;
    void* fuse_w = nullptr;
    float* fuse_b = nullptr;
    std::vector<BlockDev> jb;
    float *head_ln_w = nullptr, *head_ln_b = nullptr;
    void* corr_w = nullptr;
    float *corr_b = nullptr, *conf_w = nullptr, *conf_b = nullptr;

    // Weight-only values computed at create time.
    float* x1b = nullptr;   // [B T'][d] the queries after their self-attention, per request slot
    float* qk = nullptr;    // [H T'][dv] cross-attention queries mapped into VLM space (scaled)

    // Activations (fp32).
    float *t1 = nullptr, *xa = nullptr, *ua = nullptr, *kva = nullptr;   // [B Dm][d], kva [B Dm][2d]
    float *ql = nullptr, *ol = nullptr, *xl = nullptr, *ul = nullptr;    // [B][d]
    float* hidl = nullptr;                                                // [B][F]
    float *xj = nullptr, *xf = nullptr, *u = nullptr, *qkv = nullptr, *o = nullptr;   // [B T'] rows
    float* hid = nullptr;                                                 // [B T'][F]
    float *sc = nullptr, *gs = nullptr;                                   // [B][M][Tm], [B][M][dv]
    float *scp = nullptr, *gsp = nullptr;   // partials: [B][dv / CORR_KCHUNK][M][Tm], [B][Tm / CORR_TCHUNK][M][dv], rounded up
    float* conf_scratch = nullptr;                                        // [B]

};

namespace {

template <typename T>
jpi_status corr_alloc(jpi_corr_handle* h, T** p, size_t count) {
    void* q = nullptr;
    const size_t bytes = count * sizeof(T);
    const cudaError_t e = cudaMalloc(&q, bytes ? bytes : 16);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return cfail(JPI_ERR_OOM, "cudaMalloc(%zu bytes) failed: %s", bytes, cudaGetErrorString(e));
    }
    h->allocs.push_back(q);
    h->bytes += bytes;
    *p = static_cast<T*>(q);
    return JPI_OK;
}

// Copies an fp32 tensor of n elements (host or device) to dst: fp32 as is, or rounded to bf16.
jpi_status put(jpi_corr_handle* h, bool on_device, void* dst, bool to_bf16, const float* src, size_t n,
               const char* name) {
    if (!src) return cfail(JPI_ERR_INVALID_ARG, "weight tensor %s is NULL", name);
    const float* dsrc = src;
    if (!on_device) {
        if (!to_bf16) {
            JPI_CUDA_TRY(cudaMemcpy(dst, src, n * sizeof(float), cudaMemcpyHostToDevice));
            return JPI_OK;
        }
        JPI_CUDA_TRY(cudaMemcpy(h->staging, src, n * sizeof(float), cudaMemcpyHostToDevice));
        dsrc = h->staging;
    }
    if (to_bf16) {
        k_corr_cast<<<grid_for((long long)n), 256>>>(dsrc, static_cast<__nv_bfloat16*>(dst), (long long)n);
        JPI_CUDA_TRY(cudaGetLastError());
    } else {
        JPI_CUDA_TRY(cudaMemcpy(dst, dsrc, n * sizeof(float), cudaMemcpyDeviceToDevice));
    }
    return JPI_OK;
}

// A weight matrix (stored bf16 or fp32) and a vector (fp32) of the handle.
jpi_status put_mat(jpi_corr_handle* h, bool dev, void** dst, const float* src, size_t n, const char* name) {
    if (h->bf16) {
        __nv_bfloat16* p = nullptr;
        JPI_TRY(corr_alloc(h, &p, n));
        *dst = p;
    } else {
        float* p = nullptr;
        JPI_TRY(corr_alloc(h, &p, n));
        *dst = p;
    }
    return put(h, dev, *dst, h->bf16, src, n, name);
}

jpi_status put_vec(jpi_corr_handle* h, bool dev, float** dst, const float* src, size_t n, const char* name) {
    JPI_TRY(corr_alloc(h, dst, n));
    return put(h, dev, *dst, false, src, n, name);
}

size_t tw_bytes(const jpi_corr_handle* h) { return h->bf16 ? 2 : 4; }
const void* tw_rows(const jpi_corr_handle* h, const void* base, size_t row, size_t in) {
    return static_cast<const char*>(base) + row * in * tw_bytes(h);
}

jpi_status put_block(jpi_corr_handle* h, bool dev, BlockDev* out, const jpi_corr_block& b, bool with_mlp,
                     const char* name) {
    const size_t d = (size_t)h->d, F = (size_t)h->F;
    char nm[64];
    auto N = [&](const char* f) {
        snprintf(nm, sizeof(nm), "%s.%s", name, f);
        return nm;
    };
    JPI_TRY(put_vec(h, dev, &out->ln1_w, b.ln1_w, d, N("ln1_w")));
    JPI_TRY(put_vec(h, dev, &out->ln1_b, b.ln1_b, d, N("ln1_b")));
    if (h->bf16) {
        __nv_bfloat16* p = nullptr;
        JPI_TRY(corr_alloc(h, &p, 3 * d * d));
        out->wqkv = p;
    } else {
        float* p = nullptr;
        JPI_TRY(corr_alloc(h, &p, 3 * d * d));
        out->wqkv = p;
    }
    char* wq = static_cast<char*>(out->wqkv);
    JPI_TRY(put(h, dev, wq, h->bf16, b.wq, d * d, N("wq")));
    JPI_TRY(put(h, dev, wq + d * d * tw_bytes(h), h->bf16, b.wk, d * d, N("wk")));
    JPI_TRY(put(h, dev, wq + 2 * d * d * tw_bytes(h), h->bf16, b.wv, d * d, N("wv")));
    JPI_TRY(corr_alloc(h, &out->bqkv, 3 * d));
    JPI_TRY(put(h, dev, out->bqkv, false, b.bq, d, N("bq")));
    JPI_TRY(put(h, dev, out->bqkv + d, false, b.bk, d, N("bk")));
    JPI_TRY(put(h, dev, out->bqkv + 2 * d, false, b.bv, d, N("bv")));
    JPI_TRY(put_mat(h, dev, &out->wo, b.wo, d * d, N("wo")));
    JPI_TRY(put_vec(h, dev, &out->bo, b.bo, d, N("bo")));
    if (with_mlp) {
        JPI_TRY(put_vec(h, dev, &out->ln2_w, b.ln2_w, d, N("ln2_w")));
        JPI_TRY(put_vec(h, dev, &out->ln2_b, b.ln2_b, d, N("ln2_b")));
        JPI_TRY(put_mat(h, dev, &out->w1, b.w1, F * d, N("w1")));
        JPI_TRY(put_vec(h, dev, &out->b1, b.b1, F, N("b1")));
        JPI_TRY(put_mat(h, dev, &out->w2, b.w2, d * F, N("w2")));
        JPI_TRY(put_vec(h, dev, &out->b2, b.b2, d, N("b2")));
    }
    return JPI_OK;
}

// ---------------------------------------------------------------- launchers

// Every kernel of a call is launched with programmatic dependent launch (each waits for its
// predecessor at its start), so a kernel's launch overlaps the previous kernel's tail. The calls
// enqueue their kernels on the caller's pointers: a captured graph needs every input copied in and every
// output copied out (10 us of a compress and 12 of a predict at batch 1), and the host's 26 launches take less
// time than the kernels run. A failed launch leaves its error for the cudaGetLastError check that follows.
template <typename... KArgs, typename... Args>
void pdl(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*k)(KArgs...), Args&&... args) {
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
    (void)cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

// Whether a product can stream its weights through shared memory (k_corr_linear_pipe): bf16 rows of
// 16-byte chunks up to LP_MAX_IN, 16-byte aligned activations.
bool pipe_ok(const jpi_corr_handle* h, const float* x, int ldx, const void* w, int in) {
    return h->bf16 && in % 8 == 0 && in <= LP_MAX_IN && ldx % 4 == 0 && ((uintptr_t)x & 15) == 0 &&
           ((uintptr_t)w & 15) == 0;
}
// Whether its LayerNorm form takes `rows` rows of the module's width: every CTA computes the rows'
// statistics, up to two rows per warp; more cost what the launch saved (predict, LayerNorm in the products and
// in launches of its own, us: 12 rows 135.4 and 142.7, 16 rows 146.9 and 151.3, 20 rows 178.7 and 177.2, 24
// rows 188.0 and 184.6).
bool ln_fused(const jpi_corr_handle* h, const float* x, int ldx, const void* w, int rows) {
    return pipe_ok(h, x, ldx, w, h->d) && h->d <= 2048 && rows <= 16;
}

// By persistent CTAs, one per SM at most (plus `extra` for the confidence head).
jpi_status launch_pipe(const jpi_corr_handle* h, cudaStream_t st, int mode, LinArgs a, int extra = 0) {
    const int groups = (a.out + LP_ROWS - 1) / LP_ROWS;
    a.lin_ctas = groups < h->num_sms ? groups : h->num_sms;
    const int nst = lp_stages(a.in);
    const size_t smem = (size_t)nst * LP_ROWS * a.in * 2;
    const dim3 grid(a.lin_ctas + extra), block(256);
    const bool split = a.in <= 1024 && a.rows > LP_XR;
    if (mode == LP_LN && split) pdl(st, grid, block, smem, k_corr_linear_pipe<4, LP_LN, 2>, a);
    else if (mode == LP_LN) pdl(st, grid, block, smem, k_corr_linear_pipe<4, LP_LN, 1>, a);
    else if (mode == LP_ATTN) pdl(st, grid, block, smem, k_corr_linear_pipe<4, LP_ATTN, 1>, a);
    else if (split) pdl(st, grid, block, smem, k_corr_linear_pipe<4, LP_PLAIN, 2>, a);
    else if (nst == 4) pdl(st, grid, block, smem, k_corr_linear_pipe<4, LP_PLAIN, 1>, a);
    else pdl(st, grid, block, smem, k_corr_linear_pipe<3, LP_PLAIN, 1>, a);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

// Arguments of y [rows][out] = act(x [rows][in] w^T + bias) + res.
LinArgs lin_args(const float* x, int ldx, const void* w, const float* bias, const float* res, int ldr, float* y, int ldy,
                 int rows, int in, int out, bool gelu) {
    LinArgs a = {};
    a.x = x;
    a.ldx = ldx;
    a.w = w;
    a.bias = bias;
    a.res = res;
    a.ldr = ldr;
    a.y = y;
    a.ldy = ldy;
    a.rows = rows;
    a.in = in;
    a.out = out;
    a.gelu = gelu ? 1 : 0;
    return a;
}

jpi_status linear(const jpi_corr_handle* h, cudaStream_t st, const float* x, int ldx, const void* w,
                  const float* bias, const float* res, int ldr, float* y, int ldy, int rows, int in,
                  int out, bool gelu, int hs_items = 0) {
    if (rows <= 0 || out <= 0) return JPI_OK;
    LinArgs a = lin_args(x, ldx, w, bias, res, ldr, y, ldy, rows, in, out, gelu);
    a.hs_items = hs_items;
    a.hs_heads = h->H;
    a.hs_dh = h->Dh;
    const bool vec = in % 4 == 0 && ldx % 4 == 0 && ((uintptr_t)x & 15) == 0 &&
                     ((uintptr_t)w & (h->bf16 ? 7 : 15)) == 0;
    if (hs_items == 0 && pipe_ok(h, x, ldx, w, in)) return launch_pipe(h, st, LP_PLAIN, a);
    // Other bf16 rows of 16-byte chunks: the streaming kernel, with 2 or 4 warps per output
    // feature while that keeps at least 256 inputs a warp and brings the launch towards 2048 warps.
    if (h->bf16 && in % 8 == 0 && ldx % 4 == 0 && ((uintptr_t)x & 15) == 0 && ((uintptr_t)w & 15) == 0) {
        int ks = 1;
        while (ks < 4 && (long long)out * ks < 2048 && in % (16 * ks) == 0 && in / (2 * ks) >= 256) ks *= 2;
        const int groups = (out + 8 / ks - 1) / (8 / ks);
        const int nb = groups < 4096 ? groups : 4096;
        if (ks == 4) pdl(st, dim3(nb), dim3(256), 0, k_corr_linear16<4>, a);
        else if (ks == 2) pdl(st, dim3(nb), dim3(256), 0, k_corr_linear16<2>, a);
        else pdl(st, dim3(nb), dim3(256), 0, k_corr_linear16<1>, a);
        JPI_CUDA_TRY(cudaGetLastError());
        return JPI_OK;
    }
    const int blocks = grid_for((long long)out * 32, 256, 4096);
    if (h->bf16) {
        if (vec) pdl(st, dim3(blocks), dim3(256), 0, k_corr_linear<__nv_bfloat16, true>, a);
        else pdl(st, dim3(blocks), dim3(256), 0, k_corr_linear<__nv_bfloat16, false>, a);
    } else {
        if (vec) pdl(st, dim3(blocks), dim3(256), 0, k_corr_linear<float, true>, a);
        else pdl(st, dim3(blocks), dim3(256), 0, k_corr_linear<float, false>, a);
    }
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

jpi_status layernorm(const jpi_corr_handle* h, cudaStream_t st, const float* x, int ldx, const float* g,
                     const float* b, float* y, int ldy, int rows) {
    if (rows <= 0) return JPI_OK;
    const bool vec = h->d % 4 == 0 && ldx % 4 == 0 && ldy % 4 == 0 &&
                     (((uintptr_t)x | (uintptr_t)y | (uintptr_t)g | (uintptr_t)b) & 15) == 0;
    if (vec)
        pdl(st, dim3(grid_for((long long)rows * 32)), dim3(256), 0, k_corr_layernorm<true>, x, ldx, g, b, y, ldy, rows, h->d,
                                                                           h->cfg.ln_eps);
    else
        pdl(st, dim3(grid_for((long long)rows * 32)), dim3(256), 0, k_corr_layernorm<false>, x, ldx, g, b, y, ldy, rows, h->d,
                                                                            h->cfg.ln_eps);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

// y = act(LN(x) w^T + bias) over rows of the module's width: one launch where ln_fused, else the
// LayerNorm into u first.
jpi_status ln_linear(const jpi_corr_handle* h, cudaStream_t st, const float* x, const float* g, const float* b, float* u,
                     const void* w, const float* bias, float* y, int rows, int out, bool gelu) {
    const int d = h->d;
    if (ln_fused(h, x, d, w, rows)) {
        LinArgs a = lin_args(x, d, w, bias, nullptr, 0, y, out, rows, d, out, gelu);
        a.ln_g = g;
        a.ln_b = b;
        a.ln_eps = h->cfg.ln_eps;
        return launch_pipe(h, st, LP_LN, a);
    }
    JPI_TRY(layernorm(h, st, x, d, g, b, u, d, rows));
    return linear(h, st, u, d, w, bias, nullptr, 0, y, out, rows, d, out, gelu);
}

jpi_status attention(const jpi_corr_handle* h, cudaStream_t st, const float* q, int ldq, const float* k,
                     int ldk, const float* v, int ldv, float* o, int ldo, int B, int nq, int nk) {
    AttnSmallArgs a;
    a.q = q;
    a.ldq = ldq;
    a.k = k;
    a.ldk = ldk;
    a.v = v;
    a.ldv = ldv;
    a.o = o;
    a.ldo = ldo;
    a.B = B;
    a.nq = nq;
    a.nk = nk;
    a.H = h->H;
    a.Dh = h->Dh;
    a.scale = 1.f / sqrtf((float)h->Dh);
    const long long warps = (long long)B * h->H * nq;
    pdl(st, dim3((int)((warps + 7) / 8)), dim3(256), 0, k_corr_attn, a);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

// One pre-LN block over `rows` rows of x (rows = B n, n tokens per request), in place.
jpi_status block(const jpi_corr_handle* h, cudaStream_t st, const BlockDev& w, float* x, int B, int n) {
    const int d = h->d, rows = B * n;
    JPI_TRY(ln_linear(h, st, x, w.ln1_w, w.ln1_b, h->u, w.wqkv, w.bqkv, h->qkv, rows, 3 * d, false));
    // Attention among four tokens goes into the output product for one request (every CTA computes it:
    // more requests take longer there than in a launch of their own; predict, in the product and in its own
    // launch, us: one request 92.1 and 92.8, two 108.2 and 102.6, three 144.8 and 135.5). Which kernels run must not
    // show in a request's result, so both ways compute the same sums.
    const bool four = n == LP_XR && (h->Dh & (h->Dh - 1)) == 0 && d <= 2048 && pipe_ok(h, h->qkv, 3 * d, w.wo, d);
    if (four && B == 1) {
        LinArgs a = lin_args(h->qkv, 3 * d, w.wo, w.bo, x, d, x, d, rows, d, d, false);
        a.att_heads_dh = h->Dh;
        a.att_scale = 1.f / sqrtf((float)h->Dh);
        JPI_TRY(launch_pipe(h, st, LP_ATTN, a));
    } else {
        if (four) {
            pdl(st, dim3(B), dim3(256), 0, k_corr_attn4, (const float*)h->qkv, h->o, d, h->Dh, 1.f / sqrtf((float)h->Dh));
            JPI_CUDA_TRY(cudaGetLastError());
        } else {
            JPI_TRY(attention(h, st, h->qkv, 3 * d, h->qkv + d, 3 * d, h->qkv + 2 * d, 3 * d, h->o, d, B, n, n));
        }
        JPI_TRY(linear(h, st, h->o, d, w.wo, w.bo, x, d, x, d, rows, d, d, false));
    }
    JPI_TRY(ln_linear(h, st, x, w.ln2_w, w.ln2_b, h->u, w.w1, w.b1, h->hid, rows, h->F, true));
    JPI_TRY(linear(h, st, h->hid, h->F, w.w2, w.b2, x, d, x, d, rows, h->F, d, false));
    return JPI_OK;
}

// Weight-only part of the compressor: x1 = q0 + SA(LN1 q0) for the learned queries q0 (one copy
// per request slot), and the cross-attention queries of LN2 x1 mapped into VLM space.
jpi_status prepare(jpi_corr_handle* h, cudaStream_t st) {
    const int d = h->d, T = h->Ti;
    const BlockDev& sa = h->qf_sa;
    JPI_TRY(layernorm(h, st, h->qf_query, d, sa.ln1_w, sa.ln1_b, h->u, d, T));
    JPI_TRY(linear(h, st, h->u, d, sa.wqkv, sa.bqkv, nullptr, 0, h->qkv, 3 * d, T, d, 3 * d, false));
    JPI_TRY(attention(h, st, h->qkv, 3 * d, h->qkv + d, 3 * d, h->qkv + 2 * d, 3 * d, h->o, d, 1, T, T));
    JPI_TRY(linear(h, st, h->o, d, sa.wo, sa.bo, h->qf_query, d, h->x1b, d, T, d, d, false));
    JPI_TRY(layernorm(h, st, h->x1b, d, h->qf_ln2_w, h->qf_ln2_b, h->u, d, T));
    JPI_TRY(linear(h, st, h->u, d, h->qf_ca_wq, h->qf_ca_bq, nullptr, 0, h->o, d, T, d, d, false));
    const dim3 grid((unsigned)((h->dv + 255) / 256), (unsigned)h->H);
    const float scale = 1.f / sqrtf((float)h->Dh);
    if (h->bf16)
        pdl(st, dim3(grid), dim3(256), 0, k_corr_qk<__nv_bfloat16>, h->o, static_cast<const __nv_bfloat16*>(h->qf_ca_wk),
                                                        h->qk, T, h->Dh, d, h->dv, scale);
    else
        pdl(st, dim3(grid), dim3(256), 0, k_corr_qk<float>, h->o, static_cast<const float*>(h->qf_ca_wk), h->qk, T, h->Dh,
                                               d, h->dv, scale);
    JPI_CUDA_TRY(cudaGetLastError());
    const long long n = (long long)T * d;
    pdl(st, dim3(grid_for(n * h->B)), dim3(256), 0, k_corr_repeat, h->x1b, h->x1b, n, h->B);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

jpi_status check_corr_config(const jpi_corr_config* c) {
    if (c->width < 32 || c->width % 32 || c->width > 16384)
        return cfail(JPI_ERR_INVALID_ARG, "width must be a multiple of 32 in [32, 16384]");
    if (c->head_dim < 32 || c->head_dim % 32 || c->head_dim > 256)
        return cfail(JPI_ERR_UNSUPPORTED, "head_dim must be a multiple of 32 and at most 256");
    if (c->n_heads < 1 || c->n_heads * c->head_dim != c->width)
        return cfail(JPI_ERR_INVALID_ARG, "n_heads * head_dim must equal width");
    if (c->mlp_dim < 1 || c->d_vlm < 1 || c->action_dim < 1)
        return cfail(JPI_ERR_INVALID_ARG, "mlp_dim, d_vlm and action_dim must be >= 1");
    if (c->n_items < 1 || c->n_items > JPI_MAX_CORRECTION)
        return cfail(JPI_ERR_UNSUPPORTED, "n_items must be in [1, %d]", JPI_MAX_CORRECTION);
    if (c->n_heads * c->n_items > CORR_MAX_M)
        return cfail(JPI_ERR_UNSUPPORTED, "n_heads * n_items must be at most %d", CORR_MAX_M);
    if (c->max_delta < 1 || c->max_delta > JPI_CORR_MAX_DELTA)
        return cfail(JPI_ERR_UNSUPPORTED, "max_delta must be in [1, %d]", JPI_CORR_MAX_DELTA);
    if (c->n_joint < 0 || c->n_joint > 8) return cfail(JPI_ERR_UNSUPPORTED, "n_joint must be in [0, 8]");
    if (c->max_batch < 1 || c->max_batch > 65535 || c->max_vlm_tokens < 1)
        return cfail(JPI_ERR_INVALID_ARG, "max_batch must be in [1, 65535] and max_vlm_tokens >= 1");
    if ((long long)c->max_batch * c->n_heads * c->n_items * c->max_vlm_tokens > (1ll << 31))
        return cfail(JPI_ERR_UNSUPPORTED, "max_batch * n_heads * n_items * max_vlm_tokens is too large");
    if (c->precision != JPI_BF16 && c->precision != JPI_FP32)
        return cfail(JPI_ERR_INVALID_ARG, "unknown precision %d", (int)c->precision);
    if (!(c->ln_eps >= 0.f)) return cfail(JPI_ERR_INVALID_ARG, "ln_eps must be >= 0");
    return JPI_OK;
}

jpi_status setup(jpi_corr_handle* h, const jpi_corr_config* c, const jpi_corr_weights* w) {
    h->cfg = *c;
    h->bf16 = c->precision == JPI_BF16;
    h->d = c->width;
    h->H = c->n_heads;
    h->Dh = c->head_dim;
    h->F = c->mlp_dim;
    h->dv = c->d_vlm;
    h->Ti = c->n_items;
    h->A = c->action_dim;
    h->Dm = c->max_delta;
    h->J = c->n_joint;
    h->B = c->max_batch;
    h->Tm = c->max_vlm_tokens;
    h->M = h->H * h->Ti;
    const size_t d = (size_t)h->d, F = (size_t)h->F, dv = (size_t)h->dv, T = (size_t)h->Ti;
    const size_t B = (size_t)h->B, Dm = (size_t)h->Dm, A = (size_t)h->A, M = (size_t)h->M;
    const bool dev = w->on_device != 0;
    if (!dev) {
        size_t m = d * d;
        for (size_t v : {F * d, d * dv, Dm * d, 2 * d * d, T * d, d * A}) m = v > m ? v : m;
        JPI_TRY(corr_alloc(h, &h->staging, m));
        h->staging_elems = m;
    }

    // Q-Former compressor.
    JPI_TRY(put_vec(h, dev, &h->qf_query, w->qf_query, T * d, "qf_query"));
    JPI_TRY(put_block(h, dev, &h->qf_sa, w->qf_sa, false, "qf_sa"));
    JPI_TRY(put_vec(h, dev, &h->qf_ln2_w, w->qf_ln2_w, d, "qf_ln2_w"));
    JPI_TRY(put_vec(h, dev, &h->qf_ln2_b, w->qf_ln2_b, d, "qf_ln2_b"));
    JPI_TRY(put_mat(h, dev, &h->qf_ca_wq, w->qf_ca_wq, d * d, "qf_ca_wq"));
    JPI_TRY(put_vec(h, dev, &h->qf_ca_bq, w->qf_ca_bq, d, "qf_ca_bq"));
    JPI_TRY(put_mat(h, dev, &h->qf_ca_wk, w->qf_ca_wk, d * dv, "qf_ca_wk"));
    // qf_ca_bk adds the same amount to every score of a query; softmax cancels it.
    JPI_TRY(put_mat(h, dev, &h->qf_ca_wv, w->qf_ca_wv, d * dv, "qf_ca_wv"));
    JPI_TRY(put_vec(h, dev, &h->qf_ca_bv, w->qf_ca_bv, d, "qf_ca_bv"));
    JPI_TRY(put_mat(h, dev, &h->qf_ca_wo, w->qf_ca_wo, d * d, "qf_ca_wo"));
    JPI_TRY(put_vec(h, dev, &h->qf_ca_bo, w->qf_ca_bo, d, "qf_ca_bo"));
    JPI_TRY(put_vec(h, dev, &h->qf_ln3_w, w->qf_ln3_w, d, "qf_ln3_w"));
    JPI_TRY(put_vec(h, dev, &h->qf_ln3_b, w->qf_ln3_b, d, "qf_ln3_b"));
    JPI_TRY(put_mat(h, dev, &h->qf_w1, w->qf_mlp_w1, F * d, "qf_mlp_w1"));
    JPI_TRY(put_vec(h, dev, &h->qf_b1, w->qf_mlp_b1, F, "qf_mlp_b1"));
    JPI_TRY(put_mat(h, dev, &h->qf_w2, w->qf_mlp_w2, d * F, "qf_mlp_w2"));
    JPI_TRY(put_vec(h, dev, &h->qf_b2, w->qf_mlp_b2, d, "qf_mlp_b2"));
    JPI_TRY(put_vec(h, dev, &h->qf_lnf_w, w->qf_lnf_w, d, "qf_lnf_w"));
    JPI_TRY(put_vec(h, dev, &h->qf_lnf_b, w->qf_lnf_b, d, "qf_lnf_b"));
    // Action branch, join, joint blocks, heads.
    JPI_TRY(put_mat(h, dev, &h->act_w1, w->act_w1, d * A, "act_w1"));
    JPI_TRY(put_vec(h, dev, &h->act_b1, w->act_b1, d, "act_b1"));
    JPI_TRY(put_mat(h, dev, &h->act_w2, w->act_w2, d * d, "act_w2"));
    JPI_TRY(put_vec(h, dev, &h->act_b2, w->act_b2, d, "act_b2"));
    JPI_TRY(put_vec(h, dev, &h->act_pos, w->act_pos, Dm * d, "act_pos"));
    JPI_TRY(put_block(h, dev, &h->ab, w->ab, true, "ab"));
    JPI_TRY(put_mat(h, dev, &h->fuse_w, w->fuse_w, d * 2 * d, "fuse_w"));
    JPI_TRY(put_vec(h, dev, &h->fuse_b, w->fuse_b, d, "fuse_b"));
    h->jb.resize((size_t)h->J);
    for (int i = 0; i < h->J; ++i) {
        char nm[16];
        snprintf(nm, sizeof(nm), "jb%d", i);
        JPI_TRY(put_block(h, dev, &h->jb[(size_t)i], w->jb[i], true, nm));
    }
    JPI_TRY(put_vec(h, dev, &h->head_ln_w, w->head_ln_w, d, "head_ln_w"));
    JPI_TRY(put_vec(h, dev, &h->head_ln_b, w->head_ln_b, d, "head_ln_b"));
    JPI_TRY(put_mat(h, dev, &h->corr_w, w->corr_w, d * d, "corr_w"));
    JPI_TRY(put_vec(h, dev, &h->corr_b, w->corr_b, d, "corr_b"));
    JPI_TRY(put_vec(h, dev, &h->conf_w, w->conf_w, d, "conf_w"));
    JPI_TRY(put_vec(h, dev, &h->conf_b, w->conf_b, 1, "conf_b"));

    // Weight-only values and activations.
    JPI_TRY(corr_alloc(h, &h->x1b, B * T * d));
    JPI_TRY(corr_alloc(h, &h->qk, M * dv));
    JPI_TRY(corr_alloc(h, &h->t1, B * Dm * d));
    JPI_TRY(corr_alloc(h, &h->xa, B * Dm * d));
    JPI_TRY(corr_alloc(h, &h->ua, B * Dm * d));
    JPI_TRY(corr_alloc(h, &h->kva, B * Dm * 2 * d));
    JPI_TRY(corr_alloc(h, &h->ql, B * d));
    JPI_TRY(corr_alloc(h, &h->ol, B * d));
    JPI_TRY(corr_alloc(h, &h->xl, B * d));
    JPI_TRY(corr_alloc(h, &h->ul, B * d));
    JPI_TRY(corr_alloc(h, &h->hidl, B * F));
    JPI_TRY(corr_alloc(h, &h->xj, B * T * 2 * d));
    JPI_TRY(corr_alloc(h, &h->xf, B * T * d));
    JPI_TRY(corr_alloc(h, &h->u, B * T * d));
    JPI_TRY(corr_alloc(h, &h->qkv, B * T * 3 * d));
    JPI_TRY(corr_alloc(h, &h->o, B * T * d));
    JPI_TRY(corr_alloc(h, &h->hid, B * T * F));
    JPI_TRY(corr_alloc(h, &h->sc, B * M * (size_t)h->Tm));
    JPI_TRY(corr_alloc(h, &h->gs, B * M * dv));
    JPI_TRY(corr_alloc(h, &h->scp, B * (size_t)((dv + CORR_KCHUNK - 1) / CORR_KCHUNK) * M * h->Tm));
    JPI_TRY(corr_alloc(h, &h->gsp, B * (size_t)((h->Tm + CORR_TCHUNK - 1) / CORR_TCHUNK) * M * dv));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<float, true, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<float, true, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<float, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<float, false, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<__nv_bfloat16, true, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<__nv_bfloat16, true, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<__nv_bfloat16, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_scores<__nv_bfloat16, false, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CORR_SCORES_SMEM));
    for (auto k : {k_corr_linear_pipe<4, LP_PLAIN, 1>, k_corr_linear_pipe<4, LP_PLAIN, 2>, k_corr_linear_pipe<4, LP_LN, 1>,
                   k_corr_linear_pipe<4, LP_LN, 2>, k_corr_linear_pipe<4, LP_ATTN, 1>})
        JPI_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * LP_ROWS * 2048 * 2));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_corr_linear_pipe<3, LP_PLAIN, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      3 * LP_ROWS * LP_MAX_IN * 2));
    {
        int dev = 0;
        JPI_CUDA_TRY(cudaGetDevice(&dev));
        JPI_CUDA_TRY(cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    JPI_TRY(corr_alloc(h, &h->conf_scratch, B));

    JPI_TRY(prepare(h, nullptr));
    JPI_CUDA_TRY(cudaStreamSynchronize(nullptr));
    return JPI_OK;
}

}  // namespace

namespace {

// The compressor's kernel sequence on `st`: hvlm [batch][n_tokens][dv] -> out [batch][T'][d].
jpi_status enqueue_compress(jpi_corr_handle* h, const void* hvlm, int vlm_is_fp32, int batch, int n_tokens,
                            float* out, cudaStream_t st) {
    const int d = h->d, T = h->Ti, M = h->M, dv = h->dv, rows = batch * T;
    const int nkc = (dv + CORR_KCHUNK - 1) / CORR_KCHUNK, ntc = (n_tokens + CORR_TCHUNK - 1) / CORR_TCHUNK;
    const dim3 gs((unsigned)((n_tokens + 31) / 32), (unsigned)nkc, (unsigned)batch);
    const dim3 gw((unsigned)((dv + 255) / 256), (unsigned)ntc, (unsigned)batch);
    const int red_grid = grid_for((long long)batch * M * dv);
    if (vlm_is_fp32) {
        const float* hv = static_cast<const float*>(hvlm);
        if (dv % 4 == 0 && ((uintptr_t)hv & 15) == 0)
            pdl(st, dim3(gs), dim3(256), CORR_SCORES_SMEM, M <= 32 ? k_corr_scores<float, true, 4> : k_corr_scores<float, true, 8>, h->qk, hv, h->scp, M, n_tokens, dv);
        else
            pdl(st, dim3(gs), dim3(256), CORR_SCORES_SMEM, M <= 32 ? k_corr_scores<float, false, 4> : k_corr_scores<float, false, 8>, h->qk, hv, h->scp, M, n_tokens, dv);
        pdl(st, dim3(batch * M), dim3(256), 0, k_corr_softmax_sum, h->scp, h->sc, M, n_tokens, nkc);
        const bool pair = dv % 2 == 0 && ((uintptr_t)hv & 7) == 0;
        if (M <= 32) {
            if (pair) pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<float, 16, true>, h->sc, hv, h->gsp, M, n_tokens, dv);
            else pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<float, 16, false>, h->sc, hv, h->gsp, M, n_tokens, dv);
        } else {
            if (pair) pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<float, 32, true>, h->sc, hv, h->gsp, M, n_tokens, dv);
            else pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<float, 32, false>, h->sc, hv, h->gsp, M, n_tokens, dv);
        }
    } else {
        const __nv_bfloat16* hv = static_cast<const __nv_bfloat16*>(hvlm);
        if (dv % 4 == 0 && ((uintptr_t)hv & 7) == 0)
            pdl(st, dim3(gs), dim3(256), CORR_SCORES_SMEM, M <= 32 ? k_corr_scores<__nv_bfloat16, true, 4> : k_corr_scores<__nv_bfloat16, true, 8>, h->qk, hv, h->scp, M, n_tokens, dv);
        else
            pdl(st, dim3(gs), dim3(256), CORR_SCORES_SMEM, M <= 32 ? k_corr_scores<__nv_bfloat16, false, 4> : k_corr_scores<__nv_bfloat16, false, 8>, h->qk, hv, h->scp, M, n_tokens, dv);
        pdl(st, dim3(batch * M), dim3(256), 0, k_corr_softmax_sum, h->scp, h->sc, M, n_tokens, nkc);
        const bool pair = dv % 2 == 0 && ((uintptr_t)hv & 3) == 0;
        if (M <= 32) {
            if (pair) pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<__nv_bfloat16, 16, true>, h->sc, hv, h->gsp, M, n_tokens, dv);
            else pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<__nv_bfloat16, 16, false>, h->sc, hv, h->gsp, M, n_tokens, dv);
        } else {
            if (pair) pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<__nv_bfloat16, 32, true>, h->sc, hv, h->gsp, M, n_tokens, dv);
            else pdl(st, dim3(gw), dim3(256), 0, k_corr_wsum<__nv_bfloat16, 32, false>, h->sc, hv, h->gsp, M, n_tokens, dv);
        }
    }
    pdl(st, dim3(red_grid), dim3(256), 0, k_corr_wsum_reduce, h->gsp, h->gs, batch, M, dv, ntc);
    JPI_CUDA_TRY(cudaGetLastError());
    // out_hi = W_v,h g_hi + b_v (head-select rows of gs), then the output projection onto the
    // queries' residual, the MLP, and the output LayerNorm.
    JPI_TRY(linear(h, st, h->gs, dv, h->qf_ca_wv, h->qf_ca_bv, nullptr, 0, h->o, d, rows, dv, d, false, T));
    JPI_TRY(linear(h, st, h->o, d, h->qf_ca_wo, h->qf_ca_bo, h->x1b, d, h->xf, d, rows, d, d, false));
    JPI_TRY(ln_linear(h, st, h->xf, h->qf_ln3_w, h->qf_ln3_b, h->u, h->qf_w1, h->qf_b1, h->hid, rows, h->F, true));
    JPI_TRY(linear(h, st, h->hid, h->F, h->qf_w2, h->qf_b2, h->xf, d, h->xf, d, rows, h->F, d, false));
    JPI_TRY(layernorm(h, st, h->xf, d, h->qf_lnf_w, h->qf_lnf_b, out, d, rows));
    return JPI_OK;
}

// f_corr's kernel sequence on `st`: state, actions -> out [batch][T'][d], conf [batch].
jpi_status enqueue_predict(jpi_corr_handle* h, const float* state, const float* actions, int batch, int delta,
                           float* out, float* conf, cudaStream_t st) {
    const int d = h->d, T = h->Ti, F = h->F, ra = batch * delta, rows = batch * T;
    const BlockDev& ab = h->ab;
    // Action tokens: MLP, plus the position row of each action.
    JPI_TRY(linear(h, st, actions, h->A, h->act_w1, h->act_b1, nullptr, 0, h->t1, d, ra, h->A, d, true));
    if (pipe_ok(h, h->t1, d, h->act_w2, d)) {
        LinArgs a = lin_args(h->t1, d, h->act_w2, h->act_b2, h->act_pos, d, h->xa, d, ra, d, d, false);
        a.res_mod = delta;
        JPI_TRY(launch_pipe(h, st, LP_PLAIN, a));
    } else {
        JPI_TRY(linear(h, st, h->t1, d, h->act_w2, h->act_b2, nullptr, 0, h->xa, d, ra, d, d, false));
        pdl(st, dim3(grid_for((long long)ra * d)), dim3(256), 0, k_corr_add_pos, h->xa, h->act_pos, batch, delta, d);
        JPI_CUDA_TRY(cudaGetLastError());
    }
    // Block ab, kept at the last action of each request only: keys and values of every action,
    // the query, attention output, residual and MLP of the last.
    const size_t last = (size_t)(delta - 1) * d;
    const bool abln = ln_fused(h, h->xa, d, ab.wqkv, ra);
    if (!abln) JPI_TRY(layernorm(h, st, h->xa, d, ab.ln1_w, ab.ln1_b, h->ua, d, ra));
    const float* uin = abln ? h->xa : h->ua;
    if (pipe_ok(h, uin, d, ab.wqkv, d)) {
        // One product: its first d features (the queries) over the last actions, the rest over all.
        LinArgs a = lin_args(uin, d, ab.wqkv, ab.bqkv, nullptr, 0, h->kva - d, 2 * d, ra, d, 3 * d, false);
        a.seg_out = d;
        a.seg_rows = batch;
        a.seg_x = uin + last;
        a.seg_ldx = delta * d;
        a.seg_y = h->ql;
        a.seg_ldy = d;
        a.ln_g = ab.ln1_w;
        a.ln_b = ab.ln1_b;
        a.ln_eps = h->cfg.ln_eps;
        JPI_TRY(launch_pipe(h, st, abln ? LP_LN : LP_PLAIN, a));
    } else {
        JPI_TRY(linear(h, st, h->ua, d, tw_rows(h, ab.wqkv, (size_t)d, (size_t)d), ab.bqkv + d, nullptr, 0, h->kva,
                       2 * d, ra, d, 2 * d, false));
        JPI_TRY(linear(h, st, h->ua + last, delta * d, ab.wqkv, ab.bqkv, nullptr, 0, h->ql, d, batch, d, d, false));
    }
    JPI_TRY(attention(h, st, h->ql, d, h->kva, 2 * d, h->kva + d, 2 * d, h->ol, d, batch, 1, delta));
    JPI_TRY(linear(h, st, h->ol, d, ab.wo, ab.bo, h->xa + last, delta * d, h->xl, d, batch, d, d, false));
    JPI_TRY(ln_linear(h, st, h->xl, ab.ln2_w, ab.ln2_b, h->ul, ab.w1, ab.b1, h->hidl, batch, F, true));
    JPI_TRY(linear(h, st, h->hidl, F, ab.w2, ab.b2, h->xl, d, h->xl, d, batch, F, d, false));
    // Join: [compressed token ; action summary] projected back to the module width.
    if (pipe_ok(h, state, d, h->fuse_w, 2 * d)) {
        LinArgs a = lin_args(state, d, h->fuse_w, h->fuse_b, nullptr, 0, h->xf, d, rows, 2 * d, d, false);
        a.join = d;
        a.x2 = h->xl;
        a.x2_div = T;
        a.ldx2 = d;
        JPI_TRY(launch_pipe(h, st, LP_PLAIN, a));
    } else {
        pdl(st, dim3(grid_for((long long)rows * 2 * d)), dim3(256), 0, k_corr_join, state, h->xl, h->xj, batch, T, d);
        JPI_CUDA_TRY(cudaGetLastError());
        JPI_TRY(linear(h, st, h->xj, 2 * d, h->fuse_w, h->fuse_b, nullptr, 0, h->xf, d, rows, 2 * d, d, false));
    }
    for (int i = 0; i < h->J; ++i) JPI_TRY(block(h, st, h->jb[(size_t)i], h->xf, batch, T));
    // Heads.
    if (ln_fused(h, h->xf, d, h->corr_w, rows)) {
        LinArgs a = lin_args(h->xf, d, h->corr_w, h->corr_b, nullptr, 0, out, d, rows, d, d, false);
        a.ln_g = h->head_ln_w;
        a.ln_b = h->head_ln_b;
        a.ln_eps = h->cfg.ln_eps;
        a.conf_items = T;
        a.conf_w = h->conf_w;
        a.conf_b = h->conf_b;
        a.conf = conf;
        return launch_pipe(h, st, LP_LN, a, batch);
    }
    JPI_TRY(layernorm(h, st, h->xf, d, h->head_ln_w, h->head_ln_b, h->u, d, rows));
    JPI_TRY(linear(h, st, h->u, d, h->corr_w, h->corr_b, nullptr, 0, out, d, rows, d, d, false));
    pdl(st, dim3(batch), dim3(256), 0, k_corr_confidence, h->u, h->conf_w, h->conf_b, conf, T, d);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

}  // namespace

extern "C" {

JPI_API jpi_status jpi_corr_create(const jpi_corr_config* cfg, const jpi_corr_weights* w,
                                   jpi_corr_handle** out) {
    jpi::clear_error();
    if (!out) return cfail(JPI_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!cfg || !w) return cfail(JPI_ERR_INVALID_ARG, "config or weights is NULL");
    JPI_TRY(check_corr_config(cfg));
    if (cfg->n_joint > 0 && !w->jb) return cfail(JPI_ERR_INVALID_ARG, "joint blocks (jb) are NULL");
    jpi_corr_handle* h = new (std::nothrow) jpi_corr_handle();
    if (!h) return cfail(JPI_ERR_OOM, "host allocation failed");
    const jpi_status s = setup(h, cfg, w);
    if (s != JPI_OK) {
        cudaStreamSynchronize(nullptr);   // let any conversion in flight finish before its buffers go
        cudaGetLastError();
        for (void* p : h->allocs) cudaFree(p);
        delete h;
        return s;
    }
    *out = h;
    return JPI_OK;
}

JPI_API jpi_status jpi_corr_destroy(jpi_corr_handle* h) {
    jpi::clear_error();
    if (!h) return JPI_OK;
    cudaDeviceSynchronize();
    for (void* p : h->allocs) cudaFree(p);
    cudaGetLastError();
    delete h;
    return JPI_OK;
}

JPI_API jpi_status jpi_corr_compress(jpi_corr_handle* h, const void* h_vlm, int vlm_is_fp32, int batch,
                                     int n_tokens, float* out_state, void* stream) {
    jpi::clear_error();
    if (!h) return cfail(JPI_ERR_INVALID_ARG, "handle is NULL");
    if (!h_vlm || !out_state) return cfail(JPI_ERR_INVALID_ARG, "NULL input or output");
    if (batch < 1 || n_tokens < 1) return cfail(JPI_ERR_INVALID_ARG, "batch and n_tokens must be >= 1");
    if (batch > h->B || n_tokens > h->Tm)
        return cfail(JPI_ERR_SHAPE, "batch %d / n_tokens %d exceed the maxima %d / %d", batch, n_tokens, h->B,
                     h->Tm);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return enqueue_compress(h, h_vlm, vlm_is_fp32, batch, n_tokens, out_state, st);
}

JPI_API jpi_status jpi_corr_predict(jpi_corr_handle* h, const float* state, const float* actions, int batch,
                                    int delta, float* out_state, float* out_confidence, void* stream) {
    jpi::clear_error();
    if (!h) return cfail(JPI_ERR_INVALID_ARG, "handle is NULL");
    if (!state || !actions || !out_state) return cfail(JPI_ERR_INVALID_ARG, "NULL input or output");
    if (batch < 1 || delta < 1) return cfail(JPI_ERR_INVALID_ARG, "batch and delta must be >= 1");
    if (batch > h->B || delta > h->Dm)
        return cfail(JPI_ERR_SHAPE, "batch %d / delta %d exceed the maxima %d / %d", batch, delta, h->B, h->Dm);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return enqueue_predict(h, state, actions, batch, delta, out_state, out_confidence ? out_confidence : h->conf_scratch,
                           st);
}

JPI_API jpi_status jpi_corr_memory_usage(const jpi_corr_handle* h, long long* bytes) {
    jpi::clear_error();
    if (!h || !bytes) return cfail(JPI_ERR_INVALID_ARG, "handle or bytes is NULL");
    *bytes = (long long)h->bytes;
    return JPI_OK;
}

}  // extern "C"
