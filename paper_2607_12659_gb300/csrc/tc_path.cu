// Tensor-core path of the bf16 expert layers: tcgen05 GEMMs fed by bulk tensor copies.
//
// Every projection of a layer is a skinny GEMM Y[tokens][out] = X[tokens][K] W[out][K]^T with
// tokens = batch x (chunk + 1) (51 at batch 1). Three kernels share it by token count (the rules are
// at the thresholds in tc_prepare and at rows_narrow, big_split and resid_rows below):
//   gemm_kernel.cuh  few tokens: "swap-AB", a 128-row tile of W as the A operand (M = 128), 64 tokens
//                    of X as B (N = 64), the fp32 product in TMEM; the K range of a weight tile split
//                    over the CTAs of a cluster, which exchange fp16 partials through distributed
//                    shared memory and sum them in a fixed rank order;
//   gemm_rows.cuh    many tokens: tokens on the MMA's rows, 128 x 256 or 128 x 128 tiles over the
//                    whole K range;
//   gemm_big.cuh     O and down at token counts whose tiles would leave SMs idle: 128 x 128 tiles
//                    with a K split over a cluster, fp32 partials.
// Each loads its weight blocks with bulk tensor copies before it waits on the previous kernel
// (weights do not depend on it), then its X blocks the same way from the bf16 activation the previous
// op left in global memory. The RMSNorm-fed kinds read the scaled residual stream and apply 1 / rms
// and the norm's shift in the epilogue. Epilogues: rotary encoding + scatter into the query buffer and
// KV store (QKV), GeGLU (gate/up), or the gated residual update of the fp32 stream with the next norm's
// bf16 operand and per-token sums of squares (O, down).

#include "tc_path.h"
#include "ptx.h"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstdlib>
#include <vector>

namespace jpi {
namespace {

constexpr int NT = 64;                         // tokens per MMA (N)
constexpr int TILE_ROWS = 128;                 // weight rows per tile (M)
constexpr int KBLK = 64;                       // K elements per block: one 128-byte swizzle row
constexpr int TILE_BYTES = TILE_ROWS * KBLK * 2;
constexpr int XBLK_BYTES = NT * KBLK * 2;
constexpr int PART_BYTES = TILE_ROWS * NT * 2;  // fp16 partial of one tile (128-byte rows)
constexpr int GEMM_THREADS = 256;
constexpr uint64_t WAIT_LIMIT_NS = 200ull * 1000 * 1000;   // 0.2 s

enum GemmKind { G_QKV = 0, G_O = 1, G_GU = 2, G_DOWN = 3 };

struct GemmArgs {
    int Mt, K, nkb, kpb, splits;
    int ntiles;              // weight tiles (large-M kernel: tiles walked by the persistent CTAs)
    // RMSNorm-fed projections (QKV, gate/up): W u = rinv * (W xs) + W beta, with xs = (1 + sigma) h
    // and beta packed as tiles of 63 tokens + 1 beta row by the producer of h, and rinv from the
    // per-token sums of squares it left.
    const float* ss;         // [nslot][ss_ld]: sums of h^2 over disjoint feature ranges
    int nslot, ss_ld;
    float eps, inv_w;
    // Gated residual epilogue (O, down).
    float* hres;
    __nv_bfloat16* xs;       // operand of the next norm-fed GEMM (null: none follows)
    const float* sigma_next; // that norm's scale and shift
    const float* beta_next;
    const float* gamma;
    float* ss_out;           // slot (tile * splits + rank): this CTA's features
    int W;
    // QKV epilogue.
    __nv_bfloat16* q;
    __nv_bfloat16* kst;
    __nv_bfloat16* vst;
    const float2* rope;
    int S, H, D, P, kv_rows;
    // GeGLU epilogue.
    __nv_bfloat16* z;
    int F;
    int* err;
};

// GELU, tanh form, with the hardware tanh (PTX tanh.approx.f32, relative error about 2^-11): the
// product it enters is rounded to bf16 (2^-9) right after, and the fp32 verification mode runs the
// CUDA-core kernels with the library tanh.
__device__ __forceinline__ float gelu_tanh(float y) {
    const float k0 = 0.7978845608028654f;   // sqrt(2 / pi)
    float th;
    asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(k0 * (y + 0.044715f * y * y * y)));
    return 0.5f * y * (1.f + th);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_half2(uint32_t v) {
    __half2 b = *reinterpret_cast<__half2*>(&v);
    return __half22float2(b);
}

__device__ __forceinline__ void set_device_error(int* err, int code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ float f4get(const float4& v, int e) {
    return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w;
}
__device__ __forceinline__ float4 half4_to_float4(uint2 v) {
    const float2 lo = __half22float2(*reinterpret_cast<__half2*>(&v.x));
    const float2 hi = __half22float2(*reinterpret_cast<__half2*>(&v.y));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Shared-memory layout of one GEMM CTA (byte offsets from the 1024-aligned base).
struct GemmSmem {
    int x, recv, misc, ssred, bars, total;
};
__host__ __device__ __forceinline__ GemmSmem gemm_layout(int kpb, int splits, bool norm_in) {
    GemmSmem L;
    const int xbytes = kpb * XBLK_BYTES > PART_BYTES ? kpb * XBLK_BYTES : PART_BYTES;
    const int ssred_bytes = 2 * NT * (int)sizeof(float);
    L.x = kpb * TILE_BYTES;
    L.recv = L.x + xbytes;
    L.misc = L.recv + (splits - 1) * (TILE_ROWS / splits) * NT * 2;
    int end = L.misc + (norm_in ? 4 * NT * (int)sizeof(float) : 0);   // ss partials + rinv
    if (norm_in) {
        L.ssred = L.misc;                               // unused by the norm-fed kinds
    } else if (xbytes >= PART_BYTES + ssred_bytes) {
        L.ssred = L.x + PART_BYTES;                     // X blocks are dead once the MMA is done
    } else {
        L.ssred = end;
        end += ssred_bytes;
    }
    L.bars = (end + 7) & ~7;
    L.total = L.bars + 64;   // 4 mbarriers, the TMEM address, the error flag
    return L;
}

#include "gemm_kernel.cuh"
#include "gemm_big.cuh"
#include "gemm_rows.cuh"

// ---------------------------------------------------------------------------------------------
// Host side: packing, plans, tensor maps, launches.

size_t gemm_smem(int kpb, int splits, bool norm_in) {
    return 1024 + (size_t)gemm_layout(kpb, splits, norm_in).total;
}

// Chooses the K blocks per CTA: one wave on the device, then at most 8 CTAs per cluster (each
// extra rank adds two pushes to every CTA's exchange and a slice to every owner's sum, which
// measured slower than streaming more weight per CTA), then little weight per SM, then shared
// memory small enough (<= 113 KB) for two CTAs per SM.
bool make_plan(int rows, int K, int max_cluster, int num_sms, bool norm_in, GemmPlan* out) {
    if (rows % TILE_ROWS || K % KBLK) return false;
    GemmPlan best;
    long best_score = -1;
    const int ntiles = rows / TILE_ROWS, nkb = K / KBLK;
    for (int kpb = 1; kpb <= 8; kpb *= 2) {
        if (nkb % kpb) continue;
        const int splits = nkb / kpb;
        if (splits > std::min(max_cluster, MAX_SPLIT_K) || 64 % splits) continue;
        const size_t smem = gemm_smem(kpb, splits, norm_in);
        if (smem > 227 * 1024) continue;
        const int res = std::min(2, (int)((228 * 1024) / (smem + 1024)));
        const int ctas = ntiles * splits;
        const long waves = (ctas + (long)num_sms * res - 1) / ((long)num_sms * res);
        const long per_sm = (ctas + num_sms - 1) / num_sms;
        const long score = waves * 10000 + std::max(splits - 8, 0) * 100 + per_sm * kpb * 10 +
                           (smem > 113 * 1024 ? 5 : 0) + (ctas > num_sms ? 1 : 0);
        if (best_score < 0 || score < best_score) {
            best_score = score;
            best.rows = rows; best.K = K; best.ntiles = ntiles; best.nkb = nkb; best.kpb = kpb;
            best.splits = splits; best.ctas = ctas; best.smem = smem;
        }
    }
    if (best_score < 0) return false;
    *out = best;
    return true;
}

// fp32 [rows][K] -> bf16 tiles; source row s lands on tiled row dest_row[s] (identity if null).
__global__ void k_pack_tiles(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                             const int* __restrict__ dest_row, int rows, int K) {
    const int nkb = K / KBLK;
    const long long total = (long long)rows * K;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(i / K), k = (int)(i % K);
        const int R = dest_row ? dest_row[s] : s;
        const size_t o = ((size_t)(R / TILE_ROWS) * nkb + k / KBLK) * (TILE_ROWS * KBLK) +
                         (size_t)(R % TILE_ROWS) * KBLK + (k % KBLK);
        dst[o] = __float2bfloat16_rn(src[i]);
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

// 2D 16-bit tensor map over [rows][cols] (row-major), 128-byte swizzle, box {64 cols, box_rows}.
jpi_status make_tmap(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, CUtensorMap* map,
                     CUtensorMapDataType dtype = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16) {
    auto enc = get_encode();
    if (!enc) {
        set_error("cuTensorMapEncodeTiled is unavailable from the driver");
        return JPI_ERR_CUDA;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)KBLK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, dtype, 2, (void*)base, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
        return JPI_ERR_CUDA;
    }
    return JPI_OK;
}

template <typename T>
jpi_status tc_alloc(jpi_handle* h, T** p, size_t count) {
    void* q = nullptr;
    if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc of %zu bytes failed", count * sizeof(T));
        return JPI_ERR_OOM;
    }
    h->allocations.push_back(q);
    h->device_bytes += count * sizeof(T);
    *p = (T*)q;
    return JPI_OK;
}

// Puts one fp32 tensor (host or device) into device memory at `dst` (fp32).
jpi_status stage(float* dst, const float* src, size_t n, bool on_device) {
    if (!src) {
        set_error("a per-layer weight tensor is NULL");
        return JPI_ERR_INVALID_ARG;
    }
    JPI_CUDA_TRY(cudaMemcpy(dst, src, n * sizeof(float),
                            on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice));
    return JPI_OK;
}

jpi_status pack(const float* tmp, __nv_bfloat16* dst, const int* dmap, int rows, int K) {
    const long long total = (long long)rows * K;
    const int g = (int)std::min<long long>((total + 255) / 256, 16384);
    k_pack_tiles<<<g, 256>>>(tmp, dst, dmap, rows, K);
    JPI_CUDA_TRY(cudaGetLastError());
    return JPI_OK;
}

// Columns per epilogue item of the K-split kernel: the residual kinds take two at a split of 8 or more,
// where that is an item for every thread (four columns leave half of them idle, and each item has eight
// residual values to fetch and update), else four, so that a thread has few items. Measured: pi0.5 sizes, split 8,
// denoise at batch 1 5.09 ms with four columns, 4.90 with two (and the split-KV attention's whole-block
// copies); O of one head of 128 at W = 1024, split 1, 51 tokens 6.3 us with four, 7.4 with two.
int tw_of(int kind, const GemmPlan& pl) {
    return (kind == G_O || kind == G_DOWN) && pl.splits >= 8 ? 2 : 4;
}
using GemmFn = void (*)(CUtensorMap, CUtensorMap, GemmArgs);
GemmFn gemm_fn(int kind, const GemmPlan& pl) {
    const bool two = tw_of(kind, pl) == 2;
    switch (kind) {
        case G_QKV: return k_tc_gemm<G_QKV, 4>;
        case G_GU: return k_tc_gemm<G_GU, 4>;
        case G_O: return two ? k_tc_gemm<G_O, 2> : k_tc_gemm<G_O, 4>;
        default: return two ? k_tc_gemm<G_DOWN, 2> : k_tc_gemm<G_DOWN, 4>;
    }
}

template <int KIND>
jpi_status launch_gemm(jpi_handle* h, const GemmPlan& pl, const CUtensorMap& wmap,
                       const CUtensorMap& xmap, const GemmArgs& a, cudaStream_t st) {
    // One grid row per token tile (63 tokens + the beta row for the norm-fed kinds, else 64).
    constexpr int TT = (KIND == G_QKV || KIND == G_GU) ? XS_TOKENS : NT;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.ctas, (unsigned)std::max(1, (a.Mt + TT - 1) / TT));
    cfg.blockDim = dim3(GEMM_THREADS);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attrs[2];
    int n = 0;
    attrs[n].id = cudaLaunchAttributeClusterDimension;
    attrs[n].val.clusterDim.x = pl.splits;
    attrs[n].val.clusterDim.y = 1;
    attrs[n].val.clusterDim.z = 1;
    ++n;
    if (h->pdl) {
        attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = n;
    cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_fn(KIND, pl), wmap, xmap, a);
    if (e != cudaSuccess) {
        set_error("tensor-core GEMM launch failed: %s", cudaGetErrorString(e));
        return JPI_ERR_CUDA;
    }
    return JPI_OK;
}

// K split of the large-M residual projections: persistent CTAs over (weight tile, 128-token tile) units,
// of which they have few with a long K; splitting each unit's K range over a cluster of S CTAs fills
// the GPU. S is the one of 1, 2, 4, 8 with the least estimated time: `first` + `kb` us a k-block for the first
// wave of units, and for each further one, which overlaps with it, the longer of `next` (its exchange and
// epilogue) and `next_kb` a k-block. Fitted to 336 shapes (128 to 3264 tokens, 256 to 2048 output features, K of
// 128 to 4096): what it chooses takes 0.2% longer than the best choice on average, 5% at most. Measured,
// S = 1, 2, 4, 8, us: 1024 features, 408 tokens, K = 512 7.6, 6.1, 6.2, 13.2, K = 2048 14.4, 9.4, 8.5, 14.5, K = 4096
// 23.1, 13.5, 11.0, 16.5; 816 tokens, K = 2048 14.4, 9.6, 12.8, 20.1; 2040 tokens, K = 2048 14.6, 15.1, 22.3, 42.5.
struct BigCost {
    double first, kb, next, next_kb;
};
constexpr BigCost BIG_COST[4] = {{5.7, .27, 4.4, .29}, {5.2, .26, 4.0, .33}, {5.05, .32, 4.0, .42}, {5.5, .42, 3.9, .50}};

// Clusters of S large-M CTAs that can run at once (one CTA per SM; clusters of 8 leave some SMs
// of each GPC idle), from the occupancy query at prepare time.
int big_clusters(const jpi_handle* h, int S) {
    const int i = S == 1 ? 0 : S == 2 ? 1 : S == 4 ? 2 : 3;
    return h->big_clusters[i] > 0 ? h->big_clusters[i] : h->num_sms / S;
}

int big_split(const jpi_handle* h, int units, int nkb, double* us_out = nullptr) {
    if (us_out) *us_out = 0.;
    if (h->big_split > 0) return nkb % h->big_split == 0 ? h->big_split : 1;
    int best = 1;
    double best_us = -1.;
    for (int i = 0; i < 4; ++i) {
        const int S = 1 << i;
        if (nkb % S) continue;
        const BigCost& c = BIG_COST[i];
        const double kb = nkb / S;
        const long waves = (units + big_clusters(h, S) - 1) / big_clusters(h, S);
        const double us = c.first + c.kb * kb + (double)(waves - 1) * std::max(c.next, c.next_kb * kb);
        if (best_us < 0. || us < best_us) {
            best_us = us;
            best = S;
        }
    }
    if (us_out) *us_out = best_us;
    return best;
}

// Whether a residual projection takes the tokens-on-rows kernel (128 x 256 tiles, no K split): when its
// estimate (the same fit: 8.6 us + 0.275 a k-block, a further wave 6.5 + 0.22) is less than the best
// split's of the other kernel. Measured, this kernel and the best split, us: 1024 features, 3264 tokens, K = 2048
// 18.5 and 20.4, K = 4096 27.7 and 32.6; 2448 tokens, K = 1024 13.6 and 13.8; 2048 features, 3264 tokens, K = 512
// 19.9 and 17.8.
bool resid_rows(const jpi_handle* h, int Mt, const GemmPlan& pl) {
    if (h->resid_rows >= 0) return h->resid_rows != 0;
    double other = 0.;
    big_split(h, pl.ntiles * ((Mt + BIG_NT - 1) / BIG_NT), pl.nkb, &other);
    if (other == 0.) return false;   // a fixed split
    const long tiles = (long)((pl.ntiles + 1) / 2) * ((Mt + 127) / 128);
    const long waves = (tiles + h->num_sms - 1) / h->num_sms;
    return 8.6 + .275 * pl.nkb + (double)(waves - 1) * (6.5 + .22 * pl.nkb) < other;
}

// Whether a norm-fed projection takes 128 x 128 tiles instead of 128 x 256 ones: a wave of the narrow
// ones takes 7/11 of a wave of the wide ones (3.5 and 5.5 us at K = 1024), so while their waves
// cost no more. pi0.5 sizes, us, narrow and wide: QKV 408 tokens 7.5 and 11.3 (one wave each), 816: 7.8
// and 11.3, 1020: 12.3 and 11.5 (two waves and one), 2040: 17.1 and 18.4, 3264: 21.7 and 20.4; gate/up 204
// tokens 6.8 and 8.8, 408: 10.4 and 9.1, 816: 14.2 and 14.7, 1020: 17.8 and 15.3, 3264: 44.1 and 38.6.
// At five other widths (256 to 2048, 204 to 3264 tokens) the choice takes 0.3% longer than the better tile on
// average, 3% at most.
bool rows_narrow(const jpi_handle* h, int Mt, const GemmPlan& pl) {
    if (h->rows_tile_n > 0) return h->rows_tile_n == TILE_ROWS;
    const long ntm = (Mt + 2 * XS_TOKENS - 1) / (2 * XS_TOKENS), n = h->num_sms;
    const long narrow = (pl.ntiles * ntm + n - 1) / n, wide = ((pl.ntiles + 1) / 2 * ntm + n - 1) / n;
    return narrow * 7 <= wide * 11;
}

template <int KIND, int NW>
jpi_status launch_gemm_rows(jpi_handle* h, const GemmPlan& pl, const CUtensorMap& wmap, const CUtensorMap& xmap,
                            const GemmArgs& a, cudaStream_t st) {
    constexpr int TT = (KIND == G_QKV || KIND == G_GU) ? 2 * XS_TOKENS : 128;
    const int tiles = ((pl.ntiles + NW - 1) / NW) * std::max(1, (a.Mt + TT - 1) / TT);
    GemmArgs ar = a;
    ar.ntiles = pl.ntiles;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(tiles, h->num_sms));   // persistent, one CTA per SM
    cfg.blockDim = dim3(RT_THREADS);
    cfg.dynamicSmemBytes = RT_SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = h->pdl ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_tc_gemm_rows<KIND, NW>, wmap, xmap, ar);
    if (e != cudaSuccess) {
        set_error("tensor-core GEMM launch failed: %s", cudaGetErrorString(e));
        return JPI_ERR_CUDA;
    }
    return JPI_OK;
}

template <int KIND, int S>
jpi_status launch_big_s(jpi_handle* h, int units, const CUtensorMap& wmap, const CUtensorMap& xmap,
                        const GemmArgs& a, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    // Persistent: one CTA per SM (clusters of S that all run at once, at most one per unit).
    cfg.gridDim = dim3((unsigned)(S * std::min(units, big_clusters(h, S))));
    cfg.blockDim = dim3(BIG_THREADS);
    cfg.dynamicSmemBytes = 1024 + big_smem_bytes<S>();
    cfg.stream = st;
    cudaLaunchAttribute attrs[2];
    int n = 0;
    if (S > 1) {
        attrs[n].id = cudaLaunchAttributeClusterDimension;
        attrs[n].val.clusterDim.x = S;
        attrs[n].val.clusterDim.y = 1;
        attrs[n].val.clusterDim.z = 1;
        ++n;
    }
    if (h->pdl) {
        attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = n;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_tc_gemm_big<KIND, S>, wmap, xmap, a);
    if (e != cudaSuccess) {
        set_error("tensor-core GEMM launch failed: %s", cudaGetErrorString(e));
        return JPI_ERR_CUDA;
    }
    return JPI_OK;
}

template <int KIND>
jpi_status launch_gemm_big(jpi_handle* h, const GemmPlan& pl, const CUtensorMap& wmap,
                           const CUtensorMap& xmap, const GemmArgs& a, cudaStream_t st) {
    const int units = pl.ntiles * std::max(1, (a.Mt + BIG_NT - 1) / BIG_NT);
    GemmArgs ab = a;
    ab.ntiles = pl.ntiles;
    switch (big_split(h, units, pl.nkb)) {
        case 2: return launch_big_s<KIND, 2>(h, units, wmap, xmap, ab, st);
        case 4: return launch_big_s<KIND, 4>(h, units, wmap, xmap, ab, st);
        case 8: return launch_big_s<KIND, 8>(h, units, wmap, xmap, ab, st);
        default: return launch_big_s<KIND, 1>(h, units, wmap, xmap, ab, st);
    }
}

GemmArgs base_args(jpi_handle* h, int B, int C, const GemmPlan& pl) {
    GemmArgs a = {};
    a.Mt = B * (C + h->n_ctx());
    a.K = pl.K;
    a.nkb = pl.nkb;
    a.kpb = pl.kpb;
    a.splits = pl.splits;
    a.ss = h->ss;
    a.nslot = h->W / TILE_ROWS;
    a.ss_ld = h->maxMt;
    a.eps = h->cfg.rms_eps;
    a.inv_w = 1.f / (float)h->W;
    a.W = h->W;
    a.S = C + h->n_ctx();
    a.H = h->H;
    a.D = h->D;
    a.P = h->cur_prefix;
    a.kv_rows = h->kv_rows;
    a.F = h->F;
    a.err = h->dev_err;
    return a;
}

}  // namespace

jpi_status tc_make_tmap(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, CUtensorMap* map) {
    return make_tmap(base, rows, cols, box_rows, map);
}

bool tc_supported(const jpi_handle* h) {
    return h->W % TILE_ROWS == 0 && h->D % TILE_ROWS == 0 && h->F % 64 == 0 && h->HD % KBLK == 0 &&
           h->W / TILE_ROWS <= 64;
}

jpi_status tc_pack_layers(jpi_handle* h, const jpi_weights* w, float* tmp, bool on_device) {
    const int W = h->W, D = h->D, F = h->F, HD = h->HD, QKV = h->QKV;
    // Tiled row of every source row: QKV pairs (d, d + D/2) of each head section share a tile
    // (rows r and r + 64); gate row f and up row f share tile f / 64.
    std::vector<int> qmap(QKV), gmap(F), umap(F);
    const int hd = D / 2;
    for (int s = 0; s < QKV; ++s) {
        const int sec = s / D, dd = s % D, half = dd / hd, d = dd % hd;
        const int pair = sec * hd + d;
        qmap[s] = (pair / 64) * TILE_ROWS + half * 64 + pair % 64;
    }
    for (int f = 0; f < F; ++f) {
        gmap[f] = (f / 64) * TILE_ROWS + f % 64;
        umap[f] = (f / 64) * TILE_ROWS + 64 + f % 64;
    }
    int* dmaps = nullptr;
    JPI_TRY(tc_alloc(h, &dmaps, (size_t)QKV + 2 * F));
    JPI_CUDA_TRY(cudaMemcpy(dmaps, qmap.data(), QKV * sizeof(int), cudaMemcpyHostToDevice));
    JPI_CUDA_TRY(cudaMemcpy(dmaps + QKV, gmap.data(), F * sizeof(int), cudaMemcpyHostToDevice));
    JPI_CUDA_TRY(cudaMemcpy(dmaps + QKV + F, umap.data(), F * sizeof(int), cudaMemcpyHostToDevice));

    h->tiled.resize(h->L);
    for (int l = 0; l < h->L; ++l) {
        LayerTiled& t = h->tiled[l];
        JPI_TRY(tc_alloc(h, &t.qkv, (size_t)QKV * W));
        JPI_TRY(tc_alloc(h, &t.o, (size_t)W * HD));
        JPI_TRY(tc_alloc(h, &t.gu, (size_t)2 * F * W));
        JPI_TRY(tc_alloc(h, &t.down, (size_t)W * F));
        JPI_TRY(stage(tmp, w->wq[l], (size_t)HD * W, on_device));
        JPI_TRY(stage(tmp + (size_t)HD * W, w->wk[l], (size_t)D * W, on_device));
        JPI_TRY(stage(tmp + (size_t)(HD + D) * W, w->wv[l], (size_t)D * W, on_device));
        JPI_TRY(pack(tmp, t.qkv, dmaps, QKV, W));
        JPI_TRY(stage(tmp, w->wo[l], (size_t)W * HD, on_device));
        JPI_TRY(pack(tmp, t.o, nullptr, W, HD));
        JPI_TRY(stage(tmp, w->w_gate[l], (size_t)F * W, on_device));
        JPI_TRY(pack(tmp, t.gu, dmaps + QKV, F, W));
        JPI_TRY(stage(tmp, w->w_up[l], (size_t)F * W, on_device));
        JPI_TRY(pack(tmp, t.gu, dmaps + QKV + F, F, W));
        JPI_TRY(stage(tmp, w->w_down[l], (size_t)W * F, on_device));
        JPI_TRY(pack(tmp, t.down, nullptr, W, F));
    }
    JPI_CUDA_TRY(cudaDeviceSynchronize());
    return JPI_OK;
}

jpi_status tc_prepare(jpi_handle* h) {
    int dev = 0, sms = 0;
    JPI_CUDA_TRY(cudaGetDevice(&dev));
    JPI_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    h->num_sms = sms;
    if (attn_tc_supported(h)) JPI_TRY(attn_tc_prepare(h));
    JPI_TRY(attn_t5_prepare(h));

    int max_cluster = 16;
    for (GemmFn k : {k_tc_gemm<G_QKV, 4>, k_tc_gemm<G_O, 2>, k_tc_gemm<G_O, 4>, k_tc_gemm<G_GU, 4>, k_tc_gemm<G_DOWN, 2>,
                     k_tc_gemm<G_DOWN, 4>}) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            max_cluster = 8;
        }
        JPI_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    }
    for (auto k : {k_tc_gemm_rows<G_QKV, 1>, k_tc_gemm_rows<G_QKV, 2>, k_tc_gemm_rows<G_GU, 1>, k_tc_gemm_rows<G_GU, 2>,
                   k_tc_gemm_rows<G_O, 2>, k_tc_gemm_rows<G_DOWN, 2>})
        JPI_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RT_SMEM));
    auto big1 = {k_tc_gemm_big<G_O, 1>, k_tc_gemm_big<G_DOWN, 1>};
    for (auto k : big1)
        JPI_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<1>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_O, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<2>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_DOWN, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<2>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_O, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<4>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_DOWN, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<4>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_O, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<8>()));
    JPI_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm_big<G_DOWN, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + big_smem_bytes<8>()));
    {
        auto query = [&](const void* fn, int S, int smem) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(S * (sms / S)));
            cfg.blockDim = dim3(BIG_THREADS);
            cfg.dynamicSmemBytes = (size_t)smem;
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = S;
            at.val.clusterDim.y = 1;
            at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            return n;
        };
        h->big_clusters[0] = sms;
        h->big_clusters[1] = query((const void*)k_tc_gemm_big<G_DOWN, 2>, 2, 1024 + big_smem_bytes<2>());
        h->big_clusters[2] = query((const void*)k_tc_gemm_big<G_DOWN, 4>, 4, 1024 + big_smem_bytes<4>());
        h->big_clusters[3] = query((const void*)k_tc_gemm_big<G_DOWN, 8>, 8, 1024 + big_smem_bytes<8>());
    }
    // JPI_BIG_SPLIT=S fixes the K split of the large-M residual projections (1, 2, 4 or 8).
    const char* split_env = std::getenv("JPI_BIG_SPLIT");
    if (split_env) h->big_split = std::atoi(split_env);
    // JPI_BIG_RESID_ROWS=0 / 1 fixes the kernel of those projections (1: tokens on the MMA's rows).
    const char* rows_env = std::getenv("JPI_BIG_RESID_ROWS");
    if (rows_env) h->resid_rows = std::atoi(rows_env) != 0 ? 1 : 0;
    // JPI_BIG_TILE_N=128 / 256 fixes the tile width of the large-M QKV and gate/up projections.
    const char* tile_env = std::getenv("JPI_BIG_TILE_N");
    if (tile_env) h->rows_tile_n = std::atoi(tile_env) == TILE_ROWS ? TILE_ROWS : 2 * TILE_ROWS;
    const int rows[4] = {h->QKV, h->W, 2 * h->F, h->W};
    const int ks[4] = {h->W, h->HD, h->W, h->F};
    // The K split (and so the summation order) is chosen once per projection, for every batch
    // size: a request's result does not depend on how many other requests share its batch.
    for (int g = 0; g < 4; ++g) {
        if (!make_plan(rows[g], ks[g], max_cluster, sms, g == G_QKV || g == G_GU, &h->plans[g])) {
            set_error("no tensor-core tiling for a %d x %d projection", rows[g], ks[g]);
            return JPI_ERR_UNSUPPORTED;
        }
    }
    // A cluster of `splits` CTAs must fit on the device at this shared-memory size.
    for (int g = 0; g < 4; ++g) {
        const GemmPlan& pl = h->plans[g];
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(pl.ctas);
        cfg.blockDim = dim3(GEMM_THREADS);
        cfg.dynamicSmemBytes = pl.smem;
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = pl.splits;
        at.val.clusterDim.y = 1;
        at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int nclusters = 0;
        const void* fn = (const void*)gemm_fn(g, pl);
        if (cudaOccupancyMaxActiveClusters(&nclusters, fn, &cfg) != cudaSuccess || nclusters < 1) {
            cudaGetLastError();
            set_error("a cluster of %d CTAs with %zu bytes of shared memory does not fit", pl.splits, pl.smem);
            return JPI_ERR_UNSUPPORTED;
        }
        // The K-split kernel runs its grid once per token tile of 63 or 64; the large-M kernels take
        // over once its CTAs no longer all run at once (two per SM where the shared memory allows;
        // with one, clusters leave some SMs of a GPC idle). At pi0.5 sizes that is from 190 tokens for
        // QKV (153 tokens: 6.6 us against 7.3; 204: 10.7 against 7.4), 64 for gate/up (102: 11.1 against
        // 6.9) and 65 for down (102: 10.7 against 9.4). O would gain up to 256 tokens (255: 7.0 against
        // 8.4) but takes over at 128 at the latest: the K-split kernel's partial sums are fp16, the
        // large-M kernels' fp32. QKV takes over at 512 at the latest for the same reason, which only an
        // expert of few heads meets (W = 2048, two heads of 128, 500 tokens: 7.4 us against 10.0; W = 1024, one
        // head: 5.8 against 7.1). JPI_BIG_GEMM_MIN_TOKENS sets one threshold for all four.
        const int resident = 2 * (pl.smem + 1024) <= 228 * 1024 ? 2 * sms : nclusters * pl.splits;
        const int tt = g == G_QKV || g == G_GU ? XS_TOKENS : NT;
        h->big_min_tokens[g] = std::min(std::max(1, resident / pl.ctas) * tt + 1, g == G_QKV ? 512 : 128);
        if (const char* big_env = std::getenv("JPI_BIG_GEMM_MIN_TOKENS")) h->big_min_tokens[g] = std::atoi(big_env);
    }
    h->tmaps.resize((size_t)4 * h->L);
    for (int l = 0; l < h->L; ++l) {
        const LayerTiled& t = h->tiled[l];
        const int qkv_rows = h->QKV, o_rows = h->W, gu_rows = 2 * h->F, d_rows = h->W;
        JPI_TRY(make_tmap(t.qkv, (uint64_t)qkv_rows / TILE_ROWS * (h->W / KBLK) * TILE_ROWS, KBLK, TILE_ROWS,
                          &h->tmaps[4 * l + G_QKV]));
        JPI_TRY(make_tmap(t.o, (uint64_t)o_rows / TILE_ROWS * (h->HD / KBLK) * TILE_ROWS, KBLK, TILE_ROWS,
                          &h->tmaps[4 * l + G_O]));
        JPI_TRY(make_tmap(t.gu, (uint64_t)gu_rows / TILE_ROWS * (h->W / KBLK) * TILE_ROWS, KBLK, TILE_ROWS,
                          &h->tmaps[4 * l + G_GU]));
        JPI_TRY(make_tmap(t.down, (uint64_t)d_rows / TILE_ROWS * (h->F / KBLK) * TILE_ROWS, KBLK, TILE_ROWS,
                          &h->tmaps[4 * l + G_DOWN]));
    }
    // B operands: scaled residual stream in tiles of 63 tokens + beta, attention output and GeGLU
    // output ([rows][K] row-major).
    JPI_TRY(make_tmap(h->hx, (uint64_t)xs_tiles(h->maxMt) * 64, h->W, NT, &h->xmaps[0]));
    JPI_TRY(make_tmap(h->o, h->maxMt, h->HD, NT, &h->xmaps[1]));
    JPI_TRY(make_tmap(h->z, h->maxMt, h->F, NT, &h->xmaps[2]));
    JPI_TRY(make_tmap(h->hx, (uint64_t)xs_tiles(h->maxMt) * 64, h->W, 128, &h->xmaps_rows[0]));
    JPI_TRY(make_tmap(h->o, h->maxMt, h->HD, 128, &h->xmaps_rows[1]));
    JPI_TRY(make_tmap(h->z, h->maxMt, h->F, 128, &h->xmaps_rows[2]));
    JPI_TRY(mod_tc_prepare(h));
    // Batch-invariant mode: the K-split projections and the split-KV attention at every size.
    if (h->batch_invariant) {
        h->attn_t5_min_batch = 0;
        for (int k = 0; k < 4; ++k) h->big_min_tokens[k] = 0;
    }
    return JPI_OK;
}

jpi_status tc_launch_op(jpi_handle* h, int op, int l, int step, int B, int C, cudaStream_t st) {
    const int W = h->W;
    const float* ms = h->mods + (size_t)step * mod_rows(h->L) * W + (size_t)6 * l * W;
    const size_t kv_layer = (size_t)l * h->maxB * h->kv_rows * h->D;
    const jpi::GemmPlan* plans = h->plans;
    const int Mt = B * (C + h->n_ctx());
    // Batched launches with many tokens: one CTA per (weight tile, 128-row operand tile) over
    // the whole K range. Residual kinds then leave one sum-of-squares slot per weight tile, and
    // the norm-fed kind after them reads as many slots as its producer left.
    auto big = [&](int kind) { return h->big_min_tokens[kind] > 0 && Mt >= h->big_min_tokens[kind]; };
    auto slots_left = [&](int kind) { return big(kind) ? plans[kind].ntiles : plans[kind].ntiles * plans[kind].splits; };
    auto run = [&](auto kind_tag, const GemmPlan& pl, const CUtensorMap& wm, int xi,
                   const GemmArgs& a) -> jpi_status {
        constexpr int KIND = decltype(kind_tag)::value;
        if (!big(KIND)) return launch_gemm<KIND>(h, pl, wm, h->xmaps[xi], a, st);
        if constexpr (KIND == G_QKV || KIND == G_GU) {
            if (rows_narrow(h, Mt, pl)) return launch_gemm_rows<KIND, 1>(h, pl, wm, h->xmaps_rows[xi], a, st);
        } else if (!resid_rows(h, Mt, pl)) {
            return launch_gemm_big<KIND>(h, pl, wm, h->xmaps_rows[xi], a, st);
        }
        return launch_gemm_rows<KIND, 2>(h, pl, wm, h->xmaps_rows[xi], a, st);
    };
    using KQ = std::integral_constant<int, G_QKV>;
    using KO = std::integral_constant<int, G_O>;
    using KG = std::integral_constant<int, G_GU>;
    using KD = std::integral_constant<int, G_DOWN>;
    switch (op) {
        case 2: {
            const GemmPlan& pl = plans[G_QKV];
            GemmArgs a = base_args(h, B, C, pl);
            // Sums of squares left by the embedding (one per 128 features) or the previous
            // layer's down projection (one per CTA).
            if (l > 0) a.nslot = slots_left(G_DOWN);
            a.q = (__nv_bfloat16*)h->q;
            a.kst = (__nv_bfloat16*)h->kv_k + kv_layer;
            a.vst = (__nv_bfloat16*)h->kv_v + kv_layer;
            a.rope = h->rope_tab;
            return run(KQ{}, pl, h->tmaps[4 * l + G_QKV], 0, a);
        }
        case 3:
            // Batched launches: one CTA per 128 query rows over all keys (tcgen05, no split);
            // otherwise the split-KV kernel that spreads one request over the whole GPU.
            if (h->attn_t5 && h->attn_t5_min_batch > 0 && B >= h->attn_t5_min_batch)
                return launch_attn_t5(h, l, B, C, st);
            return attn_tc_supported(h) ? launch_attn_tc(h, l, B, C, st)
                                        : launch_op_simt(h, 3, l, step, B, C, st);
        case 4: {
            const GemmPlan& pl = plans[G_O];
            GemmArgs a = base_args(h, B, C, pl);
            a.hres = h->h;
            a.xs = (__nv_bfloat16*)h->hx;
            a.sigma_next = ms + 3 * W;   // the MLP norm of this layer
            a.beta_next = ms + 4 * W;
            a.gamma = ms + 2 * W;
            a.ss_out = h->ss;
            return run(KO{}, pl, h->tmaps[4 * l + G_O], 1, a);
        }
        case 5: {
            const GemmPlan& pl = plans[G_GU];
            GemmArgs a = base_args(h, B, C, pl);
            a.nslot = slots_left(G_O);   // left by O
            a.z = (__nv_bfloat16*)h->z;
            return run(KG{}, pl, h->tmaps[4 * l + G_GU], 0, a);
        }
        case 6: {
            const GemmPlan& pl = plans[G_DOWN];
            GemmArgs a = base_args(h, B, C, pl);
            a.hres = h->h;
            if (l + 1 < h->L) {           // the attention norm of the next layer
                a.xs = (__nv_bfloat16*)h->hx;
                a.sigma_next = ms + 6 * W;
                a.beta_next = ms + 7 * W;
            }
            a.gamma = ms + 5 * W;
            a.ss_out = h->ss;
            return run(KD{}, pl, h->tmaps[4 * l + G_DOWN], 2, a);
        }
        default:
            set_error("unknown layer op %d", op);
            return JPI_ERR_INVALID_ARG;
    }
}

jpi_status tc_launch_layer(jpi_handle* h, int l, int step, int B, int C, cudaStream_t st) {
    for (int op = 2; op <= 6; ++op) JPI_TRY(tc_launch_op(h, op, l, step, B, C, st));
    return JPI_OK;
}

void tc_release(jpi_handle*) {}

}  // namespace jpi
