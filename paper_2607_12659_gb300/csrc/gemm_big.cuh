// Large-M kernel of the residual projections (O, down) with a K split (included by tc_path.cu, inside
// jpi's anonymous namespace), for launches whose 128 x 256 tiles over the whole K range would leave
// SMs idle (gemm_rows.cuh has that kernel, and the rule that chooses).
//
// Output tile = one 128-row weight tile x one tile of 128 tokens; a cluster of S CTAs splits its K
// range. Bound by the rate at which one SM takes operands in from L2 (87-100 GB/s measured per SM
// with 128 KB under way), not by the MMAs.
// Persistent: one CTA per SM walks the tiles u = blockIdx.x, + gridDim.x, ... (weight tile
// fastest), and its roles overlap consecutive tiles:
//   warp 0  one thread streams (weight block, operand block) pairs by bulk tensor copies into a
//           ring of STAGES shared-memory stages (full/empty mbarriers), tile after tile;
//   warp 1  one thread issues the tcgen05.mma chain (M = 128, N = 128, K = 16 each) of a tile
//           into one of two TMEM accumulators (tile j into buffer j mod 2, once the epilogue has
//           read tile j - 2 out of it) and releases each stage through tcgen05.commit;
//   warps 2-9  the epilogue, two groups of four warps (group g takes accumulator columns
//           64g..64g+63, one TMEM lane = weight row per thread). After the read-out the TMEM buffer
//           goes back to the MMA thread. With a K split the partials are exchanged and summed as
//           described at BigCfg. Without one the residual rows of the tile are copied into a shared
//           fp32 tile [token][feature] with 16-byte async copies before the accumulator is waited
//           for and the accumulator rows are added into that tile. Either way the new residual, the
//           next norm's operand and each token's sum of squares are written a token row per warp
//           instruction (16 / 8 bytes per lane).
// The next kernel is released once this CTA's last accumulator is complete. All waits are
// bounded.

constexpr int BIG_NT = 128;                       // operand rows per tile
constexpr int BIG_EPI = 256;                     // epilogue threads: two groups of 4 warps
constexpr int BIG_THREADS = 64 + BIG_EPI;
constexpr int BIG_XBYTES = BIG_NT * KBLK * 2;     // 16 KB operand block
constexpr int BIG_STAGE_BYTES = TILE_BYTES + BIG_XBYTES;
constexpr int BIG_HS = BIG_NT + 4;                // [token][feature] residual stride: 16-byte rows
constexpr int BIG_YBYTES = BIG_NT * BIG_HS * 4;

// S CTAs of a cluster split the K range of each unit (S = 1: no split). Each CTA then owns
// TOK = 128 / S of the unit's tokens: it sends the fp32 partial of every other CTA's tokens to that
// CTA and sums the S partials of its own tokens in rank order. A slice is laid out [feature / 32][token]
// [32], so each epilogue warp's part of it (its 32 accumulator rows, all tokens) is one contiguous
// block, which the warp sends as soon as it has written it; a receiving warp adds the partials of its
// tokens to residual rows it holds in registers and stores the results, with no staging tile and one
// block barrier (for the CTA's own partials). The exchange buffers take shared memory from the ring,
// which keeps 4 (S = 2) or 3 stages of 32 KB in flight. What bounds a unit at these sizes is the chain
// from the accumulator to the stores: O takes 7.2 us at 153 tokens, 7.9 at 408 and 9.0 at 816, down 9.2, 10.2 and
// 12.9; whole-slice copies between block barriers and a staging tile add 1.1-2.3 us to each.
template <int S>
struct BigCfg {
    static constexpr int STAGES = S <= 2 ? 4 : 3;
    static constexpr int TOK = BIG_NT / S;                                 // tokens owned per CTA
    static constexpr int SLICE = TOK * BIG_NT * 4;                         // one fp32 slice
    static constexpr int WBLK = TOK * 32;                                  // floats of a warp's block of it
    static constexpr int YBYTES = S == 1 ? BIG_YBYTES : 0;                 // staging tile
    static constexpr int SEND = (S - 1) * SLICE;                           // outgoing slices
    static constexpr int RECV = S == 1 ? 0 : S * SLICE;                    // partials by rank (own one too)
};

template <int S>
__host__ __device__ constexpr int big_smem_bytes() {
    // stages | residual tile | send | recv | bars (full, empty, acc full[2], acc empty[2],
    // recv full, peers free) + TMEM slot + flag
    return BigCfg<S>::STAGES * BIG_STAGE_BYTES + BigCfg<S>::YBYTES + BigCfg<S>::SEND + BigCfg<S>::RECV +
           160;
}

template <int KIND, int S>
__global__ void __launch_bounds__(BIG_THREADS, 1) k_tc_gemm_big(const __grid_constant__ CUtensorMap wmap,
                                                             const __grid_constant__ CUtensorMap xmap,
                                                             const __grid_constant__ GemmArgs a) {
    using CF = BigCfg<S>;
    constexpr int STAGES = CF::STAGES;
    constexpr int TOK = CF::TOK;
    static_assert(KIND == G_O || KIND == G_DOWN, "the residual projections");
    constexpr uint32_t IDESC = ptx::idesc_bf16_f32(TILE_ROWS, BIG_NT);

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stages = smem;                                             // [stage][W 16 KB | X 16 KB]
    float* ystage = (float*)(smem + STAGES * BIG_STAGE_BYTES);          // residual tile [token][feature]
    float* sendb = (float*)((uint8_t*)ystage + CF::YBYTES);             // [S - 1][4][TOK][32] to the peers
    float* recvb = (float*)((uint8_t*)sendb + CF::SEND);                // [S][4][TOK][32] by sender rank
    uint64_t* full = (uint64_t*)((uint8_t*)recvb + CF::RECV);
    uint64_t* empty = full + STAGES;
    uint64_t* accf = empty + STAGES;   // [2] accumulator buffer holds a finished tile
    uint64_t* acce = accf + 2;         // [2] the epilogue has read it out
    uint64_t* recvf = acce + 2;        // the peers' slices of this unit have landed
    uint64_t* pfree = recvf + 1;       // every peer has summed the slices of the last unit
    uint32_t* tmem_slot = (uint32_t*)(pfree + 1);
    int* flag = (int*)(tmem_slot + 1);

    const int tid = threadIdx.x, warp = ptx::warp_index(), lane = tid & 31;
    const int rank = S == 1 ? 0 : (int)ptx::cluster_rank();
    const int nkb = a.nkb / S;                 // K blocks of this CTA
    const int kb0 = rank * nkb;
    const int ntiles = a.ntiles;
    const int nxt = (a.Mt + BIG_NT - 1) / BIG_NT;
    const int total = ntiles * nxt;
    const int u0 = (int)blockIdx.x / S, du = (int)gridDim.x / S;

    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, 2 * BIG_NT);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            ptx::mbar_init(&full[i], 1);
            ptx::mbar_init(&empty[i], 1);
        }
        ptx::mbar_init(&accf[0], 1);
        ptx::mbar_init(&accf[1], 1);
        ptx::mbar_init(&acce[0], BIG_EPI);
        ptx::mbar_init(&acce[1], BIG_EPI);
        ptx::mbar_init(recvf, 1);
        ptx::mbar_init(pfree, S > 1 ? (S - 1) * (BIG_EPI / 32) : 1);
        ptx::fence_mbar_init();
        *flag = 0;
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // Split K: every CTA of the cluster has initialised its barriers before any peer aims a copy or
    // an arrival at them (waited for before the first exchange).
    if (S > 1) ptx::cluster_arrive_relaxed();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (ptx::elect_one()) {
            const uint64_t pol = ptx::l2_policy_evict_first();
            auto load_w = [&](int tile, int kb, int s) {
                ptx::mbar_expect_tx(&full[s], (uint32_t)BIG_STAGE_BYTES);
                ptx::tma_load_2d(stages + s * BIG_STAGE_BYTES, &wmap, &full[s], 0, (tile * a.nkb + kb0 + kb) * TILE_ROWS,
                                 pol);
            };
            ptx::prefetch_tmap(&xmap);
            auto load_x = [&](int xt, int kb, int s) {
                uint8_t* xs = stages + s * BIG_STAGE_BYTES + TILE_BYTES;
                ptx::tma_load_2d(xs, &xmap, &full[s], (kb0 + kb) * KBLK, xt * BIG_NT, pol);
            };
            // Weight blocks of the first tile's first stages do not depend on the previous kernel.
            const int npre = u0 < total ? (nkb < STAGES ? nkb : STAGES) : 0;
            for (int kb = 0; kb < npre; ++kb) load_w(u0 % ntiles, kb, kb);
            ptx::grid_dep_wait();
            int it = 0;   // k-block counter over this CTA's tiles: stage it mod STAGES
            bool ok = true;
            for (int u = u0; u < total && ok; u += du) {
                const int tile = u % ntiles, xt = u / ntiles;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % STAGES, n = it / STAGES;
                    if (it < npre) {   // first tile, weights already in flight
                        load_x(xt, kb, s);
                        continue;
                    }
                    if (it >= STAGES && !ptx::mbar_wait_bounded(&empty[s], (n - 1) & 1, WAIT_LIMIT_NS)) {
                        *flag = DEV_TIMEOUT_WEIGHTS;
                        ok = false;
                        break;
                    }
                    load_w(tile, kb, s);
                    load_x(xt, kb, s);
                }
            }
            if (!ptx::ring_drain(full, STAGES, it, WAIT_LIMIT_NS)) *flag = DEV_TIMEOUT_WEIGHTS;
        }
    } else if (warp == 1) {
        if (ptx::elect_one()) {
            const uint32_t base = ptx::smem_u32(stages);
            bool good = true;
            int it = 0;
            for (int u = u0, j = 0; u < total; u += du, ++j) {
                const int buf = j & 1;
                // Tile j - 2 has been read out of this accumulator buffer.
                if (j >= 2 && !ptx::mbar_wait_bounded(&acce[buf], ((j - 2) >> 1) & 1, WAIT_LIMIT_NS)) good = false;
                ptx::tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * BIG_NT);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % STAGES, n = it / STAGES;
                    if (good && !ptx::mbar_wait_bounded(&full[s], n & 1, WAIT_LIMIT_NS)) good = false;
                    ptx::tc_fence_after();
                    if (good) {
                        const uint64_t w = ptx::desc_sw128(base + s * BIG_STAGE_BYTES), x = ptx::desc_add(w, TILE_BYTES);
#pragma unroll
                        for (int kk = 0; kk < KBLK / 16; ++kk)
                            ptx::mma_bf16(acc, ptx::desc_add(w, kk * 32), ptx::desc_add(x, kk * 32), IDESC,
                                          (kb | kk) != 0);
                    }
                    ptx::mma_commit(&empty[s]);
                }
                // Committed even after a timeout so that the epilogue wakes up.
                ptx::mma_commit(&accf[buf]);
            }
            if (!good) *flag = DEV_TIMEOUT_MMA;
        }
    } else if constexpr (S > 1) {
        // ---- epilogue with a K split: TMEM lane `row` (weight row) of the accumulator per thread ----
        const int eg = (tid - 64) >> 7;   // group: accumulator columns (tokens) 64 eg ..
        const int ew = (tid - 64) >> 5, quarter = warp & 3;
        constexpr int TW = TOK / 8;       // tokens a warp finishes: TW ew .. of this CTA's
        constexpr int NSL = 64 / TOK > 0 ? 64 / TOK : 1;   // slices a group's columns cover
        ptx::grid_dep_wait();
        bool ok = true;
        for (int u = u0, j = 0; u < total; u += du, ++j) {
            const int buf = j & 1;
            const int tile = u % ntiles, xt = u / ntiles;
            const int tok0 = xt * BIG_NT + rank * TOK + TW * ew;   // this warp's first token
            const int f0 = tile * TILE_ROWS;
            // Features 4 lane ..: the residual rows, gamma and the next norm's scale, in flight while the
            // accumulator is waited for.
            const float4 gm = *(const float4*)(a.gamma + f0 + 4 * lane);
            const float4 sg = a.xs ? *(const float4*)(a.sigma_next + f0 + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 hr[TW];
#pragma unroll
            for (int k = 0; k < TW; ++k)
                hr[k] = tok0 + k < a.Mt ? *(const float4*)(a.hres + (size_t)(tok0 + k) * a.W + f0 + 4 * lane)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            // Slices of this unit from the S - 1 peers.
            if (tid == 64) ptx::mbar_expect_tx(recvf, (uint32_t)((S - 1) * CF::SLICE));
            __syncwarp();
            if (j == 0) {
                ptx::cluster_wait();
            } else if (!ptx::mbar_wait_cluster_bounded(pfree, (j - 1) & 1, WAIT_LIMIT_NS)) {
                // (Every peer has summed the last unit's slices, so this CTA's outgoing slices, read by
                // those copies, and the peers' receive slots are free again.)
                *flag = DEV_TIMEOUT_MMA;
            }
            if (!ptx::mbar_wait_bounded(&accf[buf], (j >> 1) & 1, WAIT_LIMIT_NS)) *flag = DEV_TIMEOUT_MMA;
            __syncwarp();
            ptx::tc_fence_after();
            // This CTA's last accumulator is complete: the next kernel may start streaming its weights.
            if (u + du >= total) ptx::grid_dep_launch();
            // Accumulator column c (token c of the unit) belongs to rank c / TOK: own columns go to this
            // CTA's slot of the receive buffer, the others to the outgoing slice of their rank.
            {
                const uint32_t lane_base = tmem + (uint32_t)(buf * BIG_NT + 64 * eg) + ((uint32_t)(quarter * 32) << 16);
                uint32_t r[4][16];
#pragma unroll
                for (int c = 0; c < 4; ++c) ptx::tmem_ld_x16(lane_base + (uint32_t)(16 * c), r[c]);
                ptx::tmem_ld_wait();
                ptx::tc_fence_before();
                ptx::mbar_arrive(&acce[buf]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // 16 columns never straddle two owners (TOK >= 16).
                    const int col0 = 64 * eg + 16 * c, q = col0 / TOK;
                    float* dst = (q == rank ? recvb + (size_t)rank * TOK * BIG_NT
                                            : sendb + (size_t)(q < rank ? q : q - 1) * TOK * BIG_NT) +
                                 quarter * CF::WBLK + (col0 % TOK) * 32 + lane;
#pragma unroll
                    for (int i = 0; i < 16; ++i) dst[i * 32] = __uint_as_float(r[c][i]);
                }
            }
            // This warp's blocks of the outgoing slices, lane i to the i-th of their ranks.
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane < NSL && eg * NSL + lane != rank) {
                const int q = eg * NSL + lane;
                ptx::bulk_copy_to_cluster(
                    ptx::dsmem_map(ptx::smem_u32(recvb + (size_t)rank * TOK * BIG_NT + quarter * CF::WBLK), (uint32_t)q),
                    sendb + (size_t)(q < rank ? q : q - 1) * TOK * BIG_NT + quarter * CF::WBLK, (uint32_t)(CF::WBLK * 4),
                    ptx::dsmem_map(ptx::smem_u32(recvf), (uint32_t)q));
            }
            ptx::named_bar_sync(1, BIG_EPI);   // the CTA's own partials
            ok = ok && *flag == 0;
            // The next norm's shift in the last row of each of its token tiles (this tile's rows).
            if (a.xs && xt == 0 && ok && rank == 0 && eg == 0) {
                const int f = f0 + quarter * 32 + lane;
                const float bn = a.beta_next[f];
                for (int x = 0; x < xs_tiles(a.Mt); ++x)
                    a.xs[((size_t)x * 64 + 63) * a.W + f] = __float2bfloat16_rn(bn);
            }
            if (!ptx::mbar_wait_bounded(recvf, j & 1, WAIT_LIMIT_NS)) {
                *flag = DEV_TIMEOUT_MMA;
                ok = false;
            }
            // (A timeout may be seen by some lanes only: the warp decides together.)
            ok = __all_sync(0xffffffffu, ok);
            // Everything addressed to this CTA has landed; once all of the cluster say so every copy
            // out of it has landed too.
            if (u + du >= total) ptx::cluster_arrive_relaxed();
            // n = h + gamma * (sum of the S partials in rank order); the token's sum of squares over
            // the tile's 128 features is lane 0's butterfly total (slot `tile`).
            float4 y[TW];
#pragma unroll
            for (int k = 0; k < TW; ++k) {
                y[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < S; ++q) {
                    const float4 v = *(const float4*)(recvb + (size_t)q * TOK * BIG_NT + (lane >> 3) * CF::WBLK +
                                                      (TW * ew + k) * 32 + 4 * (lane & 7));
                    y[k].x += v.x;
                    y[k].y += v.y;
                    y[k].z += v.z;
                    y[k].w += v.w;
                }
            }
            // This warp has read its part of the receive buffer: each peer may overwrite its slot (and
            // reuse its outgoing slices) for the next unit. One lane per peer; a release, so that the reads
            // of the whole warp (ordered before it by the __syncwarp) are over before the peer's next copy.
            if (u + du < total) {
                __syncwarp();
                if (lane < S - 1) {
                    const int q = lane < rank ? lane : lane + 1;
                    ptx::mbar_arrive_cluster(ptx::dsmem_map(ptx::smem_u32(pfree), (uint32_t)q));
                }
            }
#pragma unroll
            for (int k = 0; k < TW; ++k) {
                const int t = tok0 + k;
                if (t >= a.Mt || !ok) break;
                float4 n;
                n.x = hr[k].x + gm.x * y[k].x;
                n.y = hr[k].y + gm.y * y[k].y;
                n.z = hr[k].z + gm.z * y[k].z;
                n.w = hr[k].w + gm.w * y[k].w;
                *(float4*)(a.hres + (size_t)t * a.W + f0 + 4 * lane) = n;
                if (a.xs)
                    *(uint2*)(a.xs + (size_t)xs_row(t) * a.W + f0 + 4 * lane) =
                        make_uint2(pack_bf16x2((1.f + sg.x) * n.x, (1.f + sg.y) * n.y),
                                   pack_bf16x2((1.f + sg.z) * n.z, (1.f + sg.w) * n.w));
                float sq = ((n.x * n.x + n.y * n.y) + n.z * n.z) + n.w * n.w;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (lane == 0) a.ss_out[(size_t)tile * a.ss_ld + t] = sq;
            }
            // Every warp has read the CTA's own slot before the next unit rewrites it.
            if (u + du < total) ptx::named_bar_sync(1, BIG_EPI);
        }
    } else {
        // ---- epilogue: TMEM lane `row` (weight row) of the accumulator per thread ----
        const int eg = (tid - 64) >> 7;   // group
        const int row = (warp & 3) * 32 + lane;
        ptx::grid_dep_wait();
        bool ok = true;
        // A tile's global inputs, all loads in flight together: the residual rows of the tile's
        // tokens (epilogue warp ew copies tokens 16 ew.. into the shared tile [token][feature], 16
        // bytes per lane).
        const int ew = (tid - 64) >> 5;
        float gam = 0.f;
        float4 sg4 = make_float4(0.f, 0.f, 0.f, 0.f);   // next norm's scale of features 4 lane..
        auto fetch = [&](int tile, int tok0) {
            const int f0 = tile * TILE_ROWS;
            gam = a.gamma[f0 + row];
            if (a.xs) sg4 = *(const float4*)(a.sigma_next + f0 + 4 * lane);
#pragma unroll
            for (int k = 0; k < TOK / 8; ++k) {
                const int c = (TOK / 8) * ew + k, t = tok0 + c;
                const bool in = t < a.Mt;
                ptx::cp_async_16(ptx::smem_u32(ystage + c * BIG_HS + 4 * lane),
                                 a.hres + (in ? (size_t)t * a.W + f0 + 4 * lane : 0), in);
            }
        };
        for (int u = u0, j = 0; u < total; u += du, ++j) {
            const int buf = j & 1;
            const int tile = u % ntiles, xt = u / ntiles;
            const int tok0 = xt * BIG_NT;
            fetch(tile, tok0);
            ptx::cp_async_wait_all();
            if (tid == 64 && !ptx::mbar_wait_bounded(&accf[buf], (j >> 1) & 1, WAIT_LIMIT_NS)) *flag = DEV_TIMEOUT_MMA;
            // The residual rows are published; the MMAs of the tile are done.
            ptx::named_bar_sync(1, BIG_EPI);
            ptx::tc_fence_after();
            // This CTA's last accumulator is complete: the next kernel may start streaming its weights.
            if (u + du >= total) ptx::grid_dep_launch();
            ok = ok && *flag == 0;
            {
                const uint32_t lane_base = tmem + (uint32_t)(buf * BIG_NT) + ((uint32_t)((warp & 3) * 32) << 16);
                {
                    const int f0 = tile * TILE_ROWS, f = f0 + row;
                    // n = h + gamma * y in place of h: accumulator row `row` (feature f), 32 token
                    // columns at a time, into column f of the [token][feature] tile.
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 32) {
                        uint32_t r[2][16];
                        ptx::tmem_ld_x16(lane_base + (uint32_t)(64 * eg + c0), r[0]);
                        ptx::tmem_ld_x16(lane_base + (uint32_t)(64 * eg + c0 + 16), r[1]);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            float* hp = ystage + (64 * eg + c0 + i) * BIG_HS + row;
                            *hp = *hp + gam * __uint_as_float(r[i >> 4][i & 15]);
                        }
                    }
                    ptx::tc_fence_before();
                    ptx::mbar_arrive(&acce[buf]);
                    // The next norm's shift in the last row of each of its token tiles (this tile's rows).
                    if (a.xs && xt == 0 && ok && eg == 0) {
                        const float bn = a.beta_next[f];
                        for (int x = 0; x < xs_tiles(a.Mt); ++x)
                            a.xs[((size_t)x * 64 + 63) * a.W + f] = __float2bfloat16_rn(bn);
                    }
                    ptx::named_bar_sync(1, BIG_EPI);   // the tile's new residual rows are complete
                    // Warp ew writes tokens TOK / 8 ew..: lane l the features 4 l..4 l + 3 of the new
                    // residual (16 bytes) and of the next norm's operand (8 bytes); the token's sum of
                    // squares over the tile's 128 features is lane 0's butterfly total (slot `tile`).
                    // (A timeout flag may be seen by some lanes only: the warp decides together.)
                    const bool okw = __all_sync(0xffffffffu, ok);
#pragma unroll 4
                    for (int k = 0; k < TOK / 8; ++k) {
                        const int c = (TOK / 8) * ew + k, t = tok0 + c;
                        if (t >= a.Mt || !okw) break;
                        const float4 n = *(const float4*)(ystage + c * BIG_HS + 4 * lane);
                        *(float4*)(a.hres + (size_t)t * a.W + f0 + 4 * lane) = n;
                        if (a.xs) {
                            const uint2 v = make_uint2(pack_bf16x2((1.f + sg4.x) * n.x, (1.f + sg4.y) * n.y),
                                                       pack_bf16x2((1.f + sg4.z) * n.z, (1.f + sg4.w) * n.w));
                            *(uint2*)(a.xs + (size_t)xs_row(t) * a.W + f0 + 4 * lane) = v;
                        }
                        float sq = ((n.x * n.x + n.y * n.y) + n.z * n.z) + n.w * n.w;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                        if (lane == 0) a.ss_out[(size_t)tile * a.ss_ld + t] = sq;
                    }
                }
                // Every epilogue thread is done with the residual tile.
                ptx::named_bar_sync(1, BIG_EPI);
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (tid == 0 && *flag != 0) set_device_error(a.err, *flag);   // after every role's last word on it
    if (warp == 1) ptx::tmem_dealloc(tmem, 2 * BIG_NT);
    // Split K: no copy or arrival of a peer is still aimed at this CTA when it exits (the epilogue
    // warps arrived once their last slices had landed).
    if (S > 1) {
        if (warp <= 1) {
            __syncwarp();
            ptx::cluster_wait();
            ptx::cluster_arrive_relaxed();
        }
        ptx::cluster_wait();
    }
}
