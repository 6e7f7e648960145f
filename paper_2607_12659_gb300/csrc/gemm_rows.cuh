// Large-M projection kernel with the tokens on the MMA's rows (included by tc_path.cu, inside jpi's
// anonymous namespace).
//
// Output tile = 128 operand rows (the MMA's M: 128 tokens, or for the RMSNorm-fed kinds two 64-row
// tiles of 63 tokens + one beta row) x 256 weight rows (its N: NW = 2 consecutive 128-row weight tiles)
// over the whole K range. What bounds these products is the operand bytes an SM takes in per
// multiply-add, and how many of them are in flight: a k-block brings 48 KB for 2 M multiply-adds and
// the ring keeps four of them, 192 KB, under way: about 0.39 us a k-block, 85% of the tensor peak
// inside a tile (128 x 128 tiles bring 32 KB for 1 M, 128 KB under way: 0.32 us a k-block of half the
// size). Per launch, us, 128 x 128 tiles -> these: 3264 tokens (K = 1024: QKV 2560 rows 31.5 -> 21.5,
// gate/up 8192 rows 66.3 -> 42.2; O 26.0 -> 20.4, down 39.3 -> 30.1); 408 tokens: gate/up 16.8 -> 9.8.
// NW = 1 (norm-fed kinds) is for launches of few tiles, where half of them would leave SMs idle: twice
// the CTAs, each with half the bytes and half the epilogue (QKV, 408 tokens: 40 tiles 11.3 us, 80 narrow
// ones 7.5; the launcher has the rule).
// Persistent: one CTA per SM walks the tiles u = blockIdx.x, + gridDim.x, .., the token tile fastest
// (the CTAs that run together share one weight tile, which is read from HBM once):
//   warp 0  one thread streams (operand block, weight block pair) by bulk tensor copies through the
//           ring; the weight blocks of the first stages are requested before the dependency wait;
//   warp 1  one thread issues the tcgen05.mma chain (M = 128, N = 128 NW, K = 16 each) of a tile into one
//           of two TMEM accumulators and releases each stage through tcgen05.commit;
//   warps 2-9  the epilogue: a TMEM lane is a token, so the two features that rotary coding or GeGLU
//           combine are columns of one thread. Group g of four warps takes weight tile g (NW = 1: half of
//           the one tile's pairs). Norm-fed kinds scale by the token's 1 / rms and add W beta, which is the
//           accumulator row of the beta row (TMEM lane 63): its warp hands the group's 128 values
//           over through shared memory. Every warp passes its 32 rows through 4 KB of shared memory
//           of its own (128 bytes a row, 16-byte chunks XOR-swizzled by the row), so that global
//           memory is read and written 128 bytes of four rows per instruction: with a token's row per
//           thread each instruction touched 32 lines, and those (10 per 16 columns in the residual
//           kinds) held the tile longer than its MMAs (O at batch 8: 26 us).
//           Residual kinds fetch the old residual rows one 32-column step ahead.
// All waits are bounded.

constexpr int RT_XBYTES = 128 * KBLK * 2;                       // 16 KB operand block
constexpr int RT_RING = 192 * 1024;                             // 4 stages of 48 KB, or 6 of 32 KB
constexpr int RT_EPI = 256;
constexpr int RT_THREADS = 64 + RT_EPI;
constexpr int RT_STAGING = 32 * 128;                            // one epilogue warp: 32 rows of 128 bytes
constexpr int RT_SMEM = 1024 + RT_RING + 8 * RT_STAGING + 2 * TILE_ROWS * 4 + 160;

template <int KIND, int NW>
__global__ void __launch_bounds__(RT_THREADS, 1) k_tc_gemm_rows(const __grid_constant__ CUtensorMap wmap,
                                                              const __grid_constant__ CUtensorMap xmap,
                                                              const __grid_constant__ GemmArgs a) {
    constexpr bool NORM_IN = (KIND == G_QKV || KIND == G_GU);
    constexpr int TT = NORM_IN ? 2 * XS_TOKENS : 128;   // tokens per tile
    constexpr int RT_N = NW * TILE_ROWS;                // weight rows per tile (MMA N)
    constexpr int RT_STAGE_BYTES = RT_XBYTES + NW * TILE_BYTES;
    constexpr int RT_STAGES = RT_RING / RT_STAGE_BYTES;
    constexpr uint32_t IDESC = ptx::idesc_bf16_f32(128, RT_N);
    static_assert(NW == 2 || (NW == 1 && NORM_IN), "one weight tile: norm-fed kinds only");

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* stages = smem;                                             // [stage][X 16 KB | W 16 KB each]
    uint8_t* staging = smem + RT_STAGES * RT_STAGE_BYTES;               // [8 warps][32 rows][128 B]
    float* beta_s = (float*)(staging + 8 * RT_STAGING);                 // [2 groups][128] W beta of their columns
    uint64_t* full = (uint64_t*)(beta_s + 2 * TILE_ROWS);
    uint64_t* empty = full + RT_STAGES;
    uint64_t* accf = empty + RT_STAGES;   // [2] accumulator holds a finished tile
    uint64_t* acce = accf + 2;            // [2] the epilogue has read it out
    uint32_t* tmem_slot = (uint32_t*)(acce + 2);
    int* flag = (int*)(tmem_slot + 1);

    const int tid = threadIdx.x, warp = ptx::warp_index(), lane = tid & 31;
    const int nkb = a.nkb;
    const int ntn = (a.ntiles + NW - 1) / NW, ntm = (a.Mt + TT - 1) / TT;
    const int total = ntn * ntm;
    const int u0 = (int)blockIdx.x, du = (int)gridDim.x;

    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, 2 * RT_N);
        ptx::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2 * RT_STAGES; ++i) ptx::mbar_init(&full[i], 1);
        ptx::mbar_init(&accf[0], 1);
        ptx::mbar_init(&accf[1], 1);
        ptx::mbar_init(&acce[0], RT_EPI);
        ptx::mbar_init(&acce[1], RT_EPI);
        ptx::fence_mbar_init();
        *flag = 0;
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (ptx::elect_one()) {
            const uint64_t pol = ptx::l2_policy_evict_first();
            // The weight tiles' k-blocks (rows past the last tile arrive as zeros).
            auto load_w = [&](int tn, int kb, int s) {
                uint8_t* ws = stages + s * RT_STAGE_BYTES + RT_XBYTES;
                ptx::mbar_expect_tx(&full[s], (uint32_t)RT_STAGE_BYTES);
#pragma unroll
                for (int w = 0; w < NW; ++w)
                    ptx::tma_load_2d(ws + w * TILE_BYTES, &wmap, &full[s], 0, ((NW * tn + w) * nkb + kb) * TILE_ROWS, pol);
            };
            auto load_x = [&](int tm, int kb, int s) {
                ptx::tma_load_2d_plain(stages + s * RT_STAGE_BYTES, &xmap, &full[s], kb * KBLK, tm * 128);
            };
            ptx::prefetch_tmap(&xmap);
            const int npre = u0 < total ? (nkb < RT_STAGES ? nkb : RT_STAGES) : 0;
            for (int kb = 0; kb < npre; ++kb) load_w(u0 / ntm, kb, kb);
            ptx::grid_dep_wait();
            int it = 0;
            bool ok = true;
            for (int u = u0; u < total && ok; u += du) {
                const int tm = u % ntm, tn = u / ntm;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % RT_STAGES, n = it / RT_STAGES;
                    if (it < npre) {
                        load_x(tm, kb, s);
                        continue;
                    }
                    if (it >= RT_STAGES && !ptx::mbar_wait_bounded(&empty[s], (n - 1) & 1, WAIT_LIMIT_NS)) {
                        *flag = DEV_TIMEOUT_WEIGHTS;
                        ok = false;
                        break;
                    }
                    load_w(tn, kb, s);
                    load_x(tm, kb, s);
                }
            }
            if (!ptx::ring_drain(full, RT_STAGES, it, WAIT_LIMIT_NS)) *flag = DEV_TIMEOUT_WEIGHTS;
        }
    } else if (warp == 1) {
        if (ptx::elect_one()) {
            const uint32_t base = ptx::smem_u32(stages);
            bool good = true;
            int it = 0;
            for (int u = u0, j = 0; u < total; u += du, ++j) {
                const int buf = j & 1;
                if (j >= 2 && !ptx::mbar_wait_bounded(&acce[buf], ((j - 2) >> 1) & 1, WAIT_LIMIT_NS)) good = false;
                ptx::tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * RT_N);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % RT_STAGES, n = it / RT_STAGES;
                    if (good && !ptx::mbar_wait_bounded(&full[s], n & 1, WAIT_LIMIT_NS)) good = false;
                    ptx::tc_fence_after();
                    if (good) {
                        const uint64_t x = ptx::desc_sw128(base + s * RT_STAGE_BYTES), w = ptx::desc_add(x, RT_XBYTES);
#pragma unroll
                        for (int kk = 0; kk < KBLK / 16; ++kk)
                            ptx::mma_bf16(acc, ptx::desc_add(x, kk * 32), ptx::desc_add(w, kk * 32), IDESC,
                                          (kb | kk) != 0);
                    }
                    ptx::mma_commit(&empty[s]);
                }
                // Committed even after a timeout so that the epilogue wakes up.
                ptx::mma_commit(&accf[buf]);
            }
            if (!good) *flag = DEV_TIMEOUT_MMA;
        }
    } else {
        // ---- epilogue: one token (TMEM lane) per thread; group g has weight tile g of two, or half of
        // the one tile's pairs (steps 2 g, 2 g + 1) ----
        const int g = (warp - 2) >> 2, qd = warp & 3;
        constexpr int NST = 2 * NW;                  // this group's steps of 32 columns
        const int st0 = NW == 1 ? NST * g : 0;
        const int row = qd * 32 + lane;
        const uint32_t bar_id = 1 + g;
        uint8_t* stg = staging + (warp - 2) * RT_STAGING;
        // Through the staging, lane l handles chunk l mod 8 of rows 4 i + l / 8 of the warp's 32.
        const int sr = lane >> 3, sc = lane & 7;
        auto own_chunk = [&](int c) { return (uint4*)(stg + lane * 128 + ((c ^ (lane & 7)) << 4)); };
        auto row_chunk = [&](int r, int c) { return (const uint4*)(stg + r * 128 + ((c ^ (r & 7)) << 4)); };
        // Token of row r (0 .. 127) of tile tm; -1 for beta rows and past the last token.
        auto token = [&](int tm, int r) {
            const int r64 = r & 63;
            const int t = NORM_IN ? tm * TT + (r >> 6) * XS_TOKENS + r64 : tm * TT + r;
            return t < a.Mt && !(NORM_IN && r64 == XS_TOKENS) ? t : -1;
        };
        ptx::grid_dep_wait();
        bool ok = true;
        for (int u = u0, j = 0; u < total; u += du, ++j) {
            const int buf = j & 1;
            const int tm = u % ntm, tile = NW == 2 ? 2 * (u / ntm) + g : u / ntm;   // this group's 128-row weight tile
            const bool tile_live = tile < a.ntiles;
            const int f0 = tile * TILE_ROWS;
            // Global inputs that do not depend on the product, before the accumulator is waited for.
            float rinv = 0.f;
            if (NORM_IN) {
                const int t = token(tm, row);
                float s = 0.f;
                for (int s0 = 0; s0 < a.nslot; s0 += 8) {   // slot order, eight loads in flight
                    float v[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        v[k] = t >= 0 && s0 + k < a.nslot ? a.ss[(size_t)(s0 + k) * a.ss_ld + t] : 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) s += v[k];
                }
                rinv = rsqrtf(s * a.inv_w + a.eps);
            }
            // Tokens of the rows this lane handles through the staging.
            int tk[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) tk[i] = tile_live ? token(tm, qd * 32 + 4 * i + sr) : -1;
            // QKV: head section and first pair of this weight tile's 64 pairs; each row's position.
            const int hd = KIND == G_QKV ? a.D >> 1 : 1;
            int sec = 0, d0 = 0;
            int pos[8];
            size_t dst[8];
            if (KIND == G_QKV) {
                sec = f0 / 2 / hd;
                d0 = f0 / 2 - sec * hd;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int t = tk[i] < 0 ? 0 : tk[i], b = t / a.S;
                    pos[i] = a.P + t - b * a.S;
                    dst[i] = sec < a.H ? ((size_t)t * a.H + sec) * a.D : ((size_t)b * a.kv_rows + pos[i]) * a.D;
                }
            }
            const bool rot = KIND == G_QKV && a.rope && sec <= a.H;
            __nv_bfloat16* qkv = sec < a.H ? a.q : sec == a.H ? a.kst : a.vst;
            float4 in4[8];   // QKV: (cos, sin) of two pairs; residual kinds: the old residual
            auto fetch = [&](int step) {
                if (KIND == G_QKV) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        in4[i] = rot && tk[i] >= 0 ? __ldg((const float4*)(a.rope + (size_t)pos[i] * hd + d0 + 16 * step) + sc)
                                                   : make_float4(1.f, 0.f, 1.f, 0.f);
                } else if (!NORM_IN) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        in4[i] = tk[i] >= 0 ? *(const float4*)(a.hres + (size_t)tk[i] * a.W + f0 + 32 * step + 4 * sc)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            };
            fetch(st0);
            if (!ptx::mbar_wait_bounded(&accf[buf], (j >> 1) & 1, WAIT_LIMIT_NS)) *flag = DEV_TIMEOUT_MMA;
            ptx::tc_fence_after();
            // This CTA's last accumulator is complete: the next kernel may start streaming its weights.
            if (u + du >= total) ptx::grid_dep_launch();
            const uint32_t lb = tmem + (uint32_t)(buf * RT_N + (NW == 2 ? 128 * g : 0)) + ((uint32_t)(qd * 32) << 16);
            if constexpr (NORM_IN) {
                if (qd == 1) {
                    // The beta row is this warp's lane 31 (TMEM lane 63).
#pragma unroll
                    for (int c0 = 0; c0 < 128; c0 += 32) {
                        if (NW == 1 && ((c0 >> 5) & 1) != g) continue;   // the other group's pairs
                        uint32_t r[2][16];
                        ptx::tmem_ld_x16(lb + (uint32_t)c0, r[0]);
                        ptx::tmem_ld_x16(lb + (uint32_t)(c0 + 16), r[1]);
                        ptx::tmem_ld_wait();
                        if (lane == 31) {
                            uint4* bp = (uint4*)(beta_s + 128 * g + c0);
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                bp[i] = make_uint4(r[i >> 2][4 * (i & 3)], r[i >> 2][4 * (i & 3) + 1],
                                                   r[i >> 2][4 * (i & 3) + 2], r[i >> 2][4 * (i & 3) + 3]);
                        }
                    }
                }
                ptx::named_bar_sync(bar_id, 128);
                ok = __all_sync(0xffffffffu, ok && *flag == 0);
                const float4* bt = (const float4*)(beta_s + 128 * g);
#pragma unroll
                for (int q = 0; q < NST; ++q) {
                    const int st = st0 + q;
                    // Columns 16 st.. and 64 + 16 st..: the two features of 16 pairs.
                    uint32_t r1[16], r2[16];
                    ptx::tmem_ld_x16(lb + (uint32_t)(16 * st), r1);
                    ptx::tmem_ld_x16(lb + (uint32_t)(64 + 16 * st), r2);
                    ptx::tmem_ld_wait();
                    float y1[16], y2[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 b1 = bt[4 * st + i], b2 = bt[16 + 4 * st + i];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            y1[4 * i + e] = rinv * __uint_as_float(r1[4 * i + e]) + f4get(b1, e);
                            y2[4 * i + e] = rinv * __uint_as_float(r2[4 * i + e]) + f4get(b2, e);
                        }
                    }
                    if (KIND == G_GU) {
                        // 16 features: 32 bytes of the row's 128 (64 features of z).
                        uint32_t o[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            o[i] = pack_bf16x2(gelu_tanh(y1[2 * i]) * y2[2 * i], gelu_tanh(y1[2 * i + 1]) * y2[2 * i + 1]);
                        *own_chunk(2 * st) = make_uint4(o[0], o[1], o[2], o[3]);
                        *own_chunk(2 * st + 1) = make_uint4(o[4], o[5], o[6], o[7]);
                    } else {
                        // Pairs 2 c, 2 c + 1 of the 16 as one chunk (y1, y1, y2, y2): lane sc of a row
                        // rotates chunk sc.
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            *own_chunk(c) = make_uint4(__float_as_uint(y1[2 * c]), __float_as_uint(y1[2 * c + 1]),
                                                       __float_as_uint(y2[2 * c]), __float_as_uint(y2[2 * c + 1]));
                        __syncwarp();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const uint4 v = *row_chunk(4 * i + sr, sc);
                            const float4 c = in4[i];
                            const float ua = __uint_as_float(v.x), ub = __uint_as_float(v.y);
                            const float va = __uint_as_float(v.z), vb = __uint_as_float(v.w);
                            if (tk[i] >= 0 && ok) {
                                __nv_bfloat16* p = qkv + dst[i] + d0 + 16 * st + 2 * sc;
                                *(uint32_t*)p = pack_bf16x2(ua * c.x - va * c.y, ub * c.z - vb * c.w);
                                *(uint32_t*)(p + hd) = pack_bf16x2(va * c.x + ua * c.y, vb * c.z + ub * c.w);
                            }
                        }
                        if (q < NST - 1) fetch(st + 1);
                        __syncwarp();
                    }
                }
                ptx::tc_fence_before();
                ptx::mbar_arrive(&acce[buf]);
                if (KIND == G_GU) {
                    __syncwarp();
                    if (NW == 1) {
                        // Four chunks a row: eight rows per instruction.
                        const int c = 4 * g + (lane & 3);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int r = 8 * i + (lane >> 2), t = tile_live ? token(tm, qd * 32 + r) : -1;
                            const uint4 v = *row_chunk(r, c);
                            if (t >= 0 && ok) *(uint4*)(a.z + (size_t)t * a.F + tile * 64 + 8 * c) = v;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 8 && NW == 2; ++i) {
                        const uint4 v = *row_chunk(4 * i + sr, sc);
                        if (tk[i] >= 0 && ok) *(uint4*)(a.z + (size_t)tk[i] * a.F + tile * 64 + 8 * sc) = v;
                    }
                }
                ptx::named_bar_sync(bar_id, 128);   // beta_s and the staging are rewritten by the next tile
            } else {
                ok = __all_sync(0xffffffffu, ok && *flag == 0);
                float sq[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) sq[i] = 0.f;
#pragma unroll
                for (int st = 0; st < 4; ++st) {
                    uint32_t r[2][16];
                    ptx::tmem_ld_x16(lb + (uint32_t)(32 * st), r[0]);
                    ptx::tmem_ld_x16(lb + (uint32_t)(32 * st + 16), r[1]);
                    float4 gm = make_float4(0.f, 0.f, 0.f, 0.f), sg = gm;   // of this lane's four features
                    if (tile_live) {
                        gm = __ldg((const float4*)(a.gamma + f0 + 32 * st) + sc);
                        if (a.xs) sg = __ldg((const float4*)(a.sigma_next + f0 + 32 * st) + sc);
                    }
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *own_chunk(c) = make_uint4(r[c >> 2][4 * (c & 3)], r[c >> 2][4 * (c & 3) + 1],
                                                   r[c >> 2][4 * (c & 3) + 2], r[c >> 2][4 * (c & 3) + 3]);
                    __syncwarp();
                    float4 n[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint4 v = *row_chunk(4 * i + sr, sc);
                        n[i] = make_float4(in4[i].x + gm.x * __uint_as_float(v.x), in4[i].y + gm.y * __uint_as_float(v.y),
                                           in4[i].z + gm.z * __uint_as_float(v.z), in4[i].w + gm.w * __uint_as_float(v.w));
                        sq[i] = fmaf(n[i].x, n[i].x, fmaf(n[i].y, n[i].y, fmaf(n[i].z, n[i].z, fmaf(n[i].w, n[i].w, sq[i]))));
                    }
                    if (st < 3) fetch(st + 1);   // before the stores, which would hold the loads back
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        if (tk[i] < 0 || !ok) continue;
                        *(float4*)(a.hres + (size_t)tk[i] * a.W + f0 + 32 * st + 4 * sc) = n[i];
                        if (a.xs)
                            *(uint2*)(a.xs + (size_t)xs_row(tk[i]) * a.W + f0 + 32 * st + 4 * sc) =
                                make_uint2(pack_bf16x2((1.f + sg.x) * n[i].x, (1.f + sg.y) * n[i].y),
                                           pack_bf16x2((1.f + sg.z) * n[i].z, (1.f + sg.w) * n[i].w));
                    }
                    __syncwarp();
                }
                ptx::tc_fence_before();
                ptx::mbar_arrive(&acce[buf]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    sq[i] += __shfl_xor_sync(0xffffffffu, sq[i], 1);
                    sq[i] += __shfl_xor_sync(0xffffffffu, sq[i], 2);
                    sq[i] += __shfl_xor_sync(0xffffffffu, sq[i], 4);
                    if (sc == 0 && tk[i] >= 0 && ok) a.ss_out[(size_t)tile * a.ss_ld + tk[i]] = sq[i];
                }
                // The next norm's shift in the last row of each of its token tiles.
                if (a.xs && tm == 0 && ok && tile_live) {
                    const float bn = a.beta_next[f0 + row];
                    for (int x = 0; x < xs_tiles(a.Mt); ++x)
                        a.xs[((size_t)x * 64 + 63) * a.W + f0 + row] = __float2bfloat16_rn(bn);
                }
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (tid == 0 && *flag != 0) set_device_error(a.err, *flag);   // after every role's last word on it
    if (warp == 1) ptx::tmem_dealloc(tmem, 2 * RT_N);
}
