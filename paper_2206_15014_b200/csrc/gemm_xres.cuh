// CTA-pair kernel with the activations resident, for weights in tensor-core form and reductions of at most 1024.
//
// A pair tile is 256 output channels x 192 tokens as in nm_gemm_pair_kernel, but the tiles run token-tile-major: the
// pair's token tile stays in shared memory for its whole reduction (each CTA its 96 tokens, up to 96 KB) while the weights of
// one output tile after the other stream through the ring.  Against resident weights and streamed activations:
//   * per tile and CTA 64 KB (2:4, 1024 reduction elements) of weights that all pairs share pass through L2, and not 96 KB
//     of activations; against streaming both (dense weights) the activations are not read again for every output tile;
//   * the rows of Y are written whole within a short time.
// The index metadata changes with every tile: four metadata warps (one per TMEM lane quarter, both CTAs) keep a ring of
// four buffers of 32 TMEM columns filled, one tile's reduction each.  A token tile's slices are replaced one by one as the
// last output tile's MMAs are done with them.
// What bounds it: the epilogue, and with it the loads, which wait behind its stores.  1024 -> 4096, 16384 tokens, time stamps: a stage's MMAs
// take 100-140 clocks to issue (640-830 while their operands were built per thread, see elect_one) and are handed over every 525-566, a tile of four
// stages follows the other after 5.3 k clocks with fp32 outputs, 3.7 k with bfloat16, 4.4 k with int8, of which its epilogue takes 4.7, 3.0 and
// 3.8 k; a load takes 3.7-5.3 k from issue to arrival.  16384 tokens 768 -> 3072: bfloat16 31.7 -> 28.9 us
// with staging tiles of each warp's own (narrow_tile).  Measured without gain: two MMAs of half the
// width, alternating accumulators, weights in 64-byte rows (16384 tokens 1024 -> 4096 64.6 / 62.0 us).
#pragma once

namespace nm {

constexpr int kXresMetaBufs = 4;
template <int EPI> constexpr int kXresEpiWarps = kNarrow<EPI> ? 16 : 8;
template <int EPI> constexpr int kXresThreads = 32 * (3 + kXresEpiWarps<EPI> + 4);

template <bool SPARSE>
struct XresCfg {
    static constexpr int BN = 192;
    static constexpr int KB = SPARSE ? 256 : 128;     // reduction elements per stage: 128 stored bytes of every weight row
    static constexpr int A_BYTES = kBM * 128;         // one stage of the ring
    static constexpr int B_ROWS = BN / 2;             // tokens staged by each CTA
    static constexpr int B_SUB = B_ROWS * 128;        // one 128-byte-wide slice of them
    static constexpr int SLICES = KB / 128;           // slices per stage
    static constexpr int X_RES = 8 * B_SUB;           // reductions of at most 1024
    static constexpr int MAX_KB = 1024 / KB;
    static constexpr int STORE_STAGE = 8 * 4096;
    static constexpr int STAGES = (kSmemLimit - kSmemTail - STORE_STAGE - 1024 - X_RES) / A_BYTES;
    static constexpr int SMEM = STAGES * A_BYTES + X_RES + STORE_STAGE + kSmemTail + 1024;
    static constexpr int META_COL = 2 * BN;
    static constexpr int META_SLOT = 32;              // columns of one tile's metadata (1024 reduction elements)
    static_assert(STAGES >= 4 && STAGES <= kPairMaxStages, "pipeline");
    static_assert(META_COL + kXresMetaBufs * META_SLOT <= kTmemCols, "tensor memory");
};

template <bool SPARSE, int EPI>
__global__ void __launch_bounds__(kXresThreads<EPI>, 1)
nm_gemm_xres_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                    const __grid_constant__ CUtensorMap tmap_y, const GemmParams p) {
    using Cfg = XresCfg<SPARSE>;
    constexpr int S = Cfg::STAGES, BN = Cfg::BN, MB = kXresMetaBufs, XB = Cfg::MAX_KB;
    constexpr int EW = kXresEpiWarps<EPI>, kGateWarp = 10, kMetaWarp0 = 3 + EW;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* x_res = smem + S * Cfg::A_BYTES;
    uint8_t* store_stage = x_res + Cfg::X_RES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(store_stage + Cfg::STORE_STAGE);
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };                                // leader: weight stage landed (both CTAs' bytes)
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };                         // both CTAs (multicast commit)
    auto acc_full_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };                  // both CTAs (multicast commit)
    auto acc_empty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };             // leader; arrivals from both
    auto meta_full_bar = [&](int b) { return bar0 + 8u * (2 * S + 4 + b); };             // leader; arrivals from both
    auto meta_empty_bar = [&](int b) { return bar0 + 8u * (2 * S + 4 + MB + b); };       // both CTAs (multicast commit)
    auto x_full_bar = [&](int k) { return bar0 + 8u * (2 * S + 4 + 2 * MB + k); };       // leader: activations of stage k landed
    auto x_free_bar = [&](int k) { return bar0 + 8u * (2 * S + 4 + 2 * MB + XB + k); };  // both CTAs: no MMA reads them any more
    const uint32_t drained_bar = bar0 + 8u * (2 * S + 4 + 2 * MB + 2 * XB);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 5 + 2 * MB + 2 * XB);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* never_flag = tmem_slot + 2;

    const int warp = (int)ptx::warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();
    const bool leader = rank == 0;
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int per = p.n_tiles / pairs, rem = p.n_tiles % pairs;
    const int tile_begin = pair * per + min(pair, rem), tile_count = per + (pair < rem ? 1 : 0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { ptx::mbar_init(acc_full_bar(b), 1); ptx::mbar_init(acc_empty_bar(b), 2 * EW); }
        for (int b = 0; b < MB; ++b) { ptx::mbar_init(meta_full_bar(b), 8); ptx::mbar_init(meta_empty_bar(b), 1); }
        for (int k = 0; k < XB; ++k) { ptx::mbar_init(x_full_bar(k), 1); ptx::mbar_init(x_free_bar(k), 1); }
        ptx::mbar_init(drained_bar, 1);
        *abort_flag = 0;
        *never_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_w);
        ptx::prefetch_tensormap(&tmap_x);
        if (p.tma_store) ptx::prefetch_tensormap(&tmap_y);
    }
    __syncthreads();
    ptx::cluster_arrive();   // both CTAs' barriers exist before anything remote touches them
    ptx::cluster_wait();
    if (warp == 1) {
        ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), kTmemCols);
        ptx::tmem_relinquish_pair();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = ptx::warp_uniform(*tmem_slot);
    // Set-up above overlaps the tail of the kernel before this one in the stream (when launched as its
    // programmatic dependent); nothing in global memory is read or written before this point.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    auto raise_timeout = [&]() {  // both CTAs of the pair stop: the peer's roles see the flag in their own shared memory
        *abort_flag = 1;
        ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(const_cast<uint32_t*>(abort_flag)), rank ^ 1u), 1u);
        if (p.status) atomicOr(p.status, NM_STATUS_TIMEOUT);
    };

    if (warp == 0) {
        // ------------------------------ TMA producer (both CTAs) --------------------------------
        if (lane == 0) {
            uint32_t it = 0, x_parity = 1u;  // nothing reads the resident activations before the first load
            int prev_tok = -1, o = tile_begin % p.n_out_tiles, tok = tile_begin / p.n_out_tiles;
            bool ok = true;
            const uint64_t keep = ptx::policy_evict_last();  // the weights are read again for every token tile
            for (int i = 0; i < tile_count && ok; ++i) {
                const int n0 = o * (2 * kBM) + (int)rank * kBM, t0 = tok * BN + (int)rank * Cfg::B_ROWS;
                const bool new_x = tok != prev_tok;
                for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                    if (new_x) {
                        if (!ptx::mbar_wait_bounded(x_free_bar(kb), x_parity, abort_flag, kWaitLimit)) { raise_timeout(); ok = false; break; }
                        if (leader) ptx::mbar_expect_tx(x_full_bar(kb), 2 * Cfg::SLICES * Cfg::B_SUB);  // bytes of both CTAs
                        // X is mapped as [k-slice][token][128 bytes]: all slices of the stage in one operation
                        ptx::tma_load_3d_pair_hint(ptx::smem_u32(x_res + kb * Cfg::SLICES * Cfg::B_SUB), &tmap_x, 0, t0, kb * Cfg::SLICES,
                                                   ptx::map_to_cta(x_full_bar(kb), 0), keep);
                    }
                    const int s = it % S;
                    if (!ptx::mbar_wait_bounded(empty_bar(s), ((it / S) & 1u) ^ 1u, abort_flag, kWaitLimit)) { raise_timeout(); ok = false; break; }
                    NM_TRACE_STAGE(it, 0);
                    if (NM_SKIP_STAGE(it)) continue;
                    const uint32_t dst = ptx::smem_u32(smem + s * Cfg::A_BYTES), lead_full = ptx::map_to_cta(full_bar(s), 0);
                    if (leader) ptx::mbar_expect_tx(full_bar(s), 2 * Cfg::A_BYTES);
                    ptx::tma_load_2d_pair_hint(dst, &tmap_w, kb * 128, n0, lead_full, keep);
                    NM_TRACE_STAGE(it, 1);
                }
                if (new_x) { prev_tok = tok; x_parity ^= 1u; }
                if (++o == p.n_out_tiles) { o = 0; ++tok; }
            }
            // After an expired wait (here or anywhere in the pair) nobody waits for this producer's last copies, and the stages'
            // barriers count the bytes of both CTAs: give the copies time before the CTA and its shared memory go away.
            if (!ok || *abort_flag) ptx::wait_clocks(kAbortDrain);
        }
    } else if (warp >= kMetaWarp0) {
        // ------------------------------ metadata warps (both CTAs, 2:4 only) ----------------------
        if constexpr (SPARSE) {
            const int row = (warp & 3) * 32 + lane, total_words = p.kblocks * (Cfg::KB / 32);
            const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + Cfg::META_COL;
            const uint4 kIdle = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);  // valid "positions 0,1"
            uint4 mw[8];
            // Columns past the row's metadata (the last stage may span more than the reduction) and rows past `out` get a valid
            // pattern: their products are zero or discarded.
            auto fetch = [&](int o) {
                const int n = o * (2 * kBM) + (int)rank * kBM + row;
                const uint4* src = reinterpret_cast<const uint4*>(p.meta + (size_t)(n < p.out ? n : 0) * p.mrow_words);
#pragma unroll
                for (int j = 0; j < 8; ++j) mw[j] = (n < p.out && 4 * j < p.mrow_words) ? __ldg(src + j) : kIdle;
            };
            int o = tile_begin % p.n_out_tiles;
            if (tile_count > 0) fetch(o);
            for (int i = 0; i < tile_count; ++i) {
                const int b = i % MB;
                bool got = lane != 0 || ptx::mbar_wait_bounded(meta_empty_bar(b), ((i / MB) & 1u) ^ 1u, abort_flag, kWaitLimit);
                if (!__all_sync(0xffffffffu, got)) { if (lane == 0) raise_timeout(); break; }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (4 * j < total_words) ptx::tmem_st_32x4(taddr + b * Cfg::META_SLOT + 4 * j, mw[j].x, mw[j].y, mw[j].z, mw[j].w);
                ptx::tmem_st_wait();
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(meta_full_bar(b), 0));
                if (++o == p.n_out_tiles) o = 0;
                if (i + 1 < tile_count) fetch(o);  // travels while the buffers ahead are still full
            }
        }
    } else if (warp == kGateWarp) {
        // ------------------------------ gate (leader): mbarrier waits relayed to the MMA warp ------
        if (leader) {
            uint32_t it = 0, x_phase = 0;
            int prev_tok = -1, o = tile_begin % p.n_out_tiles, tok = tile_begin / p.n_out_tiles;
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t parity) {
                if (lane == 0 && ok && !ptx::mbar_wait_bounded(bar, parity, abort_flag, kWaitLimit)) {
                    raise_timeout();
                    ptx::wait_clocks(kGateDrain);
                    ok = false;
                }
            };
            for (int i = 0; i < tile_count; ++i) {
                const int buf = i & 1;
                const bool new_x = tok != prev_tok;
                if (SPARSE) wait(meta_full_bar(i % MB), (i / MB) & 1u);
                wait(acc_empty_bar(buf), ((i >> 1) & 1u) ^ 1u);
                for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                    if (new_x) wait(x_full_bar(kb), x_phase);
                    wait(full_bar(it % S), (it / S) & 1u);
                    if (lane == 0) NM_TRACE_STAGE(it, 2);
                    __syncwarp();
                    ptx::relay_step(1 + (it & 7u), abort_flag);
                }
                if (new_x) { prev_tok = tok; x_phase ^= 1u; }
                if (++o == p.n_out_tiles) { o = 0; ++tok; }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer (leader) --------------------------------------
        if (leader) {
            // Descriptors are formed once and advanced with one add, ring positions are carried: a single thread's dependent
            // instructions cost several clocks each.
            constexpr uint32_t idesc = ptx::idesc_i8(2 * kBM, BN, SPARSE);
            const uint64_t a_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(smem), 128, ptx::kSwizzle128);
            const uint64_t b_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(x_res), 128, ptx::kSwizzle128);
            uint32_t relay = 1, s = 0;
            int o = tile_begin % p.n_out_tiles;
            NM_TRACE_ONLY(uint32_t it = 0;)
            for (int i = 0; i < tile_count; ++i) {
                const uint32_t buf = i & 1, d_tmem = tmem_base + buf * BN;
                uint32_t e = tmem_base + Cfg::META_COL + (uint32_t)(i % MB) * Cfg::META_SLOT;
                const bool last_of_x = ++o == p.n_out_tiles;  // the next tile is another token tile's
                if (last_of_x) o = 0;
                uint64_t b = b_desc0;
                for (int kb = 0; kb < p.kblocks; ++kb) {
                    ptx::named_bar_sync(relay, 64);
                    relay = (relay & 7u) + 1u;
                    if (kb == 0) ptx::tc_fence_after();  // once per tile (see the one-CTA kernel)
                    if (ptx::elect_one()) {
                        NM_TRACE_STAGE(it, 3);
                        const uint64_t a = ptx::desc_advance(a_desc0, s * Cfg::A_BYTES);
                        if constexpr (SPARSE) {
#pragma unroll
                            for (int j = 0; j < 4; ++j)  // 64 reduction elements each: 32 stored bytes of A, 64 of X
                                ptx::mma_sp_i8_pair(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, (j >> 1) * Cfg::B_SUB + 64 * (j & 1)), e + 2 * j, idesc, (kb | j) != 0);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                ptx::mma_i8_pair(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 32 * j), idesc, (kb | j) != 0);
                        }
                        ptx::tc_commit_pair(empty_bar(s), 3);   // both producers may refill the stage
                        if (last_of_x) ptx::tc_commit_pair(x_free_bar(kb), 3);  // ... and replace these activations
                        if (kb == p.kblocks - 1) {
                            ptx::tc_commit_pair(acc_full_bar(buf), 3);
                            if (SPARSE) ptx::tc_commit_pair(meta_empty_bar(i % MB), 3);
                        }
                        NM_TRACE_STAGE(it, 4);
                    }
                    __syncwarp();
                    NM_TRACE_ONLY(++it;)
                    b = ptx::desc_advance(b, Cfg::SLICES * Cfg::B_SUB);
                    e += 8;
                    if (++s == S) s = 0;
                }
            }
            if (ptx::elect_one()) {
                ptx::tc_commit_pair(drained_bar, 1);
                ptx::mbar_wait_bounded(drained_bar, 0, never_flag, kWaitLimit);
            }
            __syncwarp();
        }
    } else {
        // ------------------------------ epilogue warps (both CTAs) --------------------------------
        constexpr int EWH = EW / 4, CH = BN / 32, CI = (CH + EWH - 1) / EWH;
        const int ew = warp - 2 - (warp > kGateWarp ? 1 : 0), q = warp & 3, half = ew >> 2, row = q * 32 + lane;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16);
        float* my_stage = reinterpret_cast<float*>(store_stage + ew * 4096);
        const float sx = p.sx_dev ? *p.sx_dev : p.sx_host;
        float amax = 0.0f;
        const float rsy = EPI == EPI_Q8 ? __frcp_rn(p.sy) : 0.0f;
        uint32_t n_stores = 0;
        bool ok = true;
        auto release_acc = [&](int buf) {
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(acc_empty_bar(buf), 0));
        };
        const uint64_t stream_out = ptx::policy_evict_first();  // Y is written once and not read here
        int o = tile_begin % p.n_out_tiles, tok = tile_begin / p.n_out_tiles;
        // channel constants of a tile are fetched while the one before it is converted
        auto scale_of = [&](int tile_o) { const int n = tile_o * (2 * kBM) + (int)rank * kBM + row; return EPI != EPI_ACC && n < p.out ? p.sw[n] : 0.0f; };
        auto bias_of = [&](int tile_o) { const int n = tile_o * (2 * kBM) + (int)rank * kBM + row; return EPI != EPI_ACC && p.bias && n < p.out ? p.bias[n] : 0.0f; };
        float sw_next = 0.0f, b_next = 0.0f, ns_next[4], nb_next[4];
        if (kNarrow<EPI> && p.tma_store) narrow_fetch(p.sw, p.bias, o * (2 * kBM) + (int)rank * kBM + q * 32, lane, p.out, ns_next, nb_next);
        else { sw_next = scale_of(o); b_next = bias_of(o); }

        NM_TRACE_EPI_DECL;
        for (int i = 0; i < tile_count && ok; ++i) {
            const int buf = i & 1, n0 = o * (2 * kBM) + (int)rank * kBM, n = n0 + row, t0 = tok * BN;
            if (++o == p.n_out_tiles) { o = 0; ++tok; }
            bool got = ptx::mbar_wait_bounded(acc_full_bar(buf), (i >> 1) & 1u, abort_flag, kWaitLimit);
            ok = __all_sync(0xffffffffu, got);
            if (!ok && lane == 0) raise_timeout();
            if (EPI == EPI_BF16 && p.grouped) ok = ptx::named_bar_and(kNarrowGroup + half, 128, ok);  // the group stops together
            if (!ok) break;
            ptx::tc_fence_after();
            if (ew == 0 && lane == 0) NM_TRACE_TILE(i, 0);
            NM_TRACE_EPI_MARK();
            const bool n_ok = n < p.out;
            if (!p.tma_store) {
                const float c_n = __fmul_rn(sx, sw_next), b_n = b_next;
                sw_next = scale_of(o); b_next = bias_of(o);
                direct_tile<EPI>(lane_taddr + buf * BN, BN, p.tokens - t0, half, EWH, c_n, b_n, p.sy, rsy,
                                 reinterpret_cast<typename EpiOut<EPI>::type*>(kF32<EPI> ? (void*)p.Y : EPI == EPI_ACC ? (void*)p.ACC : p.NARROW), t0, n, p.out, amax,
                                 [&] { release_acc(buf); });
                continue;
            }
            if constexpr (kNarrow<EPI>) {
                float nc[4], nb[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) { nc[k] = __fmul_rn(sx, ns_next[k]); nb[k] = nb_next[k]; }
                narrow_fetch(p.sw, p.bias, o * (2 * kBM) + (int)rank * kBM + q * 32, lane, p.out, ns_next, nb_next);
                constexpr int SUBS = BN / 16 / EWH, PER = Cfg::STORE_STAGE / EW;
                if (EPI == EPI_BF16 && p.grouped)
                    narrow_group_tile<16>(lane_taddr + buf * BN, BN, p.tokens - t0, half, EWH, kNarrowGroup + half, ptx::smem_u32(store_stage) + half * 8192, n_stores,
                                          q, lane, nc, nb, &tmap_y, n0, t0, p.out, stream_out, [&] { release_acc(buf); });
                else
                narrow_tile<EPI, SUBS, kNarrowStage<EPI, PER, SUBS>, 1, 1, true>(lane_taddr + buf * BN, p.tokens - t0, half, EWH, ptx::smem_u32(store_stage) + ew * PER,
                    lane, nc, nb, p.sy, rsy, p.in, &tmap_y, n0 + q * 32, t0, p.out, stream_out, [&] { release_acc(buf); });
                if (ew == 0 && lane == 0) { NM_TRACE_TILE(i, 1); NM_TRACE_EPI_FLUSH(i); }
                continue;
            }
            if constexpr (!kNarrow<EPI>) {
                const float c_n = __fmul_rn(sx, sw_next), b_n = b_next;
                sw_next = scale_of(o); b_next = bias_of(o);
                const int nact = min(CH, (p.tokens - t0 + 31) >> 5);
                // chunks are read one ahead of their conversion
                uint32_t r[2][32];
                if (half >= nact) release_acc(buf);
                else ptx::tmem_ld_32x32(lane_taddr + buf * BN + half * 32, r[0]);
#pragma unroll
                for (int ci = 0; ci < CI; ++ci) {
                    const int c = half + ci * EWH, tc0 = t0 + c * 32;
                    if (c < nact) {
                        ptx::tmem_ld_wait();
                        NM_TRACE_EPI_ADD(0);
                        if (c + EWH >= nact) release_acc(buf);
                        else ptx::tmem_ld_32x32(lane_taddr + buf * BN + (c + EWH) * 32, r[(ci + 1) & 1]);
                        const int jmax = n_ok ? min(32, p.tokens - tc0) : 0;  // outputs of this lane that exist
                        using OT = typename EpiOut<EPI>::type;
                        auto conv = [&](int j) -> OT {
                            float y_abs;
                            const OT o = epi_convert<EPI>(r[ci & 1][j], c_n, b_n, y_abs);
                            if constexpr (EPI == EPI_F32MAX) amax = fmaxf(amax, j < jmax ? y_abs : 0.0f);
                            return o;
                        };
#pragma unroll
                        for (int h = 0; h < 2; ++h) {  // 16 tokens per store, alternating staging tiles
                            if (tc0 + 16 * h >= p.tokens) continue;  // warp-uniform (and the same in all warps of a group)
                            OT* sb = reinterpret_cast<OT*>(my_stage + (n_stores & 1u) * 512);
                            if (lane == 0) ptx::bulk_wait_group_read<1>();  // the store that last used this tile has read it
                            __syncwarp();
                            NM_TRACE_EPI_ADD(1);
#pragma unroll
                            for (int j = 0; j < 16; ++j) sb[j * 32 + lane] = conv(16 * h + j);
                            NM_TRACE_EPI_ADD(2);
                            ptx::fence_proxy_async_smem();
                            __syncwarp();
                            NM_TRACE_EPI_ADD(3);
                            if (lane == 0) {
                                ptx::tma_store_2d_hint(&tmap_y, n0 + q * 32, tc0 + 16 * h, ptx::smem_u32(sb), stream_out);
                                ptx::bulk_commit_group();
                            }
                            NM_TRACE_EPI_ADD(4);
                            ++n_stores;
                        }
                    }
                }
            }
            if (ew == 0 && lane == 0) { NM_TRACE_TILE(i, 1); NM_TRACE_EPI_FLUSH(i); }
        }
        if (lane == 0) ptx::bulk_wait_group_read<0>();  // the stores have read the staging tiles
        if (EPI == EPI_F32MAX) {
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, s));
            if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(p.absmax), __float_as_uint(amax));
        }
    }

    // Neither CTA may release TMEM or exit while the other can still reach into it.
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_arrive();
    ptx::cluster_wait();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

}  // namespace nm
