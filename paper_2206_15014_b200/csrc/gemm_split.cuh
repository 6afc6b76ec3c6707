// One-CTA tiles whose reduction is split over a cluster, for problems with fewer tiles than SMs.
//
// A tile is 128 output channels x BN tokens as in nm_gemm_kernel; the `splits` CTAs of a cluster each multiply their share of
// the k-blocks.  Then CTA r of the cluster gets the tokens [r, r + 1) * BN / splits of everyone's accumulator (int32, 16-byte stores
// into its shared memory), adds them (whole numbers: any order gives the same) and finishes those tokens.
// What bounds such a problem is the chain of one CTA: index metadata, k-blocks that each take a load's latency over the depth of
// the ring, the epilogue.  A split shortens the first two for one exchange through distributed shared memory: 384 tokens 4096 -> 1024
// (eight output tiles) 11.9 us unsplit, 7.3 in clusters of four with 96 tokens, 8.7 in pairs; 1 token 8192 -> 1024 19.7 -> 5.6.
//   warp 0      TMA producer
//   warp 1      allocates TMEM; one lane waits for the stages and issues the MMAs
//   warps 2-9   index metadata of the CTA's k-blocks into TMEM (the first four), exchange, epilogue with direct stores
//   warps 10-21 (XF: weights not in tensor-core form) three groups of four build the weight tiles as in nm_gemm_kernel
// An expired wait: the MMA warp issues nothing more, so no stage comes free after the one that was missed and nobody goes round the ring
// beyond it; the epilogue warps, which wait in vain for the accumulator, set the flag of every CTA of the cluster between its two
// barriers, and no CTA of it writes outputs.
#pragma once

namespace nm {

constexpr int kSplitThreads = 32 * 10;
template <bool XF> constexpr int kSplitThreadsOf = kSplitThreads + (XF ? 32 * 4 * kBuildGroups : 0);
constexpr int kSplitMaxKb = 32;   // k-blocks of a CTA: their metadata (4 columns each) lies beside the accumulator

template <bool SPARSE, int BN>
struct SplitCfg {
    static constexpr int A_ROW = SPARSE ? 64 : 128;
    static constexpr int A_BYTES = kBM * A_ROW;
    static constexpr int B_BYTES = BN * 128;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int RECV = kBM * BN * 4;  // partial sums of the other CTAs: (splits - 1) * BN / splits columns
    static constexpr int FIT = (kSmemLimit - kSmemTail - RECV - 1024) / STAGE;
    static constexpr int STAGES = FIT < 8 ? FIT : 8;
    static constexpr int SMEM = STAGES * STAGE + RECV + kSmemTail + 1024;
    static constexpr int META_COL = BN;
    static_assert(META_COL + 4 * kSplitMaxKb <= kTmemCols, "tensor memory");
    static_assert(STAGE % 1024 == 0 && A_BYTES % 1024 == 0, "swizzle alignment");
};

template <bool SPARSE, int BN, int EPI, bool XF>
__global__ void __launch_bounds__(kSplitThreadsOf<XF>, 1)
nm_gemm_split_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x, const GemmParams p,
                     const int splits) {
    using Cfg = SplitCfg<SPARSE, BN>;
    constexpr int S = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* recv = smem + S * Cfg::STAGE;
    uint64_t* bars = reinterpret_cast<uint64_t*>(recv + Cfg::RECV);
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    const uint32_t acc_full_bar = bar0 + 8u * (2 * S), meta_bar = acc_full_bar + 8u, drained_bar = acc_full_bar + 16u;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 3);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* never_flag = tmem_slot + 2;  // stays 0: for the drain wait after an abort
    uint32_t* lut = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(bars) + 512);  // XF: slot tables (xform.cuh)

    const int warp = (int)ptx::warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_ctarank();
    const int tile = blockIdx.x / splits, out_tile = tile / p.n_tok_tiles;
    const int n0 = out_tile * kBM, t0 = (tile - out_tile * p.n_tok_tiles) * BN;
    const int kb_begin = rank * p.kblocks / splits, kb_count = (rank + 1) * p.kblocks / splits - kb_begin;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { ptx::mbar_init(full_bar(s), XF ? 5 : 1); ptx::mbar_init(empty_bar(s), 1); }
        ptx::mbar_init(acc_full_bar, 1);
        ptx::mbar_init(meta_bar, 4);
        ptx::mbar_init(drained_bar, 1);
        *abort_flag = 0;
        *never_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_w);
        ptx::prefetch_tensormap(&tmap_x);
    }
    if (XF) xf::build_lut(lut, threadIdx.x, blockDim.x);
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(tmem_slot), kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = ptx::warp_uniform(*tmem_slot);
    ptx::cluster_arrive();  // the others' shared memory may be written once all of them run (waited for before the exchange)
    ptx::grid_dep_wait();   // nothing in global memory is read or written before this point
    ptx::grid_dep_launch();

    auto raise_timeout = [&]() {
        *abort_flag = 1;
        if (p.status) atomicOr(p.status, NM_STATUS_TIMEOUT);
    };

    if (warp == 0) {
        if (lane == 0) {
            for (int it = 0; it < kb_count; ++it) {
                const int s = it % S, kb = kb_begin + it;
                if (!ptx::mbar_wait_bounded(empty_bar(s), ((it / S) & 1u) ^ 1u, abort_flag, kWaitLimit)) { raise_timeout(); break; }
                if (NM_SKIP_STAGE((uint32_t)it)) continue;
                const uint32_t a_dst = ptx::smem_u32(smem + s * Cfg::STAGE);
                ptx::mbar_expect_tx(full_bar(s), XF ? Cfg::B_BYTES : Cfg::STAGE);
                if (!XF) ptx::tma_load_2d(a_dst, &tmap_w, kb * Cfg::A_ROW, n0, full_bar(s));
                ptx::tma_load_2d(a_dst + Cfg::A_BYTES, &tmap_x, kb * 128, t0, full_bar(s));
            }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = ptx::idesc_i8(kBM, BN, SPARSE);
        const uint64_t a_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(smem), SPARSE ? 64 : 128, SPARSE ? ptx::kSwizzle64 : ptx::kSwizzle128);
        const uint64_t b_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(smem) + Cfg::A_BYTES, 128, ptx::kSwizzle128);
        bool go = true;
        if (SPARSE) {
            go = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(meta_bar, 0, abort_flag, kWaitLimit));
            ptx::tc_fence_after();
        }
        uint32_t s = 0, parity = 0;
        for (int it = 0; it < kb_count && go; ++it) {
            go = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(full_bar(s), parity, abort_flag, kWaitLimit));
            if (!go) break;
            if (ptx::elect_one()) {
                const uint64_t a = ptx::desc_advance(a_desc0, s * Cfg::STAGE), b = ptx::desc_advance(b_desc0, s * Cfg::STAGE);
                if constexpr (SPARSE) {
#pragma unroll
                    for (int j = 0; j < 2; ++j)  // 64 logical k each: 32 stored bytes of A, 64 of B
                        ptx::mma_sp_i8(tmem_base, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 64 * j),
                                       tmem_base + Cfg::META_COL + it * 4 + 2 * j, idesc, (it | j) != 0);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)  // 32 k each
                        ptx::mma_i8(tmem_base, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 32 * j), idesc, (it | j) != 0);
                }
                ptx::tc_commit(empty_bar(s));
            }
            __syncwarp();
            if (++s == S) { s = 0; parity ^= 1u; }
        }
        if (ptx::elect_one()) {
            if (go) ptx::tc_commit(acc_full_bar);
            else raise_timeout();
            ptx::tc_commit(drained_bar);  // everything issued has retired before TMEM is released
            ptx::mbar_wait_bounded(drained_bar, 0, never_flag, kWaitLimit);
        }
        __syncwarp();
    } else if (XF && warp >= kSplitThreads / 32) {
        // one thread builds one row of a k-block; group g takes k-blocks g, g + G, ... (see nm_gemm_kernel)
        constexpr int G = kBuildGroups;
        static_assert(S > G, "every group needs a stage of its own in flight");
        const int bw = warp - kSplitThreads / 32, grp = bw >> 2, tr = (bw & 3) * 32 + lane, nr = n0 + tr;
        const int cb = xf::code_bytes(p.pat), mb = xf::meta_bytes(p.pat);
        const bool row_ok = nr < p.out;
        const uint8_t* v = p.values + (size_t)(row_ok ? nr : 0) * p.vrow_bytes + (size_t)kb_begin * cb;
        const uint8_t* m = reinterpret_cast<const uint8_t*>(p.meta) + (size_t)(row_ok ? nr : 0) * p.mrow_bytes + (size_t)kb_begin * mb;
        xf::Raw cur = xf::load_raw(p.pat, v + (size_t)grp * cb, m + (size_t)grp * mb, row_ok && grp < kb_count);
        for (int it = grp; it < kb_count; it += G) {
            const xf::Raw nxt = xf::load_raw(p.pat, v + (size_t)(it + G) * cb, m + (size_t)(it + G) * mb, row_ok && it + G < kb_count);
            const bool got = lane != 0 || ptx::mbar_wait_bounded(empty_bar(it % S), ((it / S) & 1u) ^ 1u, abort_flag, kWaitLimit);
            if (!__all_sync(0xffffffffu, got)) { if (lane == 0) raise_timeout(); break; }
            uint32_t w[SPARSE ? 16 : 32];
            xf::build_row<SPARSE>(p.pat, cur, lut, w);
            xf::store_row<SPARSE>(smem + (it % S) * Cfg::STAGE, tr, w);
            ptx::fence_proxy_async_smem();  // the MMA reads the tile through the async proxy
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(full_bar(it % S));
            cur = nxt;
        }
    } else {
        const int ew = warp - 2, q = warp & 3, half = ew >> 2, row = q * 32 + lane, n = n0 + row;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16);
        const int slice = BN / splits, chunks = slice >> 3;  // tokens that a CTA finishes, in chunks of eight
        float c_n = 0.0f, b_n = 0.0f;
        if (SPARSE && half == 0) {
            // index metadata of this lane's weight row for the CTA's k-blocks, several pieces in flight together; rows past the end get a
            // valid "positions 0,1" pattern, their products are discarded
            constexpr int kBatch = XF ? 4 : 8;
            const uint4 idle = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
            const int piece = XF ? xf::meta_bytes(p.pat) : 16;  // stored bytes of a k-block
            const uint8_t* src = reinterpret_cast<const uint8_t*>(p.meta) + (size_t)(n < p.out ? n : 0) * (XF ? p.mrow_bytes : 4 * p.mrow_words) + (size_t)kb_begin * piece;
            for (int c0 = 0; c0 < kb_count; c0 += kBatch) {
                uint4 w[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    w[j] = idle;
                    if (n < p.out && c0 + j < kb_count) w[j] = XF ? xf::meta_raw(p.pat, src + (size_t)(c0 + j) * piece) : xf::ldg16(src + (size_t)(c0 + j) * piece);
                }
                if constexpr (XF) {
#pragma unroll
                    for (int j = 0; j < kBatch; ++j)
                        if (n < p.out && c0 + j < kb_count) w[j] = xf::hw_meta(p.pat, w[j], lut);
                }
#pragma unroll
                for (int j = 0; j < kBatch; ++j)
                    if (c0 + j < kb_count) ptx::tmem_st_32x4(lane_taddr + Cfg::META_COL + 4 * (c0 + j), w[j].x, w[j].y, w[j].z, w[j].w);
            }
            ptx::tmem_st_wait();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(meta_bar);
        }
        if (EPI != EPI_ACC) {
            const float sx = p.sx_dev ? *p.sx_dev : p.sx_host;
            c_n = n < p.out ? __fmul_rn(sx, p.sw[n]) : 0.0f;
            b_n = n < p.out && p.bias ? p.bias[n] : 0.0f;
        }
        const bool ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(acc_full_bar, 0, abort_flag, kWaitLimit));
        if (!ok && lane == 0) raise_timeout();
        ptx::tc_fence_after();
        __syncwarp();
        ptx::cluster_wait();
        if (__builtin_expect(ok, 1)) {
            // The other CTAs' tokens: [sender][chunk][two halves of four tokens][128 channels] of 16 bytes at the receiver.
            const uint32_t base = ptx::smem_u32(recv) + (uint32_t)row * 16u;
            for (int u = half; u < (splits - 1) * chunks; u += 2) {
                const int d = u / chunks, ch = u - d * chunks;
                const int to = rank + 1 + d < splits ? rank + 1 + d : rank + 1 + d - splits;
                const int col = to * slice + ch * 8;
                if (t0 + col >= p.tokens) continue;  // nobody will read them (the same for the whole warp)
                uint32_t r[8];
                ptx::tmem_ld_32x8(lane_taddr + col, r);
                ptx::tmem_ld_wait();
                // this CTA is the receiver's number splits - 2 - d
                const uint32_t dst = ptx::map_to_cta(base + (uint32_t)(((splits - 2 - d) * chunks + ch) * 2) * (kBM * 16u), (uint32_t)to);
                ptx::st_cluster_v4(dst, r[0], r[1], r[2], r[3]);
                ptx::st_cluster_v4(dst + kBM * 16u, r[4], r[5], r[6], r[7]);
            }
        } else if (lane < splits) {
            // no sums from here: everyone's flag, so that nobody finishes tokens from what was never sent
            ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32((const void*)abort_flag), (uint32_t)lane), 1u);
        }
        __syncwarp();
        ptx::cluster_arrive();
        ptx::cluster_wait();
        const bool whole = *abort_flag == 0u;  // every CTA has sent its sums; otherwise nothing is stored
        const float rsy = EPI == EPI_Q8 ? __frcp_rn(p.sy) : 0.0f;
        float amax = 0.0f;
        using OT = typename EpiOut<EPI>::type;
        OT* const Y = reinterpret_cast<OT*>(kF32<EPI> ? (void*)p.Y : EPI == EPI_ACC ? (void*)p.ACC : p.NARROW);
        for (int ch = half; ch < chunks; ch += 2) {
            const int col = rank * slice + ch * 8, t = t0 + col;
            if (t >= p.tokens) break;
            uint32_t r[8];
            ptx::tmem_ld_32x8(lane_taddr + col, r);
            ptx::tmem_ld_wait();
            for (int d = 0; d < splits - 1; ++d) {
                const uint4* part = reinterpret_cast<const uint4*>(recv) + (size_t)((d * chunks + ch) * 2) * kBM + row;
                const uint4 a = part[0], b = part[kBM];
                r[0] += a.x; r[1] += a.y; r[2] += a.z; r[3] += a.w;
                r[4] += b.x; r[5] += b.y; r[6] += b.z; r[7] += b.w;
            }
            const int jmax = whole && n < p.out ? min(8, p.tokens - t) : 0;
            OT* dst = Y + (size_t)t * p.out + n;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                OT o;
                if constexpr (EPI == EPI_Q8) {
                    float worst = 0.0f;
                    o = epi_convert_q8_fast(r[j], c_n, b_n, rsy, worst);
                    if (!(worst <= 0.49996948f)) o = (OT)(int8_t)quantise8_exact_call(__fmaf_rn((float)(int)r[j], c_n, b_n), p.sy);
                } else {
                    float y_abs;
                    o = epi_convert<EPI>(r[j], c_n, b_n, y_abs);
                    if constexpr (EPI == EPI_F32MAX) amax = fmaxf(amax, j < jmax ? y_abs : 0.0f);
                }
                if (j < jmax) dst[(size_t)j * p.out] = o;
            }
        }
        if (EPI == EPI_F32MAX) {
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, s));
            if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(p.absmax), __float_as_uint(amax));
        }
    }
    if (warp < 2 || warp >= kSplitThreads / 32) {  // the cluster's barriers of the others; apart, so that the builders hold nothing of the epilogue's
        __syncwarp();
        ptx::cluster_wait();
        ptx::cluster_arrive();
        ptx::cluster_wait();
    }
    // after an expired wait copies may still be on their way into this CTA's shared memory
    if (threadIdx.x == 0 && *abort_flag) ptx::wait_clocks(kAbortDrain);
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace nm
