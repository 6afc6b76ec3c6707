// Integer N:M linear layer on tcgen05 tensor cores with the dequantisation epilogue fused in.
//
// The sparse operand of tcgen05.mma.sp is A, so the kernel computes D = Wq * X^T: a tile is
// 128 output channels (TMEM lanes) x BN tokens (TMEM columns).  In TMEM one lane therefore holds
// one output channel, whose scale and bias are per-thread constants in the epilogue.
//
// One persistent CTA per SM walks a contiguous range of tiles ordered output-tile-major, so the
// weight tile (and its metadata) changes at most a few times per CTA.
//   warp 0      TMA producer: X tile and W tile of every 128-wide k-block into a ring of stages
//   warp 1      allocates TMEM; one lane issues tcgen05.mma[.sp] and commits to mbarriers.  It never
//               polls an mbarrier itself: a wait in the issuing thread leaves the tensor pipe idle for
//               its whole latency, so readiness reaches it through hardware named barriers
//   warps 2-9   copy the index metadata of the current 128 output channels into TMEM
//               (tcgen05.st, once per output tile, whole K), then run the epilogue of tile i
//               (tcgen05.ld -> fma -> shared staging -> TMA store) while the MMAs of tile i+1 fill
//               the other accumulator; two warps share a TMEM lane quarter and alternate chunks
//   warp 10     gate: waits on the "stage full" / "accumulator free" / "metadata ready" mbarriers and
//               relays each k-block to warp 1 with bar.arrive
//   warps 11-   (only for weights that are not stored in the tensor core's form: 4-bit codes, 1:4, 2:8,
//               1:8, 4:8) groups of four warps build the weight tile of every k-block in shared
//               memory from the packed codes and metadata (xform.cuh), the groups taking k-blocks
//               round-robin; the producer then loads X only
// Every mbarrier wait is bounded; on expiry the CTA raises NM_STATUS_TIMEOUT, drains and exits.
#include "common.cuh"
#include "sm100_ptx.cuh"
#include "xform.cuh"
#include "tmap.cuh"
#include "tileplan.cuh"
#include <cuda.h>
#include <cuda_runtime.h>
#include <mutex>
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <initializer_list>

namespace nm {

constexpr int kBM = 128;            // output channels per tile (MMA M)
constexpr int kKB = 128;            // reduction elements per pipeline stage
constexpr int kEpiWarps = 8;        // epilogue warps when the weights come straight from TMA (two per TMEM lane quarter)
constexpr int kEpiWarpsXf = 8;      // with the weight-building warps present
constexpr int kBuildGroups = 3;     // groups of four weight-building warps; group g takes k-blocks g, g + groups, ...
constexpr int kGemmThreads = 32 * (3 + kEpiWarps);        // producer, MMA, epilogue warps, gate
constexpr int kXformThreads = 32 * (3 + kEpiWarpsXf + 4 * kBuildGroups); // ... plus the warps that build the weight tiles
constexpr int kTmemCols = 512;
constexpr int kSmemLimit = 232448;  // 227 KB of dynamic shared memory per CTA
constexpr int kSmemTail = 2048;     // barriers, TMEM slot, abort flag, slot tables
constexpr int kStoreStage = 8 * 4096;  // per epilogue warp two [16 tokens][32 channels] fp32 staging tiles, used alternately
constexpr int kMaxStages = 7;       // the relay cycles through 8 named barriers
#ifndef NM_WAIT_LIMIT
#define NM_WAIT_LIMIT (1ll << 31)
#endif
constexpr long long kAbortDrain = 1ll << 17;  // SM clocks a producer of a CTA pair waits after an expired wait so that its copies in flight land
// ... and its gate waits after one before it lets the MMA warp run on (see relay_step): a role in a wait looks at the abort flag
// at every 64th poll, a poll that fails takes about 7800 clocks (measured), so all of them have left after half a million.
constexpr long long kGateDrain = 1ll << 21;
constexpr long long kWaitLimit = NM_WAIT_LIMIT;  // SM clocks per device-side wait (about a second; test builds shorten it)

// What the epilogue writes: y = fma(acc, sx * sw[o], b[o]) as fp32; the raw int32 accumulators; y re-quantised
// to 8 bits with a scale fixed ahead of time (Eq. 5, b = 8); y rounded to bfloat16.
enum { EPI_F32 = 0, EPI_ACC = 1, EPI_Q8 = 2, EPI_BF16 = 3, EPI_F32MAX = 4 };  // EPI_F32MAX: fp32 and the running max|y|
template <int EPI> constexpr bool kF32 = EPI == EPI_F32 || EPI == EPI_F32MAX;
template <int EPI> struct EpiOut { using type = uint32_t; };          // fp32 / int32 move as 32-bit patterns
template <> struct EpiOut<EPI_Q8> { using type = uint8_t; };
template <> struct EpiOut<EPI_BF16> { using type = uint16_t; };
// EPI_Q8 a value at a time (split kernel, direct stores), without a branch: the code from the reciprocal rsy = RN(1 / sy), exact unless the product sits
// within 2^-15 of a rounding tie (6 values in 100000), where only the IEEE division decides.  `worst` keeps the largest
// distance of a product from its rounded integer; beyond 0.49996948 the caller takes the code from the exact quantiser.  The clamp to [-128.49, 127.49] before the add of 1.5 * 2^23 (whose own rounding rounds to
// the nearest-even integer) leaves nothing to clamp afterwards, and the low byte of the sum's bit pattern
// 0x4B400000 + code is the code.
__device__ __forceinline__ uint8_t epi_convert_q8_fast(uint32_t acc, float c_n, float b_n, float rsy, float& worst) {
    constexpr float kMagic = 12582912.0f;
    const float y = __fmaf_rn((float)(int)acc, c_n, b_n);
    const float qc = fminf(fmaxf(__fmul_rn(y, rsy), -128.49f), 127.49f);
    const float t = __fadd_rn(qc, kMagic);
    worst = fmaxf(worst, fabsf(__fsub_rn(qc, __fsub_rn(t, kMagic))));
    return (uint8_t)__float_as_uint(t);
}

// The exact quantiser as a call: the repair of near-ties runs for a few values in 10^5, its code stays out of the loops.
__device__ __noinline__ int quantise8_exact_call(float y, float sy) { return quantise8_exact(y, sy); }

// Narrow outputs leave through [tokens][32 channels] tiles of the warp's own (narrow_tile), or [tokens][128 channels] tiles that the four warps of a
// TMEM-lane-quarter group fill together (narrow_group_tile): there a named barrier per group orders the fills against the one warp
// that issues the TMA store, kNarrowAgree + half makes the group take a timed-out wait together so that nobody is left alone on it.
template <int EPI> constexpr bool kNarrow = EPI == EPI_Q8 || EPI == EPI_BF16;
constexpr uint32_t kNarrowGroup = 9, kNarrowAgree = 13;  // named barriers: one per group from kNarrowGroup on

// One output element from an accumulator: fp32 value y, then the narrowing the epilogue kind asks for.
template <int EPI>
__device__ __forceinline__ typename EpiOut<EPI>::type epi_convert(uint32_t acc, float c_n, float b_n, float& y_abs) {
    static_assert(EPI != EPI_Q8, "epi_convert_q8_fast or narrow_convert");
    if constexpr (EPI == EPI_ACC) {
        y_abs = 0.0f;
        return acc;
    } else {
        const float y = __fmaf_rn((float)(int)acc, c_n, b_n);
        y_abs = fabsf(y);
        if constexpr (kF32<EPI>) {
            return __float_as_uint(y);
        } else {
            uint16_t h;
            asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(y));
            return h;
        }
    }
}

// Four codes of the exact quantiser, for the few values in 10^5 next to a rounding tie: a call, out of the loops' way.
__device__ __noinline__ uint32_t quantise8_exact4(float y0, float y1, float y2, float y3, float sy) {
    return (uint32_t)(quantise8_exact(y0, sy) & 0xff) | (uint32_t)(quantise8_exact(y1, sy) & 0xff) << 8 |
           (uint32_t)(quantise8_exact(y2, sy) & 0xff) << 16 | (uint32_t)(quantise8_exact(y3, sy) & 0xff) << 24;
}

// 16 tokens of a warp's 32 channels, as the two loads of the stmatrix layout left them in r, converted: two bfloat16 or four codes a word.
template <int EPI>
__device__ __forceinline__ void narrow_convert(const uint32_t* r, uint32_t* pk, const float (&c)[4], const float (&b)[4], float sy, float rsy, float far) {
    constexpr float kMagic = 12582912.0f;
    const uint64_t c01[2] = {ptx::pack_f32x2(c[0], c[0]), ptx::pack_f32x2(c[2], c[2])}, c23[2] = {ptx::pack_f32x2(c[1], c[1]), ptx::pack_f32x2(c[3], c[3])};
    const uint64_t b01[2] = {ptx::pack_f32x2(b[0], b[0]), ptx::pack_f32x2(b[2], b[2])}, b23[2] = {ptx::pack_f32x2(b[1], b[1]), ptx::pack_f32x2(b[3], b[3])};
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // k = 2 * (lane half) + column group
        const uint32_t* x = r + 4 * k;
        const uint64_t y01 = ptx::fma_f32x2(ptx::pack_f32x2((float)(int)x[0], (float)(int)x[1]), c01[k >> 1], b01[k >> 1]);
        const uint64_t y23 = ptx::fma_f32x2(ptx::pack_f32x2((float)(int)x[2], (float)(int)x[3]), c23[k >> 1], b23[k >> 1]);
        float y0, y1, y2, y3;
        ptx::unpack_f32x2(y01, y0, y1);
        ptx::unpack_f32x2(y23, y2, y3);
        if constexpr (EPI == EPI_BF16) {
            pk[2 * k] = ptx::cvt_bf16x2(y0, y1);
            pk[2 * k + 1] = ptx::cvt_bf16x2(y2, y3);
        } else {
            const uint64_t rs2 = ptx::pack_f32x2(rsy, rsy), magic2 = ptx::pack_f32x2(kMagic, kMagic), minus2 = ptx::pack_f32x2(-1.0f, -1.0f);
            const uint64_t t01 = ptx::fma_f32x2(y01, rs2, magic2), t23 = ptx::fma_f32x2(y23, rs2, magic2);
            float d0, d1, d2, d3, t[4];
            ptx::unpack_f32x2(ptx::fma_f32x2(y01, rs2, ptx::fma_f32x2(t01, minus2, magic2)), d0, d1);
            ptx::unpack_f32x2(ptx::fma_f32x2(y23, rs2, ptx::fma_f32x2(t23, minus2, magic2)), d2, d3);
            ptx::unpack_f32x2(t01, t[0], t[1]);
            ptx::unpack_f32x2(t23, t[2], t[3]);
            auto code = [&](int i) { return __float_as_int(t[i]) - 0x4B400000; };
            pk[k] = ptx::pack_sat_s8(code(0), code(1), ptx::pack_sat_s8(code(2), code(3), 0u));
            if (!(ptx::max_abs_nan(d2, d3, ptx::max_abs_nan(d0, d1, far)) <= 0.49996948f)) pk[k] = quantise8_exact4(y0, y1, y2, y3, sy);
        }
    }
}

// The same words, transposed into a tile [16 tokens][32 channels] in the 64-byte (bfloat16) or 32-byte swizzle of the store's tensor map, so that
// no two rows of a matrix meet in a bank.
template <int EPI>
__device__ __forceinline__ void narrow_fill(uint32_t tile, const uint32_t* pk, int lane) {
    const uint32_t token = lane & 7;
    if constexpr (EPI == EPI_BF16) {
#pragma unroll
        for (int g = 0; g < 2; ++g)  // matrix i: channels 8 i .. 8 i + 7, eight tokens
            ptx::stmatrix_trans_b16(tile + (8 * g + token) * 64 + (((lane >> 3) ^ (token >> 1)) << 4), pk[2 * g], pk[2 * g + 1], pk[4 + 2 * g], pk[4 + 2 * g + 1]);
    } else {  // matrix i: channels 16 (i % 2) .. + 15, tokens 8 (i / 2) .. + 7
        ptx::stmatrix_trans_b8(tile + (8 * (lane >> 4) + token) * 32 + ((((lane >> 3) & 1) ^ (token >> 2)) << 4), pk[0], pk[2], pk[1], pk[3]);
    }
}

// 1 where a product of a thread's four channels in narrow_tile could leave the range in which int8 codes are taken from bits (then every
// code comes from the exact division), 0 otherwise: an accumulator is at most in * 2^14, a product then below 2^23.  A bound per tile, which
// nothing waits for before the first check, instead of a clamp per value: a scale that small (200 times under one that spreads the
// outputs over the codes) saturates nearly every output.
template <int EPI>
__device__ __forceinline__ float narrow_far(float rsy, const float (&c)[4], const float (&b)[4], int in) {
    if (EPI != EPI_Q8) return 0.0f;
    const float c_max = ptx::max_abs_nan(c[0], c[1], ptx::max_abs_nan(c[2], c[3], 0.0f)), b_max = ptx::max_abs_nan(b[0], b[1], ptx::max_abs_nan(b[2], b[3], 0.0f));
    return (c_max * ((float)in * 16384.0f) + b_max) * rsy < 8388608.0f ? 0.0f : 1.0f;
}

// Tiles of 16 tokens that BYTES of staging memory hold, of the SUBS that a warp has to do at most.
template <int EPI, int BYTES, int SUBS> constexpr int kNarrowStage = BYTES / (EPI == EPI_BF16 ? 1024 : 512) < SUBS ? BYTES / (EPI == EPI_BF16 ? 1024 : 512) : SUBS;

// A warp's 32 channels of an output tile as int8 or bfloat16.  The groups of four warps (one per TMEM lane quarter) share the tile's tokens evenly.
//
// The warp reads 16 tokens from the accumulator in the fragment layout of stmatrix (a thread has two neighbouring tokens of four channels),
// converts them in pairs, and writes them transposed, 16 bytes of a token's row at a time, into staging tiles of its own, in rounds of
// as many as its staging memory holds.  With a lane per channel every value took a conversion and a store instruction of its own: 4
// instructions for a bfloat16, 11 for an exact int8 code, 2.2 and 5.3 so.  No warp waits for another: staging tiles shared by the four
// warps of a group (rows of 128 channels) took a barrier or two a round, and 300 clocks for the group to agree on an expired wait; 16384
// tokens 768 -> 3072 bfloat16 31.7 -> 28.9 us (35.0 with a lane per channel), int8 outputs over 263 shapes and formats 0.96 of the time.
// int8: t = fma(y, rsy, 1.5 * 2^23) rounds the product to the nearest-even integer, which saturates to the code; `d` is the product's
// distance from it, and within 2^-15 of a tie (or NaN) the IEEE division decides.  Below -1.5 * 2^23 t turns negative and the integer
// that its bits give, less those of 1.5 * 2^23, wraps round to the other end: narrow_far.
//
// acc: TMEM address of the tile's first column in this warp's lane quarter.  c, b: scale and bias of channels lane / 4 + 8 i of the quarter.
// valid: tokens of the tile that exist.  n: the warp's first channel.  LD: pieces of 16 tokens that it has in registers together.
// release(): it has read its accumulator.
template <int EPI, int SUBS, int STAGE, int BUFS, int LD, bool HINT, typename Release>
__device__ __forceinline__ void narrow_tile(uint32_t acc, int valid, int group, int groups, uint32_t stage, int lane, const float (&c)[4], const float (&b)[4],
                                            float sy, float rsy, int in, const CUtensorMap* tmap_y, int n, int t0, int out, uint64_t policy, Release release) {
    constexpr uint32_t TILE = EPI == EPI_BF16 ? 1024 : 512;
    const float far = narrow_far<EPI>(rsy, c, b, in);
    const int all = min((valid + 15) >> 4, SUBS * groups), share = (all + groups - 1) / groups;
    const int first = group * share, last = min(first + share, all);
    if (first >= last) { release(); return; }
    uint32_t buf = 0;
#pragma unroll 1
    for (int u = first; u < last; u += STAGE) {
        const uint32_t tile = stage + buf * (STAGE * TILE);
#pragma unroll
        for (int h = 0; h < STAGE; h += LD) {
            if (u + h >= last) break;
            uint32_t r[LD][16];
#pragma unroll
            for (int k = 0; k < LD; ++k) {  // past the last 16 tokens: other columns, not used
                ptx::tmem_ld_16x256x2(acc + 16 * (u + h + k), r[k]);
                ptx::tmem_ld_16x256x2(acc + (16u << 16) + 16 * (u + h + k), r[k] + 8);
            }
            ptx::tmem_ld_wait();
            if (u + h + LD >= last) release();
            uint32_t pk[LD][EPI == EPI_Q8 ? 4 : 8];
#pragma unroll
            for (int k = 0; k < LD; ++k) narrow_convert<EPI>(r[k], pk[k], c, b, sy, rsy, far);
            if (h == 0) {  // the stores that last used the staging tiles have read them
                if (lane == 0) {
                    if (BUFS == 1 || u == first) ptx::bulk_wait_group_read<0>();
                    else ptx::bulk_wait_group_read<1>();
                }
                __syncwarp();
            }
#pragma unroll
            for (int k = 0; k < LD; ++k)
                if (h + k < STAGE) narrow_fill<EPI>(tile + (h + k) * TILE, pk[k], lane);
        }
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && n < out) {
            for (int h = 0; h < min(STAGE, last - u); ++h) {
                if (HINT) ptx::tma_store_2d_hint(tmap_y, n, t0 + 16 * (u + h), tile + h * TILE, policy);
                else ptx::tma_store_2d(tmap_y, n, t0 + 16 * (u + h), tile + h * TILE);
            }
            ptx::bulk_commit_group();
        }
        __syncwarp();
        if (BUFS == 2) buf ^= 1u;
    }
}

// The same for bfloat16 with the four warps of a group sharing staging tiles [UNIT tokens][128 channels], two in turn, so that the rows
// that leave are whole 128-byte lines and not halves of them: where Y goes to HBM as fast as it can the halves cost more than the group's
// barriers.  The 512-channel kernel always (with halves 1.008 of the time with packed 4-bit codes, up to 1.038), the pair kernels for shorter reductions from
// 192 MB of Y on (32768 tokens 1024 -> 3072 64.3 us so, 66.1 with halves; 1024 -> 4096 with 4-bit codes 108.9 / 112.4,
// with dense weights 104.0 / 112.3; below it the halves are
// better: 16384 tokens 1024 -> 4096 40.3 / 38.6).
constexpr size_t kNarrowGroupBytes = (size_t)192 << 20;
template <int UNIT, typename Release>
__device__ __forceinline__ void narrow_group_tile(uint32_t acc, int columns, int valid, int group, int groups, uint32_t bar, uint32_t stage, uint32_t& n_stores,
                                                  int q, int lane, const float (&c)[4], const float (&b)[4], const CUtensorMap* tmap_y, int n0, int t0,
                                                  int out, uint64_t policy, Release release) {
    constexpr uint32_t ROW = 128, BOX = UNIT * ROW, TILE = 2 * BOX;  // two boxes of 64 channels
    const int units = (min(valid, columns) + UNIT - 1) / UNIT;       // units that hold tokens (the same for the whole group)
    if (group >= units) release();
#pragma unroll 1
    for (int u = group; u < units; u += groups) {
        const uint32_t tile = stage + (n_stores & 1u) * TILE;
#pragma unroll
        for (int h = 0; h < UNIT / 16; ++h) {
            uint32_t r[16], pk[8];
            ptx::tmem_ld_16x256x2(acc + u * UNIT + 16 * h, r);
            ptx::tmem_ld_16x256x2(acc + (16u << 16) + u * UNIT + 16 * h, r + 8);
            ptx::tmem_ld_wait();
            if (h == UNIT / 16 - 1 && u + groups >= units) release();
            narrow_convert<EPI_BF16>(r, pk, c, b, 0.0f, 0.0f, 0.0f);
            if (h == 0) {
                if (q == 0 && lane == 0) ptx::bulk_wait_group_read<1>();  // the store before the last has read this tile
                ptx::named_bar_sync(bar, 128);
            }
            const uint32_t token = lane & 7;
#pragma unroll
            for (int g = 0; g < 2; ++g)  // as in narrow_fill
                ptx::stmatrix_trans_b16(tile + (q >> 1) * BOX + (16 * h + 8 * g + token) * ROW + ((((q & 1) * 4 + (lane >> 3)) ^ token) << 4),
                                        pk[2 * g], pk[2 * g + 1], pk[4 + 2 * g], pk[4 + 2 * g + 1]);
        }
        ptx::fence_proxy_async_smem();
        ptx::named_bar_sync(bar, 128);
        if (q == 0 && lane == 0) {
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                if (x && n0 + 64 * x >= out) break;
                ptx::tma_store_2d_hint(tmap_y, n0 + 64 * x, t0 + u * UNIT, tile + x * BOX, policy);
            }
            ptx::bulk_commit_group();
        }
        ++n_stores;
    }
}

// One output tile where TMA cannot store the rows of Y (not whole units of 16 bytes): a lane per channel, 32 tokens of an accumulator at a
// time, stored straight from the registers.  Staged in shared memory and written by rows of 128 channels, with a quarter of the partial
// sectors, it was slower: bfloat16 1024 -> 1002, 8192 tokens, packed 4-bit codes 28 us against 18, fp32 23 against 17.  Out of the kernels' main
// loops, so that those stay short.  EIGHTS: of the last tokens no more than there are, to eight, in the one-CTA kernel without builder warps: 18
// tokens 128 -> 2687 bfloat16, dense weights 2.63 -> 2.39 us, 2:4 2.78 -> 2.55.  The kernels with builder warps pay for more code with fetching it
// (1 % of every other call), int8 codes gain nothing, being a branch each.
template <int EPI, bool EIGHTS = false, typename Release>
__device__ __forceinline__ void direct_tile(uint32_t acc, int columns, int valid, int group, int groups, float c_n, float b_n, float sy, float rsy,
                                            typename EpiOut<EPI>::type* Y, int t0, int n, int out, float& amax, Release release) {
    using OT = typename EpiOut<EPI>::type;
    const int chunks = (min(valid, columns) + 31) >> 5;
    if (group >= chunks) release();
#pragma unroll 1
    for (int c = group; c < chunks; c += groups) {
        uint32_t r[32];
        ptx::tmem_ld_32x32(acc + c * 32, r);
        ptx::tmem_ld_wait();
        if (c + groups >= chunks) release();
        const int count = min(32, valid - c * 32);
        OT* dst = Y + (size_t)(t0 + c * 32) * out + n;
        auto conv = [&](int j) -> OT {
            float y_abs = 0.0f;
            OT o;
            if constexpr (EPI == EPI_Q8) {
                float worst = 0.0f;
                o = epi_convert_q8_fast(r[j], c_n, b_n, rsy, worst);
                if (!(worst <= 0.49996948f)) o = (OT)(int8_t)quantise8_exact_call(__fmaf_rn((float)(int)r[j], c_n, b_n), sy);
            } else {
                o = epi_convert<EPI>(r[j], c_n, b_n, y_abs);
            }
            if constexpr (EPI == EPI_F32MAX) amax = fmaxf(amax, y_abs);
            return o;
        };
        if (n < out) {
            if (count == 32) {  // no branch per store
#pragma unroll
                for (int j = 0; j < 32; ++j) dst[(size_t)j * out] = conv(j);
            } else {
#pragma unroll
                for (int g = 0; g < 32; g += 8) {
                    if (EIGHTS && g >= count) break;
#pragma unroll
                    for (int j = g; j < g + 8; ++j)
                        if (j < count) dst[(size_t)j * out] = conv(j);
                }
            }
        }
        __syncwarp();
    }
}

// Weight scale and bias of the four channels of a thread in narrow_tile; `first` is the lane quarter's first channel.
__device__ __forceinline__ void narrow_fetch(const float* sw, const float* bias, int first, int lane, int out, float (&s)[4], float (&b)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int n = first + (lane >> 2) + 8 * i;
        s[i] = n < out ? sw[n] : 0.0f;
        b[i] = n < out && bias ? bias[n] : 0.0f;
    }
}
__device__ __forceinline__ void narrow_constants(const float* sw, const float* bias, float sx, int first, int lane, int out, float (&c)[4], float (&b)[4]) {
    narrow_fetch(sw, bias, first, lane, out, c, b);
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = __fmul_rn(sx, c[i]);
}
// Pieces of metadata (16 bytes: one row, one 128-wide k-block) that a metadata warp of the one-CTA kernel has in flight (four
// in the forms with weight-building warps, which are short of registers).  One at a time, each load waited for before its
// store to TMEM, they held up the first MMA: 384 tokens 1024 -> 3072 7.6 -> 6.6 us, 4096 -> 1024 16.8 -> 14.7, 64 tokens
// 4096 -> 4096 18.1 -> 14.9.
template <bool XF> constexpr int kMetaBatchOf = XF ? 4 : 8;
// Metadata that has to be converted goes piece by piece all the same where the four copies of the conversion cost more (fetching
// their code) than the loads' latency: rows of at most this many words (reductions of at most 768), and the metadata of an output
// tile that is not the CTA's first.  Over the shapes with 256, 640 and 768 reduction elements 4, 3 and 2 % less than in batches (3000
// tokens 256 -> 256 1:4 / 8 bit 6.5 -> 5.9 us); from 1024 on batches are the faster ones, by up to 9 %.  32768 tokens 1152 -> 640 1:4 / 8
// bit, where a few CTAs change their output tile, 44.2 -> 41.6.
constexpr int kMetaShort = 24;

// Where the weight operand comes from: TMA (already in tensor-core form), built per k-block into the
// stage ring, or built once per output tile into a resident region (reduction length <= kResidentKB k-blocks).
enum { W_TMA = 0, W_BUILD = 1, W_RESIDENT = 2 };
constexpr int kResidentKB = 8;

struct GemmParams {
    int tokens, out, in;
    int n_tok_tiles, n_tiles, kblocks;
    int n_out_tiles, band;  // pair kernel: tiles are ordered band by band (see tile_coord)
    const uint32_t* meta;  // canonical metadata [out, mrow_words] (sparse modes)
    int mrow_words;
    const uint8_t* values; // packed codes (transform modes)
    int vrow_bytes, mrow_bytes, pat;
    int tma_store;         // 1: epilogue writes through shared memory + TMA; 0: direct stores
    int grouped;           // 1: narrow_group_tile (pair kernels, bfloat16)
    const float* sw;
    const float* bias;
    const float* sx_dev;
    float sx_host;
    float* Y;
    int32_t* ACC;
    void* NARROW;          // int8 (EPI_Q8) or bfloat16 (EPI_BF16) output [tokens, out]
    float sy;              // static output scale of EPI_Q8
    float* absmax;
    uint32_t* status;
    unsigned long long* trace;  // NM_TRACE builds: time stamps of CTA 0 (see nm_debug_set_trace); NULL otherwise
    int skip_stage;             // NM_TEST_HOOKS builds: CTA 0's producer leaves this pipeline stage unissued (-1: none)
};

// Time stamps for profiling, compiled in with -DNM_TRACE only (a second library, never the product's):
// CTA 0 writes clock64() into row `it` (one row of 8 words per pipeline stage, kTraceStages rows) or, for
// per-tile events, into row kTraceStages + tile.  The kernels' work is unchanged.
constexpr int kTraceStages = 512, kTraceTiles = 64;
// Test hook, compiled in with -DNM_TEST_HOOKS only (the library the timeout test loads, never the product's): CTA 0's
// producer skips pipeline stage `skip_stage` -- nothing is armed, nothing is copied, no address is touched -- so that
// the stage's "full" barrier never completes and the bounded waits downstream run out.
#ifdef NM_TEST_HOOKS
#define NM_SKIP_STAGE(it) (p.skip_stage >= 0 && blockIdx.x == 0 && (it) == (uint32_t)p.skip_stage)
#else
#define NM_SKIP_STAGE(it) false
#endif

#ifdef NM_TRACE
#define NM_TRACE_ONLY(x) x
#define NM_TRACE_STAGE(it, col) do { if (p.trace && blockIdx.x == 0 && (it) < (uint32_t)kTraceStages) p.trace[8 * (size_t)(it) + (col)] = clock64(); } while (0)
#define NM_TRACE_TILE(i, col) do { if (p.trace && blockIdx.x == 0 && (i) < kTraceTiles) p.trace[8 * (size_t)(kTraceStages + (i)) + (col)] = clock64(); } while (0)
// Phases of the first epilogue warp's work on a tile, summed per tile into columns 3..7 of the tile's row: waiting for the
// accumulator chunk, waiting for the staging tile to be free, converting and filling it, the proxy fence, issuing the store.
#define NM_TRACE_EPI_DECL long long tr_t = clock64(), tr_acc[5] = {0, 0, 0, 0, 0}
#define NM_TRACE_EPI_MARK() do { tr_t = clock64(); } while (0)
#define NM_TRACE_EPI_ADD(k) do { const long long tr_now = clock64(); tr_acc[k] += tr_now - tr_t; tr_t = tr_now; } while (0)
#define NM_TRACE_EPI_FLUSH(i) do { if (p.trace && blockIdx.x == 0 && (i) < kTraceTiles) { for (int k = 0; k < 5; ++k) { p.trace[8 * (size_t)(kTraceStages + (i)) + 3 + k] = tr_acc[k]; tr_acc[k] = 0; } } } while (0)
#else
#define NM_TRACE_ONLY(x)
#define NM_TRACE_STAGE(it, col) do { } while (0)
#define NM_TRACE_TILE(i, col) do { } while (0)
#define NM_TRACE_EPI_DECL do { } while (0)
#define NM_TRACE_EPI_MARK() do { } while (0)
#define NM_TRACE_EPI_ADD(k) do { } while (0)
#define NM_TRACE_EPI_FLUSH(i) do { } while (0)
#endif

template <bool SPARSE, int BN, bool RESIDENT = false>
struct GemmCfg {
    static constexpr int A_ROW = SPARSE ? 64 : 128;   // bytes of one weight row per stage
    static constexpr int A_BYTES = kBM * A_ROW;
    static constexpr int B_BYTES = BN * 128;
    static constexpr int A_RES = RESIDENT ? kResidentKB * A_BYTES : 0;  // whole-K weight tile kept across token tiles
    static constexpr int B_OFF = RESIDENT ? 0 : A_BYTES;                // X tile within a stage
    static constexpr int STAGE = B_OFF + B_BYTES;
    static constexpr int FIT = (kSmemLimit - kSmemTail - kStoreStage - 1024 - A_RES) / STAGE;
    static constexpr int STAGES = FIT < kMaxStages ? FIT : kMaxStages;
    static constexpr int SMEM = STAGES * STAGE + A_RES + kStoreStage + kSmemTail + 1024;
    static constexpr int META_COL = 2 * BN;           // first TMEM column of the metadata
    static constexpr int META_COLS = kTmemCols - 2 * BN;
    static_assert(STAGES >= 3, "pipeline too shallow");
    static_assert(BN % 32 == 0 && BN >= 32 && BN <= 256, "token tile");
};

// GROUPED: bfloat16 tiles through narrow_group_tile; a kernel of its own, since its code beside the other's cost every call 1 %.
template <bool SPARSE, int BN, int EPI, int WSRC, bool GROUPED = false>
__global__ void __launch_bounds__(WSRC != W_TMA ? kXformThreads : kGemmThreads, 1)
nm_gemm_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
               const __grid_constant__ CUtensorMap tmap_y, const GemmParams p) {
    constexpr bool XF = WSRC != W_TMA, RES = WSRC == W_RESIDENT;
    static_assert(!GROUPED || (EPI == EPI_BF16 && RES), "see store_grouped");
    using Cfg = GemmCfg<SPARSE, BN, RES>;
    constexpr int S = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* a_res = smem + S * Cfg::STAGE;  // resident weight tile: kResidentKB k-blocks of A_BYTES
    uint8_t* store_stage = a_res + Cfg::A_RES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(store_stage + kStoreStage);
    // bars[0..S) full, [S..2S) empty, then acc_full[2], acc_empty[2], meta_ready, drained, a_full, a_free
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto acc_full_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };
    auto acc_empty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };
    const uint32_t meta_bar = bar0 + 8u * (2 * S + 4);
    const uint32_t drained_bar = bar0 + 8u * (2 * S + 5);
    const uint32_t a_full_bar = bar0 + 8u * (2 * S + 6);  // resident weight tile built (all builder warps)
    const uint32_t a_free_bar = bar0 + 8u * (2 * S + 7);  // ... and no longer read by any MMA
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 8);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* never_flag = tmem_slot + 2;  // stays 0: for the drain waits after an abort
    uint32_t* lut = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(bars) + 512);

    constexpr int EW = XF ? kEpiWarpsXf : kEpiWarps, kGateWarp = 2 + EW;
    const int warp = (int)ptx::warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int per = p.n_tiles / gridDim.x, rem = p.n_tiles % gridDim.x;
    const int tile_begin = blockIdx.x * per + min((int)blockIdx.x, rem);
    const int tile_count = per + ((int)blockIdx.x < rem ? 1 : 0);

    if (threadIdx.x == 0) {
        // a stage is full when its TMA bytes have landed and, in transform mode, the four warps building it are done
        for (int s = 0; s < S; ++s) { ptx::mbar_init(full_bar(s), WSRC == W_BUILD ? 5 : 1); ptx::mbar_init(empty_bar(s), 1); }
        ptx::mbar_init(a_full_bar, 4 * kBuildGroups);
        ptx::mbar_init(a_free_bar, 1);
        for (int b = 0; b < 2; ++b) { ptx::mbar_init(acc_full_bar(b), 1); ptx::mbar_init(acc_empty_bar(b), XF ? kEpiWarpsXf : kEpiWarps); }
        ptx::mbar_init(meta_bar, 4);
        ptx::mbar_init(drained_bar, 1);
        *abort_flag = 0;
        *never_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_w);
        ptx::prefetch_tensormap(&tmap_x);
        if (p.tma_store) ptx::prefetch_tensormap(&tmap_y);
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
    // Set-up above overlaps the tail of the kernel before this one in the stream (when launched as its
    // programmatic dependent); nothing in global memory is read or written before this point.
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    auto raise_timeout = [&]() {
        *abort_flag = 1;
        if (p.status) atomicOr(p.status, NM_STATUS_TIMEOUT);
    };

    if (warp == 0) {
        // ------------------------------ TMA producer ------------------------------------------
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int i = 0; i < tile_count && ok; ++i) {
                const int tile = tile_begin + i;
                const int n0 = (tile / p.n_tok_tiles) * kBM, t0 = (tile % p.n_tok_tiles) * BN;
                for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                    const int s = it % S;
                    if (!ptx::mbar_wait_bounded(empty_bar(s), ((it / S) & 1u) ^ 1u, abort_flag, kWaitLimit)) {
                        raise_timeout(); ok = false; break;
                    }
                    if (NM_SKIP_STAGE(it)) continue;
                    const uint32_t a_dst = ptx::smem_u32(smem + s * Cfg::STAGE);
                    ptx::mbar_expect_tx(full_bar(s), XF ? Cfg::B_BYTES : Cfg::STAGE);
                    if (!XF) ptx::tma_load_2d(a_dst, &tmap_w, kb * Cfg::A_ROW, n0, full_bar(s));
                    ptx::tma_load_2d(a_dst + Cfg::B_OFF, &tmap_x, kb * 128, t0, full_bar(s));
                }
            }
            if (!ok) {
                // let copies already in flight land before the CTA goes away
                const uint32_t first = it > (uint32_t)S ? it - S : 0;
                for (uint32_t j = first; j < it; ++j)
                    ptx::mbar_wait_bounded(full_bar(j % S), (j / S) & 1u, never_flag, kWaitLimit >> 4);
            }
        }
    } else if (XF && warp >= kGateWarp + 1) {
        // ------------------------------ weight-tile builders (transform modes) ------------------
        // One thread builds one row of a k-block.  The work of one k-block is a long dependent chain
        // (unpack, table lookups, byte permutes, stores, fence), so several groups of four warps
        // take the k-blocks round-robin: group g builds pipeline steps g, g + G, g + 2G, ...
        constexpr int G = kBuildGroups;
        static_assert(RES || S > G, "every group needs a stage of its own in flight");
        const int bw = warp - (kGateWarp + 1), grp = bw >> 2;
        const int tr = (bw & 3) * 32 + lane;  // row of the 128-row weight tile
        const int cb = xf::code_bytes(p.pat), mb = xf::meta_bytes(p.pat);
        const uint8_t* meta8 = reinterpret_cast<const uint8_t*>(p.meta);
        if constexpr (RES) {
            // Short reductions: the whole-K weight tile of an output tile is built once and stays in
            // shared memory for all token tiles of that output tile; the ring then carries X only.
            int prev_out_tile = -1;
            uint32_t free_parity = 1u;  // nothing reads the region before the first build
            for (int i = 0; i < tile_count; ++i) {
                const int out_tile = (tile_begin + i) / p.n_tok_tiles;
                if (out_tile == prev_out_tile) continue;
                prev_out_tile = out_tile;
                const int n = out_tile * kBM + tr;
                const bool row_ok = n < p.out;
                const uint8_t* v = p.values + (size_t)(row_ok ? n : 0) * p.vrow_bytes;
                const uint8_t* m = meta8 + (size_t)(row_ok ? n : 0) * p.mrow_bytes;
                xf::Raw cur = xf::load_raw(p.pat, v + (size_t)grp * cb, m + (size_t)grp * mb, row_ok && grp < p.kblocks);
                // the MMAs of the previous output tile have finished reading the region
                bool got = lane != 0 || ptx::mbar_wait_bounded(a_free_bar, free_parity, abort_flag, kWaitLimit);
                free_parity ^= 1u;
                if (!__all_sync(0xffffffffu, got)) { if (lane == 0) raise_timeout(); break; }
                for (int kb = grp; kb < p.kblocks; kb += G) {
                    const int nkb = kb + G;
                    xf::Raw nxt = xf::load_raw(p.pat, v + (size_t)nkb * cb, m + (size_t)nkb * mb, row_ok && nkb < p.kblocks);
                    uint32_t w[SPARSE ? 16 : 32];
                    xf::build_row<SPARSE>(p.pat, cur, lut, w);
                    xf::store_row<SPARSE>(a_res + kb * Cfg::A_BYTES, tr, w);
                    cur = nxt;
                }
                ptx::fence_proxy_async_smem();  // the MMA reads the tile through the async proxy
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(a_full_bar);
            }
        } else {
        // position of a pipeline step: tile index i within this CTA's range, k-block kb; row pointers follow i
        struct Pos { int i, kb; const uint8_t* v; const uint8_t* m; bool ok; };
        auto locate = [&](Pos& q) {  // row pointers and validity for tile q.i
            q.ok = q.i < tile_count;
            const int n = q.ok ? ((tile_begin + q.i) / p.n_tok_tiles) * kBM + tr : 0;
            q.ok = q.ok && n < p.out;
            q.v = p.values + (size_t)n * p.vrow_bytes;
            q.m = meta8 + (size_t)n * p.mrow_bytes;
        };
        auto advance = [&](Pos& q) {  // G pipeline steps further
            q.kb += G;
            if (q.kb >= p.kblocks) {
                do { q.kb -= p.kblocks; ++q.i; } while (q.kb >= p.kblocks);
                locate(q);
            }
        };
        Pos at{0, 0, nullptr, nullptr, false};
        at.kb = grp;
        while (at.kb >= p.kblocks) { at.kb -= p.kblocks; ++at.i; }
        locate(at);
        int s = grp % S;
        uint32_t parity = 1u;  // of the empty barrier: the first pass over the ring finds every stage free
        xf::Raw cur = xf::load_raw(p.pat, at.v + (size_t)at.kb * cb, at.m + (size_t)at.kb * mb, at.ok);
        while (at.i < tile_count) {
            // fetch this group's next k-block before working on the current one
            Pos nx = at;
            advance(nx);
            xf::Raw nxt = xf::load_raw(p.pat, nx.v + (size_t)nx.kb * cb, nx.m + (size_t)nx.kb * mb, nx.ok);
            bool got = lane != 0 || ptx::mbar_wait_bounded(empty_bar(s), parity, abort_flag, kWaitLimit);
            if (!__all_sync(0xffffffffu, got)) { if (lane == 0) raise_timeout(); break; }
            uint32_t w[SPARSE ? 16 : 32];
            xf::build_row<SPARSE>(p.pat, cur, lut, w);
            xf::store_row<SPARSE>(smem + s * Cfg::STAGE, tr, w);
            ptx::fence_proxy_async_smem();  // the MMA reads the tile through the async proxy
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(full_bar(s));
            cur = nxt;
            at = nx;
            s += G;
            if (s >= S) { s -= S; parity ^= 1u; }
        }
        }
    } else if (warp == kGateWarp) {
        // ------------------------------ gate: mbarrier waits relayed to the MMA warp ------------
        // Runs its full trip count even after a timeout (then without waiting), so that the MMA
        // warp, which blocks on the named barriers, always gets its arrivals.
        uint32_t it = 0, meta_phase = 0, a_phase = 0;
        int prev_out_tile = -1;
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity) {
            if (lane == 0 && ok && !ptx::mbar_wait_bounded(bar, parity, abort_flag, kWaitLimit)) {
                raise_timeout();
                ptx::wait_clocks(kGateDrain);
                ok = false;
            }
        };
        for (int i = 0; i < tile_count; ++i) {
            const int tile = tile_begin + i, out_tile = tile / p.n_tok_tiles, buf = i & 1;
            if (out_tile != prev_out_tile) {
                if (SPARSE) { wait(meta_bar, meta_phase); meta_phase ^= 1u; }
                if (RES) { wait(a_full_bar, a_phase); a_phase ^= 1u; }
                prev_out_tile = out_tile;
            }
            wait(acc_empty_bar(buf), ((i >> 1) & 1u) ^ 1u);
            for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                wait(full_bar(it % S), (it / S) & 1u);
                __syncwarp();
                ptx::relay_step(1 + (it & 7u), abort_flag);
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ---------------------------------------------
        constexpr uint32_t idesc = ptx::idesc_i8(kBM, BN, SPARSE);
        const uint64_t a_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(RES ? a_res : smem), SPARSE ? 64 : 128, SPARSE ? ptx::kSwizzle64 : ptx::kSwizzle128);
        const uint64_t b_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(smem) + Cfg::B_OFF, 128, ptx::kSwizzle128);
        uint32_t s = 0, relay = 1;
        int tok = tile_begin % p.n_tok_tiles;
        for (int i = 0; i < tile_count; ++i) {
            const uint32_t buf = i & 1, d_tmem = tmem_base + buf * BN;
            const bool last_of_out_tile = RES && ++tok == p.n_tok_tiles;  // the next tile is another output tile's
            if (last_of_out_tile) tok = 0;
            for (int kb = 0; kb < p.kblocks; ++kb) {
                ptx::named_bar_sync(relay, 64);  // stage s holds k-block kb (and, for kb = 0, the
                relay = (relay & 7u) + 1u;       // accumulator is free and the metadata in place)
                // The tcgen05 fence orders the MMAs after other threads' TMEM accesses (accumulator read
                // back, metadata stores): needed once per tile.  Executed every stage it drains the MMA
                // pipe (measured ~585 clk per stage); the staged operands are ordered by the mbarrier.
                if (kb == 0) ptx::tc_fence_after();
                if (ptx::elect_one()) {
                    const uint64_t a = ptx::desc_advance(a_desc0, RES ? kb * Cfg::A_BYTES : s * Cfg::STAGE), b = ptx::desc_advance(b_desc0, s * Cfg::STAGE);
                    if constexpr (SPARSE) {
#pragma unroll
                        for (int j = 0; j < 2; ++j)  // 64 logical k each: 32 stored bytes of A, 64 of B
                            ptx::mma_sp_i8(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 64 * j),
                                           tmem_base + Cfg::META_COL + kb * 4 + 2 * j, idesc, (kb | j) != 0);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)  // 32 k each
                            ptx::mma_i8(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 32 * j), idesc, (kb | j) != 0);
                    }
                    ptx::tc_commit(empty_bar(s));  // stage reusable once these MMAs have read it
                    if (kb == p.kblocks - 1) {
                        ptx::tc_commit(acc_full_bar(buf));
                        if (last_of_out_tile) ptx::tc_commit(a_free_bar);  // the builders may overwrite the weight tile
                    }
                }
                __syncwarp();
                if (++s == S) s = 0;
            }
        }
        if (ptx::elect_one()) {  // everything issued has retired before TMEM is released
            ptx::tc_commit(drained_bar);
            ptx::mbar_wait_bounded(drained_bar, 0, never_flag, kWaitLimit);
        }
        __syncwarp();
    } else {
        // ------------------------------ metadata + epilogue warps ------------------------------
        // Warp w may touch TMEM lanes 32 * (w % 4) ... + 31.  With eight warps two share a lane quarter
        // and take alternate 32-column chunks of the accumulator.
        constexpr int EWH = EW / 4;               // warps per lane quarter
        constexpr int CH = BN / 32;               // chunks per accumulator
        constexpr int CI = (CH + EWH - 1) / EWH;  // chunks per warp
        const int ew = warp - 2, q = warp & 3, half = ew >> 2, row = q * 32 + lane;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16);
        float* my_stage = reinterpret_cast<float*>(store_stage + ew * 4096);
        const float sx = p.sx_dev ? *p.sx_dev : p.sx_host;
        float amax = 0.0f, c_n = 0.0f, b_n = 0.0f;
        const float rsy = EPI == EPI_Q8 ? __frcp_rn(p.sy) : 0.0f;
        int scaled_out_tile = -1;
        uint32_t n_stores = 0;
        int narrow_out_tile = -1;  // whose constants nc, nb are (narrow outputs)
        float nc[4], nb[4];
        bool ok = true;

        // Index metadata of this lane's weight row for the whole reduction; rows past the end get a valid "positions 0,1" pattern,
        // their products are discarded.  The form with resident built weights always goes piece by piece, and fetches the channel
        // constants behind the wait for the accumulator: with batches, and the constants in front of it, int8 and bfloat16 outputs took
        // 2 % more over all shapes and up to 11 % (32768 tokens 256 -> 256 1:4 / 8 bit bfloat16 13.5 us against 12.1, 12000 tokens
        // 512 -> 2048 2:4 / 4 bit 26.1 against 24.2).
        auto load_meta = [&](int out_tile, bool first) {
            const int n = out_tile * kBM + row;
            const bool row_ok = n < p.out;
            const uint4 idle = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
            const uint8_t* src = reinterpret_cast<const uint8_t*>(p.meta) + (size_t)(row_ok ? n : 0) * (XF ? p.mrow_bytes : 4 * p.mrow_words);
            const int piece = XF ? xf::meta_bytes(p.pat) : 16;  // stored bytes of a k-block
            if (RES || (XF && (!first || p.mrow_words <= kMetaShort))) {
                for (int c = 0; c < p.mrow_words; c += 4) {
                    uint4 w = idle;
                    if (row_ok) w = xf::hw_meta(p.pat, xf::meta_raw(p.pat, src + (size_t)(c >> 2) * piece), lut);
                    ptx::tmem_st_32x4(lane_taddr + Cfg::META_COL + c, w.x, w.y, w.z, w.w);
                }
            } else {
                constexpr int kMetaBatch = kMetaBatchOf<XF>;
                for (int c0 = 0; c0 < p.mrow_words; c0 += 4 * kMetaBatch) {  // all loads of a batch are in flight together
                    uint4 mw[kMetaBatch];
#pragma unroll
                    for (int j = 0; j < kMetaBatch; ++j) {
                        mw[j] = idle;
                        if (row_ok && c0 + 4 * j < p.mrow_words) {
                            if constexpr (XF) mw[j] = xf::meta_raw(p.pat, src + (size_t)((c0 >> 2) + j) * piece);
                            else mw[j] = xf::ldg16(src + (size_t)((c0 >> 2) + j) * 16);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kMetaBatch; ++j) {
                        if (c0 + 4 * j < p.mrow_words) {
                            uint4 w = mw[j];
                            if constexpr (XF) w = row_ok ? xf::hw_meta(p.pat, mw[j], lut) : idle;
                            ptx::tmem_st_32x4(lane_taddr + Cfg::META_COL + c0 + 4 * j, w.x, w.y, w.z, w.w);
                        }
                    }
                }
            }
            ptx::tmem_st_wait();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(meta_bar);
        };
        auto release_acc = [&](int buf) {  // this warp has read all it needs from the accumulator
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(acc_empty_bar(buf));
        };

        for (int i = 0; i < tile_count && ok; ++i) {
            const int tile = tile_begin + i, out_tile = tile / p.n_tok_tiles, buf = i & 1;
            const int n0 = out_tile * kBM, n = n0 + row, t0 = (tile % p.n_tok_tiles) * BN;
            if (SPARSE && i == 0 && half == 0) load_meta(out_tile, true);
            if (!(RES && SPARSE) && EPI != EPI_ACC && !(kNarrow<EPI> && p.tma_store) && out_tile != scaled_out_tile) {  // channel constants: once per output tile
                scaled_out_tile = out_tile;
                c_n = n < p.out ? __fmul_rn(sx, p.sw[n]) : 0.0f;
                b_n = n < p.out && p.bias ? p.bias[n] : 0.0f;
            }
            if (kNarrow<EPI> && p.tma_store && out_tile != narrow_out_tile) {
                narrow_out_tile = out_tile;
                narrow_constants(p.sw, p.bias, sx, n0 + q * 32, lane, p.out, nc, nb);
            }
            bool got = ptx::mbar_wait_bounded(acc_full_bar(buf), (i >> 1) & 1u, abort_flag, kWaitLimit);
            ok = __all_sync(0xffffffffu, got);
            if (!ok && lane == 0) raise_timeout();
            if constexpr (GROUPED) ok = ptx::named_bar_and(kNarrowAgree + half, 128, ok);  // the group stops together
            if (!ok) break;
            ptx::tc_fence_after();
            if (SPARSE && half == 0 && i + 1 < tile_count) {
                const int next_out_tile = (tile + 1) / p.n_tok_tiles;
                if (next_out_tile != out_tile) load_meta(next_out_tile, false);  // MMAs of this output tile are done
            }
            const bool n_ok = n < p.out;
            if (RES && SPARSE && EPI != EPI_ACC && !(kNarrow<EPI> && p.tma_store) && out_tile != scaled_out_tile) {  // (see load_meta)
                scaled_out_tile = out_tile;
                c_n = n_ok ? __fmul_rn(sx, p.sw[n]) : 0.0f;
                b_n = n_ok && p.bias ? p.bias[n] : 0.0f;
            }
            if (!p.tma_store) {
                direct_tile<EPI, !XF && EPI != EPI_Q8>(lane_taddr + buf * BN, BN, p.tokens - t0, half, EWH, c_n, b_n, p.sy, rsy,
                                 reinterpret_cast<typename EpiOut<EPI>::type*>(kF32<EPI> ? (void*)p.Y : EPI == EPI_ACC ? (void*)p.ACC : p.NARROW), t0, n, p.out, amax,
                                 [&] { release_acc(buf); });
                continue;
            }
            if constexpr (GROUPED) {
                narrow_group_tile<16>(lane_taddr + buf * BN, BN, p.tokens - t0, half, EWH, kNarrowGroup + half, ptx::smem_u32(store_stage) + half * 8192, n_stores,
                                      q, lane, nc, nb, &tmap_y, n0, t0, p.out, ptx::policy_evict_first(), [&] { release_acc(buf); });
                continue;
            } else if constexpr (kNarrow<EPI>) {
                constexpr int SUBS = (BN / 16 + EWH - 1) / EWH;
                narrow_tile<EPI, SUBS, kNarrowStage<EPI, kStoreStage / kEpiWarps, SUBS>, 1, 1, false>(lane_taddr + buf * BN, p.tokens - t0, half, EWH,
                    ptx::smem_u32(store_stage) + ew * (kStoreStage / kEpiWarps), lane, nc, nb, p.sy, rsy, p.in, &tmap_y, n0 + q * 32, t0, p.out, 0, [&] { release_acc(buf); });
                continue;
            }
            if constexpr (!kNarrow<EPI>) {
                const int nact = min(CH, (p.tokens - t0 + 31) >> 5);  // chunks that hold tokens (warp-uniform)
                // Accumulator chunks are read one ahead of their conversion (two register buffers); the
                // transform kernels, short of registers with their extra warps, read each chunk when it is due.
                constexpr int RB = XF ? 1 : 2;
                uint32_t r[RB][32];
                if (half >= nact) release_acc(buf);
                else if (RB == 2) ptx::tmem_ld_32x32(lane_taddr + buf * BN + half * 32, r[0]);
#pragma unroll
                for (int ci = 0; ci < CI; ++ci) {
                    const int c = half + ci * EWH, tc0 = t0 + c * 32;
                    if (c < nact) {
                        if (RB == 1) ptx::tmem_ld_32x32(lane_taddr + buf * BN + c * 32, r[0]);
                        ptx::tmem_ld_wait();
                        if (c + EWH >= nact) release_acc(buf);
                        else if (RB == 2) ptx::tmem_ld_32x32(lane_taddr + buf * BN + (c + EWH) * 32, r[(ci + 1) & (RB - 1)]);
                        // conversion of accumulator column j of this chunk; jmax = outputs of this lane that exist
                        const int jmax = n_ok ? min(32, p.tokens - tc0) : 0;
                        using OT = typename EpiOut<EPI>::type;
                        auto conv = [&](int j) -> OT {
                            float y_abs;
                            const OT o = epi_convert<EPI>(r[ci & (RB - 1)][j], c_n, b_n, y_abs);
                            if constexpr (EPI == EPI_F32MAX) amax = fmaxf(amax, j < jmax ? y_abs : 0.0f);
                            return o;
                        };
                        // two stores of 16 tokens each, through alternating staging tiles: while one is
                        // being read by its TMA store the other is filled
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (tc0 + 16 * h >= p.tokens) continue;  // warp-uniform (and the same in all warps of a group)
                            OT* sb = reinterpret_cast<OT*>(my_stage + (n_stores & 1u) * 512);
                            if (lane == 0) ptx::bulk_wait_group_read<1>();  // the store before the last has read this tile
                            __syncwarp();
#pragma unroll
                            for (int j = 0; j < 16; ++j) sb[j * 32 + lane] = conv(16 * h + j);
                            ptx::fence_proxy_async_smem();
                            __syncwarp();
                            if (lane == 0) {
                                ptx::tma_store_2d(&tmap_y, n0 + q * 32, tc0 + 16 * h, ptx::smem_u32(sb));
                                ptx::bulk_commit_group();
                            }
                            ++n_stores;
                        }
                    }
                }
            }
        }
        if (lane == 0) ptx::bulk_wait_group_read<0>();  // the stores have read the staging tiles
        if (EPI == EPI_F32MAX) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(p.absmax), __float_as_uint(amax));
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ---------------------------------------------------------------------------------------------
// CTA-pair variant (cluster of two, tcgen05 cta_group::2) for weights already in tensor-core form.
// A pair tile is 256 output channels x BN tokens.  Each CTA stages its own 128 weight rows and HALF of
// the X tile (BN/2 tokens); one MMA issued by the leader CTA (cluster rank 0) spans both CTAs: every
// CTA's tensor core accumulates its 128 rows over all BN tokens, taking the other half of X from the
// peer's shared memory.  Per MAC this moves 0.63x the bytes of the one-CTA kernel through L2 and
// through each SM's shared-memory port.
// Protocol differences: both producers' TMA bytes are counted on the LEADER's "full" barrier; the
// leader's commits are multicast to the "empty" / "accumulator full" barriers of both CTAs; the
// peer's epilogue and metadata warps arrive remotely on the leader's barriers; the pair synchronises
// as a cluster before the first remote operation and before TMEM is released.
// ---------------------------------------------------------------------------------------------
constexpr int kPairThreads = 32 * (3 + kEpiWarps);
constexpr int kPairBuildWarps = 8;  // two groups of four (one thread per weight row of the CTA) taking alternate 128-wide k-blocks
template <bool BUILD> constexpr int kPairThreadsOf = kPairThreads + (BUILD ? 32 * kPairBuildWarps : 0);
// Narrow outputs from resident weights: the epilogue sets the pace there and is a chain of waits (accumulator read, staging
// tile, fence, store issue) that eight warps do not overlap; sixteen epilogue warps in four groups take 16-token units.
// The second eight sit behind the gate warp, where the builder warps of the BUILD form are.
template <int EPI, bool RES, bool BUILD> constexpr int kPairEpiWarps = (kNarrow<EPI> && RES && !BUILD) ? 16 : kEpiWarps;
template <int EPI, bool RES, bool BUILD> constexpr int kPairThreadsFor = kPairThreadsOf<BUILD> + 32 * (kPairEpiWarps<EPI, RES, BUILD> - kEpiWarps);
constexpr int kPairMaxStages = 7;   // the relay cycles through 8 named barriers (ids 1-8; 9-14 serve the narrow-output epilogue)

constexpr int kPairResStages = 4;   // stages of weights a CTA can keep resident (1024 reduction elements at 2:4)

template <bool SPARSE, int BN, bool RES = false>
struct PairCfg {
    // A stage holds 128 stored bytes of every weight row (256 reduction elements when 2:4 compressed,
    // 128 when dense) and the matching 128-byte-wide slices of X: one TMA operation each, four MMAs.
    static constexpr int KB = SPARSE ? 256 : 128;
    static constexpr int A_ROW = 128;
    static constexpr int A_BYTES = kBM * A_ROW;
    static constexpr int B_ROWS = BN / 2;            // tokens staged by each CTA
    static constexpr int B_SUB = B_ROWS * 128;       // one 128-byte-wide slice of the X half tile
    static constexpr int B_BYTES = B_SUB * (KB / 128);
    // RES: the whole-K weight rows of the CTA stay in shared memory across the token tiles of an
    // output tile; the ring then carries X only and holds more of it.
    static constexpr int A_RES = RES ? kPairResStages * A_BYTES : 0;
    static constexpr int B_OFF = RES ? 0 : A_BYTES;
    static constexpr int STAGE = B_OFF + B_BYTES;
    // Epilogue staging: two [16 tokens][32 channels] fp32 tiles per warp where the epilogue sets the pace
    // (short reductions, RES); one where the main loop does and a fifth stage in the ring is worth more.
    static constexpr int STORE_BUFS = RES ? 2 : 1;
    static constexpr int STORE_STAGE = kEpiWarps * STORE_BUFS * 2048;
    static constexpr int FIT = (kSmemLimit - kSmemTail - STORE_STAGE - 1024 - A_RES) / STAGE;
    static constexpr int STAGES = FIT < kPairMaxStages ? FIT : kPairMaxStages;
    static constexpr int SMEM = STAGES * STAGE + A_RES + STORE_STAGE + kSmemTail + 1024;
    static_assert(STAGES >= 3, "pipeline too shallow");
    static constexpr int META_COL = 2 * BN;
    static constexpr int META_COLS = kTmemCols - 2 * BN;
    static_assert(B_SUB % 1024 == 0, "X half tile must keep the swizzle alignment");
    static_assert(BN % 32 == 0 && BN <= 256, "token tile");
};

// Index metadata of one weight row (this lane's) into TMEM columns taddr .. taddr + total_words - 1: `row_words` words from
// the row, eight pieces of four in flight together, then the valid pattern "positions 0,1": the last stage may span more
// reduction elements than the row has, and rows past `out` (row_words = 0) must hold valid patterns too; their
// products are zero or discarded.  A function of its own: inlined into the epilogue's loop the batch cost more through the
// instruction cache than it saved (16384 tokens 1024 -> 4096 61.4 us before, 62.7 inlined, 60.1 so; 1024 -> 1024 21.8 / 21.8 /
// 21.3; 49152 tokens 1024 -> 1024 bfloat16 42.0 -> 40.8).  Not with int8 outputs (12288 tokens 768 -> 3072 42.0 / 42.5) and not
// in the BUILD form.
__device__ __noinline__ void meta_to_tmem(const uint4* src, int row_words, int total_words, uint32_t taddr) {
    for (int c0 = 0; c0 < total_words; c0 += 32) {
        uint4 w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            w[j] = c0 + 4 * j < row_words ? __ldg(src + (c0 >> 2) + j) : make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (c0 + 4 * j < total_words) ptx::tmem_st_32x4(taddr + c0 + 4 * j, w[j].x, w[j].y, w[j].z, w[j].w);
    }
    ptx::tmem_st_wait();
    ptx::tc_fence_before();
}

// BUILD (with RES, sparse target): the weights are not stored in the tensor core's form (packed 4-bit codes, 1:4, 2:8,
// 1:8).  Instead of a TMA copy, eight builder warps rebuild the CTA's 128 weight rows for the whole reduction in the resident
// region once per output tile (xform.cuh: widening, placement into 2-of-4 slots), and the metadata warps derive the
// hardware metadata from the canonical one; everything else is the resident-weight kernel.
template <bool SPARSE, int BN, int EPI, bool RES, bool BUILD = false>
__global__ void __launch_bounds__(kPairThreadsFor<EPI, RES, BUILD>, 1)
nm_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                    const __grid_constant__ CUtensorMap tmap_y, const GemmParams p,
                    const __grid_constant__ PairSchedule sched) {
    using Cfg = PairCfg<SPARSE, BN, RES>;
    constexpr int S = Cfg::STAGES;
    constexpr int EW = kPairEpiWarps<EPI, RES, BUILD>, kGateWarp = 2 + kEpiWarps;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* a_res = smem + S * Cfg::STAGE;  // resident weight rows: kPairResStages stages of A_BYTES
    uint8_t* store_stage = a_res + Cfg::A_RES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(store_stage + Cfg::STORE_STAGE);
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };              // used in the leader
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };       // both CTAs (multicast commit)
    auto acc_full_bar = [&](int b) { return bar0 + 8u * (2 * S + b); };   // both CTAs (multicast commit)
    auto acc_empty_bar = [&](int b) { return bar0 + 8u * (2 * S + 2 + b); };  // leader; arrivals from both
    const uint32_t meta_bar = bar0 + 8u * (2 * S + 4);                 // leader; arrivals from both
    const uint32_t drained_bar = bar0 + 8u * (2 * S + 5);
    const uint32_t a_full_bar = bar0 + 8u * (2 * S + 6);               // leader: resident weights of both CTAs landed
    const uint32_t a_free_bar = bar0 + 8u * (2 * S + 7);               // both CTAs (multicast commit): no MMA reads them any more
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 8);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* never_flag = tmem_slot + 2;
    uint32_t* lut = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(bars) + 512);  // BUILD: slot tables (xform.cuh)
    static_assert(!BUILD || (RES && SPARSE), "weights are rebuilt only in the resident-weight, sparse-target form");

    const int warp = (int)ptx::warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();
    const bool leader = rank == 0;
    const int pair = blockIdx.x >> 1;
    const int tile_begin = sched.start[pair];
    const int tile_count = sched.start[pair + 1] - tile_begin;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { ptx::mbar_init(acc_full_bar(b), 1); ptx::mbar_init(acc_empty_bar(b), 2 * EW); }
        ptx::mbar_init(meta_bar, 8);
        ptx::mbar_init(drained_bar, 1);
        ptx::mbar_init(a_full_bar, BUILD ? 2 * kPairBuildWarps : 1);  // the builder warps of both CTAs, or the TMA bytes
        ptx::mbar_init(a_free_bar, 1);
        *abort_flag = 0;
        *never_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_w);
        ptx::prefetch_tensormap(&tmap_x);
        if (p.tma_store) ptx::prefetch_tensormap(&tmap_y);
    }
    if (BUILD) xf::build_lut(lut, threadIdx.x, blockDim.x);
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
            uint32_t it = 0, free_parity = 1u;  // nothing reads the resident region before the first load
            int prev_out_tile = -1;
            bool ok = true;
            const uint64_t keep = ptx::policy_evict_last();  // X is read again for every output tile
            for (int i = 0; i < tile_count && ok; ++i) {
                const int tile = tile_begin + i;
                const TileCoord tc = tile_coord(tile, p.n_tok_tiles, p.n_out_tiles, p.band);
                const int n0 = tc.o * (2 * kBM) + (int)rank * kBM;
                const int t0 = tc.t * BN + (int)rank * Cfg::B_ROWS;
                if (RES && !BUILD && tc.o != prev_out_tile) {
                    // new output tile: once the MMAs of the previous one are done, fetch this CTA's weight rows for the whole reduction
                    prev_out_tile = tc.o;
                    if (!ptx::mbar_wait_bounded(a_free_bar, free_parity, abort_flag, kWaitLimit)) {
                        raise_timeout(); ok = false; break;
                    }
                    free_parity ^= 1u;
                    const uint32_t lead_a_full = ptx::map_to_cta(a_full_bar, 0);
                    if (leader) ptx::mbar_expect_tx(a_full_bar, 2 * p.kblocks * Cfg::A_BYTES);  // bytes of both CTAs
                    for (int kb = 0; kb < p.kblocks; ++kb)
                        ptx::tma_load_2d_pair(ptx::smem_u32(a_res + kb * Cfg::A_BYTES), &tmap_w, kb * Cfg::A_ROW, n0, lead_a_full);
                }
                for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                    const int s = it % S;
                    if (!ptx::mbar_wait_bounded(empty_bar(s), ((it / S) & 1u) ^ 1u, abort_flag, kWaitLimit)) {
                        raise_timeout(); ok = false; break;
                    }
                    NM_TRACE_STAGE(it, 0);
                    if (NM_SKIP_STAGE(it)) continue;
                    const uint32_t a_dst = ptx::smem_u32(smem + s * Cfg::STAGE);
                    const uint32_t lead_full = ptx::map_to_cta(full_bar(s), 0);
                    if (leader) ptx::mbar_expect_tx(full_bar(s), 2 * Cfg::STAGE);  // bytes of both CTAs
                    if (!RES) ptx::tma_load_2d_pair(a_dst, &tmap_w, kb * Cfg::A_ROW, n0, lead_full);
                    // X is mapped as [k-slice][token][128 bytes]: both slices of the stage in one operation
                    ptx::tma_load_3d_pair_hint(a_dst + Cfg::B_OFF, &tmap_x, 0, t0, kb * (Cfg::KB / 128), lead_full, keep);
                    NM_TRACE_STAGE(it, 1);
                }
            }
            // After an expired wait (here or anywhere in the pair) nobody waits for this producer's last copies, and the stages'
            // barriers count the bytes of both CTAs: give the copies time before the CTA and its shared memory go away.
            if (!ok || *abort_flag) ptx::wait_clocks(kAbortDrain);
        }
    } else if (BUILD && warp > kGateWarp) {
        // ------------------------------ weight builders (both CTAs) ------------------------------
        // One thread = one of the CTA's 128 weight rows; group g builds the 128-wide k-blocks g, g + 2, ... of the row
        // into the resident region (two k-blocks per 128-byte row of a stage), once per output tile.
        const int bw = warp - (kGateWarp + 1), grp = bw >> 2, tr = (bw & 3) * 32 + lane;
        const int cb = xf::code_bytes(p.pat), mb = xf::meta_bytes(p.pat);
        const uint8_t* meta8 = reinterpret_cast<const uint8_t*>(p.meta);
        const int kb_real = p.in >> 7, kb_all = 2 * p.kblocks;  // k-blocks of the reduction / of the stages (a last half stage gets zeros)
        const uint32_t lead_a_full = ptx::map_to_cta(a_full_bar, 0);
        int prev_out_tile = -1;
        uint32_t free_parity = 1u;  // nothing reads the region before the first build
        for (int i = 0; i < tile_count; ++i) {
            const int out_tile = tile_coord(tile_begin + i, p.n_tok_tiles, p.n_out_tiles, p.band).o;
            if (out_tile == prev_out_tile) continue;
            prev_out_tile = out_tile;
            const int n = out_tile * (2 * kBM) + (int)rank * kBM + tr;
            const bool row_ok = n < p.out;
            const uint8_t* v = p.values + (size_t)(row_ok ? n : 0) * p.vrow_bytes;
            const uint8_t* m = meta8 + (size_t)(row_ok ? n : 0) * p.mrow_bytes;
            xf::Raw cur = xf::load_raw(p.pat, v + (size_t)grp * cb, m + (size_t)grp * mb, row_ok && grp < kb_real);
            // the MMAs of the previous output tile have finished reading the region
            bool got = lane != 0 || ptx::mbar_wait_bounded(a_free_bar, free_parity, abort_flag, kWaitLimit);
            free_parity ^= 1u;
            if (!__all_sync(0xffffffffu, got)) { if (lane == 0) raise_timeout(); break; }
            for (int kb = grp; kb < kb_all; kb += 2) {
                const int nkb = kb + 2;
                xf::Raw nxt = xf::load_raw(p.pat, v + (size_t)nkb * cb, m + (size_t)nkb * mb, row_ok && nkb < kb_real);
                uint32_t w[16];
                xf::build_row<true>(p.pat, cur, lut, w);
                xf::store_half_row128(a_res + (kb >> 1) * Cfg::A_BYTES, tr, kb & 1, w);
                cur = nxt;
            }
            ptx::fence_proxy_async_smem();  // the MMA reads the tile through the async proxy
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(lead_a_full);
        }
    } else if (warp == kGateWarp) {
        // ------------------------------ gate (leader): mbarrier waits relayed to the MMA warp ------
        if (leader) {
            uint32_t it = 0, meta_phase = 0, a_phase = 0;
            int prev_out_tile = -1;
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t parity) {
                if (lane == 0 && ok && !ptx::mbar_wait_bounded(bar, parity, abort_flag, kWaitLimit)) {
                    raise_timeout();
                    ptx::wait_clocks(kGateDrain);
                    ok = false;
                }
            };
            for (int i = 0; i < tile_count; ++i) {
                const int tile = tile_begin + i, out_tile = tile_coord(tile, p.n_tok_tiles, p.n_out_tiles, p.band).o, buf = i & 1;
                if (out_tile != prev_out_tile) {
                    if (SPARSE) { wait(meta_bar, meta_phase); meta_phase ^= 1u; }
                    if (RES) { wait(a_full_bar, a_phase); a_phase ^= 1u; }
                    prev_out_tile = out_tile;
                }
                wait(acc_empty_bar(buf), ((i >> 1) & 1u) ^ 1u);
                for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
                    wait(full_bar(it % S), (it / S) & 1u);
                    if (lane == 0) NM_TRACE_STAGE(it, 2);
                    __syncwarp();
                    ptx::relay_step(1 + (it & 7u), abort_flag);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer (leader) --------------------------------------
        if (leader) {
            constexpr uint32_t idesc = ptx::idesc_i8(2 * kBM, BN, SPARSE);
            const uint64_t a_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(RES ? a_res : smem), 128, ptx::kSwizzle128);
            const uint64_t b_desc0 = ptx::smem_desc_kmajor(ptx::smem_u32(smem) + Cfg::B_OFF, 128, ptx::kSwizzle128);
            uint32_t s = 0, relay = 1;
            NM_TRACE_ONLY(uint32_t it = 0;)
            for (int i = 0; i < tile_count; ++i) {
                const uint32_t buf = i & 1, d_tmem = tmem_base + buf * BN;
                const bool last_of_out_tile = RES && (tile_begin + i + 1 >= p.n_tiles ||
                    tile_coord(tile_begin + i + 1, p.n_tok_tiles, p.n_out_tiles, p.band).o != tile_coord(tile_begin + i, p.n_tok_tiles, p.n_out_tiles, p.band).o);
                for (int kb = 0; kb < p.kblocks; ++kb) {
                    ptx::named_bar_sync(relay, 64);
                    relay = (relay & 7u) + 1u;
                    if (kb == 0) ptx::tc_fence_after();  // once per tile (see the one-CTA kernel)
                    if (ptx::elect_one()) {
                        NM_TRACE_STAGE(it, 3);
                        const uint64_t a = ptx::desc_advance(a_desc0, RES ? kb * Cfg::A_BYTES : s * Cfg::STAGE), b = ptx::desc_advance(b_desc0, s * Cfg::STAGE);
                        if constexpr (SPARSE) {
#pragma unroll
                            for (int j = 0; j < 4; ++j)  // 64 reduction elements each: 32 stored bytes of A, 64 of X
                                ptx::mma_sp_i8_pair(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, (j >> 1) * Cfg::B_SUB + 64 * (j & 1)),
                                                    tmem_base + Cfg::META_COL + kb * 8 + 2 * j, idesc, (kb | j) != 0);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                ptx::mma_i8_pair(d_tmem, ptx::desc_advance(a, 32 * j), ptx::desc_advance(b, 32 * j), idesc, (kb | j) != 0);
                        }
                        ptx::tc_commit_pair(empty_bar(s), 3);   // both producers may refill the stage
                        if (kb == p.kblocks - 1) {
                            ptx::tc_commit_pair(acc_full_bar(buf), 3);
                            if (last_of_out_tile) ptx::tc_commit_pair(a_free_bar, 3);  // both producers may replace the weights
                        }
                        NM_TRACE_STAGE(it, 4);
                    }
                    __syncwarp();
                    if (++s == S) s = 0;
                    NM_TRACE_ONLY(++it;)
                }
            }
            if (ptx::elect_one()) {
                ptx::tc_commit_pair(drained_bar, 1);
                ptx::mbar_wait_bounded(drained_bar, 0, never_flag, kWaitLimit);
            }
            __syncwarp();
        }
    } else {
        // ------------------------------ metadata + epilogue warps (both CTAs) ----------------------
        constexpr int EWH = EW / 4, CH = BN / 32, CI = (CH + EWH - 1) / EWH;
        const int ew = warp - 2 - (warp > kGateWarp ? 1 : 0), q = warp & 3, half = ew >> 2, row = q * 32 + lane;
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16);
        constexpr int NB = Cfg::STORE_BUFS;
        float* my_stage = reinterpret_cast<float*>(store_stage + ew * (NB * 2048));
        const float sx = p.sx_dev ? *p.sx_dev : p.sx_host;
        const uint32_t lead_meta = ptx::map_to_cta(meta_bar, 0);
        float amax = 0.0f, c_n = 0.0f, b_n = 0.0f;
        const float rsy = EPI == EPI_Q8 ? __frcp_rn(p.sy) : 0.0f;
        int scaled_out_tile = -1;
        uint32_t n_stores = 0;
        int narrow_out_tile = -1;  // whose constants nc, nb are (narrow outputs)
        float nc[4], nb[4];
        bool ok = true;

        auto load_meta = [&](int out_tile) {
            const int n = out_tile * (2 * kBM) + (int)rank * kBM + row;
            if constexpr (BUILD || EPI == EPI_Q8) {
                for (int c = 0; c < p.kblocks * (Cfg::KB / 32); c += 4) {
                    uint4 w = make_uint4(0x44444444u, 0x44444444u, 0x44444444u, 0x44444444u);  // as in meta_to_tmem
                    if (n < p.out && c < p.mrow_words) {
                        if constexpr (BUILD) w = xf::hw_meta(p.pat, xf::meta_raw(p.pat, reinterpret_cast<const uint8_t*>(p.meta) + (size_t)n * p.mrow_bytes + (size_t)(c >> 2) * xf::meta_bytes(p.pat)), lut);
                        else w = __ldg(reinterpret_cast<const uint4*>(p.meta + (size_t)n * p.mrow_words) + (c >> 2));
                    }
                    ptx::tmem_st_32x4(lane_taddr + Cfg::META_COL + c, w.x, w.y, w.z, w.w);
                }
                ptx::tmem_st_wait();
                ptx::tc_fence_before();
            } else {
                const uint4* src = reinterpret_cast<const uint4*>(p.meta + (size_t)(n < p.out ? n : 0) * p.mrow_words);
                meta_to_tmem(src, n < p.out ? p.mrow_words : 0, p.kblocks * (Cfg::KB / 32), lane_taddr + Cfg::META_COL);
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(lead_meta);
        };
        auto release_acc = [&](int buf) {
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(acc_empty_bar(buf), 0));
        };
        const uint64_t stream_out = ptx::policy_evict_first();  // Y is written once and not read here

        NM_TRACE_EPI_DECL;
        for (int i = 0; i < tile_count && ok; ++i) {
            const TileCoord tc = tile_coord(tile_begin + i, p.n_tok_tiles, p.n_out_tiles, p.band);
            const int out_tile = tc.o, tok_tile = tc.t, buf = i & 1;
            const int n0 = out_tile * (2 * kBM) + (int)rank * kBM, n = n0 + row, t0 = tok_tile * BN;
            if (SPARSE && i == 0 && half == 0) load_meta(out_tile);
            if (kNarrow<EPI> && p.tma_store && out_tile != narrow_out_tile) {
                narrow_out_tile = out_tile;
                narrow_constants(p.sw, p.bias, sx, n0 + q * 32, lane, p.out, nc, nb);
            }
            bool got = ptx::mbar_wait_bounded(acc_full_bar(buf), (i >> 1) & 1u, abort_flag, kWaitLimit);
            ok = __all_sync(0xffffffffu, got);
            if (!ok && lane == 0) raise_timeout();
            if (EPI == EPI_BF16 && p.grouped) ok = ptx::named_bar_and(EW == 16 ? kNarrowGroup + half : kNarrowAgree + half, 128, ok);  // the group stops together
            if (!ok) break;
            ptx::tc_fence_after();
            if (ew == 0 && lane == 0) NM_TRACE_TILE(i, 0);
            NM_TRACE_EPI_MARK();
            // the next tile starts a new output tile: its metadata can go in now, the MMAs of this one are done
            if (SPARSE && half == 0 && i + 1 < tile_count) {
                const int next_out_tile = tile_coord(tile_begin + i + 1, p.n_tok_tiles, p.n_out_tiles, p.band).o;
                if (next_out_tile != out_tile) load_meta(next_out_tile);
            }
            const bool n_ok = n < p.out;
            if (EPI != EPI_ACC && !(kNarrow<EPI> && p.tma_store) && out_tile != scaled_out_tile) {  // channel constants: fetched once per output tile
                scaled_out_tile = out_tile;
                c_n = n_ok ? __fmul_rn(sx, p.sw[n]) : 0.0f;
                b_n = n_ok && p.bias ? p.bias[n] : 0.0f;
            }
            if (!p.tma_store) {
                direct_tile<EPI>(lane_taddr + buf * BN, BN, p.tokens - t0, half, EWH, c_n, b_n, p.sy, rsy,
                                 reinterpret_cast<typename EpiOut<EPI>::type*>(kF32<EPI> ? (void*)p.Y : EPI == EPI_ACC ? (void*)p.ACC : p.NARROW), t0, n, p.out, amax,
                                 [&] { release_acc(buf); });
                continue;
            }
            if constexpr (kNarrow<EPI>) {
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
                const int nact = min(CH, (p.tokens - t0 + 31) >> 5);
                // chunks are read one ahead of their conversion; with the builder warps present registers are short and
                // every chunk is read when it is due
                constexpr int RB = BUILD ? 1 : 2;
                uint32_t r[RB][32];
                if (half >= nact) release_acc(buf);
                else if (RB == 2) ptx::tmem_ld_32x32(lane_taddr + buf * BN + half * 32, r[0]);
#pragma unroll
                for (int ci = 0; ci < CI; ++ci) {
                    const int c = half + ci * EWH, tc0 = t0 + c * 32;
                    if (c < nact) {
                        if (RB == 1) ptx::tmem_ld_32x32(lane_taddr + buf * BN + c * 32, r[0]);
                        ptx::tmem_ld_wait();
                        NM_TRACE_EPI_ADD(0);
                        if (c + EWH >= nact) release_acc(buf);
                        else if (RB == 2) ptx::tmem_ld_32x32(lane_taddr + buf * BN + (c + EWH) * 32, r[(ci + 1) & (RB - 1)]);
                        const int jmax = n_ok ? min(32, p.tokens - tc0) : 0;  // outputs of this lane that exist
                        using OT = typename EpiOut<EPI>::type;
                        auto conv = [&](int j) -> OT {
                            float y_abs;
                            const OT o = epi_convert<EPI>(r[ci & (RB - 1)][j], c_n, b_n, y_abs);
                            if constexpr (EPI == EPI_F32MAX) amax = fmaxf(amax, j < jmax ? y_abs : 0.0f);
                            return o;
                        };
#pragma unroll
                        for (int h = 0; h < 2; ++h) {  // 16 tokens per store, alternating staging tiles
                            if (tc0 + 16 * h >= p.tokens) continue;  // warp-uniform (and the same in all warps of a group)
                            OT* sb = reinterpret_cast<OT*>(my_stage + (NB == 2 ? (n_stores & 1u) * 512 : 0));
                            if (lane == 0) ptx::bulk_wait_group_read<NB - 1>();  // the store that last used this tile has read it
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
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
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

#include "gemm_wide.cuh"
#include "gemm_xres.cuh"
#include "gemm_split.cuh"

namespace nm {

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
// Kernel-choice overrides for measurements and tests (nm_debug_set_option); all zero = the library's own choice.
struct DebugOptions {
    int no_pair;      // one-CTA kernels only
    int no_resident;  // always stream the weights through the stage ring
    int no_wide;      // never the 512-channel pair kernel
    int wide_any;     // the 512-channel pair kernel whenever the shape allows it, however few tiles there are
    int wide_bn;      // token-tile width of that kernel: 224 or 192 (0 = automatic)
    int xres;         // the pair kernel with resident activations: 1 = whenever the shape allows it, 2 = never
    int split;        // reduction split over a cluster: 1000 * CTAs + token-tile width, 1 = never (0 = automatic)
    int grouped;      // bfloat16 tiles shared by four warps: 1 = always, 2 = never
    int one_bn;       // token-tile width of the one-CTA kernel (0 = automatic)
    int band;         // band size of the streamed pair kernel's tile order (0 = automatic)
    int skip_stage;   // NM_TEST_HOOKS builds: 1 + the pipeline stage CTA 0's producer leaves out (0 = none)
};
static DebugOptions g_opt = {};
int g_no_pdl = 0;

// Trace buffer of NM_TRACE builds (device, kTraceStages + kTraceTiles rows of 8 u64), handed to every GEMM launch.
static unsigned long long* g_trace_buffer = nullptr;

struct LinearArgs {
    const int8_t* X; int tokens; const nm_packed_t* W;
    float sx; const float* sx_dev; const float* sw; const float* bias;
    float* Y; int32_t* ACC; float* absmax; uint32_t* status; cudaStream_t stream;
    void* NARROW = nullptr; float sy = 1.0f;
};

// Tensor map of the output for the epilogue's TMA stores ([16 tokens][32 channels] boxes).  The epilogue stores
// through TMA when the output can be described by a tensor map (16-byte aligned base and row pitch);
// otherwise *tma_store is cleared, the threads store directly and the map describes X as a stand-in.
template <int EPI>
static int make_store_map(CUtensorMap* ty, const LinearArgs& a, bool* tma_store, uint32_t box_rows = 16, bool grouped = false) {
    const nm_packed_t& W = *a.W;
    constexpr uint32_t es = (uint32_t)sizeof(typename EpiOut<EPI>::type);
    void* ybase = kF32<EPI> ? (void*)a.Y : EPI == EPI_ACC ? (void*)a.ACC : a.NARROW;
    *tma_store = aligned(ybase, 16) && ((size_t)W.out * es) % 16 == 0;
    const CUtensorMapDataType dt = kF32<EPI> ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : EPI == EPI_ACC ? CU_TENSOR_MAP_DATA_TYPE_INT32
                                 : EPI == EPI_Q8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    if (!*tma_store)
        return make_map(ty, a.X, (uint64_t)a.tokens, (uint64_t)W.in / 4, 16, 32, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_DATA_TYPE_INT32, 4);
    // narrow outputs: in the swizzle of narrow_fill or narrow_group_tile
    return make_map(ty, ybase, (uint64_t)a.tokens, (uint64_t)W.out, box_rows, grouped ? 64 : 32,
                    grouped ? CU_TENSOR_MAP_SWIZZLE_128B : EPI == EPI_BF16 ? CU_TENSOR_MAP_SWIZZLE_64B : EPI == EPI_Q8 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE, dt, es);
}

// Whether bfloat16 outputs leave through narrow_group_tile.  The one-CTA kernel with resident weights: from 80 MB of Y at eight k-blocks
// (weights for the sparse form), or 24 MB at six and more (for the dense one); below, and with shorter reductions, whose tiles follow one another
// faster, the warps' own tiles are the better ones.  Over 800 shapes, shared / own in us: 16384 tokens 1024 -> 3072 2:4 / 4 bit 41.4 / 43.8, 32768
// tokens 1024 -> 4096 109 / 118, 24000 tokens 896 -> 4096 4:8 / 4 bit 94 / 115, 16384 tokens 768 -> 2304 4:4 / 4 bit 33.6 / 38.7; not taken:
// 16384 tokens 896 -> 3072 2:4 / 4 bit 42.3 / 39.8, 8192 tokens 640 -> 3072 4:4 / 4 bit 24.9 / 23.7, 16384 tokens 256 -> 4096 2:4 / 4 bit 45.6 / 33.7.
template <int EPI, bool RES = false, bool SPARSE = false>
static bool store_grouped(const LinearArgs& a) {
    if (EPI != EPI_BF16 || g_opt.grouped == 2) return false;
    if (g_opt.grouped == 1) return true;
    const size_t bytes = (size_t)a.tokens * a.W->out * 2;
    if (!RES) return bytes >= kNarrowGroupBytes;
    return SPARSE ? a.W->in >= 1024 && bytes >= (size_t)80 << 20 : a.W->in >= 768 && bytes >= (size_t)24 << 20;
}

template <bool SPARSE, int BN, int EPI, int WSRC>
static int launch_gemm(const LinearArgs& a) {
    constexpr bool XF = WSRC != W_TMA;
    using Cfg = GemmCfg<SPARSE, BN, WSRC == W_RESIDENT>;
    const nm_packed_t& W = *a.W;
    CUtensorMap tw, tx, ty;
    // transform modes build the weight tile in shared memory and never use this map: describe X instead
    int rc = XF ? make_map(&tw, a.X, (uint64_t)a.tokens, (uint64_t)W.in, BN, 128, CU_TENSOR_MAP_SWIZZLE_128B)
                : make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)(SPARSE ? W.in / 2 : W.in), kBM, Cfg::A_ROW,
                           SPARSE ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    rc = make_map(&tx, a.X, (uint64_t)a.tokens, (uint64_t)W.in, BN, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    bool tma_store = false;
    constexpr bool kBothForms = WSRC == W_RESIDENT && EPI == EPI_BF16;
    const bool grouped = kBothForms && store_grouped<EPI, true, SPARSE>(a);
    rc = make_store_map<EPI>(&ty, a, &tma_store, 16, grouped);
    if (rc != NM_OK) return rc;
    GemmParams p{};
    p.tma_store = tma_store ? 1 : 0;
    p.tokens = a.tokens; p.out = W.out; p.in = W.in;
    p.n_tok_tiles = (a.tokens + BN - 1) / BN;
    p.n_tiles = p.n_tok_tiles * ((W.out + kBM - 1) / kBM);
    p.kblocks = W.in / kKB;
    p.meta = (const uint32_t*)W.meta; p.mrow_words = W.in / 32;  // hardware metadata words per row (4 per k-block)
    p.values = (const uint8_t*)W.values;
    p.vrow_bytes = (int)values_row_bytes(W.in, W.n, W.m, W.bits);
    p.mrow_bytes = (int)meta_row_words(W.in, W.n, W.m) * 4;
    p.pat = xf::pattern_of(W.n, W.m, W.bits);
    p.sw = a.sw; p.bias = a.bias; p.sx_dev = a.sx_dev; p.sx_host = a.sx;
    p.Y = a.Y; p.ACC = a.ACC; p.NARROW = a.NARROW; p.sy = a.sy; p.absmax = a.absmax; p.status = a.status; p.trace = g_trace_buffer; p.skip_stage = g_opt.skip_stage - 1;
    auto fn = nm_gemm_kernel<SPARSE, BN, EPI, WSRC>;
    if constexpr (kBothForms) {
        if (grouped && tma_store) fn = nm_gemm_kernel<SPARSE, BN, EPI, WSRC, true>;
    }
    NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, Cfg::SMEM));
    const int grid = p.n_tiles < sm_count() ? p.n_tiles : sm_count();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(XF ? kXformThreads : kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = a.stream;
    // as for the pair kernel: set-up may overlap the previous kernel's tail, global memory waits for it
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 0 : 1;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, tw, tx, ty, p));
    return NM_OK;
}

// The plan costs a pass over all tiles on the host; layers are launched again and again with the same shape, so
// the last few plans are kept.
static int cached_pair_plan(int n_tok_tiles, int n_out_tiles, int pairs, bool resident, int band_request, PairSchedule& out) {
    struct Entry { int key[5]; int band; PairSchedule sched; bool used; };
    static Entry cache[8];
    static unsigned next = 0;
    static std::mutex mu;
    const int key[5] = {n_tok_tiles, n_out_tiles, pairs, resident ? 1 : 0, band_request};
    std::lock_guard<std::mutex> lock(mu);
    for (Entry& e : cache)
        if (e.used && std::equal(key, key + 5, e.key)) { out = e.sched; return e.band; }
    Entry& e = cache[next++ % 8];
    std::copy(key, key + 5, e.key);
    e.band = plan_pair_tiles(n_tok_tiles, n_out_tiles, pairs, resident, band_request, e.sched.start);
    e.used = true;
    out = e.sched;
    return e.band;
}

template <bool SPARSE, int BN, int EPI, bool RES, bool BUILD = false>
static int launch_gemm_pair(const LinearArgs& a) {
    using Cfg = PairCfg<SPARSE, BN, RES>;
    const nm_packed_t& W = *a.W;
    CUtensorMap tw, tx, ty;
    // rebuilt weights are read by the builder warps, not by TMA: the weight map then describes X as a stand-in
    int rc = BUILD ? make_map(&tw, a.X, (uint64_t)a.tokens, (uint64_t)W.in, kBM, 128, CU_TENSOR_MAP_SWIZZLE_128B)
                   : make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)(SPARSE ? W.in / 2 : W.in), kBM, Cfg::A_ROW,
                              CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    rc = make_map_x3(&tx, a.X, (uint64_t)a.tokens, (uint64_t)W.in, Cfg::B_ROWS, Cfg::KB / 128);
    if (rc != NM_OK) return rc;
    bool tma_store = false;
    const bool grouped = store_grouped<EPI>(a);
    rc = make_store_map<EPI>(&ty, a, &tma_store, 16, grouped);
    if (rc != NM_OK) return rc;
    GemmParams p{};
    p.tma_store = tma_store ? 1 : 0;
    p.grouped = grouped ? 1 : 0;
    p.tokens = a.tokens; p.out = W.out; p.in = W.in;
    p.n_tok_tiles = (a.tokens + BN - 1) / BN;
    p.n_out_tiles = (W.out + 2 * kBM - 1) / (2 * kBM);
    p.n_tiles = p.n_tok_tiles * p.n_out_tiles;
    p.kblocks = (W.in + Cfg::KB - 1) / Cfg::KB;
    p.meta = (const uint32_t*)W.meta; p.mrow_words = W.in / 32;
    p.values = (const uint8_t*)W.values;
    p.vrow_bytes = (int)values_row_bytes(W.in, W.n, W.m, W.bits);
    p.mrow_bytes = (int)meta_row_words(W.in, W.n, W.m) * 4;
    p.pat = xf::pattern_of(W.n, W.m, W.bits);
    p.sw = a.sw; p.bias = a.bias; p.sx_dev = a.sx_dev; p.sx_host = a.sx;
    p.Y = a.Y; p.ACC = a.ACC; p.NARROW = a.NARROW; p.sy = a.sy; p.absmax = a.absmax; p.status = a.status; p.trace = g_trace_buffer; p.skip_stage = g_opt.skip_stage - 1;
    auto fn = nm_gemm_pair_kernel<SPARSE, BN, EPI, RES, BUILD>;
    NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, Cfg::SMEM));
    int pairs = p.n_tiles < sm_count() / 2 ? p.n_tiles : sm_count() / 2;
    if (pairs > kMaxPairs) pairs = kMaxPairs;
    // Contiguous tile ranges of about equal cost: a tile costs 1, entering a new output tile inside a range
    // costs `crossing` tiles (weights resident: ~1, the reload waits for the MMAs to drain; streamed: metadata only).
    // Streamed weights: a change of output tile only costs the metadata, so the tiles are banded by about
    // one pair's share and neighbouring pairs share X tiles in L2.  Resident weights: long runs.
    PairSchedule sched;
    p.band = cached_pair_plan(p.n_tok_tiles, p.n_out_tiles, pairs, RES, g_opt.band, sched);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(kPairThreadsFor<EPI, RES, BUILD>, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    // the kernel's set-up may start while the previous kernel of the stream drains; it waits for that kernel
    // (griddepcontrol.wait) before its first access to global memory
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 1 : 2;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, tw, tx, ty, p, sched));
    return NM_OK;
}

// Wide pair kernel (512 channels x BN tokens per pair): 2:4 weights streamed, 8-bit codes or (W4) packed 4-bit ones.
template <int BN, int EPI, bool W4 = false>
static int launch_gemm_wide(const LinearArgs& a) {
    using Cfg = WideCfg<BN, W4>;
    const nm_packed_t& W = *a.W;
    CUtensorMap tw, tx, ty;
    // packed 4-bit codes: two stages of a row at a time
    int rc = W4 ? make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)W.in / 4, Cfg::A_ROWS, 64, CU_TENSOR_MAP_SWIZZLE_64B)
                : make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)W.in / 2, Cfg::A_ROWS, Cfg::A_ROW, CU_TENSOR_MAP_SWIZZLE_64B);
    if (rc != NM_OK) return rc;
    rc = make_map(&tx, a.X, (uint64_t)a.tokens, (uint64_t)W.in, Cfg::B_ROWS, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    bool tma_store = false;
    rc = make_store_map<EPI>(&ty, a, &tma_store, EPI == EPI_Q8 ? 16 : 32, EPI == EPI_BF16);
    if (rc != NM_OK) return rc;
    GemmParams p{};
    p.tma_store = tma_store ? 1 : 0;
    p.tokens = a.tokens; p.out = W.out; p.in = W.in;
    p.n_tok_tiles = (a.tokens + BN - 1) / BN;
    p.n_out_tiles = (W.out + 2 * Cfg::A_ROWS - 1) / (2 * Cfg::A_ROWS);
    p.n_tiles = p.n_tok_tiles * p.n_out_tiles;
    p.kblocks = W.in / Cfg::KB;
    p.meta = (const uint32_t*)W.meta; p.mrow_words = W.in / 32;
    p.values = (const uint8_t*)W.values; p.vrow_bytes = (int)values_row_bytes(W.in, W.n, W.m, W.bits);
    p.sw = a.sw; p.bias = a.bias; p.sx_dev = a.sx_dev; p.sx_host = a.sx;
    p.Y = a.Y; p.ACC = a.ACC; p.NARROW = a.NARROW; p.sy = a.sy; p.absmax = a.absmax; p.status = a.status; p.trace = g_trace_buffer; p.skip_stage = g_opt.skip_stage - 1;
    auto fn = nm_gemm_wide_kernel<BN, EPI, W4>;
    NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, Cfg::SMEM));
    int pairs = p.n_tiles < sm_count() / 2 ? p.n_tiles : sm_count() / 2;
    if (pairs > kMaxPairs) pairs = kMaxPairs;
    PairSchedule sched;
    p.band = cached_pair_plan(p.n_tok_tiles, p.n_out_tiles, pairs, false, 0, sched);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(kWideThreadsOf<W4>, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 1 : 2;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, tw, tx, ty, p, sched));
    return NM_OK;
}

// Pair kernel with resident activations (gemm_xres.cuh).
template <bool SPARSE, int EPI>
static int launch_gemm_xres(const LinearArgs& a) {
    using Cfg = XresCfg<SPARSE>;
    const nm_packed_t& W = *a.W;
    CUtensorMap tw, tx, ty;
    int rc = make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)(SPARSE ? W.in / 2 : W.in), kBM, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    rc = make_map_x3(&tx, a.X, (uint64_t)a.tokens, (uint64_t)W.in, Cfg::B_ROWS, Cfg::SLICES);
    if (rc != NM_OK) return rc;
    bool tma_store = false;
    const bool grouped = store_grouped<EPI>(a);
    rc = make_store_map<EPI>(&ty, a, &tma_store, 16, grouped);
    if (rc != NM_OK) return rc;
    GemmParams p{};
    p.tma_store = tma_store ? 1 : 0;
    p.grouped = grouped ? 1 : 0;
    p.tokens = a.tokens; p.out = W.out; p.in = W.in;
    p.n_tok_tiles = (a.tokens + Cfg::BN - 1) / Cfg::BN;
    p.n_out_tiles = (W.out + 2 * kBM - 1) / (2 * kBM);
    p.n_tiles = p.n_tok_tiles * p.n_out_tiles;
    p.kblocks = (W.in + Cfg::KB - 1) / Cfg::KB;
    p.meta = (const uint32_t*)W.meta; p.mrow_words = W.in / 32;
    p.sw = a.sw; p.bias = a.bias; p.sx_dev = a.sx_dev; p.sx_host = a.sx;
    p.Y = a.Y; p.ACC = a.ACC; p.NARROW = a.NARROW; p.sy = a.sy; p.absmax = a.absmax; p.status = a.status; p.trace = g_trace_buffer; p.skip_stage = g_opt.skip_stage - 1;
    auto fn = nm_gemm_xres_kernel<SPARSE, EPI>;
    NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, Cfg::SMEM));
    const int pairs = p.n_tiles < sm_count() / 2 ? p.n_tiles : sm_count() / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(kXresThreads<EPI>, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 1 : 2;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, tw, tx, ty, p));
    return NM_OK;
}

// One-CTA tiles with the reduction split over clusters of `splits` CTAs (gemm_split.cuh).
template <bool SPARSE, int BN, int EPI, bool XF>
static int launch_gemm_split(const LinearArgs& a, int splits) {
    using Cfg = SplitCfg<SPARSE, BN>;
    const nm_packed_t& W = *a.W;
    CUtensorMap tw, tx;
    // rebuilt weights are not read by TMA: the weight map then describes X as a stand-in
    int rc = XF ? make_map(&tw, a.X, (uint64_t)a.tokens, (uint64_t)W.in, BN, 128, CU_TENSOR_MAP_SWIZZLE_128B)
                : make_map(&tw, W.values, (uint64_t)W.out, (uint64_t)(SPARSE ? W.in / 2 : W.in), kBM, Cfg::A_ROW,
                           SPARSE ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    rc = make_map(&tx, a.X, (uint64_t)a.tokens, (uint64_t)W.in, BN, 128, CU_TENSOR_MAP_SWIZZLE_128B);
    if (rc != NM_OK) return rc;
    GemmParams p{};
    p.tokens = a.tokens; p.out = W.out; p.in = W.in;
    p.n_tok_tiles = (a.tokens + BN - 1) / BN;
    p.n_tiles = p.n_tok_tiles * ((W.out + kBM - 1) / kBM);
    p.kblocks = W.in / kKB;
    p.meta = (const uint32_t*)W.meta; p.mrow_words = W.in / 32;
    p.values = (const uint8_t*)W.values;
    p.vrow_bytes = (int)values_row_bytes(W.in, W.n, W.m, W.bits);
    p.mrow_bytes = (int)meta_row_words(W.in, W.n, W.m) * 4;
    p.pat = xf::pattern_of(W.n, W.m, W.bits);
    p.sw = a.sw; p.bias = a.bias; p.sx_dev = a.sx_dev; p.sx_host = a.sx;
    p.Y = a.Y; p.ACC = a.ACC; p.NARROW = a.NARROW; p.sy = a.sy; p.absmax = a.absmax; p.status = a.status; p.skip_stage = g_opt.skip_stage - 1;
    auto fn = nm_gemm_split_kernel<SPARSE, BN, EPI, XF>;
    NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, Cfg::SMEM));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.n_tiles * splits), 1, 1);
    cfg.blockDim = dim3(kSplitThreadsOf<XF>, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)splits; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 1 : 2;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, tw, tx, p, splits));
    return NM_OK;
}

// Where the kernel with resident activations is the faster pair kernel.  At least two output tiles (with one the activations
// are not read twice), and then by measurement, this kernel / the other one in us:
//  - dense weights, which the other kernel streams besides the activations: always (6144 tokens 768 -> 768 9.3 / 9.9, 768 -> 3072
//    19.2 / 21.7, 12288 tokens 1024 -> 4096 bfloat16 44.2 / 45.3), except for narrow outputs whose rows are not 16-byte
//    aligned (20000 tokens 1024 -> 1500 bfloat16 30.5 / 30.2);
//  - 2:4 weights: up to 896 reduction elements (6144 tokens 768 -> 768 7.7 / 8.6, 768 -> 2304 13.0 / 13.4, 9000 tokens 512 -> 2048
//    14.8 / 16.0); at 1024 only while a pair has few tiles, then the fill of the resident weights of the other kernel is what counts
//    (5000 tokens 1024 -> 1024 8.2 / 9.4; 16384 tokens 1024 -> 4096, 19 tiles, 64.0 / 56.8; 49152 tokens 1024 -> 1024 bfloat16, 14
//    tiles, 43.6 / 40.0);
//  - int8 outputs of 2:4 weights: a few tiles (3977 tokens 768 -> 3072, 3 tiles, 12.0 / 13.1).
// The lines were drawn when a stage's MMAs took 430-550 clocks to issue (now 70-150, see elect_one); measured since over 432 shapes, either
// kernel forced is no better than the rule in the mean (this one 1.002, the other 1.07), but it loses at 16384 tokens 1024 -> 3072
// (45.8 / 43.2), 40000 tokens 768 -> 3072 bfloat16 (82.0 / 79.5), 49152 tokens 768 -> 1024 bfloat16 (37.3 / 33.8), and with int8 outputs of more
// tiles (16384 tokens 768 -> 3072 34.7 / 36.1, 4096 tokens 1024 -> 4096 15.4 / 16.7).
template <bool SPARSE, int EPI>
static bool use_xres(const LinearArgs& a) {
    const nm_packed_t& W = *a.W;
    if (W.in > 1024 || g_opt.xres == 2 || g_opt.no_resident) return false;
    if (g_opt.xres == 1) return true;
    const long long out_tiles = (W.out + 2 * kBM - 1) / (2 * kBM), pairs = sm_count() / 2;
    const long long per_pair = (out_tiles * ((a.tokens + 191) / 192) + pairs - 1) / pairs;
    if (out_tiles < 2) return false;
    if (!SPARSE) return !kNarrow<EPI> || (size_t)W.out * sizeof(typename EpiOut<EPI>::type) % 16 == 0;
    if (EPI == EPI_Q8) return per_pair <= 4;
    return W.in <= 896 || per_pair <= (EPI == EPI_BF16 ? 8 : 16);
}

// Whether the one-CTA kernel has at most one 192-token tile for every SM.  It then beats the pair kernels where their larger
// tiles leave SMs idle or need a second round: 3977 tokens 3072 -> 768 (126 tiles of 128 x 192; 42 of 512 x 192) 11.6 against 14.6 us, packed 4-bit codes
// 15.9 against 20.8; 4500 tokens (144 tiles) 11.4 / 14.6; 5000 tokens 2560 -> 640 10.1 / 13.1.  With a second wave it loses: 5500 tokens 3072 ->
// 768 (174 tiles) 17.8 / 14.5.  Against the 256-channel kernels, before their MMAs were issued by an elected lane: 5000 tokens 640 -> 640 (135 tiles; 81
// of 256 x 192 on 74 pairs) 7.3 / 9.5, dense 2560 -> 640 14.0 / 19.1, 9000 tokens 896 -> 384 8.6 / 10.6, packed 4-bit codes 5000 tokens 640 -> 640 9.3 / 12.3.
static bool one_wave(const LinearArgs& a) {
    const long long tiles = (long long)((a.W->out + kBM - 1) / kBM) * ((a.tokens + 191) / 192);
    return tiles <= sm_count() && a.W->in / 32 <= kTmemCols - 2 * 192;
}

// Token-tile width of the wide kernel: the one whose slowest pair has the least to do (tiles per pair, rounded
// up, times the tile width); 0 = the wide kernel does not apply (short reductions keep their weights resident in
// the 256-channel kernel; a matrix of at most 256 channels would leave one of the two blocks idle; small problems stay on the other
// kernels).  It / the 256-channel kernel in us: 16384 tokens 4096 -> 1024 fp32 40.8 / 49.2, bfloat16 35.8 / 44.6, int8 36.7 / 52.1, packed 4-bit codes
// 51.9 / 78.5; over 165 shapes the other takes 1.12 of its time.  The line of half the pairs is older than the present issue of the MMAs and
// loses where the last round of its large tiles is nearly empty or few pairs have one: 9000 tokens 3072 -> 768 24.6 / 17.2, 16384 tokens 2048 -> 4096
// int8 94.6 / 76.9, 4096 tokens 4096 -> 4096 64 / 55.
static int wide_bn(const LinearArgs& a) {
    if (g_opt.no_wide || g_opt.no_pair) return 0;
    const nm_packed_t& W = *a.W;
    if (W.in <= kPairResStages * PairCfg<true, 192>::KB || W.out <= 2 * kBM) return 0;
    if (one_wave(a) && !g_opt.wide_any) return 0;
    const long long pairs = sm_count() / 2, out_tiles = (W.out + 4 * kBM - 1) / (4 * kBM);
    int best = 0;
    long long best_cost = 0;
    for (int bn : {224, 192}) {
        if (g_opt.wide_bn && bn != g_opt.wide_bn) continue;
        const long long tiles = out_tiles * ((a.tokens + bn - 1) / bn);
        if (2 * tiles < pairs && !g_opt.wide_any) continue;  // measured: with half the pairs busy it still beats the 256-channel kernel
        const long long cost = ((tiles + pairs - 1) / pairs) * bn;
        if (!best || cost < best_cost) { best = bn; best_cost = cost; }
    }
    return best;
}

// The pair kernel pays off when there is enough work for every SM pair; small problems stay on one CTA.
template <bool SPARSE>
static bool use_pair(const LinearArgs& a) {
    if (g_opt.no_pair) return false;
    const long long tiles = (long long)((a.W->out + 2 * kBM - 1) / (2 * kBM)) * ((a.tokens + 191) / 192);
    const bool fits = !SPARSE || a.W->in / 32 <= PairCfg<SPARSE, 192>::META_COLS;
    if (tiles > sm_count() / 2 && one_wave(a)) return false;  // a second round of pair tiles against one of small tiles
    return fits && tiles >= sm_count() / 2;
}

// Pair kernel with the weights streamed through the ring, or (2:4, reduction up to 1024) kept resident.
template <bool SPARSE, int EPI>
static int pick_pair(const LinearArgs& a) {
    if (use_xres<SPARSE, EPI>(a)) return launch_gemm_xres<SPARSE, EPI>(a);
    if constexpr (SPARSE) {
        if (a.W->in <= kPairResStages * PairCfg<true, 192>::KB && !g_opt.no_resident)
            return launch_gemm_pair<true, 192, EPI, true>(a);
    }
    return launch_gemm_pair<SPARSE, 192, EPI, false>(a);
}

// Token-tile width of the one-CTA kernel: the one whose slowest CTA has the least to do, a tile costing its width plus `fixed`
// tokens (what a tile costs however narrow it is: its weights, barriers, start and end); the wider one on equality.
// The widest that still fills the SMs, the rule before, left half of a last wave idle: 2085 tokens 1024 -> 1002 dense
// 8.7 -> 7.0 us (64 -> 128), 2000 tokens 3072 -> 768 int8 17.4 -> 13.4 and 2500 tokens 2560 -> 640 15.1 -> 11.2 (64 -> 96),
// 384 tokens 1024 -> 4096 8.5 -> 6.9 (64 -> 128), 900 tokens 768 -> 3072 dense 8.8 -> 7.9 (128 -> 192), 128 tokens 768 -> 768
// 5.1 -> 4.7 (64 -> 32).  The choice was the best of the five, or within 2 % of it, on 24 shapes.
template <bool SPARSE>
static int one_cta_bn(const LinearArgs& a, std::initializer_list<int> widths, int fixed) {
    const long long out_tiles = (a.W->out + kBM - 1) / kBM, sms = sm_count();
    int best = 0;
    long long best_cost = 0;
    for (int bn : widths) {
        if (SPARSE && a.W->in / 32 > kTmemCols - 2 * bn) continue;  // the metadata of the reduction beside two accumulators
        if (g_opt.one_bn && bn != g_opt.one_bn) continue;
        const long long tiles = out_tiles * ((a.tokens + bn - 1) / bn);
        const long long cost = ((tiles + sms - 1) / sms) * (bn + fixed);
        if (!best || cost < best_cost) { best = bn; best_cost = cost; }
    }
    return best;
}

// Clusters of `splits` one-CTA tiles that the current device runs at a time (74, 33 and 14 of 2, 4 and 8 CTAs): one more goes into a second
// round, which costs what the split gains.  Asked once per device; 0, that is no split, also where the device does not say.
static int resident_clusters(int splits) {
    static std::mutex mu;
    static int known[64][3] = {};  // 1 + the answer
    const int at = splits == 2 ? 0 : splits == 4 ? 1 : 2;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    int& n = known[dev][at];
    if (n == 0) {
        using Cfg = SplitCfg<true, 64>;
        auto fn = nm_gemm_split_kernel<true, 64, EPI_F32, false>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)splits, 1, 1);
        cfg.blockDim = dim3(kSplitThreads, 1, 1);
        cfg.dynamicSmemBytes = Cfg::SMEM;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)splits; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int fit = 0;
        if (allow_dynamic_smem((const void*)fn, Cfg::SMEM) != cudaSuccess || cudaOccupancyMaxActiveClusters(&fit, (const void*)fn, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        n = 1 + std::max(fit, 0);
    }
    return n - 1;
}

// Where the reduction is split, and how: 1000 * CTAs + token-tile width, or 0.  A split costs its k-blocks, each the tile's width
// plus 256 tokens, and an exchange of 12 times the width; it is taken where that is at most 0.9 of the unsplit kernel's k-blocks
// at the same rate.  Over 299 shapes (1 to 1000 tokens, reductions of 384 to 8192) 0.70 of the unsplit time in the geometric mean, 1.03 at the
// worst, the best of all splits 0.697: 384 tokens 4096 -> 1024 11.9 -> 7.3 us, 64 tokens 768 -> 768 4.5 -> 3.6, 1 token 8192 -> 1024 19.7 -> 5.6;
// not taken: 384 tokens 1024 -> 3072 5.9 / 6.6.
// Formats rebuilt on the way (xf) pay 384 tokens a k-block for the builders, every cluster more the more of them rebuild the same weights, and
// the unsplit kernel has an epilogue of its own to be compared with: 0.63 of the unsplit time over 141 shapes, formats and outputs, 1.017 at the
// worst: 1 token 8192 -> 1536 1:4 / 8 bit 39.9 -> 9.6 us, 384 tokens 1024 -> 1024 1:4 / 8 bit 8.4 -> 7.0, 128 tokens 768 -> 768 2:4 / 4 bit 5.8 -> 4.7;
// not taken: a reduction of three k-blocks (1 token 384 -> 1536, 4:4 / 4 bit 4.25 / 4.51), 200 tokens 1024 -> 4096, 2:4 / 4 bit 7.3 / 8.3.
// `resident(splits)`: clusters of that size that run at a time.
template <bool SPARSE, bool XF, typename Resident>
static int split_plan(const LinearArgs& a, Resident resident) {
    constexpr bool xf = XF;
    const int unsplit_bn = XF ? one_cta_bn<SPARSE>(a, {192, 128, 64}, 160) : one_cta_bn<SPARSE>(a, {192, 128, 96, 64, 32}, 64);
    if (g_opt.split == 1 || g_opt.one_bn || (g_opt.skip_stage && !g_opt.split)) return 0;  // the test hook counts the stages of an unsplit tile
    const int kblocks = a.W->in / kKB, out_tiles = (a.W->out + kBM - 1) / kBM;
    const long long unsplit = xf ? (long long)kblocks * (unsplit_bn + 384) + 4 * unsplit_bn : (long long)kblocks * (unsplit_bn + 256);
    long long best_cost = 0;
    int best = 0;
    for (int splits : {2, 4, 8})
        for (int bn : {32, 64, 96, 128}) {
            const int plan = 1000 * splits + bn, per = (kblocks + splits - 1) / splits;
            if ((bn / splits) % 8 || kblocks < splits || per > kSplitMaxKb) continue;
            if (g_opt.split && plan != g_opt.split) continue;
            const long long clusters = (long long)out_tiles * ((a.tokens + bn - 1) / bn);
            if (clusters * splits > sm_count()) continue;
            const long long cost = xf ? (long long)per * (bn + 384) + 12 * bn + 12 * clusters * splits : (long long)per * (bn + 256) + 12 * bn;
            const bool gains = xf ? cost <= unsplit && kblocks > 3 : 10 * cost <= 9 * unsplit;
            if (g_opt.split ? resident(splits) < 1 : !gains || clusters > resident(splits)) continue;
            if (!best || cost < best_cost) { best = plan; best_cost = cost; }
        }
    return best;
}

template <bool SPARSE, int EPI, bool XF>
static int pick_split(const LinearArgs& a, int plan) {
    const int splits = plan / 1000;
    switch (plan % 1000) {
        case 128: return launch_gemm_split<SPARSE, 128, EPI, XF>(a, splits);
        case 96: return launch_gemm_split<SPARSE, 96, EPI, XF>(a, splits);
        case 64: return launch_gemm_split<SPARSE, 64, EPI, XF>(a, splits);
        default: return launch_gemm_split<SPARSE, 32, EPI, XF>(a, splits);
    }
}

template <bool SPARSE, int EPI, bool XF>
static int pick_bn(const LinearArgs& a) {
    if (const int plan = split_plan<SPARSE, XF>(a, resident_clusters)) return pick_split<SPARSE, EPI, XF>(a, plan);
    if (g_opt.split > 1) return NM_ERR_UNSUPPORTED;  // a split was asked for that this problem cannot have
    const int out_tiles = (a.W->out + kBM - 1) / kBM, sms = sm_count();
    if constexpr (!XF) {
        switch (one_cta_bn<SPARSE>(a, {192, 128, 96, 64, 32}, 64)) {
            case 192: return launch_gemm<SPARSE, 192, EPI, W_TMA>(a);
            case 128: return launch_gemm<SPARSE, 128, EPI, W_TMA>(a);
            case 96: return launch_gemm<SPARSE, 96, EPI, W_TMA>(a);
            case 64: return launch_gemm<SPARSE, 64, EPI, W_TMA>(a);
            default: return launch_gemm<SPARSE, 32, EPI, W_TMA>(a);
        }
    } else {
        // Sparse-target formats with a short reduction and work for every SM pair: the CTA-pair kernel with the weights
        // rebuilt once per output tile into its resident region (32-bit outputs).
        if constexpr (SPARSE && (kF32<EPI> || EPI == EPI_ACC)) {
            const long long pair_tiles = (long long)((a.W->out + 2 * kBM - 1) / (2 * kBM)) * ((a.tokens + 191) / 192);
            if (a.W->in <= kPairResStages * PairCfg<true, 192>::KB && pair_tiles >= sms / 2 && !(pair_tiles > sms / 2 && one_wave(a)) &&
                !g_opt.no_pair && !g_opt.no_resident)
                return launch_gemm_pair<true, 192, EPI, true, true>(a);
        }
        // Short reductions with many token tiles per output tile: build each weight tile once and keep it.
        constexpr int BNR = SPARSE ? 192 : 128;
        if (a.W->in / kKB <= kResidentKB && (long long)out_tiles * ((a.tokens + BNR - 1) / BNR) >= sms && !g_opt.no_resident)
            return launch_gemm<SPARSE, BNR, EPI, W_RESIDENT>(a);
        switch (one_cta_bn<SPARSE>(a, {192, 128, 64}, 160)) {
            case 192: return launch_gemm<SPARSE, 192, EPI, W_BUILD>(a);
            case 128: return launch_gemm<SPARSE, 128, EPI, W_BUILD>(a);
            default: return launch_gemm<SPARSE, 64, EPI, W_BUILD>(a);
        }
    }
}

static int check_linear(int tokens, int out, int in, int n, int m, int bits) {
    int rc = check_pattern(out, in, n, m, bits);
    if (rc != NM_OK) return rc;
    if (tokens < 0) return NM_ERR_SHAPE;
    if (in % kKB) return NM_ERR_SHAPE;          // reduction length: whole 128-wide k-blocks
    if (in > 8192) return NM_ERR_UNSUPPORTED;   // metadata of one output tile must fit in TMEM
    return NM_OK;
}

// Token-tile width of the 512-channel kernel where it takes the problem (2:4 with 8-bit or packed 4-bit codes), or 0.
static int takes_wide(const LinearArgs& a, bool xform, bool sparse) {
    return sparse && (!xform || xf::pattern_of(a.W->n, a.W->m, a.W->bits) == xf::P24_4) ? wide_bn(a) : 0;
}

template <int EPI>
static int run_linear_epi(const LinearArgs& a, bool xform, bool sparse) {
    if (const int bn = takes_wide(a, xform, sparse)) {
        if (bn == 224) return xform ? launch_gemm_wide<224, EPI, true>(a) : launch_gemm_wide<224, EPI>(a);
        return xform ? launch_gemm_wide<192, EPI, true>(a) : launch_gemm_wide<192, EPI>(a);
    }
    if (xform) return sparse ? pick_bn<true, EPI, true>(a) : pick_bn<false, EPI, true>(a);
    if (sparse) return use_pair<true>(a) ? pick_pair<true, EPI>(a) : pick_bn<true, EPI, false>(a);
    return use_pair<false>(a) ? pick_pair<false, EPI>(a) : pick_bn<false, EPI, false>(a);
}

static int run_linear(const LinearArgs& a, int epi) {
    if (!a.W) return NM_ERR_NULL;
    const nm_packed_t& W = *a.W;
    int rc = check_linear(a.tokens, W.out, W.in, W.n, W.m, W.bits);
    if (rc != NM_OK) return rc;
    const int pat = xf::pattern_of(W.n, W.m, W.bits);
    const bool xform = pat != xf::PNONE;
    const bool sparse = xform ? xf::sparse_target(pat) : W.n != W.m;  // tensor-core form of the weights
    if (!a.X || !W.values || (W.n != W.m && !W.meta)) return NM_ERR_NULL;
    if (epi != EPI_ACC && !a.sw) return NM_ERR_NULL;
    if (epi == EPI_F32 && !a.Y) return NM_ERR_NULL;
    if (epi == EPI_ACC && !a.ACC) return NM_ERR_NULL;
    if ((epi == EPI_Q8 || epi == EPI_BF16) && !a.NARROW) return NM_ERR_NULL;
    if (epi == EPI_Q8 && !(a.sy >= 1.17549435e-38f && a.sy <= 3.402823466e38f)) return NM_ERR_SHAPE;  // positive, normal, finite
    if (!aligned(a.X, 16) || !aligned(W.values, 16) || (W.meta && !aligned(W.meta, 16))) return NM_ERR_ALIGN;
    if ((a.Y && !aligned(a.Y, 4)) || (a.ACC && !aligned(a.ACC, 4))) return NM_ERR_ALIGN;
    if (epi == EPI_BF16 && !aligned(a.NARROW, 2)) return NM_ERR_ALIGN;
    if (a.tokens == 0 || W.out == 0) return NM_OK;
    switch (epi) {
        case EPI_F32: return a.absmax ? run_linear_epi<EPI_F32MAX>(a, xform, sparse) : run_linear_epi<EPI_F32>(a, xform, sparse);
        case EPI_ACC: return run_linear_epi<EPI_ACC>(a, xform, sparse);
        case EPI_Q8: return run_linear_epi<EPI_Q8>(a, xform, sparse);
        default: return run_linear_epi<EPI_BF16>(a, xform, sparse);
    }
}

}  // namespace nm

extern "C" {

int nm_pair_tile_plan(int n_tok_tiles, int n_out_tiles, int pairs, int resident, int band_request, int* start,
                      int* tile_out, int* tile_tok) {
    if (!start) return NM_ERR_NULL;
    if (n_tok_tiles < 1 || n_out_tiles < 1 || pairs < 1 || pairs > nm::kMaxPairs ||
        (long long)n_tok_tiles * n_out_tiles > 0x7fffffffll || pairs > n_tok_tiles * n_out_tiles)
        return NM_ERR_SHAPE;
    const int band = nm::plan_pair_tiles(n_tok_tiles, n_out_tiles, pairs, resident != 0, band_request, start);
    for (int t = 0; t < n_tok_tiles * n_out_tiles; ++t) {
        const nm::TileCoord c = nm::tile_coord(t, n_tok_tiles, n_out_tiles, band);
        if (tile_out) tile_out[t] = c.o;
        if (tile_tok) tile_tok[t] = c.t;
    }
    return band;
}

int nm_split_plan(int tokens, int out, int in, int n, int m, int bits, const int* clusters) {
    const int rc = nm::check_linear(tokens, out, in, n, m, bits);
    if (rc != NM_OK) return rc;
    if (tokens == 0 || out == 0) return 0;
    const nm_packed_t W{out, in, n, m, bits, nullptr, nullptr};
    nm::LinearArgs a{};
    a.tokens = tokens; a.W = &W;
    const int pat = nm::xf::pattern_of(n, m, bits);
    const bool xform = pat != nm::xf::PNONE, sparse = xform ? nm::xf::sparse_target(pat) : n != m;
    auto resident = [&](int splits) { return clusters ? clusters[splits == 2 ? 0 : splits == 4 ? 1 : 2] : nm::resident_clusters(splits); };
    if (nm::takes_wide(a, xform, sparse)) return 0;
    if (xform) return sparse ? nm::split_plan<true, true>(a, resident) : nm::split_plan<false, true>(a, resident);
    if (sparse) return nm::use_pair<true>(a) ? 0 : nm::split_plan<true, false>(a, resident);
    return nm::use_pair<false>(a) ? 0 : nm::split_plan<false, false>(a, resident);
}

int nm_debug_set_option(const char* name, int value) {
    if (!name) return NM_ERR_NULL;
    struct { const char* name; int* slot; } table[] = {
        {"no_pdl", &nm::g_no_pdl}, {"no_pair", &nm::g_opt.no_pair}, {"no_resident", &nm::g_opt.no_resident},
        {"no_wide", &nm::g_opt.no_wide}, {"wide_any", &nm::g_opt.wide_any}, {"wide_bn", &nm::g_opt.wide_bn},
        {"one_bn", &nm::g_opt.one_bn}, {"split", &nm::g_opt.split}, {"xres", &nm::g_opt.xres}, {"grouped", &nm::g_opt.grouped}, {"band", &nm::g_opt.band}, {"pack_form", &nm::g_pack_form}};
    for (auto& e : table)
        if (!strcmp(name, e.name)) { *e.slot = value; return NM_OK; }
#ifdef NM_TEST_HOOKS
    if (!strcmp(name, "skip_stage")) { nm::g_opt.skip_stage = value; return NM_OK; }
    if (!strcmp(name, "skip_pack_copy")) return nm::pack_set_skip_unit(value - 1);
#endif
    return NM_ERR_UNSUPPORTED;
}

int nm_debug_set_trace(unsigned long long* buffer) {
#ifdef NM_TRACE
    nm::g_trace_buffer = buffer;
    return NM_OK;
#else
    (void)buffer;
    return NM_ERR_UNSUPPORTED;
#endif
}

int nm_int_linear_check(int tokens, int out, int in, int n, int m, int bits) {
    return nm::check_linear(tokens, out, in, n, m, bits);
}

size_t nm_int_linear_workspace_bytes(int, int, int, int, int, int) { return 0; }

int nm_int_linear(const int8_t* X, int tokens, const nm_packed_t* W, float sx, const float* sw,
                  const float* bias, float* Y, void*, size_t, uint32_t* status, void* stream) {
    nm::LinearArgs a{X, tokens, W, sx, nullptr, sw, bias, Y, nullptr, nullptr, status, (cudaStream_t)stream};
    return nm::run_linear(a, nm::EPI_F32);
}

int nm_int_linear_dsx(const int8_t* X, int tokens, const nm_packed_t* W, const float* sx_dev,
                      const float* sw, const float* bias, float* Y, float* absmax_out, void*, size_t,
                      uint32_t* status, void* stream) {
    if (!sx_dev) return NM_ERR_NULL;
    nm::LinearArgs a{X, tokens, W, 0.0f, sx_dev, sw, bias, Y, nullptr, absmax_out, status, (cudaStream_t)stream};
    return nm::run_linear(a, nm::EPI_F32);
}

int nm_int_linear_q8(const int8_t* X, int tokens, const nm_packed_t* W, float sx, const float* sw,
                     const float* bias, float sy, int8_t* Yq, void*, size_t, uint32_t* status, void* stream) {
    nm::LinearArgs a{X, tokens, W, sx, nullptr, sw, bias, nullptr, nullptr, nullptr, status, (cudaStream_t)stream};
    a.NARROW = Yq; a.sy = sy;
    return nm::run_linear(a, nm::EPI_Q8);
}

int nm_int_linear_bf16(const int8_t* X, int tokens, const nm_packed_t* W, float sx, const float* sw,
                       const float* bias, uint16_t* Ybf16, void*, size_t, uint32_t* status, void* stream) {
    nm::LinearArgs a{X, tokens, W, sx, nullptr, sw, bias, nullptr, nullptr, nullptr, status, (cudaStream_t)stream};
    a.NARROW = Ybf16;
    return nm::run_linear(a, nm::EPI_BF16);
}

int nm_int_linear_acc(const int8_t* X, int tokens, const nm_packed_t* W, int32_t* ACC, void*, size_t,
                      uint32_t* status, void* stream) {
    nm::LinearArgs a{X, tokens, W, 1.0f, nullptr, nullptr, nullptr, nullptr, ACC, nullptr, status, (cudaStream_t)stream};
    return nm::run_linear(a, nm::EPI_ACC);
}

}  // extern "C"
