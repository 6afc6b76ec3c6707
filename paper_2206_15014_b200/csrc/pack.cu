// N:M magnitude projection + per-channel symmetric quantisation + packing (one HBM pass).
//
// Work decomposition: a row is covered by 1, 2, 4 ... 32 warps of the same block, a warp by up to four steps of 256
// consecutive weights, of which every lane holds eight (32 bytes: one load per operand and step).  Eight consecutive weights
// are whole groups of four or eight, so everything after the row maximum is lane-local and stays in registers; the
// codes and the index fields of a step are one store each, coalesced over the warp.
#include "common.cuh"
#include "sm100_ptx.cuh"
#include <cuda_runtime.h>
#include <vector>
#include <mutex>
#include <algorithm>
#include <cstdlib>

namespace nm {

struct PackJobDev {
    const float* W;
    const float* U;
    uint8_t* values;
    uint32_t* meta;
    float* scales;
    int out, in;
    int wpr_log2;         // log2(warps per row)
    unsigned unit_begin;  // first block of this job inside the launch
    unsigned vrow_bytes;  // bytes of one row of values
    unsigned mrow_words;  // words of one row of metadata
};

// Dense outputs of one job of a batched ADMM step (parallel to the PackJobDev table).
struct DenseOutDev {
    float* Z;
    float* U_next;
};

// Job tables of up to kInlineJobs entries travel as a kernel parameter: no table in device memory, no
// host-to-device copy in front of the launch.  A single matrix is a table of one.
static constexpr int kInlineJobs = 8;
struct PackJobInline {
    PackJobDev j[kInlineJobs];
};

static constexpr int kPackMinWarps = 4;
#ifndef NM_WAIT_LIMIT
#define NM_WAIT_LIMIT (1ll << 31)
#endif
static constexpr long long kPackWaitLimit = NM_WAIT_LIMIT;  // SM clocks a warp waits for its staged chunk (about a second)

// Test hook, compiled in with -DNM_TEST_HOOKS only (the library the timeout test loads, never the product's): in the
// staged form, warp 0 of block 0 leaves the copies of its unit number `d_pack_skip_unit` (counted per block) unissued --
// nothing is armed, nothing is copied, no address is touched -- so that the wait for that chunk runs out.
#ifdef NM_TEST_HOOKS
__device__ int d_pack_skip_unit = -1;
int pack_set_skip_unit(int unit) {
    NM_CUDA_TRY(cudaMemcpyToSymbol(d_pack_skip_unit, &unit, sizeof(unit)));
    return NM_OK;
}
#define NM_PACK_SKIP(iter) (blockIdx.x == 0 && w == 0 && (iter) == d_pack_skip_unit)
#else
#define NM_PACK_SKIP(iter) false
#endif
// group_mode of pack_kernel: scale per row from the row itself; only fold the row maxima per group into
// `scales`; take the scales found in `scales`.
enum { kGroupNone = 0, kGroupMaxPass = 1, kGroupScalesGiven = 2 };

// Eight consecutive floats that are not read again: one 32-byte access, or two of 16 bytes where the rows are only aligned to those.
__device__ __forceinline__ void ld8(const float* p, float* x) {
    asm volatile("ld.global.cs.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]) : "l"(p) : "memory");
}
__device__ __forceinline__ void ld4(const float* p, float* x) {
    const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
    x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
}
__device__ __forceinline__ void st8(float* p, const float* x) {
    asm volatile("st.global.cs.v8.f32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]),
                 "f"(x[5]), "f"(x[6]), "f"(x[7]), "l"(p) : "memory");
}
__device__ __forceinline__ void st4(float* p, const float* x) { __stcs(reinterpret_cast<float4*>(p), make_float4(x[0], x[1], x[2], x[3])); }
// n = 1, and 2 of 8: the kept values and their positions straight from one or two passes of
// "largest magnitude, first one on equality" (strict >), positions ascending.
template <int N, int M>
__device__ __forceinline__ void select_passes(const float* v, float* sel, unsigned* selp) {
    float best = fabsf(v[0]), bv = v[0];
    unsigned bi = 0;
#pragma unroll
    for (int j = 1; j < M; ++j) {
        const float aj = fabsf(v[j]);
        const bool gt = aj > best;
        best = gt ? aj : best;
        bv = gt ? v[j] : bv;
        bi = gt ? (unsigned)j : bi;
    }
    if constexpr (N == 1) {
        sel[0] = bv; selp[0] = bi;
    } else {
        float best2 = -1.0f, bv2 = 0.0f;  // magnitudes are >= 0
        unsigned bj = 0;
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const float aj = fabsf(v[j]);
            const bool gt = (aj > best2) && ((unsigned)j != bi);
            best2 = gt ? aj : best2;
            bv2 = gt ? v[j] : bv2;
            bj = gt ? (unsigned)j : bj;
        }
        const bool sw = bj < bi;
        sel[0] = sw ? bv2 : bv; selp[0] = sw ? bj : bi;
        sel[1] = sw ? bv : bv2; selp[1] = sw ? bi : bj;
    }
}

// Two of four by a tournament on the pairs (0,1) and (2,3).  With "larger magnitude first, lower index first
// among equals" the two kept positions are 0 and 1 when the smaller of the first pair is >= the larger of the
// second, 2 and 3 when the smaller of the second pair is > the larger of the first, and otherwise the larger of
// each pair (the first one of a pair on equality).  Kept values in ascending position; returns the index nibble.
__device__ __forceinline__ unsigned select_2_of_4(const float* v, float* sel) {
    const bool i01 = fabsf(v[1]) > fabsf(v[0]), i23 = fabsf(v[3]) > fabsf(v[2]);
    const float w01 = i01 ? v[1] : v[0], l01 = i01 ? v[0] : v[1], w23 = i23 ? v[3] : v[2], l23 = i23 ? v[2] : v[3];
    const bool both01 = fabsf(l01) >= fabsf(w23), both23 = fabsf(l23) > fabsf(w01);
    sel[0] = both01 ? v[0] : (both23 ? v[2] : w01);
    sel[1] = both01 ? v[1] : (both23 ? v[3] : w23);
    const unsigned mixed = (i01 ? 9u : 8u) + (i23 ? 4u : 0u);
    return both01 ? 0x4u : (both23 ? 0xEu : mixed);
}

// Bit mask of the positions kept in one group (2 of 4 in the search, 4 of 8): position i is kept iff fewer than N others beat it,
// where j beats i when |v_j| > |v_i|, or |v_j| == |v_i| and j < i.
template <int N, int M>
__device__ __forceinline__ unsigned keep_mask(const float* a) {
    if constexpr (N == 4 && M == 8) {
        // Four of eight: the fourth largest magnitude T from a selection network (both halves sorted with five
        // compare-exchanges each, then the four maxima of a bitonic half-cleaner hold the four largest and their
        // minimum is T), the support as a >= T.  Equal magnitudes at the threshold make that more than four
        // positions; only then does the rank network below decide (lower index first).
        auto cx = [](float& hi, float& lo) { const float h = fmaxf(hi, lo), l = fminf(hi, lo); hi = h; lo = l; };
        float x0 = a[0], x1 = a[1], x2 = a[2], x3 = a[3], y0 = a[4], y1 = a[5], y2 = a[6], y3 = a[7];
        cx(x0, x1); cx(x2, x3); cx(x0, x2); cx(x1, x3); cx(x1, x2);   // x0 >= x1 >= x2 >= x3
        cx(y0, y1); cx(y2, y3); cx(y0, y2); cx(y1, y3); cx(y1, y2);   // y0 >= y1 >= y2 >= y3
        const float T = fminf(fminf(fmaxf(x0, y3), fmaxf(x1, y2)), fminf(fmaxf(x2, y1), fmaxf(x3, y0)));
        unsigned mask = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) mask |= (a[i] >= T ? 1u : 0u) << i;
        if (__popc(mask) == N) return mask;
    }
    int rank[M];
#pragma unroll
    for (int i = 0; i < M; ++i) rank[i] = 0;
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
        for (int j = i + 1; j < M; ++j) {
            bool ge = a[i] >= a[j];  // i (the lower index) beats j on >=, j beats i otherwise
            rank[j] += ge ? 1 : 0;
            rank[i] += ge ? 0 : 1;
        }
    unsigned mask = 0;
#pragma unroll
    for (int i = 0; i < M; ++i) mask |= (rank[i] < N ? 1u : 0u) << i;
    return mask;
}

// ---------------------------------------------------------------------------------------------
// ADMM-Dist scale (Sec. 3.3.1, "Minimize Quantization Distance"): per output channel the scale that
// minimises the squared distance E_j between the N:M-projected channel and its quantised form, searched
// over the candidates s_j = fl32(s_max * (64 - j) / 64), j = 0 .. ncand-1 (s_max = the ADMM-Max scale;
// lowest j on equal distance).  The decision is taken on distances held in double, in two steps:
//
// 1. Bounds of every candidate's distance, in units of s_max: y = |v| / s_max.
//    4 bits (dist_bounds4): with the nearest codes E_j = sum y^2 - 2 s_j * sum over the thresholds (k - 1/2) s_j of what lies above
//    them, sum of (y - threshold)+.  The values go, rounded to 2^-16, into bins of 1/32, each with its count and the sum of its
//    remainders, and sums over the higher bins give all (value - threshold)+ but those of the bin that holds the threshold; these lie
//    between max(0, f - c t) and f (1 - t / width) (c values of remainders f in sum, the threshold at t; both bounds of a
//    convex function with given mean), exact for one value.  All thresholds are multiples of 1/128, so everything is whole
//    numbers.  That is a pass over the values and 8 lookups per candidate in place of 32 evaluations of every value.  1.2 to 1.5
//    of 32 candidates are left on rows of Gaussian weights; bins of 1/16 left 2 to 3.
//    8 bits: the row's largest value alone rules out all candidates but the first few (3 to 16; see there); those are evaluated in single
//    precision: code magnitude k = min(rne(y * 64 / (64 - j)), end code of v's sign), d = y - k * (64 - j) / 64, sum of d * d: five
//    operations per candidate and kept value, four of them as packed pairs, sums (at most 80 roundings of non-negative terms)
//    good to 2^-17 relative.
//    Per value |d| is within eps = 2^(b - 1) * 2^-19 of the exact distance: y and 64 / (64 - j) carry relative errors of 1.5 * 2^-23
//    and 2^-24 and the real scale s_j one of 2^-24, which move d by less than 2^(b - 1) * 2^-21 when the code is the true one; the
//    code differs only where the quotient is within 2^(b - 1) * 3 * 2^-23 of a tie, and there the two
//    distances differ by twice that; the rounding to 2^-16 adds 2^-17, half of eps.  By the triangle inequality the root of the exact E_j
//    is within eps * sqrt(values) of the root of the computed one.
// 2. A candidate whose lower bound exceeds another's upper bound cannot win.  Usually one is left; otherwise those that are left are
//    evaluated in double from the fp32 weights (code from the IEEE quotient, d = v - s_j * code and E += d * d as two FMAs, s_j * code
//    being exact in double) and compared.  Scales outside [2^-126, 2^125] and non-finite rows skip step 1.
//
// A row spans `wpr` warps; the partial sums of its warps are added in a fixed order, so the result is
// deterministic.  85 M weights at 2:4 / 4 bit and 32 candidates, search and projection: 461 us with all candidates in single precision,
// 281 so (80 shapes and formats from 64 to 4096 rows 0.40 to 0.95).  What bounds it: instructions (61 % of the issue slots in an earlier
// state), their fetching among the stalls.
// ---------------------------------------------------------------------------------------------
template <int N, int M>
__device__ __forceinline__ void kept_values(const float* v, float* sel) {
    if constexpr (N == M) {
#pragma unroll
        for (int p = 0; p < M; ++p) sel[p] = v[p];
    } else if constexpr ((N == 1) || (N == 2 && M == 8)) {
        unsigned selp[N];
        select_passes<N, M>(v, sel, selp);
    } else if constexpr (N == 2) {
        (void)select_2_of_4(v, sel);
    } else {
        float a[M];
#pragma unroll
        for (int p = 0; p < M; ++p) a[p] = fabsf(v[p]);
        const unsigned mask = keep_mask<N, M>(a);
        {
#pragma unroll
            for (int c = 0; c < N; ++c) sel[c] = 0.0f;
#pragma unroll
            for (int p = 0; p < M; ++p) {
                const bool kept = (mask >> p) & 1u;
                const int before = __popc(mask & ((1u << p) - 1u));
#pragma unroll
                for (int c = 0; c < N; ++c)
                    if (c <= p && (M - p) >= (N - c)) sel[c] = (kept && before == c) ? v[p] : sel[c];
            }
        }
    }
}


// Distance of candidate j in double over the warp's part of the row (every lane returns the sum over the lanes), from the lane's `count` kept
// values, value i at x[32 i].  A short loop over shared memory: few rows come here, and unrolled over registers its code kept the
// rest of the kernel out of the instruction cache.  Codes from RN(1 / s_j) as in pack_row, the IEEE division only next to a tie.  Four values
// at a time, their codes and distances independent of one another: a row with several candidates left is a small matrix's last one, and
// value by value it took the latency of every step: 256 x 1024 dense 4 bit 13.8 -> 11.1 us, 1024 x 1024 14.9 -> 12.2, 4096 x 1024 2:4 17.7 -> 15.9.
template <int BITS>
__device__ __noinline__ double dist_exact(const float* x, int count, float smax, int j) {
    constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
    constexpr float kLo = -(float)(1 << (BITS - 1)) - 0.49f, kHi = qmax + 0.49f;
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
    const float sj = __fmul_rn(smax, (float)(64 - j) * 0.015625f), rs = __frcp_rn(sj);
    const bool fast_ok = sj >= 1.17549435e-38f && sj <= 4.25e37f;
    const double nsd = -(double)sj;
    double e[2] = {0.0, 0.0};
    for (int i = 0; i < count; i += 4) {  // values past `count` are zeros and add nothing
        float xi[4], t[4], worst = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) xi[k] = x[32 * (i + k)];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = __fmaf_rn(xi[k], rs, kMagic);
            worst = ptx::max_abs_nan(__fmaf_rn(xi[k], rs, -__fsub_rn(t[k], kMagic)), 0.0f, worst);
            t[k] = fminf(fmaxf(t[k], kMagic - qmax - 1.0f), kMagic + qmax);
        }
        if (!(worst <= 0.49996948f) || !fast_ok) {
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] = __fadd_rn(fminf(fmaxf(__fdiv_rn(xi[k], sj), kLo), kHi), kMagic);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // the code as a double: 2^52 + 2^31 + code is whole
            const double r = __dsub_rn(__hiloint2double(0x43300000, (__float_as_int(t[k]) - 0x4B400000) ^ (int)0x80000000), 4503601774854144.0);
            const double d = fma(nsd, r, (double)xi[k]);
            e[k & 1] = fma(d, d, e[k & 1]);
        }
    }
    double sum = e[0] + e[1];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    return sum;
}

// Bins of dist_bounds4, per warp: 128 of the tail of the negative values, 256 of all; each counts its values and sums their remainders.
constexpr int kTailBins = 128, kAllBins = 256, kTailFirst = 123;
struct DistBins {
    uint32_t bin[kTailBins + kAllBins];  // count << 21 | sum of remainders
    uint2 above[kTailBins + kAllBins];   // count and sum of the values in higher bins, permuted so that lanes store side by side
};

// Step 1 of the search at 4 bits: bounds of every candidate's distance (lane j: candidate j), less the sum of squares `q` of the warp's
// values that all candidates share, in units of s_max^2.  See above.
template <int N, int M>
__device__ __forceinline__ void dist_bounds4(const float* x, int steps, int lane, float smax, DistBins& h, double& lo, double& hi, float& q) {
    constexpr int KS = 8 / M * N;
    constexpr float kMagic = 12582912.0f;
    uint4* zero = reinterpret_cast<uint4*>(h.bin);
#pragma unroll
    for (int i = 0; i < (kTailBins + kAllBins) / 128; ++i) zero[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    const float r0 = __frcp_rn(smax);
    q = 0.0f;
#pragma unroll
    for (int st = 0; st < 4; ++st)
        if (st < steps) {  // steps beyond the warp's columns hold zeros
#pragma unroll
            for (int i = 0; i < KS; ++i) {
                const float t = __fmaf_rn(fabsf(__fmul_rn(x[st * KS + i], r0)), 65536.0f, kMagic);
                const int y = __float_as_int(t) - 0x4B400000;  // magnitude in units of s_max / 65536, at most 7 * 65536
                const float yf = __fsub_rn(t, kMagic);
                q = __fmaf_rn(yf, yf, q);
                if (y >= 16384) {  // the lowest threshold of all candidates is 33 * 512
                    const uint32_t w = (uint32_t)(y & 2047) | (1u << 21);
                    atomicAdd(&h.bin[kTailBins + (y >> 11)], w);
                    if (x[st * KS + i] < 0.0f && y >= kTailFirst * 2048) atomicAdd(&h.bin[(y >> 11) - kTailFirst], w);
                }
            }
        }
    __syncwarp();
    // sums over the higher bins: lane l has bins 8 l .. 8 l + 7 of all values and 4 l .. 4 l + 3 of the tail
    {
        uint32_t wa[8], wt[4];
        *reinterpret_cast<uint4*>(wa) = *reinterpret_cast<const uint4*>(h.bin + kTailBins + 8 * lane);
        *reinterpret_cast<uint4*>(wa + 4) = *reinterpret_cast<const uint4*>(h.bin + kTailBins + 8 * lane + 4);
        *reinterpret_cast<uint4*>(wt) = *reinterpret_cast<const uint4*>(h.bin + 4 * lane);
        uint32_t sa[8], st[4], sum_a = 0, sum_t = 0, cnt = 0;  // cnt: tail << 16 | all (at most 1024 each)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sa[i] = (wa[i] >> 21) * (uint32_t)((8 * lane + i) << 11) + (wa[i] & 0x1FFFFFu);
            sum_a += sa[i]; cnt += wa[i] >> 21;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            st[i] = (wt[i] >> 21) * (uint32_t)((4 * lane + i + kTailFirst) << 11) + (wt[i] & 0x1FFFFFu);
            sum_t += st[i]; cnt += (wt[i] >> 21) << 16;
        }
        uint32_t xa = sum_a, xt = sum_t, xc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t ua = __shfl_down_sync(0xffffffffu, xa, o), ut = __shfl_down_sync(0xffffffffu, xt, o), uc = __shfl_down_sync(0xffffffffu, xc, o);
            if (lane + o < 32) { xa += ua; xt += ut; xc += uc; }
        }
        xa -= sum_a; xt -= sum_t; xc -= cnt;
        uint32_t ca = xc & 0xFFFFu, ct = xc >> 16;
#pragma unroll
        for (int i = 7; i >= 0; --i) {
            h.above[kTailBins + i * 32 + lane] = make_uint2(ca, xa);
            ca += wa[i] >> 21; xa += sa[i];
        }
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            h.above[i * 32 + lane] = make_uint2(ct, xt);
            ct += wt[i] >> 21; xt += st[i];
        }
    }
    __syncwarp();
    // sum of (value - threshold) over the values above each of the candidate's thresholds
    const uint32_t m = 64u - (uint32_t)lane;
    uint32_t g_lo = 0, g_hi = 0;
    auto threshold = [&](uint32_t u, uint32_t word, uint2 above) {  // u: the threshold in units of s_max / 128
        const uint32_t part = u & 3u, c = word >> 21, f = word & 0x1FFFFFu;  // where it stands in its bin; the bin's values
        const uint32_t full = above.y - u * 512u * above.x;
        const uint32_t l = (uint32_t)max(0, (int)(f - c * part * 512u)), up = (f * (4u - part) + 3u) >> 2;
        g_lo += full + l;
        g_hi += full + (c == 1u ? l : up);
    };
#pragma unroll
    for (uint32_t k = 1; k <= 7; ++k) {
        const uint32_t u = (2u * k - 1u) * m, b = u >> 2;
        threshold(u, h.bin[kTailBins + b], h.above[kTailBins + ((b & 7u) << 5) + (b >> 3)]);
    }
    const uint32_t u8 = 15u * m, b8 = (u8 >> 2) - kTailFirst;
    threshold(u8, h.bin[b8], h.above[((b8 & 3u) << 5) + (b8 >> 2)]);
    lo = -4.76837158203125e-7 * (double)m * (double)g_hi;  // 2 s_j / 65536 = m * 2^-21
    hi = -4.76837158203125e-7 * (double)m * (double)g_lo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    q *= 2.3283064365386963e-10f;  // 2^-32
}

template <int N, int M> constexpr int kKeptBytes = 32 / M * N * 128;  // kept values of a warp

// Winning candidate of this warp's row.  `red_e` holds 32 doubles per warp of the block, `bins` (4 bits) one DistBins, `kept` this warp's
// kept values (ALIAS: in the place of the bins, once nobody reads them).  Every warp of the block calls it (block-wide barriers when a
// row spans warps).
template <int N, int M, int BITS, bool ALIAS>
__device__ __forceinline__ int dist_search(const float* v, int steps, int lane, int w, int wpr, int row_in_block, bool row_ok,
                                           float smax, bool bad, int ncand, double* red_e, DistBins* bins, float* kept) {
    constexpr int KN = 32 / M * N, KS = KN / 4;       // kept values per lane, and per step
    constexpr float qend = (float)(1 << (BITS - 1));  // magnitude of the negative end code
    constexpr float kMagic = 12582912.0f;             // 1.5 * 2^23: adding it rounds to the nearest-even integer
    constexpr float kEps = qend * 1.9073486328125e-6f;  // 2^(b - 1) * 2^-19
    const float inf = __int_as_float(0x7f800000);
    const bool usable = !bad && smax >= 1.17549435e-38f && smax <= 4.25e37f;  // 1 / s_max is a normal number
    const float slack = kEps * sqrtf((float)(KN * 32 * wpr));
    bool left = lane < ncand;
    float x[KN];  // the lane's kept values, for step 2 in shared memory
#pragma unroll
    for (int g = 0; g < 32 / M; ++g) {
        float group[M];  // opaque copies: the selection of pack_row is otherwise shared with this one and kept over the search, in spilled registers
#pragma unroll
        for (int i = 0; i < M; ++i) { group[i] = v[g * M + i]; asm volatile("" : "+f"(group[i])); }
        kept_values<N, M>(group, x + g * N);
    }
    if constexpr (!ALIAS) {
#pragma unroll
        for (int i = 0; i < KN; ++i) kept[i * 32 + lane] = x[i];
    }
    if constexpr (BITS == 4) {
        double lo = 0.0, hi = 0.0;
        float q = 0.0f;
        if (usable && row_ok) dist_bounds4<N, M>(x, steps, lane, smax, bins[w], lo, hi, q);
        if (wpr > 1) {
            double* mine = reinterpret_cast<double*>(bins[w].above);
            __syncwarp();
            mine[lane] = lo;
            mine[32 + lane] = hi;
            if (lane == 0) mine[64] = (double)q;
            __syncthreads();
            lo = hi = 0.0;
            q = 0.0f;
            for (int c = 0; c < wpr; ++c) {
                const double* part = reinterpret_cast<const double*>(bins[row_in_block * wpr + c].above);
                lo += part[lane];
                hi += part[32 + lane];
                q += (float)part[64];
            }
            if (ALIAS) __syncthreads();
        }
        if constexpr (ALIAS) {
            static_assert(kKeptBytes<N, M> <= (int)sizeof(DistBins), "kept values in the place of the bins");
            __syncwarp();
#pragma unroll
            for (int i = 0; i < KN; ++i) kept[i * 32 + lane] = x[i];
        }
        // |root of the exact distance - root of the distance of the values as binned| <= slack
        const float root = sqrtf(fmaxf(q * 1.0000077f + (float)hi, 0.0f) + 1e-3f * slack);
        const double margin = 1.001 * (double)(slack * (2.0f * root + slack));
        lo -= margin;
        hi = lane < ncand ? hi + margin : 1e300;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) hi = fmin(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        left = left && (!usable || lo <= hi);
    } else {
        // the row's largest value alone makes candidate j's distance at least (2 j - 1)^2 (its quotient is beyond the end code, 127 or
        // 128), that of candidate 0 is at most a quarter per kept value
        const int last = (int)((0.5003f * sqrtf((float)(KS * 32 * steps * wpr)) + 1.0003f) * 0.5f) + 1;
        const int eval = min(ncand, last + 1);
        float mine = inf;  // lane j: candidate j's distance in units of s_max^2
        if (usable && row_ok) {
            uint64_t y[KN / 2];
            float lim[KN];
            {
                const float r0 = __frcp_rn(smax);
#pragma unroll
                for (int i = 0; i < KN; ++i) lim[i] = kMagic + (x[i] < 0.0f ? qend : qend - 1.0f);
#pragma unroll
                for (int i = 0; i < KN / 2; ++i) y[i] = ptx::pack_f32x2(fabsf(__fmul_rn(x[2 * i], r0)), fabsf(__fmul_rn(x[2 * i + 1], r0)));
            }
            const float my_inv = __frcp_rn((float)(64 - lane) * 0.015625f);  // 64 / (64 - j) of candidate j = lane
            const uint64_t magic2 = ptx::pack_f32x2(kMagic, kMagic), nmagic2 = ptx::pack_f32x2(-kMagic, -kMagic);
            // two candidates a trip, their sums over the lanes by a transposing butterfly: lane l ends up with candidate
            // 2 g + l / 16 of trip g and keeps trip l % 16's
            constexpr int kTrip = 2, kLanes = 32 / kTrip;
            float kept = inf;
#pragma unroll 1
            for (int g = 0; kTrip * g < eval; ++g) {
                float e[kTrip];
#pragma unroll
                for (int k = 0; k < kTrip; ++k) {
                    const float inv = __shfl_sync(0xffffffffu, my_inv, kTrip * g + k);
                    const float na = (float)(kTrip * g + k - 64) * 0.015625f;  // -(64 - j) / 64
                    const uint64_t inv2 = ptx::pack_f32x2(inv, inv), na2 = ptx::pack_f32x2(na, na);
                    uint64_t acc = 0;
                    auto add = [&](int i) {
                        float t0, t1;
                        ptx::unpack_f32x2(ptx::fma_f32x2(y[i], inv2, magic2), t0, t1);
                        const uint64_t code = ptx::add_f32x2(ptx::pack_f32x2(fminf(t0, lim[2 * i]), fminf(t1, lim[2 * i + 1])), nmagic2);
                        const uint64_t d = ptx::fma_f32x2(na2, code, y[i]);
                        acc = ptx::fma_f32x2(d, d, acc);
                    };
                    if constexpr (KS >= 4) {
#pragma unroll
                        for (int st = 0; st < 4; ++st)
                            if (st < steps) {  // steps beyond the warp's columns hold zeros
#pragma unroll
                                for (int i = st * KS / 2; i < (st + 1) * KS / 2; ++i) add(i);
                            }
                    } else {
#pragma unroll
                        for (int i = 0; i < KN / 2; ++i) add(i);
                    }
                    float a0, a1;
                    ptx::unpack_f32x2(acc, a0, a1);
                    e[k] = a0 + a1;
                }
                const bool up = lane & kLanes;
                const float keep = up ? e[1] : e[0], give = up ? e[0] : e[1];
                e[0] = keep + __shfl_xor_sync(0xffffffffu, give, kLanes);
#pragma unroll
                for (int o = kLanes / 2; o > 0; o >>= 1) e[0] += __shfl_xor_sync(0xffffffffu, e[0], o);
                if (lane % kLanes == g) kept = e[0];
            }
            mine = __shfl_sync(0xffffffffu, kept, (lane % kTrip) * kLanes + lane / kTrip);  // candidate j to lane j
        }
        if (wpr > 1) {
            float* red_f = reinterpret_cast<float*>(red_e);
            red_f[w * 32 + lane] = mine;
            __syncthreads();
            mine = 0.0f;
            for (int c = 0; c < wpr; ++c) mine += red_f[(row_in_block * wpr + c) * 32 + lane];
            __syncthreads();  // the array is used again below
        }
        // candidates that the bounds leave
        const float root = sqrtf(mine), lo = fmaxf(root - slack, 0.0f);
        float best = lane < ncand ? (root + slack) * (root + slack) * 1.0000153f : inf;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
        left = left && (!usable || lo * lo * 0.9999847f <= best);
    }
    const unsigned mask = row_ok ? __ballot_sync(0xffffffffu, left) : 1u;
    const bool single = (mask & (mask - 1u)) == 0u;
    if (single && wpr == 1) return __ffs(mask) - 1;
    double exact = __longlong_as_double(0x7ff0000000000000ll);
    if (!single) {
        for (unsigned m = mask; m; m &= m - 1u) {
            const int j = __ffs(m) - 1;
            const double e = dist_exact<BITS>(kept + lane, KS * steps, smax, j);
            if (lane == j) exact = e;
        }
    }
    if (wpr > 1) {
        red_e[w * 32 + lane] = exact;
        __syncthreads();
        if (single) return __ffs(mask) - 1;
        exact = 0.0;
        for (int c = 0; c < wpr; ++c) exact += red_e[(row_in_block * wpr + c) * 32 + lane];
    }
    int bj = lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double oe = __shfl_xor_sync(0xffffffffu, exact, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        const bool take = (oe < exact) || (oe == exact && oj < bj);
        exact = take ? oe : exact;
        bj = take ? oj : bj;
    }
    bj = __shfl_sync(0xffffffffu, bj, 0);
    return bj < ncand ? bj : 0;  // only when every distance is NaN or infinite (non-finite input)
}

// Where a warp stands inside a unit of a job.  A "unit" is what one block does at a time: `warps >> wpr_log2` rows of one job.
struct UnitPos {
    long long row;
    int first, steps, elems;  // first column of the warp, its steps of 256 columns, its columns inside the row (0 when the row does not exist)
    int chunk, row_in_block;
    bool row_ok;
};

__device__ __forceinline__ UnitPos unit_pos(const PackJobDev& job, unsigned unit, int w, int warps) {
    UnitPos u;
    const int wpr = 1 << job.wpr_log2;
    u.row_in_block = w >> job.wpr_log2;
    u.chunk = w & (wpr - 1);
    u.row = (long long)(unit - job.unit_begin) * (warps >> job.wpr_log2) + u.row_in_block;
    u.row_ok = u.row < job.out;
    u.steps = (((job.in + 255) >> 8) + wpr - 1) >> job.wpr_log2;  // at most 4
    u.first = u.chunk * u.steps * 256;
    u.elems = u.row_ok ? max(0, min(u.steps * 256, job.in - u.first)) : 0;
    return u;
}

// The job whose units contain `unit` (tables ascend in unit_begin) and its number in the table.
__device__ __forceinline__ PackJobDev find_job(const PackJobDev* __restrict__ jobs, int njobs, const PackJobInline& inl,
                                               unsigned unit, int& index) {
    PackJobDev job;
    if (jobs) {
        int lo = 0, hi = njobs - 1;  // last job whose unit_begin <= unit
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (jobs[mid].unit_begin <= unit) lo = mid; else hi = mid - 1;
        }
        job = jobs[lo];
        index = lo;
    } else {
        // table in the kernel's parameters (a single matrix is a table of one)
        int lo = 0;
#pragma unroll
        for (int i = 1; i < kInlineJobs; ++i)
            if (i < njobs && inl.j[i].unit_begin <= unit) lo = i;
        job = inl.j[0];
#pragma unroll
        for (int i = 1; i < kInlineJobs; ++i)
            if (lo == i) job = inl.j[i];
        index = lo;
    }
    return job;
}

// Units of a job in a launch whose blocks have `warps` warps.
__device__ __forceinline__ unsigned units_of(const PackJobDev& job, int warps) {
    const int rpb = warps >> job.wpr_log2;
    return (unsigned)((job.out + rpb - 1) / rpb);
}

// Maximum magnitude of the row that this warp works on, from the lanes' shares `v` (zeros outside the row).  `bad`: the warp's part
// holds a value that is not finite; the maximum of such a row leaves its NaNs out.  `red`: one slot per warp of the
// block.  Every warp of the block calls it (block-wide barrier when a row spans warps).
__device__ __forceinline__ float row_max(const float* v, int lane, int w, int wpr, int row_in_block, float* red,
                                         uint32_t* status, bool& bad) {
    float amax = 0.0f;
#pragma unroll
    for (int i = 0; i < 16; ++i) amax = ptx::max_abs_nan(v[2 * i], v[2 * i + 1], amax);
    bad = __any_sync(0xffffffffu, !(amax <= 3.402823466e+38f));
    if (bad) {
        if (lane == 0 && status) atomicOr(status, NM_STATUS_NONFINITE);
        amax = 0.0f;
#pragma unroll
        for (int i = 0; i < 32; ++i) amax = fmaxf(amax, fabsf(v[i]));
    }
    amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));
    if (wpr > 1) {
        if (lane == 0) red[w] = amax;
        __syncthreads();
        for (int c = 0; c < wpr; ++c) amax = fmaxf(amax, red[row_in_block * wpr + c]);
    }
    return amax;
}

// The code of x at the scale s as a float, 1.5 * 2^23 + OFFSET + code, from the IEEE quotient (Eq. 5: rounded half to even, clamped).
template <int BITS, int OFFSET>
__device__ __noinline__ float code_exact(float x, float s) {
    constexpr float kLo = -(float)(1 << (BITS - 1)) - 0.49f, kHi = (float)((1 << (BITS - 1)) - 1) + 0.49f;
    return __fadd_rn(fminf(fmaxf(__fdiv_rn(x, s), kLo), kHi), 12582912.0f + (float)OFFSET);
}

template <int BYTES>
__device__ __forceinline__ void store_lane(uint8_t* dst, const unsigned* w) {
    if constexpr (BYTES == 1) *dst = (uint8_t)w[0];
    else if constexpr (BYTES == 2) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)w[0];
    else if constexpr (BYTES == 4) *reinterpret_cast<uint32_t*>(dst) = w[0];
    else { static_assert(BYTES == 8, "lane share"); *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]); }
}

// Everything after the row maximum (row_max): `v` holds the lane's share of V = W + U (eight values per step, zeros outside the row).
//
// N == M: dense (quantise only, no metadata), processed in groups of 4.
// DENSE_OUT: the ADMM step / STE forward form.  Besides (or instead of: values, meta and scales may then be
// null) the packed outputs the kernel writes Z = s * code as dense fp32, zero where pruned, and, when
// U_next is not null, the dual update U_next = (W + U) - Z, both as coalesced as the loads.
// CLIP: the scale may be smaller than the row's maximum asks for (a searched scale), so codes are clamped; a scale from the
// row's or its group's maximum leaves nothing to clamp.
//
// Codes: t = fma(v, RN(1 / s), 1.5 * 2^23) rounds the product to the nearest-even integer, r = t - 1.5 * 2^23 is that
// integer, and f = fma(v, RN(1 / s), -r) its distance.  The product is within 2^-16 of the IEEE quotient over the code range,
// so the code is the quotient's unless |f| is within 2^-15 of a half (6 values in 100000), which is looked at
// once per step; those lanes, and rows with a scale outside the range where RN(1 / s) is a normal number or with a
// non-finite value, take the division.
template <int N, int M, int BITS, bool DENSE_OUT, bool CLIP>
__device__ __forceinline__ void pack_row(const PackJobDev& job, const UnitPos& up, int lane, const float* v, float s, bool bad,
                                         const uint16_t* pos48, float* scratch, float* __restrict__ Zout,
                                         float* __restrict__ Unext, bool wide) {
    constexpr bool kDense = (N == M);
    constexpr int G = 8 / M;                           // groups per lane and step
    constexpr int F = (M == 4) ? 2 : 4;                // metadata field width
    constexpr int KS = G * N;                          // kept values per lane and step
    constexpr int VBITS = KS * BITS;                   // value bits per lane and step (4 .. 64)
    constexpr int VWORDS = (VBITS + 31) / 32;
    constexpr int MBITS = kDense ? 0 : KS * F;         // metadata bits per lane and step (0, 4, 8, 16)
    constexpr int kOffset = BITS == 4 ? 8 : 0;         // 4-bit codes are collected as unsigned nibbles code + 8
    constexpr float kMagic = 12582912.0f + (float)kOffset;
    constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
    const long long row = up.row;
    const float rs = __frcp_rn(s);  // correctly rounded reciprocal, once per row
    const bool fast_ok = !bad && (s >= 1.17549435e-38f) && (s <= 4.25e37f);  // rs is a normal number

    const unsigned mrow_bytes = job.mrow_words * 4u;
    uint8_t* const vrow = (!DENSE_OUT || job.values) ? job.values + (size_t)row * job.vrow_bytes : nullptr;
    uint8_t* const mrow = kDense || (DENSE_OUT && !job.meta) ? nullptr : reinterpret_cast<uint8_t*>(job.meta + (size_t)row * job.mrow_words);
    constexpr int VB = VBITS >= 8 ? VBITS / 8 : 1;     // bytes of a lane's (or pair of lanes') codes
    const bool vec_ok = VB == 1 || (job.vrow_bytes % VB == 0);  // the values start on a 16-byte boundary

#pragma unroll
    for (int st = 0; st < 4; ++st) {
        if (st >= up.steps) break;
        const int col = up.first + st * 256 + lane * 8;             // first column of this lane
        const int nvals = max(0, min(8, job.in - col));             // columns inside the row: 0, 4 or 8
        const float* x8 = v + st * 8;
        float sel[KS];
        unsigned mbits = 0;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float* x = x8 + g * M;
            float* k = sel + g * N;
            if constexpr (kDense) {
#pragma unroll
                for (int p = 0; p < M; ++p) k[p] = x[p];
            } else if constexpr (N == 2 && M == 4) {
                mbits |= select_2_of_4(x, k) << (4 * g);
            } else if constexpr (N == 4) {
                // four of eight: the keep mask indexes a table whose entry is the four positions, i.e. the group's
                // metadata; the kept values are fetched by position from a column of shared memory of this lane
                float a[M];
#pragma unroll
                for (int p = 0; p < M; ++p) { a[p] = fabsf(x[p]); scratch[p * 32 + lane] = x[p]; }
                mbits = pos48[keep_mask<N, M>(a)];
#pragma unroll
                for (int c = 0; c < 4; ++c) k[c] = scratch[((mbits >> (4 * c)) & 7u) * 32 + lane];
            } else {
                unsigned selp[N];
                select_passes<N, M>(x, k, selp);
#pragma unroll
                for (int c = 0; c < N; ++c) mbits |= selp[c] << ((g * N + c) * F);
            }
        }
        float t[KS], worst = 0.0f;
#pragma unroll
        for (int c = 0; c < KS; ++c) {
            t[c] = __fmaf_rn(sel[c], rs, kMagic);
            worst = fmaxf(worst, fabsf(__fmaf_rn(sel[c], rs, -__fsub_rn(t[c], kMagic))));
            if (CLIP) t[c] = fminf(fmaxf(t[c], kMagic - qmax - 1.0f), kMagic + qmax);
        }
        if (!(worst <= 0.49996948f) || !fast_ok) {
#pragma unroll
            for (int c = 0; c < KS; ++c) t[c] = code_exact<BITS, kOffset>(sel[c], s);
        }
        if (nvals == 0) {  // past the end of the row: zeros in the metadata's padding
#pragma unroll
            for (int c = 0; c < KS; ++c) t[c] = kMagic;
            mbits = 0;
        } else if (M == 4 && nvals == 4) {
            mbits &= (1u << (MBITS / 2)) - 1u;
        }

        // ---- dense outputs (ADMM step) -----------------------------------------------------------
        if constexpr (DENSE_OUT) {
            float z[8];
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int p = 0; p < M; ++p) {
                    if constexpr (kDense) {
                        z[g * M + p] = __fmul_rn(s, __fsub_rn(t[g * M + p], kMagic));
                    } else {
                        float zp = 0.0f;
#pragma unroll
                        for (int c = 0; c < N; ++c) {
                            const unsigned pos = (mbits >> ((g * N + c) * F)) & (unsigned)(M - 1);
                            zp = pos == (unsigned)p ? __fmul_rn(s, __fsub_rn(t[g * N + c], kMagic)) : zp;
                        }
                        z[g * M + p] = zp;
                    }
                }
            float* zp = Zout + (size_t)row * job.in + col;
            if (wide) {
                if (nvals == 8) st8(zp, z);
            } else {
                if (nvals >= 4) st4(zp, z);
                if (nvals == 8) st4(zp + 4, z + 4);
            }
            if (Unext) {
                float* np = Unext + (size_t)row * job.in + col;
                float u[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) u[i] = __fsub_rn(x8[i], z[i]);  // (W + U) - Z
                if (wide) {
                    if (nvals == 8) st8(np, u);
                } else {
                    if (nvals >= 4) st4(np, u);
                    if (nvals == 8) st4(np + 4, u + 4);
                }
            }
        }

        // ---- packed outputs ------------------------------------------------------------------------
        const int unit8 = col >> 3;  // number of the lane's eight columns in the row
        if (vrow) {
            unsigned vw[VWORDS];
            if constexpr (BITS == 8) {
                auto b = [&](int c) { return __float_as_uint(t[c < KS ? c : 0]); };
#pragma unroll
                for (int i = 0; i < VWORDS; ++i)  // the low bytes of up to four codes
                    vw[i] = __byte_perm(__byte_perm(b(4 * i), b(4 * i + 1), 0x0040), __byte_perm(b(4 * i + 2), b(4 * i + 3), 0x0040), 0x5410);
            } else {
                // sum of (0x4B400000 + nibble) << 4 c, less the sum of the constants, modulo 2^32
                unsigned acc = 0, base = 0, flip = 0;
#pragma unroll
                for (int c = 0; c < KS; ++c) {
                    acc += __float_as_uint(t[c]) << (4 * c);
                    base += 0x4B400000u << (4 * c);
                    flip |= 8u << (4 * c);
                }
                vw[0] = (acc - base) ^ flip;  // code + 8 to two's complement
            }
            if constexpr (VBITS == 4) {  // two lanes share a byte
                const unsigned other = __shfl_down_sync(0xffffffffu, vw[0], 1);
                if ((lane & 1) == 0 && nvals > 0) vrow[unit8 >> 1] = (uint8_t)(vw[0] | (other << 4));
            } else {
                uint8_t* dst = vrow + (size_t)unit8 * (VBITS / 8);
                if (nvals == 8 && vec_ok) store_lane<VB>(dst, vw);
                else {
                    const int nb = nvals * VBITS / 64;
#pragma unroll
                    for (int i = 0; i < VB; ++i)
                        if (i < nb) dst[i] = (uint8_t)(vw[i >> 2] >> ((i & 3) * 8));
                }
            }
        }
        if constexpr (!kDense) {
            if (mrow) {
                if constexpr (MBITS == 4) {
                    const unsigned other = __shfl_down_sync(0xffffffffu, mbits, 1);
                    if ((lane & 1) == 0 && (unsigned)(unit8 >> 1) < mrow_bytes) mrow[unit8 >> 1] = (uint8_t)(mbits | (other << 4));
                } else {
                    constexpr int MB = MBITS / 8;
                    if ((unsigned)unit8 * MB < mrow_bytes) store_lane<MB>(mrow + (size_t)unit8 * MB, &mbits);
                }
            }
        }
    }
}

// From the loaded row to its outputs.  `red`: this unit's slots for row_max.  Every warp of the block calls it.
template <int N, int M, int BITS, bool DENSE_OUT, bool DIST = false>
__device__ __forceinline__ void pack_finish(const PackJobDev& job, const UnitPos& up, int lane, int w, const float* v,
                                            float* red, const uint16_t* pos48, float* scratch, uint32_t* status,
                                            float* __restrict__ Zout, float* __restrict__ Unext, bool wide, int group_mode, int group_rows,
                                            double* red_e = nullptr, DistBins* bins = nullptr, float* kept = nullptr) {
    const int wpr = 1 << job.wpr_log2;
    bool bad;
    const float amax = row_max(v, lane, w, wpr, up.row_in_block, red, status, bad);

    // ---- group-wise scales, first pass: fold this row's maximum into the first entry of its group -----
    if (group_mode == kGroupMaxPass) {
        if (up.row_ok && up.chunk == 0 && lane == 0) {
            const int G = (group_rows <= 0 || group_rows > job.out) ? job.out : group_rows;
            atomicMax(reinterpret_cast<unsigned*>(job.scales) + (size_t)(up.row / G) * G, __float_as_uint(amax));
        }
        return;
    }

    // ---- ADMM-Max scale ---------------------------------------------------------------------
    constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
    float s;
    if (!DIST && group_mode == kGroupScalesGiven) {
        // one scale per row, equal within a group of rows, or searched before (rows of more than 4096 weights)
        if (!up.row_ok) return;
        s = job.scales[up.row];
        pack_row<N, M, BITS, DENSE_OUT, true>(job, up, lane, v, s, bad, pos48, scratch, Zout, Unext, wide);
        return;
    }
    s = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
    if constexpr (DIST) {  // group_rows carries the number of candidate scales
        const int best = dist_search<N, M, BITS, false>(v, up.steps, lane, w, wpr, up.row_in_block, up.row_ok, s, bad, group_rows, red_e, bins, kept);
        s = __fmul_rn(s, (float)(64 - best) * 0.015625f);
    }
    if (!up.row_ok) return;
    if (up.chunk == 0 && lane == 0 && (!DENSE_OUT || job.scales)) job.scales[up.row] = s;
    pack_row<N, M, BITS, DENSE_OUT, DIST>(job, up, lane, v, s, bad, pos48, scratch, Zout, Unext, wide);
}

// Loads the lane's share of V = W + U straight from global memory.  `wide`: 32-byte accesses are aligned and rows end on them.
__device__ __forceinline__ void load_global(const PackJobDev& job, const UnitPos& up, int lane, bool wide, float* v) {
    const size_t at = (size_t)(up.row_ok ? up.row : 0) * job.in + up.first + lane * 8;
    const float* W = job.W + at;
    const float* U = job.U ? job.U + at : nullptr;
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = 0.0f;
    const int mine = up.elems - lane * 8;  // columns from this lane's first one to the end of the warp's part
    if (wide) {
#pragma unroll
        for (int st = 0; st < 4; ++st)
            if (st * 256 < mine) ld8(W + st * 256, v + st * 8);
        if (U) {
#pragma unroll
            for (int st = 0; st < 4; ++st)
                if (st * 256 < mine) {
                    float u[8];
                    ld8(U + st * 256, u);
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[st * 8 + i] = __fadd_rn(v[st * 8 + i], u[i]);
                }
        }
    } else {
#pragma unroll
        for (int h = 0; h < 8; ++h)
            if ((h >> 1) * 256 + (h & 1) * 4 < mine) ld4(W + (h >> 1) * 256 + (h & 1) * 4, v + h * 4);
        if (U) {
#pragma unroll
            for (int h = 0; h < 8; ++h)
                if ((h >> 1) * 256 + (h & 1) * 4 < mine) {
                    float u[4];
                    ld4(U + (h >> 1) * 256 + (h & 1) * 4, u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[h * 4 + i] = __fadd_rn(v[h * 4 + i], u[i]);
                }
        }
    }
}

// The same from the part of the row that the bulk copies left in shared memory (`wbuf`, `ubuf`: up to 1024 floats each).
// Every other group of four lanes reads its two 16-byte halves in the other order, so that no two lanes of a
// quarter warp meet in a bank.
__device__ __forceinline__ void load_staged(const PackJobDev& job, const UnitPos& up, int lane, const float* wbuf,
                                            const float* ubuf, float* v) {
    const bool swap = lane & 4;
    const int a = lane * 8 + (swap ? 4 : 0), b = lane * 8 + (swap ? 0 : 4);
#pragma unroll
    for (int st = 0; st < 4; ++st) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (st * 256 + a < up.elems) x = *reinterpret_cast<const float4*>(wbuf + st * 256 + a);
        if (st * 256 + b < up.elems) y = *reinterpret_cast<const float4*>(wbuf + st * 256 + b);
        if (job.U) {
            if (st * 256 + a < up.elems) {
                const float4 u = *reinterpret_cast<const float4*>(ubuf + st * 256 + a);
                x.x = __fadd_rn(x.x, u.x); x.y = __fadd_rn(x.y, u.y); x.z = __fadd_rn(x.z, u.z); x.w = __fadd_rn(x.w, u.w);
            }
            if (st * 256 + b < up.elems) {
                const float4 u = *reinterpret_cast<const float4*>(ubuf + st * 256 + b);
                y.x = __fadd_rn(y.x, u.x); y.y = __fadd_rn(y.y, u.y); y.z = __fadd_rn(y.z, u.z); y.w = __fadd_rn(y.w, u.w);
            }
        }
        float* o = v + st * 8;
        o[0] = swap ? y.x : x.x; o[1] = swap ? y.y : x.y; o[2] = swap ? y.z : x.z; o[3] = swap ? y.w : x.w;
        o[4] = swap ? x.x : y.x; o[5] = swap ? x.y : y.y; o[6] = swap ? x.z : y.z; o[7] = swap ? x.w : y.w;
    }
}

// Whether the rows of a job can be moved in 32-byte accesses.
__device__ __forceinline__ bool wide_rows(const PackJobDev& job, const float* Z, const float* U_next) {
    return (((uintptr_t)job.W | (uintptr_t)job.U | (uintptr_t)Z | (uintptr_t)U_next) & 31u) == 0 && (job.in & 7) == 0;
}

// Four of eight: table from the 8-bit keep mask to its four positions (4-bit fields, ascending), which is also the group's
// metadata.
__device__ __forceinline__ void fill_positions(uint16_t* pos48) {
    for (unsigned mk = threadIdx.x; mk < 256; mk += blockDim.x) {
        unsigned r = 0, c = 0;
#pragma unroll
        for (unsigned p8 = 0; p8 < 8; ++p8)
            if ((mk >> p8) & 1u) { r |= p8 << (4 * (c & 3u)); ++c; }
        pos48[mk] = (uint16_t)r;
    }
}

// Forms of the kernel.  kDirect: one block = one unit, global loads.  kStaged2: persistent, two buffers of up to 1024 values
// of W and U per warp (16 KB); every warp fetches its part of its NEXT unit with two bulk copies into the other buffer
// while it works on the current one, so that loading and arithmetic overlap inside a warp and not only between
// blocks that happen to be out of step.
enum { kDirect = 0, kStaged2 = 1 };
constexpr int kStagedBlocksPerSm = 3;
// Resident blocks of four warps that the registers are cut for (kDirect).  Eight (64 registers) for the plain projection: with five
// or six, more of a warp's loads are in flight, but 85 M weights in four formats take 125 / 116 us instead of 104, the
// 24-layer sweep 436 / 441 instead of 403.  Dense outputs six (738 us; five and four the same).  The search four, and
// six where a lane keeps at most eight values or the codes have 4 bits.
template <int N, int M, int BITS, bool DENSE_OUT, bool DIST>
constexpr int kDirectBlocksPerSm = DIST ? (32 / M * N <= 8 || BITS == 4 ? 6 : 4) : DENSE_OUT ? 6 : 8;

constexpr int kFewBlocksPerSm = 5;  // the plain projection of two operands where no SM gets more blocks (see pick_bits)

template <int N, int M, int BITS, int MAXT, bool DENSE_OUT = false, int PIPE = kDirect, bool DIST = false,
          int PER_SM = kDirectBlocksPerSm<N, M, BITS, DENSE_OUT, DIST>>
__global__ void __launch_bounds__(MAXT, PIPE != kDirect ? kStagedBlocksPerSm : (MAXT == 128 ? PER_SM : 1))
pack_kernel(const PackJobDev* __restrict__ jobs, int njobs, const __grid_constant__ PackJobInline inl, uint32_t* status,
            float* __restrict__ Zout, float* __restrict__ Unext, const DenseOutDev* __restrict__ dense_jobs,
            int group_mode, int group_rows, unsigned nunits, bool chained) {
    static_assert(PIPE == kDirect || (MAXT == 128 && N <= 2 && !DENSE_OUT && !DIST), "see staged_form");
    // staged: [warps][2 buffers][W, U][1024] floats.  Then (DIST) [warps][32] doubles, (4 bits) [warps] DistBins, [warps][kept values][32], [2][warps] floats for the row maximum, (4:8) the
    // position table and [warps][8][32] floats, (staged) [warps][2] mbarriers and the abort flag.
    extern __shared__ float4 tile[];
    const int warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint8_t* at = reinterpret_cast<uint8_t*>(tile) + (PIPE == kStaged2 ? warps * 16384 : 0);
    double* red_e = reinterpret_cast<double*>(at);
    if (DIST) at += warps * 256;
    DistBins* bins = reinterpret_cast<DistBins*>(at);
    if (DIST && BITS == 4) at += warps * sizeof(DistBins);
    float* kept = reinterpret_cast<float*>(at) + w * (32 * (32 / M * N));
    if (DIST) at += warps * kKeptBytes<N, M>;
    float* red = reinterpret_cast<float*>(at);
    at += warps * 8;
    uint16_t* pos48 = nullptr;
    float* scratch = nullptr;
    // a kernel launched as this one's programmatic dependent may begin its set-up on SMs this grid has left
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (N == 4 && M == 8) {
        pos48 = reinterpret_cast<uint16_t*>(at);
        at += 512;
        scratch = reinterpret_cast<float*>(at) + w * 256;
        at += warps * 1024;
        fill_positions(pos48);
        __syncthreads();
    }

    if constexpr (PIPE == kDirect) {
        int index = 0;
        const PackJobDev job = find_job(jobs, njobs, inl, blockIdx.x, index);
        if constexpr (DENSE_OUT) {
            if (jobs) { Zout = dense_jobs[index].Z; Unext = dense_jobs[index].U_next; }
        }
        const UnitPos up = unit_pos(job, blockIdx.x, w, warps);
        const bool wide = wide_rows(job, Zout, Unext);
        float v[32];
        load_global(job, up, lane, wide, v);
        pack_finish<N, M, BITS, DENSE_OUT, DIST>(job, up, lane, w, v, red, pos48, scratch, status, Zout, Unext, wide, group_mode,
                                                group_rows, red_e, bins, kept);
    } else {
        uint64_t* bars = reinterpret_cast<uint64_t*>(at);                 // [warps][2]
        volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bars + 2 * warps);
        float* mybuf = reinterpret_cast<float*>(tile) + w * 4096;         // [buffer][W, U][1024]
        const uint32_t bar0 = ptx::smem_u32(bars + 2 * w);
        if (lane == 0) {
            ptx::mbar_init(bar0, 1);
            ptx::mbar_init(bar0 + 8, 1);
            if (threadIdx.x == 0) *abort_flag = 0;
            ptx::fence_mbar_init();
        }
        __syncthreads();
        // every lane calls it; lane 0 issues one bulk copy per operand, completion counted in bytes on the buffer's barrier
        auto issue = [&](const PackJobDev& j, const UnitPos& up, int buf, int iter) {
            if (up.elems == 0) return;      // the same for the whole warp; the unit then waits for nothing
            if (NM_PACK_SKIP(iter)) return;
            ptx::fence_proxy_async_smem();  // this lane's generic accesses to the buffer before the copy's writes
            __syncwarp();                   // the buffer's last reader is done
            if (lane == 0) {
                const uint32_t bytes = (uint32_t)up.elems * 4u, bar = bar0 + 8u * buf;
                const size_t first = (size_t)up.row * j.in + up.first;
                ptx::mbar_expect_tx(bar, j.U ? 2 * bytes : bytes);
                ptx::bulk_load(ptx::smem_u32(mybuf + buf * 2048), j.W + first, bytes, bar);
                if (j.U) ptx::bulk_load(ptx::smem_u32(mybuf + buf * 2048 + 1024), j.U + first, bytes, bar);
            }
        };
        int index = 0;
        unsigned unit = blockIdx.x;
        PackJobDev job{};
        UnitPos up{};
        if (unit < nunits) {
            job = find_job(jobs, njobs, inl, unit, index);
            up = unit_pos(job, unit, w, warps);
            issue(job, up, 0, 0);
        }
        uint32_t phase = 0;  // bit b: parity of buffer b's next completion
        // The slots of the row maximum alternate over the units whose rows span warps: only those pass the block's barrier, so
        // the one before the last has been read by every warp when its slots are written again.  (Alternating over all units
        // would reuse them after an odd number of one-warp units, which no barrier separates.)
        unsigned spanning = 0;
        for (int it = 0; unit < nunits; ++it, unit += gridDim.x) {
            const int buf = it & 1;
            // the next unit's part goes into the other buffer while this one is worked on
            const unsigned next = unit + gridDim.x;
            PackJobDev njob = job;
            UnitPos nup{};
            if (next < nunits) {
                if (next - job.unit_begin >= units_of(job, warps)) njob = find_job(jobs, njobs, inl, next, index);
                nup = unit_pos(njob, next, w, warps);
                issue(njob, nup, buf ^ 1, it + 1);
            }
            if (up.elems != 0) {
                if (!ptx::mbar_wait_bounded(bar0 + 8u * buf, (phase >> buf) & 1u, abort_flag, kPackWaitLimit)) {
                    // recorded; the unit is then worked on with whatever the buffer holds (in bounds, results void)
                    *abort_flag = 1u;
                    if (status) atomicOr(status, NM_STATUS_TIMEOUT);
                }
                phase ^= 1u << buf;
            }
            float v[32];
            load_staged(job, up, lane, mybuf + buf * 2048, mybuf + buf * 2048 + 1024, v);
            pack_finish<N, M, BITS, DENSE_OUT>(job, up, lane, w, v, red + (spanning & 1u) * warps, pos48, scratch, status, Zout, Unext,
                                              wide_rows(job, Zout, Unext), group_mode, group_rows);
            spanning += job.wpr_log2 != 0 ? 1u : 0u;
            job = njob; up = nup;
        }
        // after an expired wait a copy may still be on its way into this block's shared memory
        if (*abort_flag) ptx::wait_clocks(1 << 17);
    }
    // Launched as the programmatic dependent of another launch of the same call (see launch_batched): the two work on
    // different matrices, so only the end is ordered, for whatever follows in the stream.
    if (chained) ptx::grid_dep_wait();
}

// ---------------------------------------------------------------------------------------------
// Group-wise scales in one pass: a cluster of blocks holds a whole group of rows in registers, the blocks exchange their
// maxima through distributed shared memory, and every warp goes on with its row at the group's scale.  W and U are read
// once; folding the maxima of all groups first and packing in a second launch read them twice (75 M weights, 2:4 / 4 bit, groups of 32
// rows: 232 us, 154 so).  What bounds it: a cluster loads, meets
// at its barrier and packs in turn, with two to four blocks an SM to overlap that (DRAM at 45 %).
// A unit is one group (`group_rows` rows, those past the matrix idle); it fills gridDim / units blocks, the cluster.
// ---------------------------------------------------------------------------------------------
template <int N, int M, int BITS, bool DENSE_OUT>
__global__ void __launch_bounds__(512, DENSE_OUT ? 1 : 2)
pack_group_kernel(const PackJobDev* __restrict__ jobs, int njobs, const __grid_constant__ PackJobInline inl, uint32_t* status,
                  float* __restrict__ Zout, float* __restrict__ Unext, const DenseOutDev* __restrict__ dense_jobs,
                  int group_rows, unsigned cluster, bool chained) {
    // [warps] maxima, [8] maxima of the cluster's blocks, (4:8) position table and [warps][8][32] floats
    extern __shared__ float4 tile[];
    const int warps = blockDim.x >> 5, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float* red = reinterpret_cast<float*>(tile);
    uint32_t* peers = reinterpret_cast<uint32_t*>(red + 16);
    uint16_t* pos48 = reinterpret_cast<uint16_t*>(peers + 8);
    float* scratch = reinterpret_cast<float*>(pos48 + 256) + w * 256;
    ptx::cluster_arrive();  // the other blocks' shared memory may be written once all of them run
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (N == 4 && M == 8) fill_positions(pos48);  // ordered by the barrier below
    const unsigned unit = blockIdx.x / cluster, rank = blockIdx.x % cluster;
    int index = 0;
    const PackJobDev job = find_job(jobs, njobs, inl, unit, index);
    if constexpr (DENSE_OUT) {
        if (jobs) { Zout = dense_jobs[index].Z; Unext = dense_jobs[index].U_next; }
    }
    const int wpr = 1 << job.wpr_log2, gw = (int)rank * warps + w;  // warp of the group
    UnitPos up;
    up.chunk = gw & (wpr - 1);
    up.row_in_block = w >> job.wpr_log2;
    up.row = (long long)(unit - job.unit_begin) * group_rows + (gw >> job.wpr_log2);
    up.row_ok = up.row < job.out;
    up.steps = (((job.in + 255) >> 8) + wpr - 1) >> job.wpr_log2;
    up.first = up.chunk * up.steps * 256;
    up.elems = up.row_ok ? max(0, min(up.steps * 256, job.in - up.first)) : 0;
    const bool wide = wide_rows(job, Zout, Unext);
    float v[32];
    load_global(job, up, lane, wide, v);
    bool bad;
    float amax = row_max(v, lane, w, 1, 0, red, status, bad);  // of this warp's part
    if (lane == 0) red[w] = amax;
    __syncthreads();
    ptx::cluster_wait();
    if (w == 0) {
        amax = lane < warps ? red[lane] : 0.0f;
        const uint32_t block_max = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
        if (lane < (int)cluster) ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(peers + rank), (uint32_t)lane), block_max);
    }
    __syncwarp();
    ptx::cluster_arrive();
    ptx::cluster_wait();
    amax = 0.0f;
    for (unsigned c = 0; c < cluster; ++c) amax = fmaxf(amax, __uint_as_float(peers[c]));
    if (up.row_ok) {
        constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
        const float s = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
        if (up.chunk == 0 && lane == 0) job.scales[up.row] = s;
        pack_row<N, M, BITS, DENSE_OUT, false>(job, up, lane, v, s, bad, pos48, scratch, Zout, Unext, wide);
    }
    if (chained) ptx::grid_dep_wait();  // as in pack_kernel
}

// ---------------------------------------------------------------------------------------------
// Group-wise scales: rows r with the same r / group_rows share one ADMM-Max scale.  A first pass folds
// max |W + U| of every row into the first entry of its group in `scales` (non-negative floats order like
// their bit patterns, so an unsigned atomicMax does it); a second turns each group's maximum into the
// scale and writes it to all rows of the group (one thread per group: reads before it writes).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) group_absmax_kernel(const float* __restrict__ W, const float* __restrict__ U,
                                                           int out, int in, int group_rows, float* scales) {
    const int row = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= out) return;
    const int in4 = in >> 2;
    const float4* W4 = reinterpret_cast<const float4*>(W) + (size_t)row * in4;
    const float4* U4 = U ? reinterpret_cast<const float4*>(U) + (size_t)row * in4 : nullptr;
    float a = 0.0f;
    for (int f = lane; f < in4; f += 32) {
        float4 v = __ldg(W4 + f);  // read again by the projection pass: keep it cached
        if (U4) {
            const float4 u = __ldg(U4 + f);
            v.x = __fadd_rn(v.x, u.x); v.y = __fadd_rn(v.y, u.y); v.z = __fadd_rn(v.z, u.z); v.w = __fadd_rn(v.w, u.w);
        }
        a = fmaxf(a, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
    if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(scales) + (size_t)(row / group_rows) * group_rows, __float_as_uint(a));
}

__global__ void __launch_bounds__(128) group_scale_kernel(int out, int group_rows, int bits, float* scales) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long first = g * group_rows;
    if (first >= out) return;
    const float a = scales[first];
    const float qmax = (float)((1 << (bits - 1)) - 1);
    const float s = (a == 0.0f) ? 1.0f : __fdiv_rn(a, qmax);
    const long long last = min((long long)out, first + group_rows);
    for (long long r = first; r < last; ++r) scales[r] = s;
}

// Batched form over a job table: block j serves job j.  phase 0 clears the scales (the maxima are folded
// in by the pack kernel's kGroupMaxPass), phase 1 turns each group's maximum into the scale of its rows.
__global__ void __launch_bounds__(256) group_prepare_kernel(const PackJobDev* __restrict__ jobs, int group_rows,
                                                            int bits, int phase) {
    const PackJobDev job = jobs[blockIdx.x];
    if (phase == 0) {
        for (int r = threadIdx.x; r < job.out; r += blockDim.x) job.scales[r] = 0.0f;
        return;
    }
    const int G = (group_rows <= 0 || group_rows > job.out) ? job.out : group_rows;
    const float qmax = (float)((1 << (bits - 1)) - 1);
    for (long long first = (long long)threadIdx.x * G; first < job.out; first += (long long)blockDim.x * G) {
        const float a = job.scales[first];
        const float s = (a == 0.0f) ? 1.0f : __fdiv_rn(a, qmax);
        const long long last = min((long long)job.out, first + G);
        for (long long r = first; r < last; ++r) job.scales[r] = s;
    }
}

static int launch_group_scales(const float* W, const float* U, int out, int in, int bits, int group_rows,
                               float* scales, cudaStream_t stream) {
    const int G = group_rows <= 0 ? out : (group_rows > out ? out : group_rows);
    NM_CUDA_TRY(cudaMemsetAsync(scales, 0, (size_t)out * sizeof(float), stream));
    group_absmax_kernel<<<(out + 3) / 4, 128, 0, stream>>>(W, U, out, in, G, scales);
    NM_CUDA_TRY(cudaGetLastError());
    const int ngroups = (out + G - 1) / G;
    group_scale_kernel<<<(ngroups + 127) / 128, 128, 0, stream>>>(out, G, bits, scales);
    NM_CUDA_TRY(cudaGetLastError());
    return NM_OK;
}

// The search alone (nm_dist_scales), and in front of the projection for rows of more than 4096 weights, whose blocks have too
// few registers per thread for both: writes the winning scale to `scales`.
template <int N, int M, int BITS, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 128 ? 4 : 1) dist_scale_kernel(const PackJobDev* __restrict__ jobs, int njobs,
                                                                              const __grid_constant__ PackJobInline inl,
                                                                              uint32_t* status, int ncand,
                                                                              int32_t* __restrict__ cand_out) {
    extern __shared__ float4 tile[];  // [warps][32] doubles, (4 bits) [warps] DistBins, [warps][kept values][32], [warps] floats
    const int warps = blockDim.x >> 5;
    double* red_e = reinterpret_cast<double*>(tile);
    DistBins* bins = reinterpret_cast<DistBins*>(red_e + warps * 32);
    constexpr bool kAlias = BITS == 4 && MAXT > 128;  // up to 32 warps: room for only one of the two
    float* kept = kAlias ? reinterpret_cast<float*>(bins + (threadIdx.x >> 5)) : reinterpret_cast<float*>(bins + (BITS == 4 ? warps : 0)) + (threadIdx.x >> 5) * (kKeptBytes<N, M> / 4);
    float* red = kAlias ? reinterpret_cast<float*>(bins + warps) : reinterpret_cast<float*>(bins + (BITS == 4 ? warps : 0)) + warps * (kKeptBytes<N, M> / 4);
    int index = 0;
    const PackJobDev job = find_job(jobs, njobs, inl, blockIdx.x, index);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const UnitPos up = unit_pos(job, blockIdx.x, w, warps);
    const int wpr = 1 << job.wpr_log2;
    float v[32];
    load_global(job, up, lane, wide_rows(job, nullptr, nullptr), v);
    bool bad;
    const float amax = row_max(v, lane, w, wpr, up.row_in_block, red, status, bad);
    constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
    const float smax = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, qmax);
    const int bj = dist_search<N, M, BITS, kAlias>(v, up.steps, lane, w, wpr, up.row_in_block, up.row_ok, smax, bad, ncand, red_e, bins, kept);
    if (up.row_ok && up.chunk == 0 && lane == 0) {
        job.scales[up.row] = __fmul_rn(smax, (float)(64 - bj) * 0.015625f);
        if (cand_out) cand_out[up.row] = bj;
    }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
using PackFnPtr = void (*)(const PackJobDev*, int, const PackJobInline, uint32_t*, float*, float*, const DenseOutDev*, int, int, unsigned, bool);
struct PackFn { PackFnPtr fn; int form; size_t search = 0; };  // kernel, its form (kDirect, kStaged2), shared memory of the scale search per warp

// nm_debug_set_option("pack_form"): 0 = automatic, 2 = kStaged2 wherever it exists (blocks of four warps, 1:4, 2:4, 1:8 and 2:8, no
// dense outputs), anything else = kDirect.
int g_pack_form = 0;

// What the matrices of a launch have in common: some have no U; all have one; ... and rows of a multiple of 1024 weights; ... and rows of
// 1024, 2048 or 4096, which fill the staged form's buffers.
enum { kOneOperand = 0, kTwoOperands = 1, kThousands = 2, kFullBuffers = 3 };
static int operands_of(const nm_pack_job_t& j) {
    if (!j.U) return kOneOperand;
    if (j.in % 1024) return kTwoOperands;
    return (j.in & (j.in - 1)) == 0 && j.in <= 4096 ? kFullBuffers : kThousands;
}

// Whether a launch of `blocks` blocks of four warps takes the staged form: two operands, more blocks than kDirect keeps resident, which
// otherwise start together and alternate between loading and arithmetic.  Staged / direct in us, one matrix, W and U:
//   rows of 1024, 2048, 4096, whatever their number: 6.3 M weights of 1:4 / 4 bit in rows of 4096 12.5 / 14.3, 2:8 / 8 bit 14.2 / 15.9, 2:4 / 8
//   bit 13.4 / 15.2; 50 M 67 / 75, 79 / 84, 71 / 82; 50 M in rows of 1024 71 / 72, 75 / 82, 75 / 79;
//   several matrices only up to six rounds, beyond them the direct form's blocks are out of step by themselves (24 layers of BERT-large
//   457 / 414, 4 layers 92 / 86);
//   2:4 in rows of 3072 up to six rounds (17 M 30.5 / 31.6); 2:8 there and more rounds lose (17 M 33.2 / 32.1, 2:4 50 M 81 / 78).
// Up to one round the direct form is the faster one (4.2 M of 1:4 / 4 bit 10.3 / 9.8), as with one operand (25 M 37.3 / 25.2) and in rows
// of other lengths (of 384 and 1536, 11 M 37.3 / 27.4).
template <int N, int M>
static bool staged_form(int operands, unsigned blocks, int njobs) {
    const unsigned resident = (unsigned)sm_count() * 8u;
    if (operands < kThousands || blocks <= resident) return false;
    if (operands == kFullBuffers && njobs <= 1) return true;
    return blocks <= 6u * resident && (operands == kFullBuffers || (N == 2 && M == 4));
}

template <int N, int M, bool DENSE_OUT>
static PackFn pick_bits(int bits, int warps, unsigned blocks, int operands, int njobs) {
    if (warps <= kPackMinWarps) {
        if constexpr (N <= 2 && !DENSE_OUT) {
            if (g_pack_form == 2 || (g_pack_form == 0 && staged_form<N, M>(operands, blocks, njobs)))
                return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 128, false, kStaged2>, kStaged2}
                                 : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 128, false, kStaged2>, kStaged2};
        }
        // Two operands and at most kFewBlocksPerSm blocks an SM: the instance with the registers to have both operands' loads in flight
        // together (1.0 M weights of 1:4 / 4 bit in rows of 4096 5.6 -> 5.1 us, 2.1 M of 2:4 / 8 bit in rows of 3072 6.9 -> 6.4).
        if constexpr (!DENSE_OUT) {
            if (operands != kOneOperand && blocks <= (unsigned)(sm_count() * kFewBlocksPerSm))
                return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 128, false, kDirect, false, kFewBlocksPerSm>, kDirect}
                                 : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 128, false, kDirect, false, kFewBlocksPerSm>, kDirect};
        }
        return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 128, DENSE_OUT>, kDirect}
                         : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 128, DENSE_OUT>, kDirect};
    }
    if constexpr (DENSE_OUT) {  // the dense outputs need ~128 registers: blocks of at most 512 threads get them
        if (warps <= 16)
            return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 512, true>, kDirect} : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 512, true>, kDirect};
    }
    return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 1024, DENSE_OUT>, kDirect} : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 1024, DENSE_OUT>, kDirect};
}

template <bool DENSE_OUT = false>
static PackFn pick_kernel(int n, int m, int bits, int warps, unsigned blocks, int operands, int njobs = 1) {
    if (n == m) return pick_bits<4, 4, DENSE_OUT>(bits, warps, blocks, operands, njobs);
    if (m == 4) return n == 1 ? pick_bits<1, 4, DENSE_OUT>(bits, warps, blocks, operands, njobs) : pick_bits<2, 4, DENSE_OUT>(bits, warps, blocks, operands, njobs);
    if (n == 1) return pick_bits<1, 8, DENSE_OUT>(bits, warps, blocks, operands, njobs);
    if (n == 2) return pick_bits<2, 8, DENSE_OUT>(bits, warps, blocks, operands, njobs);
    return pick_bits<4, 8, DENSE_OUT>(bits, warps, blocks, operands, njobs);
}

static int validate_job(const nm_pack_job_t& j) {
    int rc = check_pattern(j.out, j.in, j.n, j.m, j.bits);
    if (rc != NM_OK) return rc;
    if (!j.W || !j.values || !j.scales) return NM_ERR_NULL;
    if (j.n != j.m && !j.meta) return NM_ERR_NULL;
    if (j.in % 4) return NM_ERR_SHAPE;
    if (j.n == j.m && j.in % 4) return NM_ERR_SHAPE;
    if (j.in > 32768) return NM_ERR_UNSUPPORTED;
    if (!aligned(j.W, 16) || (j.U && !aligned(j.U, 16)) || !aligned(j.values, 16) ||
        (j.meta && !aligned(j.meta, 4)) || !aligned(j.scales, 4))
        return NM_ERR_ALIGN;
    return NM_OK;
}

static int wpr_log2_of(int in) {
    int chunks = (in + 1023) / 1024, l = 0;
    while ((1 << l) < chunks) ++l;
    return l;
}

static PackJobDev to_dev(const nm_pack_job_t& j) {
    PackJobDev d;
    d.W = j.W; d.U = j.U; d.values = (uint8_t*)j.values; d.meta = (uint32_t*)j.meta; d.scales = j.scales;
    d.out = j.out; d.in = j.in; d.wpr_log2 = wpr_log2_of(j.in); d.unit_begin = 0;
    d.vrow_bytes = (unsigned)values_row_bytes(j.in, j.n, j.m, j.bits);
    d.mrow_words = (unsigned)meta_row_words(j.in, j.n, j.m);
    return d;
}

// jobs_dev != nullptr: table of njobs entries in device memory; else the first njobs (>= 1) entries of `inl`.
static int launch_table(PackFn k, const PackJobDev* jobs_dev, int njobs, const PackJobInline& inl, unsigned blocks,
                        int warps, uint32_t* status, cudaStream_t stream, float* Z, float* U_next,
                        const DenseOutDev* dense_jobs, int group_mode, int group_rows, bool chained = false) {
    // buffers and barriers of the staged form, distances of the search, row-maximum slots, the 4:8 tables (see the kernel)
    const bool staged = k.form == kStaged2;
    const size_t smem = (size_t)warps * ((staged ? 16384 + 16 : 0) + k.search + 2 * sizeof(float) + 1024) + 512 + 16;
    const PackFnPtr fn = k.fn;
    if (smem > 48 * 1024) NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, 227 * 1024));
    const unsigned grid = staged ? std::min(blocks, (unsigned)(sm_count() * kStagedBlocksPerSm)) : blocks;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(warps * 32, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = chained ? 1 : 0;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, jobs_dev, njobs, inl, status, Z, U_next, dense_jobs, group_mode, group_rows, blocks, chained));
    return NM_OK;
}

static int launch(PackFn fn, const PackJobDev* jobs_dev, int njobs, const PackJobDev& single,
                  unsigned blocks, int warps, uint32_t* status, cudaStream_t stream,
                  float* Z = nullptr, float* U_next = nullptr, const DenseOutDev* dense_jobs = nullptr,
                  int group_mode = kGroupNone, int group_rows = 0, bool chained = false) {
    PackJobInline inl{};
    inl.j[0] = single;
    return launch_table(fn, jobs_dev, njobs, inl, blocks, warps, status, stream, Z, U_next, dense_jobs, group_mode, group_rows, chained);
}

// Cluster of pack_group_kernel for groups of `group_rows` rows of 1 << wpr_log2 warps: blocks of four to sixteen warps, at most
// eight (the portable cluster size), rows whole in a block; blocks of at most eight warps where that is possible, so
// that several clusters share an SM.  False: no such cluster (a group of fewer than four warps or more than 128, or an awkward
// factor), the two-pass route.
static bool group_cluster(int group_rows, int wpr_log2, int* warps, int* cluster) {
    const long long gw = (long long)group_rows << wpr_log2;
    if (group_rows <= 0 || wpr_log2 > 2 || gw < 4 || gw > 128) return false;
    for (int limit = 8; limit <= 16; limit += 8)
        for (int c = 1; c <= 8; ++c) {
            const int bw = (int)gw / c;
            if (gw % c || bw > limit || bw < 4 || bw % (1 << wpr_log2)) continue;
            *warps = bw; *cluster = c;
            return true;
        }
    return false;
}

using GroupFn = void (*)(const PackJobDev*, int, const PackJobInline, uint32_t*, float*, float*, const DenseOutDev*, int, unsigned, bool);

template <bool DENSE_OUT>
static GroupFn pick_group(int n, int m, int bits) {
    const bool b8 = bits == 8;
    if (n == m) return b8 ? pack_group_kernel<4, 4, 8, DENSE_OUT> : pack_group_kernel<4, 4, 4, DENSE_OUT>;
    if (m == 4 && n == 1) return b8 ? pack_group_kernel<1, 4, 8, DENSE_OUT> : pack_group_kernel<1, 4, 4, DENSE_OUT>;
    if (m == 4) return b8 ? pack_group_kernel<2, 4, 8, DENSE_OUT> : pack_group_kernel<2, 4, 4, DENSE_OUT>;
    if (n == 1) return b8 ? pack_group_kernel<1, 8, 8, DENSE_OUT> : pack_group_kernel<1, 8, 4, DENSE_OUT>;
    if (n == 2) return b8 ? pack_group_kernel<2, 8, 8, DENSE_OUT> : pack_group_kernel<2, 8, 4, DENSE_OUT>;
    return b8 ? pack_group_kernel<4, 8, 8, DENSE_OUT> : pack_group_kernel<4, 8, 4, DENSE_OUT>;
}

// `units` groups; the jobs of a launch have the same n, m, bits and warps per row.
template <bool DENSE_OUT>
static int launch_group(int n, int m, int bits, int warps, int cluster, const PackJobDev* jobs_dev, int njobs, const PackJobDev& single,
                        unsigned units, uint32_t* status, cudaStream_t stream, float* Z, float* U_next,
                        const DenseOutDev* dense_jobs, int group_rows, bool chained = false) {
    PackJobInline inl{};
    inl.j[0] = single;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(units * (unsigned)cluster, 1, 1);
    cfg.blockDim = dim3(warps * 32, 1, 1);
    cfg.dynamicSmemBytes = 96 + (n == 4 && m == 8 ? 512 + (size_t)warps * 1024 : 0);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = chained ? 2 : 1;
    NM_CUDA_TRY(cudaLaunchKernelEx(&cfg, pick_group<DENSE_OUT>(n, m, bits), jobs_dev, njobs, inl, status, Z, U_next, dense_jobs,
                                   group_rows, (unsigned)cluster, chained));
    return NM_OK;
}

// One matrix, group-wise scales: one pass where a cluster holds a group, otherwise maxima, scales, projection.
template <bool DENSE_OUT>
static int launch_grouped_single(const nm_pack_job_t& j, int group_rows, uint32_t* status, cudaStream_t stream,
                                 float* Z = nullptr, float* U_next = nullptr) {
    PackJobDev d = to_dev(j);
    int warps = 0, cluster = 0;
    if (group_cluster(group_rows, d.wpr_log2, &warps, &cluster)) {
        const unsigned units = (unsigned)(((long long)j.out + group_rows - 1) / group_rows);
        return launch_group<DENSE_OUT>(j.n, j.m, j.bits, warps, cluster, nullptr, 0, d, units, status, stream, Z, U_next, nullptr, group_rows);
    }
    int rc = launch_group_scales(j.W, j.U, j.out, j.in, j.bits, group_rows, j.scales, stream);
    if (rc != NM_OK) return rc;
    warps = std::max(kPackMinWarps, 1 << d.wpr_log2);
    const int rows_per_block = warps >> d.wpr_log2;
    const unsigned blocks = (unsigned)((j.out + rows_per_block - 1) / rows_per_block);
    return launch(pick_kernel<DENSE_OUT>(j.n, j.m, j.bits, warps, blocks, operands_of(j)), nullptr, 0, d, blocks, warps, status, stream,
                  Z, U_next, nullptr, kGroupScalesGiven, group_rows);
}

// Shared memory per warp of the scale search.
static constexpr size_t dist_smem(int bits, int kept_bytes, bool alias = false) {
    return 32 * sizeof(double) + (bits == 4 ? sizeof(DistBins) : 0) + (alias && bits == 4 ? 0 : (size_t)kept_bytes);
}

using DistFn = void (*)(const PackJobDev*, int, const PackJobInline, uint32_t*, int, int32_t*);

template <int N, int M>
static DistFn pick_dist_bits(int bits, int warps) {
    if (warps <= kPackMinWarps)
        return bits == 8 ? (DistFn)dist_scale_kernel<N, M, 8, 128> : (DistFn)dist_scale_kernel<N, M, 4, 128>;
    if (warps <= 16)  // the row's values and the kept ones beside them need up to ~128 registers
        return bits == 8 ? (DistFn)dist_scale_kernel<N, M, 8, 512> : (DistFn)dist_scale_kernel<N, M, 4, 512>;
    return bits == 8 ? (DistFn)dist_scale_kernel<N, M, 8, 1024> : (DistFn)dist_scale_kernel<N, M, 4, 1024>;
}

static DistFn pick_dist(int n, int m, int bits, int warps) {
    if (n == m) return pick_dist_bits<4, 4>(bits, warps);
    if (m == 4) return n == 1 ? pick_dist_bits<1, 4>(bits, warps) : pick_dist_bits<2, 4>(bits, warps);
    if (n == 1) return pick_dist_bits<1, 8>(bits, warps);
    if (n == 2) return pick_dist_bits<2, 8>(bits, warps);
    return pick_dist_bits<4, 8>(bits, warps);
}

static int launch_dist(DistFn fn, size_t search, const PackJobDev* jobs_dev, int njobs, const PackJobDev& single, unsigned blocks,
                       int warps, uint32_t* status, cudaStream_t stream, int ncand, int32_t* cand) {
    const size_t smem = (size_t)warps * (search + sizeof(float));
    const int most = warps <= kPackMinWarps ? kPackMinWarps : warps <= 16 ? 16 : 32;  // warps that share this kernel (pick_dist_bits)
    if (smem > 48 * 1024) NM_CUDA_TRY(allow_dynamic_smem((const void*)fn, most * (int)(search + sizeof(float))));
    PackJobInline inl{};
    inl.j[0] = single;
    fn<<<blocks, warps * 32, smem, stream>>>(jobs_dev, njobs, inl, status, ncand, cand);
    NM_CUDA_TRY(cudaGetLastError());
    return NM_OK;
}

// Search and projection in one kernel (blocks of four warps): the row stays in registers from the one to the other, so W and U are
// read once.
template <int N, int M, bool DENSE_OUT>
static PackFn pick_dist_pack_bits(int bits) {
    return bits == 8 ? PackFn{(PackFnPtr)pack_kernel<N, M, 8, 128, DENSE_OUT, kDirect, true>, kDirect, dist_smem(8, kKeptBytes<N, M>)}
                     : PackFn{(PackFnPtr)pack_kernel<N, M, 4, 128, DENSE_OUT, kDirect, true>, kDirect, dist_smem(4, kKeptBytes<N, M>)};
}

template <bool DENSE_OUT>
static PackFn pick_dist_pack(int n, int m, int bits) {
    if (n == m) return pick_dist_pack_bits<4, 4, DENSE_OUT>(bits);
    if (m == 4) return n == 1 ? pick_dist_pack_bits<1, 4, DENSE_OUT>(bits) : pick_dist_pack_bits<2, 4, DENSE_OUT>(bits);
    if (n == 1) return pick_dist_pack_bits<1, 8, DENSE_OUT>(bits);
    if (n == 2) return pick_dist_pack_bits<2, 8, DENSE_OUT>(bits);
    return pick_dist_pack_bits<4, 8, DENSE_OUT>(bits);
}

// One matrix: the ADMM-Dist scales into job.scales (and the winning candidate numbers into `cand`).
static int launch_dist_single(const nm_pack_job_t& j, int ncand, int32_t* cand, uint32_t* status, cudaStream_t stream) {
    PackJobDev d = to_dev(j);
    const int warps = std::max(kPackMinWarps, 1 << d.wpr_log2);
    const int rows_per_block = warps >> d.wpr_log2;
    const unsigned blocks = (unsigned)((j.out + rows_per_block - 1) / rows_per_block);
    return launch_dist(pick_dist(j.n, j.m, j.bits, warps), dist_smem(j.bits, 32 / (j.n == j.m ? 4 : j.m) * (j.n == j.m ? 4 : j.n) * 128, warps > kPackMinWarps), nullptr, 0, d, blocks, warps, status, stream, ncand, cand);
}

// One matrix: search and projection.
template <bool DENSE_OUT>
static int launch_dist_project_single(const nm_pack_job_t& j, int ncand, uint32_t* status, cudaStream_t stream,
                                      float* Z = nullptr, float* U_next = nullptr) {
    PackJobDev d = to_dev(j);
    const int warps = std::max(kPackMinWarps, 1 << d.wpr_log2);
    const int rows_per_block = warps >> d.wpr_log2;
    const unsigned blocks = (unsigned)((j.out + rows_per_block - 1) / rows_per_block);
    if (warps <= kPackMinWarps)
        return launch(pick_dist_pack<DENSE_OUT>(j.n, j.m, j.bits), nullptr, 0, d, blocks, warps, status, stream, Z, U_next, nullptr,
                      kGroupNone, ncand);
    int rc = launch_dist_single(j, ncand, nullptr, status, stream);
    if (rc != NM_OK) return rc;
    return launch(pick_kernel<DENSE_OUT>(j.n, j.m, j.bits, warps, blocks, operands_of(j)), nullptr, 0, d, blocks, warps, status, stream, Z, U_next,
                  nullptr, kGroupScalesGiven, 0);
}

// Whether the launches of a call work on separate buffers: no output of a job of one launch overlaps a buffer of a job of
// another.  `table` holds the jobs launch by launch, `first` the number of each launch's first one; `dense` is parallel to
// `table` or NULL.  One pass over the buffers by address; of those before a buffer it remembers, among the outputs and among all, the
// one that reaches furthest and the furthest of another launch.
static bool separate_launches(const std::vector<PackJobDev>& table, const DenseOutDev* dense, const std::vector<size_t>& first) {
    struct Span { uintptr_t begin, end; size_t launch; bool out; };
    std::vector<Span> spans;
    spans.reserve(table.size() * (dense ? 7 : 5));
    size_t launch = 0;
    for (size_t i = 0; i < table.size(); ++i) {
        while (launch + 1 < first.size() && i >= first[launch + 1]) ++launch;
        const PackJobDev& j = table[i];
        auto add = [&](const void* p, size_t row_bytes, bool out) {
            if (p && row_bytes) spans.push_back(Span{(uintptr_t)p, (uintptr_t)p + row_bytes * (size_t)j.out, launch, out});
        };
        add(j.W, (size_t)j.in * 4, false);
        add(j.U, (size_t)j.in * 4, false);
        add(j.values, j.vrow_bytes, true);
        add(j.meta, (size_t)j.mrow_words * 4, true);
        add(j.scales, 4, true);
        if (dense) {
            add(dense[i].Z, (size_t)j.in * 4, true);
            add(dense[i].U_next, (size_t)j.in * 4, true);
        }
    }
    std::sort(spans.begin(), spans.end(), [](const Span& x, const Span& y) { return x.begin < y.begin; });
    struct Reach {
        uintptr_t end[2] = {0, 0};  // the furthest, and the furthest of a launch other than that one's
        size_t launch = 0;          // launch of end[0]
        uintptr_t of_others(size_t l) const { return l == launch ? end[1] : end[0]; }
        void take(const Span& s) {
            if (s.launch == launch) { end[0] = std::max(end[0], s.end); return; }
            if (s.end > end[0]) { end[1] = end[0]; end[0] = s.end; launch = s.launch; }
            else end[1] = std::max(end[1], s.end);
        }
    } outs, all;
    for (const Span& s : spans) {
        if ((s.out ? all : outs).of_others(s.launch) > s.begin) return false;
        all.take(s);
        if (s.out) outs.take(s);
    }
    return true;
}

// Shared by the batched entry points: groups the jobs that can share one launch (same pattern, code width
// and block size), writes the device job table(s) into `ws` and launches one kernel per group.
template <bool DENSE_OUT>
static int launch_batched(const nm_pack_job_t* jobs, const DenseOutDev* dense, int njobs, void* ws,
                          uint32_t* status, cudaStream_t s, bool grouped = false, int group_rows = 0,
                          int dist_ncand = 0) {
    // Group jobs that can share one launch: same (n == m ? dense : n, m), bits and block size.  Where a cluster of blocks holds a
    // group of rows (group_cluster) the block size follows from the warps per row.
    struct Key { int n, m, bits, warps, cluster, operands; };
    std::vector<Key> keys;
    std::vector<std::vector<int>> groups;
    for (int i = 0; i < njobs; ++i) {
        const nm_pack_job_t& j = jobs[i];
        if (j.out == 0 || j.in == 0) continue;
        const int wl = nm::wpr_log2_of(j.in);
        Key k{j.n == j.m ? 4 : j.n, j.n == j.m ? 4 : j.m, j.bits, std::max(nm::kPackMinWarps, 1 << wl), 0, operands_of(j)};
        int gw = 0, gc = 0;
        if (grouped && group_cluster(group_rows, wl, &gw, &gc)) { k.warps = gw; k.cluster = gc; }
        size_t g = 0;
        for (; g < keys.size(); ++g)
            if (keys[g].n == k.n && keys[g].m == k.m && keys[g].bits == k.bits && keys[g].warps == k.warps && keys[g].cluster == k.cluster &&
                (!k.cluster || nm::wpr_log2_of(jobs[groups[g][0]].in) == wl)) break;
        if (g == keys.size()) { keys.push_back(k); groups.emplace_back(); }
        keys[g].operands = std::min(keys[g].operands, k.operands);
        groups[g].push_back(i);
    }
    std::vector<nm::PackJobDev> table;
    std::vector<DenseOutDev> dense_table;  // same order as `table`
    table.reserve(njobs);
    std::vector<unsigned> group_blocks(keys.size());
    std::vector<size_t> group_first(keys.size());
    for (size_t g = 0; g < keys.size(); ++g) {
        unsigned blocks = 0;
        group_first[g] = table.size();
        for (int i : groups[g]) {
            nm::PackJobDev d = nm::to_dev(jobs[i]);
            const int rows_per_block = keys[g].cluster ? group_rows : keys[g].warps >> d.wpr_log2;
            d.unit_begin = blocks;
            unsigned long long nb = ((unsigned long long)d.out + rows_per_block - 1) / rows_per_block;
            if ((blocks + nb) * (keys[g].cluster ? keys[g].cluster : 1) > 0x7fffffffull) return NM_ERR_UNSUPPORTED;
            blocks += (unsigned)nb;
            table.push_back(d);
            if (DENSE_OUT) dense_table.push_back(dense[i]);
        }
        group_blocks[g] = blocks;
    }
    // Launches after the first start while the one before them drains, and each ends only after the one before it (72 matrices in
    // four formats 104 -> 90 us, with group-wise scales 179 -> 139), unless one's outputs overlap another's buffers (two jobs of
    // different formats on the same U, one of them in place): those run one after the other, in the order of the launches.
    // Looked at when the first launch is under way.
    bool separate = false;
    // Small plain batches: every group's table fits in the kernel's parameters, nothing is copied to `ws`.
    if (!DENSE_OUT && !grouped && dist_ncand == 0) {
        bool fits = true;
        for (size_t g = 0; g < keys.size(); ++g) fits = fits && groups[g].size() <= (size_t)kInlineJobs;
        if (fits) {
            for (size_t g = 0; g < keys.size(); ++g) {
                if (g == 1) separate = !g_no_pdl && separate_launches(table, nullptr, group_first);
                PackJobInline inl{};
                for (size_t i = 0; i < groups[g].size(); ++i) inl.j[i] = table[group_first[g] + i];
                int rc = nm::launch_table(nm::pick_kernel<DENSE_OUT>(keys[g].n, keys[g].m, keys[g].bits, keys[g].warps, group_blocks[g], keys[g].operands, (int)groups[g].size()), nullptr,
                                          (int)groups[g].size(), inl, group_blocks[g], keys[g].warps, status, s, nullptr,
                                          nullptr, nullptr, kGroupNone, 0, g > 0 && separate);
                if (rc != NM_OK) return rc;
            }
            return NM_OK;
        }
    }
    // The job table goes to `ws` with an asynchronous copy from this function's own (pageable) vector.  Launched
    // eagerly the source is staged before the call returns, so `table` may go away.  Under stream capture the
    // copy node would keep the host pointer and every replay of the graph would read freed memory (and the
    // kernels would follow whatever pointers they find there): such a call is refused before anything is enqueued.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    NM_CUDA_TRY(cudaStreamIsCapturing(s, &capture));
    if (capture != cudaStreamCaptureStatusNone) return NM_ERR_UNSUPPORTED;
    NM_CUDA_TRY(cudaMemcpyAsync(ws, table.data(), table.size() * sizeof(nm::PackJobDev),
                                cudaMemcpyHostToDevice, s));
    // the dense-output table follows the job table (njobs entries were reserved for each)
    DenseOutDev* dense_dev = reinterpret_cast<DenseOutDev*>(reinterpret_cast<PackJobDev*>(ws) + njobs);
    if (DENSE_OUT)
        NM_CUDA_TRY(cudaMemcpyAsync(dense_dev, dense_table.data(), dense_table.size() * sizeof(DenseOutDev),
                                    cudaMemcpyHostToDevice, s));
    if (grouped) {
        // group-wise scales: clear, fold the row maxima per group (a first pass of the same kernel), finish
        for (size_t g = 0; g < keys.size(); ++g) {
            if (keys[g].cluster) continue;
            const nm::PackJobDev* dev = reinterpret_cast<const nm::PackJobDev*>(ws) + group_first[g];
            group_prepare_kernel<<<(unsigned)groups[g].size(), 256, 0, s>>>(dev, group_rows, keys[g].bits, 0);
            NM_CUDA_TRY(cudaGetLastError());
            int rc = nm::launch(nm::pick_kernel<DENSE_OUT>(keys[g].n, keys[g].m, keys[g].bits, keys[g].warps, group_blocks[g], keys[g].operands, (int)groups[g].size()), dev,
                                (int)groups[g].size(), nm::PackJobDev{}, group_blocks[g], keys[g].warps, status, s,
                                nullptr, nullptr, DENSE_OUT ? dense_dev + group_first[g] : nullptr, kGroupMaxPass, group_rows);
            if (rc != NM_OK) return rc;
            group_prepare_kernel<<<(unsigned)groups[g].size(), 256, 0, s>>>(dev, group_rows, keys[g].bits, 1);
            NM_CUDA_TRY(cudaGetLastError());
        }
    }
    for (size_t g = 0; g < keys.size(); ++g) {
        const nm::PackJobDev* dev = reinterpret_cast<const nm::PackJobDev*>(ws) + group_first[g];
        const Key& k = keys[g];
        const int count = (int)groups[g].size();
        const DenseOutDev* dense_g = DENSE_OUT ? dense_dev + group_first[g] : nullptr;
        if (g == 1) separate = !g_no_pdl && separate_launches(table, DENSE_OUT ? dense_table.data() : nullptr, group_first);
        const bool chained = g > 0 && separate && (grouped ? k.cluster && keys[g - 1].cluster
                                                             : dist_ncand == 0 || (k.warps <= kPackMinWarps && keys[g - 1].warps <= kPackMinWarps));
        int rc;
        if (k.cluster) {
            rc = nm::launch_group<DENSE_OUT>(k.n, k.m, k.bits, k.warps, k.cluster, dev, count, nm::PackJobDev{}, group_blocks[g], status, s,
                                             nullptr, nullptr, dense_g, group_rows, chained);
        } else if (dist_ncand > 0 && k.warps <= kPackMinWarps) {  // ADMM-Dist: search and projection in one kernel
            rc = nm::launch(nm::pick_dist_pack<DENSE_OUT>(k.n, k.m, k.bits), dev, count, nm::PackJobDev{}, group_blocks[g], k.warps,
                            status, s, nullptr, nullptr, dense_g, kGroupNone, dist_ncand, chained);
        } else {
            if (dist_ncand > 0) {  // the search writes every job's scales, the projection takes them
                rc = nm::launch_dist(nm::pick_dist(k.n, k.m, k.bits, k.warps), nm::dist_smem(k.bits, 32 / (k.n == k.m ? 4 : k.m) * (k.n == k.m ? 4 : k.n) * 128, k.warps > nm::kPackMinWarps), dev, count, nm::PackJobDev{}, group_blocks[g], k.warps,
                                     status, s, dist_ncand, nullptr);
                if (rc != NM_OK) return rc;
            }
            rc = nm::launch(nm::pick_kernel<DENSE_OUT>(k.n, k.m, k.bits, k.warps, group_blocks[g], k.operands, count), dev, count, nm::PackJobDev{},
                            group_blocks[g], k.warps, status, s, nullptr, nullptr, dense_g,
                            (grouped || dist_ncand > 0) ? kGroupScalesGiven : kGroupNone, group_rows, chained);
        }
        if (rc != NM_OK) return rc;
    }
    return NM_OK;
}

static int validate_admm(const float* W, const float* U, int out, int in, int n, int m, int bits, const float* Z,
                         const float* U_next, const void* values, const void* meta, const float* scales) {
    int rc = check_pattern(out, in, n, m, bits);
    if (rc != NM_OK) return rc;
    if (!W || !Z) return NM_ERR_NULL;
    if (in % 4) return NM_ERR_SHAPE;
    if (in > 32768) return NM_ERR_UNSUPPORTED;
    if (!aligned(W, 16) || (U && !aligned(U, 16)) || !aligned(Z, 16) || (U_next && !aligned(U_next, 16)) ||
        (values && !aligned(values, 16)) || (meta && !aligned(meta, 4)) || (scales && !aligned(scales, 4)))
        return NM_ERR_ALIGN;
    return NM_OK;
}

}  // namespace nm

extern "C" {

int nm_project_pack(const float* W, const float* U, int out, int in, int n, int m, int bits,
                    void* values, void* meta, float* scales, uint32_t* status, void* stream) {
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    int rc = nm::validate_job(j);
    if (rc != NM_OK) return rc;
    if (out == 0 || in == 0) return NM_OK;
    nm::PackJobDev d = nm::to_dev(j);
    int warps = std::max(nm::kPackMinWarps, 1 << d.wpr_log2);
    int rows_per_block = warps >> d.wpr_log2;
    unsigned blocks = (unsigned)((out + rows_per_block - 1) / rows_per_block);
    return nm::launch(nm::pick_kernel(n, m, bits, warps, blocks, nm::operands_of(j)), nullptr, 0, d, blocks, warps, status, (cudaStream_t)stream);
}

int nm_admm_project(const float* W, const float* U, int out, int in, int n, int m, int bits, float* Z,
                    float* U_next, void* values, void* meta, float* scales, uint32_t* status, void* stream) {
    int rc = nm::validate_admm(W, U, out, in, n, m, bits, Z, U_next, values, meta, scales);
    if (rc != NM_OK) return rc;
    if (out == 0 || in == 0) return NM_OK;
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    nm::PackJobDev d = nm::to_dev(j);
    int warps = std::max(nm::kPackMinWarps, 1 << d.wpr_log2);
    int rows_per_block = warps >> d.wpr_log2;
    unsigned blocks = (unsigned)((out + rows_per_block - 1) / rows_per_block);
    return nm::launch(nm::pick_kernel<true>(n, m, bits, warps, blocks, nm::operands_of(j)), nullptr, 0, d, blocks, warps, status,
                      (cudaStream_t)stream, Z, U_next);
}

int nm_project_pack_grouped(const float* W, const float* U, int out, int in, int n, int m, int bits,
                            int group_rows, void* values, void* meta, float* scales, uint32_t* status,
                            void* stream) {
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    int rc = nm::validate_job(j);
    if (rc != NM_OK) return rc;
    if (out == 0 || in == 0) return NM_OK;
    return nm::launch_grouped_single<false>(j, group_rows, status, (cudaStream_t)stream);
}

int nm_admm_project_grouped(const float* W, const float* U, int out, int in, int n, int m, int bits,
                            int group_rows, float* Z, float* U_next, void* values, void* meta, float* scales,
                            uint32_t* status, void* stream) {
    int rc = nm::validate_admm(W, U, out, in, n, m, bits, Z, U_next, values, meta, scales);
    if (rc != NM_OK) return rc;
    if (!scales) return NM_ERR_NULL;  // also the scratch of the group maxima
    if (out == 0 || in == 0) return NM_OK;
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    return nm::launch_grouped_single<true>(j, group_rows, status, (cudaStream_t)stream, Z, U_next);
}

int nm_dist_scales(const float* W, const float* U, int out, int in, int n, int m, int bits, int ncand,
                   float* scales, int32_t* cand, uint32_t* status, void* stream) {
    int rc = nm::check_pattern(out, in, n, m, bits);
    if (rc != NM_OK) return rc;
    if (ncand < 1 || ncand > NM_DIST_MAX_CANDIDATES) return NM_ERR_SHAPE;
    if (!W || !scales) return NM_ERR_NULL;
    if (in % 4) return NM_ERR_SHAPE;
    if (in > 32768) return NM_ERR_UNSUPPORTED;
    if (!nm::aligned(W, 16) || (U && !nm::aligned(U, 16)) || !nm::aligned(scales, 4) || (cand && !nm::aligned(cand, 4)))
        return NM_ERR_ALIGN;
    if (out == 0 || in == 0) return NM_OK;
    nm_pack_job_t j{W, U, out, in, n, m, bits, nullptr, nullptr, scales};
    return nm::launch_dist_single(j, ncand, cand, status, (cudaStream_t)stream);
}

int nm_project_pack_dist(const float* W, const float* U, int out, int in, int n, int m, int bits, int ncand,
                         void* values, void* meta, float* scales, uint32_t* status, void* stream) {
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    int rc = nm::validate_job(j);
    if (rc != NM_OK) return rc;
    if (ncand < 1 || ncand > NM_DIST_MAX_CANDIDATES) return NM_ERR_SHAPE;
    if (out == 0 || in == 0) return NM_OK;
    return nm::launch_dist_project_single<false>(j, ncand, status, (cudaStream_t)stream);
}

int nm_admm_project_dist(const float* W, const float* U, int out, int in, int n, int m, int bits, int ncand,
                         float* Z, float* U_next, void* values, void* meta, float* scales, uint32_t* status,
                         void* stream) {
    int rc = nm::validate_admm(W, U, out, in, n, m, bits, Z, U_next, values, meta, scales);
    if (rc != NM_OK) return rc;
    if (!scales) return NM_ERR_NULL;  // the search hands its result to the projection through it
    if (ncand < 1 || ncand > NM_DIST_MAX_CANDIDATES) return NM_ERR_SHAPE;
    if (out == 0 || in == 0) return NM_OK;
    nm_pack_job_t j{W, U, out, in, n, m, bits, values, meta, scales};
    return nm::launch_dist_project_single<true>(j, ncand, status, (cudaStream_t)stream, Z, U_next);
}

int nm_project_pack_dist_batched(const nm_pack_job_t* jobs, int njobs, int ncand, void* ws, size_t ws_bytes,
                                 uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (ncand < 1 || ncand > NM_DIST_MAX_CANDIDATES) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_pack_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    for (int i = 0; i < njobs; ++i) {
        int rc = nm::validate_job(jobs[i]);
        if (rc != NM_OK) return rc;
    }
    return nm::launch_batched<false>(jobs, nullptr, njobs, ws, status, (cudaStream_t)stream, false, 0, ncand);
}

size_t nm_pack_workspace_bytes(int njobs) {
    return njobs <= 0 ? 0 : (size_t)njobs * sizeof(nm::PackJobDev);
}

int nm_project_pack_batched(const nm_pack_job_t* jobs, int njobs, void* ws, size_t ws_bytes,
                            uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_pack_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    for (int i = 0; i < njobs; ++i) {
        int rc = nm::validate_job(jobs[i]);
        if (rc != NM_OK) return rc;
    }
    return nm::launch_batched<false>(jobs, nullptr, njobs, ws, status, (cudaStream_t)stream);
}

int nm_admm_project_grouped_batched(const nm_admm_job_t* jobs, int njobs, int group_rows, void* ws,
                                    size_t ws_bytes, uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_admm_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    std::vector<nm_pack_job_t> pj(njobs);
    std::vector<nm::DenseOutDev> dj(njobs);
    for (int i = 0; i < njobs; ++i) {
        const nm_admm_job_t& a = jobs[i];
        int rc = nm::validate_admm(a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.Z, a.U_next, a.values, a.meta, a.scales);
        if (rc != NM_OK) return rc;
        if (!a.scales) return NM_ERR_NULL;  // also the scratch of the group maxima
        pj[i] = nm_pack_job_t{a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.values, a.meta, a.scales};
        dj[i] = nm::DenseOutDev{a.Z, a.U_next};
    }
    return nm::launch_batched<true>(pj.data(), dj.data(), njobs, ws, status, (cudaStream_t)stream, true, group_rows);
}

int nm_project_pack_grouped_batched(const nm_pack_job_t* jobs, int njobs, int group_rows, void* ws,
                                    size_t ws_bytes, uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_pack_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    for (int i = 0; i < njobs; ++i) {
        int rc = nm::validate_job(jobs[i]);
        if (rc != NM_OK) return rc;
    }
    return nm::launch_batched<false>(jobs, nullptr, njobs, ws, status, (cudaStream_t)stream, true, group_rows);
}

int nm_admm_project_dist_batched(const nm_admm_job_t* jobs, int njobs, int ncand, void* ws, size_t ws_bytes,
                                 uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (ncand < 1 || ncand > NM_DIST_MAX_CANDIDATES) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_admm_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    std::vector<nm_pack_job_t> pj(njobs);
    std::vector<nm::DenseOutDev> dj(njobs);
    for (int i = 0; i < njobs; ++i) {
        const nm_admm_job_t& a = jobs[i];
        int rc = nm::validate_admm(a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.Z, a.U_next, a.values, a.meta, a.scales);
        if (rc != NM_OK) return rc;
        if (!a.scales) return NM_ERR_NULL;  // the search hands its result to the projection through it
        pj[i] = nm_pack_job_t{a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.values, a.meta, a.scales};
        dj[i] = nm::DenseOutDev{a.Z, a.U_next};
    }
    return nm::launch_batched<true>(pj.data(), dj.data(), njobs, ws, status, (cudaStream_t)stream, false, 0, ncand);
}

size_t nm_admm_workspace_bytes(int njobs) {
    return njobs <= 0 ? 0 : (size_t)njobs * (sizeof(nm::PackJobDev) + sizeof(nm::DenseOutDev));
}

int nm_admm_project_batched(const nm_admm_job_t* jobs, int njobs, void* ws, size_t ws_bytes,
                            uint32_t* status, void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (njobs == 0) return NM_OK;
    if (!jobs) return NM_ERR_NULL;
    if (!ws || ws_bytes < nm_admm_workspace_bytes(njobs)) return NM_ERR_WORKSPACE;
    if (!nm::aligned(ws, 16)) return NM_ERR_ALIGN;
    std::vector<nm_pack_job_t> pj(njobs);
    std::vector<nm::DenseOutDev> dj(njobs);
    for (int i = 0; i < njobs; ++i) {
        const nm_admm_job_t& a = jobs[i];
        int rc = nm::validate_admm(a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.Z, a.U_next, a.values, a.meta, a.scales);
        if (rc != NM_OK) return rc;
        pj[i] = nm_pack_job_t{a.W, a.U, a.out, a.in, a.n, a.m, a.bits, a.values, a.meta, a.scales};
        dj[i] = nm::DenseOutDev{a.Z, a.U_next};
    }
    return nm::launch_batched<true>(pj.data(), dj.data(), njobs, ws, status, (cudaStream_t)stream);
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Batched projection without any caller-provided or library-allocated scratch.
// The job table lives in a fixed device array that is part of the loaded library image.
// ---------------------------------------------------------------------------------------------
namespace nm {

constexpr int kNoAllocMaxJobs = 1024;  // 1024 jobs x 64 bytes = 64 KB held on every GPU that loads the library
static __device__ __align__(256) unsigned char g_noalloc_job_table[kNoAllocMaxJobs * sizeof(PackJobDev)];

// In host code `g_noalloc_job_table` is only a handle; its device address has to be asked for,
// once per device, with that device current.
static int noalloc_table_address(void** out) {
    static void* cached[64] = {nullptr};
    static std::mutex mu;
    int dev = 0;
    NM_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return record_text_error("device ordinal beyond 63");
    std::lock_guard<std::mutex> lock(mu);
    if (!cached[dev]) {
        void* p = nullptr;
        NM_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_job_table));
        cached[dev] = p;
    }
    *out = cached[dev];
    return NM_OK;
}

}  // namespace nm

extern "C" int nm_project_pack_batched_noalloc(const nm_pack_job_t* jobs, int njobs, uint32_t* status,
                                               void* stream) {
    if (njobs < 0) return NM_ERR_SHAPE;
    if (njobs > nm::kNoAllocMaxJobs) return NM_ERR_UNSUPPORTED;  // beyond NM_NOALLOC_MAX_JOBS
    if (njobs == 0) return NM_OK;
    void* table = nullptr;
    int rc = nm::noalloc_table_address(&table);
    if (rc != NM_OK) return rc;
    return nm_project_pack_batched(jobs, njobs, table, sizeof(nm::g_noalloc_job_table), status, stream);
}
