// Shared host-side helpers of the nmsparse library (error bookkeeping, pattern validation).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include "../../include/nmsparse.h"

namespace nm {

// Records the text of a failed CUDA call for nm_last_cuda_error(); returns NM_ERR_CUDA.
int record_cuda_error(cudaError_t e, const char* where);
int record_text_error(const char* text);

#define NM_CUDA_TRY(expr)                                                 \
    do {                                                                  \
        cudaError_t e__ = (expr);                                         \
        if (e__ != cudaSuccess) return nm::record_cuda_error(e__, #expr); \
    } while (0)

// Field width of one metadata entry.
__host__ __device__ inline int meta_field_bits(int m) { return m == 4 ? 2 : 4; }

// NM_OK when (out, in, n, m, bits) is a pattern the library packs.
int check_pattern(int out, int in, int n, int m, int bits);

// Bytes of one row of packed values / u32 words of one row of metadata.
inline size_t values_row_bytes(int in, int n, int m, int bits) { return (size_t)(in / m) * n * bits / 8; }
inline size_t meta_row_words(int in, int n, int m) {
    if (n == m) return 0;
    return ((size_t)(in / m) * n * meta_field_bits(m) + 31) / 32;
}

// Form of the projection kernel forced by nm_debug_set_option("pack_form") (0 = automatic).
extern int g_pack_form;
// nm_debug_set_option("no_pdl"): no launch of the library carries the programmatic-dependent-launch attribute.
extern int g_no_pdl;

#ifdef NM_TEST_HOOKS
// Timeout test only: the unit (per block) whose copies warp 0 of block 0 of the staged projection kernel leaves unissued.
int pack_set_skip_unit(int unit);
#endif

// cudaFuncSetAttribute(max dynamic shared memory) once per kernel and device instead of on every launch; `bytes`: the most that a launch of `fn` takes.
cudaError_t allow_dynamic_smem(const void* fn, int bytes);

// Multiprocessors of the current device (cached per device; 148 when the query fails).
int sm_count();

inline bool aligned(const void* p, size_t a) { return ((uintptr_t)p % a) == 0; }

#ifdef __CUDACC__
// The 8-bit code of v at the scale s from the IEEE quotient: clamped to [-128.49, 127.49] before the add of 1.5 * 2^23, whose own
// rounding rounds to the nearest-even integer, it leaves nothing to clamp afterwards (a quotient beyond the range, infinite
// included, rounds to the end code either way).
__device__ __forceinline__ int quantise8_exact(float v, float s) {
    constexpr float kMagic = 12582912.0f;
    const float qc = fminf(fmaxf(__fdiv_rn(v, s), -128.49f), 127.49f);
    return __float_as_int(__fadd_rn(qc, kMagic)) - 0x4B400000;
}
#endif

}  // namespace nm
