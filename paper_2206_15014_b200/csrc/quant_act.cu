// Dynamic per-tensor symmetric 8-bit activation quantiser: |max| reduction and the quantise pass.
#include "common.cuh"
#include "sm100_ptx.cuh"
#include <cuda_runtime.h>

namespace nm {

// Both kernels read eight consecutive floats per thread and step (32 bytes; two 16-byte loads where the tensor is only aligned to
// those), kUnroll steps in flight, coalesced over the warp.  They are launched as programmatic dependents: their blocks start
// while the kernel before them in the stream drains, and touch global memory only once it has finished.
constexpr int kActThreads = 256, kUnroll = 4;

__device__ __forceinline__ void load8(const float* p, bool wide, float* x) {
    if (wide) {
        asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7]) : "l"(p) : "memory");
    } else {
        const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    }
}

// Non-negative floats order like their bit patterns, so an unsigned atomicMax folds the maximum.
__global__ void __launch_bounds__(kActThreads) absmax_kernel(const float* Y, size_t count, float* absmax) {
    ptx::grid_dep_launch();  // a dependent kernel may begin its set-up early
    ptx::grid_dep_wait();
    const size_t n8 = count >> 3, stride = (size_t)gridDim.x * kActThreads;
    const bool wide = ((uintptr_t)Y & 31u) == 0;
    float a = 0.0f;
    for (size_t i = (size_t)blockIdx.x * kActThreads + threadIdx.x; i < n8; i += kUnroll * stride) {
        float x[kUnroll][8];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (i + u * stride < n8) load8(Y + 8 * (i + u * stride), wide, x[u]);
            else {
#pragma unroll
                for (int j = 0; j < 8; ++j) x[u][j] = 0.0f;
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
#pragma unroll
            for (int j = 0; j < 8; ++j) a = fmaxf(a, fabsf(x[u][j]));
    }
    if (blockIdx.x == 0 && threadIdx.x < (count & 7)) a = fmaxf(a, fabsf(Y[(n8 << 3) + threadIdx.x]));
    a = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(a)));
    __shared__ float red[kActThreads / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kActThreads / 32; ++i) a = fmaxf(a, red[i]);
        atomicMax(reinterpret_cast<unsigned*>(absmax), __float_as_uint(a));
    }
}

__device__ __noinline__ int quantise8(float y, float s) {
    int q = __float2int_rn(__fdiv_rn(y, s));  // IEEE division, round half to even
    return max(-128, min(127, q));
}

// Four codes from t = fma(y, RN(1 / s), 1.5 * 2^23), whose rounding gives the nearest-even integer of the product; the
// product is within 2^-16 of the IEEE quotient over the code range, so only where it lies within 2^-15 of a half (6 values in
// 100000), is NaN or is too large for the trick does the division decide.
__device__ __forceinline__ unsigned pack4(const float* y, float s, float rs, bool fast_ok) {
    constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23 = 0x4B400000: the low byte of the sum is the code
    float t[4], worst = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        t[j] = __fmaf_rn(y[j], rs, kMagic);
        const float f = fabsf(__fmaf_rn(y[j], rs, -__fsub_rn(t[j], kMagic)));
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(worst) : "f"(worst), "f"(f));
        t[j] = fminf(fmaxf(t[j], kMagic - 128.0f), kMagic + 127.0f);
    }
    if (!(fast_ok && worst <= 0.49996948f))
        return (unsigned)(quantise8(y[0], s) & 0xff) | ((unsigned)(quantise8(y[1], s) & 0xff) << 8) |
               ((unsigned)(quantise8(y[2], s) & 0xff) << 16) | ((unsigned)(quantise8(y[3], s) & 0xff) << 24);
    return __byte_perm(__byte_perm(__float_as_uint(t[0]), __float_as_uint(t[1]), 0x0040),
                       __byte_perm(__float_as_uint(t[2]), __float_as_uint(t[3]), 0x0040), 0x5410);
}

__global__ void __launch_bounds__(kActThreads, 4) quantize_act_kernel(const float* Y, size_t count, const float* absmax,
                                                                      int8_t* Xq, float* sx_out) {
    ptx::grid_dep_launch();  // a dependent kernel may begin its set-up early
    ptx::grid_dep_wait();
    const size_t n8 = count >> 3, stride = (size_t)gridDim.x * kActThreads;
    const bool wide = ((uintptr_t)Y & 31u) == 0;
    size_t i = (size_t)blockIdx.x * kActThreads + threadIdx.x;
    float x[kUnroll][8];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
        if (i + u * stride < n8) load8(Y + 8 * (i + u * stride), wide, x[u]);
    const float a = *absmax;
    const float s = (a == 0.0f) ? 1.0f : __fdiv_rn(a, 127.0f);
    const float rs = __frcp_rn(s);
    const bool fast_ok = s >= 1.17549435e-38f && s <= 4.25e37f;  // rs is a normal number
    if (sx_out && blockIdx.x == 0 && threadIdx.x == 0) *sx_out = s;
    while (i < n8) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (i + u * stride < n8)
                *reinterpret_cast<uint2*>(Xq + 8 * (i + u * stride)) =
                    make_uint2(pack4(x[u], s, rs, fast_ok), pack4(x[u] + 4, s, rs, fast_ok));
        i += kUnroll * stride;
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
            if (i + u * stride < n8) load8(Y + 8 * (i + u * stride), wide, x[u]);
    }
    if (blockIdx.x == 0 && threadIdx.x < (count & 7)) {
        size_t k = (n8 << 3) + threadIdx.x;
        Xq[k] = (int8_t)quantise8(Y[k], s);
    }
}

// One step per thread for small tensors, the device's resident blocks for large ones.
static int grid_for(size_t count) {
    size_t blocks = ((count >> 3) + kActThreads - 1) / kActThreads;
    size_t cap = (size_t)sm_count() * 4;
    return (int)(blocks < 1 ? 1 : (blocks > cap ? cap : blocks));
}

template <typename... P, typename... A>
static cudaError_t launch_dependent(void (*kernel)(P...), int grid, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kActThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_no_pdl ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace nm

extern "C" {

int nm_absmax(const float* Y, size_t count, float* absmax, void* stream) {
    if (!absmax || (!Y && count)) return NM_ERR_NULL;
    if (count == 0) return NM_OK;
    if (!nm::aligned(Y, 16) || !nm::aligned(absmax, 4)) return NM_ERR_ALIGN;
    NM_CUDA_TRY(nm::launch_dependent(nm::absmax_kernel, nm::grid_for(count), (cudaStream_t)stream, Y, count, absmax));
    return NM_OK;
}

int nm_quantize_act(const float* Y, size_t count, const float* absmax, int8_t* Xq, float* sx_out,
                    void* stream) {
    if (!absmax || ((!Y || !Xq) && count)) return NM_ERR_NULL;
    if (count && (!nm::aligned(Y, 16) || !nm::aligned(Xq, 16))) return NM_ERR_ALIGN;
    if (sx_out == absmax) return NM_ERR_SHAPE;  // one thread writes the scale while the others still read the maximum
    NM_CUDA_TRY(nm::launch_dependent(nm::quantize_act_kernel, nm::grid_for(count), (cudaStream_t)stream, Y, count, absmax, Xq, sx_out));
    return NM_OK;
}

}  // extern "C"
