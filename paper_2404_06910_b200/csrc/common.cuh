// Shared host/device helpers of the library: error reporting, argument checks,
// storage-type loads.  Nothing here is used by (or shared with) the CPU oracle.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>

#include "../../include/sp.h"

namespace sp {

// ---- thread-local error message ---------------------------------------------------
char *error_buffer();                       // 512 bytes, thread local (api.cu)
int fail(int code, const char *fmt, ...);   // formats the message, returns code

#define SP_REQUIRE(cond, code, ...)                     \
    do {                                                \
        if (!(cond)) return ::sp::fail((code), __VA_ARGS__); \
    } while (0)

#define SP_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t e__ = (call);                                                       \
        if (e__ != cudaSuccess)                                                         \
            return ::sp::fail(SP_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e__)); \
    } while (0)

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool aligned256(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }
inline int elt_bytes(int dtype) { return dtype == SP_F32 ? 4 : 2; }
__host__ __device__ constexpr size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int check_layout(const sp_layout *lay);     // host-visible fields only (api.cu)
void rope_inv_freq(double base, int rot_dim, double *out);   // [rot_dim / 2] (api.cu)

// Device status word codes (first 4 bytes of a workspace).
enum : uint32_t { STATUS_OK = 0, STATUS_TIMEOUT = 1, STATUS_BAD_LAYOUT = 2 };

#ifdef __CUDACC__
// One rotation (a, b) -> (a cos - b sin, a sin + b cos) with its roundings spelled out, so that every kernel that
// rotates the same pair with the same (cos, sin) stores the same bits.
__device__ __forceinline__ void rope_rotate(float a, float b, float c, float s, float &na, float &nb)
{
    na = __fmaf_rn(a, c, -__fmul_rn(b, s));
    nb = __fmaf_rn(a, s, __fmul_rn(b, c));
}
#endif
int num_sms();                              // multiprocessors of the current device (api.cu)

// ---- programmatic dependent launch -------------------------------------------------
// Every kernel of the library is launched as a programmatic dependent of what precedes it in the stream: its blocks may be
// scheduled, and set themselves up, while the last blocks of the kernel before are still running, which takes launch latency
// and ramp-up off every boundary of a chain of short kernels.  In return every thread of every kernel calls
// pdl_wait() before it touches global memory; after it, everything earlier in the stream is complete and visible.
// Its blocks may run while an earlier kernel still writes what they read after the wait, so nothing is read through the
// non-coherent path or a pointer promised not to alias (no ld.global.nc, __ldg or __restrict__): both may be fetched ahead of it.
// pdl_trigger() lets the next kernel's blocks in as soon as all blocks of this one have started.  One prompt of 20 documents,
// whole step: 93 -> 83 us; 4 documents in fp32: 39 -> 29.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
int launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, unsigned cluster_x, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster_x; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster_x > 1 ? 2 : 1;
    SP_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    return SP_OK;
}
#endif

// ---- device helpers ----------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Loads 8 consecutive elements (bf16: one 16-byte load) or 4 (fp32) as floats.
template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ __forceinline__ static void load(const __nv_bfloat16 *p, float (&f)[8]) {
        const uint4 w = *reinterpret_cast<const uint4 *>(p);
        f[0] = bf16_lo(w.x); f[1] = bf16_hi(w.x); f[2] = bf16_lo(w.y); f[3] = bf16_hi(w.y);
        f[4] = bf16_lo(w.z); f[5] = bf16_hi(w.z); f[6] = bf16_lo(w.w); f[7] = bf16_hi(w.w);
    }
};
template <> struct Vec<float> {
    static constexpr int N = 4;
    __device__ __forceinline__ static void load(const float *p, float (&f)[4]) {
        const float4 w = *reinterpret_cast<const float4 *>(p);
        f[0] = w.x; f[1] = w.y; f[2] = w.z; f[3] = w.w;
    }
};

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void store_val(float *p, float x) { *p = x; }
__device__ __forceinline__ void store_val(__nv_bfloat16 *p, float x) { *p = __float2bfloat16_rn(x); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&t);
}

// Two probabilities as sums of two bf16 numbers each: hi is p cut off behind 8 bits, lo the rest (16 bits in all).  lo is never
// negative, and the 2^-23 p in it, less than p's own rounding, keeps it above zero where p is: the products with an Inf in V
// are then infinities of one sign, as that of p would be, and not NaN.
__device__ __forceinline__ void split_bf16(float p0, float p1, uint32_t &hi, uint32_t &lo) {
    const uint32_t a = __float_as_uint(p0) & 0xffff0000u, b = __float_as_uint(p1) & 0xffff0000u;
    hi = __byte_perm(a, b, 0x7632);
    lo = pack_bf16x2(fmaf(p0, 1.f + 0x1p-23f, -__uint_as_float(a)), fmaf(p1, 1.f + 0x1p-23f, -__uint_as_float(b)));
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
#endif  // __CUDACC__

}  // namespace sp
