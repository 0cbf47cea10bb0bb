// k_pack2.cuh -- arithmetic on pairs of FP32 values (two neighbouring columns of one row) held in
// one 64-bit register pair: the packed instructions of sm_100 and later (add / mul / fma .f32x2)
// round each half exactly as the scalar instruction does, and issue once for both halves.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tvl1_device.cuh"

namespace tvl1 {

using pair2 = unsigned long long;  // low word: the even column, high word: the odd one

__device__ __forceinline__ pair2 pk(float a, float b) {
    pair2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(pair2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ float lo2(pair2 v) {
    float a, b;
    upk(v, a, b);
    return a;
}
__device__ __forceinline__ float hi2(pair2 v) {
    float a, b;
    upk(v, a, b);
    return b;
}
__device__ __forceinline__ pair2 bc2(float a) { return pk(a, a); }
__device__ __forceinline__ pair2 add2(pair2 a, pair2 b) {
    pair2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair2 sub2(pair2 a, pair2 b) {
    pair2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair2 mul2(pair2 a, pair2 b) {
    pair2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair2 fma2(pair2 a, pair2 b, pair2 c) {
    pair2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ pair2 neg2(pair2 a) {
    float x, y;
    upk(a, x, y);
    return pk(-x, -y);
}

// ~0 or 0 (opaque to the compiler, which would turn the masking back into selects).
__device__ __forceinline__ unsigned mask_of(bool on) {
    unsigned m = on ? ~0u : 0u;
    asm("" : "+r"(m));
    return m;
}
// x where the mask is ~0, +0 where it is 0: one logic instruction, which runs beside the FMA pipe
// (a floating-point select does not).
__device__ __forceinline__ float keep(float x, unsigned m) { return __uint_as_float(__float_as_uint(x) & m); }

// Both halves rounded to storage type T and back.
template <typename T> __device__ __forceinline__ pair2 round2(pair2 v) {
    float a, b;
    upk(v, a, b);
    return pk(storage_round<T>(a), storage_round<T>(b));
}
template <> __device__ __forceinline__ pair2 round2<float>(pair2 v) { return v; }

// A pair of stored values at element offset o (even, 8- or 4-byte aligned).
template <typename T> __device__ __forceinline__ pair2 ld_pair(const void *base, size_t o);
template <> __device__ __forceinline__ pair2 ld_pair<float>(const void *base, size_t o) {
    const float2 v = *reinterpret_cast<const float2 *>(reinterpret_cast<const float *>(base) + o);
    return pk(v.x, v.y);
}
template <> __device__ __forceinline__ pair2 ld_pair<__half>(const void *base, size_t o) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(reinterpret_cast<const __half *>(base) + o));
    return pk(v.x, v.y);
}
template <> __device__ __forceinline__ pair2 ld_pair<__nv_bfloat16>(const void *base, size_t o) {
    const float2 v = __bfloat1622float2(
        *reinterpret_cast<const __nv_bfloat162 *>(reinterpret_cast<const __nv_bfloat16 *>(base) + o));
    return pk(v.x, v.y);
}
template <typename T> __device__ __forceinline__ void st_pair(void *base, size_t o, pair2 v);
template <> __device__ __forceinline__ void st_pair<float>(void *base, size_t o, pair2 v) {
    float a, b;
    upk(v, a, b);
    *reinterpret_cast<float2 *>(reinterpret_cast<float *>(base) + o) = make_float2(a, b);
}
template <> __device__ __forceinline__ void st_pair<__half>(void *base, size_t o, pair2 v) {
    float a, b;
    upk(v, a, b);
    *reinterpret_cast<__half2 *>(reinterpret_cast<__half *>(base) + o) = __floats2half2_rn(a, b);
}
template <> __device__ __forceinline__ void st_pair<__nv_bfloat16>(void *base, size_t o, pair2 v) {
    float a, b;
    upk(v, a, b);
    *reinterpret_cast<__nv_bfloat162 *>(reinterpret_cast<__nv_bfloat16 *>(base) + o) = __floats2bfloat162_rn(a, b);
}

// Arrival at, and wait on, a named barrier of this block that `n` threads take part in (whole
// warps): the arriving warps do not wait, and their earlier shared-memory writes are visible to
// the waiting ones.
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_wait(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// 1 / max(1, sqrt(n2)) per half: rsqrt.approx of max(n2, 1), which is exactly 1 inside the ball and
// the value of rsqrtf(n2) outside (n2 > 1 is a normal number, where the flushing and the
// non-flushing instruction agree).  A NaN n2 gives 1, as the comparison n2 > 1 does.
__device__ __forceinline__ pair2 ball_scale2(pair2 n2) {
    float a, b, fa, fb;
    upk(n2, a, b);
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(fa) : "f"(fmaxf(a, 1.f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(fb) : "f"(fmaxf(b, 1.f)));
    return pk(fa, fb);
}

}  // namespace tvl1
