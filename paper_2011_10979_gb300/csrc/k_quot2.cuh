// k_quot2.cuh -- quotients by a divisor that stays the same over many divisions, without dividing: from the
// correctly rounded reciprocal, a faithful quotient and one remainder step more, which makes it correctly rounded
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
// 1990).  That holds while neither the remainders nor the quotient underflow.  Numerators below 2^-80 -- the
// flow and the illumination decay geometrically into regions without data and reach the subnormal numbers -- are
// first scaled by 2^64, and the quotient scaled back: where it is subnormal that rounds a second time, which only
// goes wrong from the middle between two numbers, where the remainder's sign decides.
#pragma once
#include "k_pack2.cuh"

namespace tvl1 {

constexpr float QUOT_SMALL = 0x1p-80f;
// QUOT_SMALL as 2 |x| in integers, for the minimum of (2 |x| - 1) over several x: zero wraps around.
constexpr unsigned QUOT_SMALL_BITS = 2u * 0x17800000u;

// The scale of a numerator and its inverse.
struct QuotScale {
    float up, down;
};
__device__ __forceinline__ QuotScale quot_scale(float x) {
    const bool small = fabsf(x) < QUOT_SMALL;
    return {small ? 0x1p64f : 1.f, small ? 0x1p-64f : 1.f};
}
// q scaled back, q the correctly rounded quotient of the scaled numerator x by e.
__device__ __forceinline__ float quot_unscale(float q, float x, float e, QuotScale s) {
    const float t = q * s.down, r = fmaf(-e, q, x), d = fmaf(t, -s.up, q);
    const bool beyond = fabsf(d) == 0x1p-86f && r != 0.f && (__float_as_int(r) ^ __float_as_int(d)) >= 0;
    return beyond ? t + copysignf(0x1p-149f, d) : t;
}

// x / e per half, e in (2^-100, 2^40) with rc its reciprocal (0 and rc 0: the quotient is 0), |x| at most 2^100;
// SCALED: whatever the numerators, else zero or at least QUOT_SMALL.
template <bool SCALED> __device__ __forceinline__ pair2 quot2(pair2 x, pair2 e, pair2 rc) {
    QuotScale s0{1.f, 1.f}, s1{1.f, 1.f};
    if (SCALED) {
        float a, b;
        upk(x, a, b);
        s0 = quot_scale(a);
        s1 = quot_scale(b);
        x = mul2(x, pk(s0.up, s1.up));
    }
    const pair2 ne = neg2(e);
    pair2 q = mul2(x, rc);
    q = fma2(fma2(ne, q, x), rc, q);
    q = fma2(fma2(ne, q, x), rc, q);
    if (!SCALED) return q;
    return pk(quot_unscale(lo2(q), lo2(x), lo2(e), s0), quot_unscale(hi2(q), hi2(x), hi2(e), s1));
}

// The proximal step's t = -rho / |e|^2, or -+ sl0 where |rho| > thr = sl0 |e|^2 per half.
template <bool SCALED> __device__ __forceinline__ pair2 prox_quot2(pair2 rho, pair2 e2, pair2 rc, pair2 thr, float sl0) {
    float r0, r1, s0, s1, q0, q1;
    upk(rho, r0, r1);
    upk(thr, s0, s1);
    upk(quot2<SCALED>(rho, e2, rc), q0, q1);
    // |t| first, then the sign of -rho
    auto sgn = [](float m, float x) {
        return __uint_as_float((__float_as_uint(m) & 0x7fffffffu) | (~__float_as_uint(x) & 0x80000000u));
    };
    return pk(sgn(fabsf(r0) > s0 ? sl0 : q0, r0), sgn(fabsf(r1) > s1 ? sl0 : q1, r1));
}
// The same with divisions, for any divisor.
__device__ __forceinline__ pair2 prox_div2(pair2 rho, pair2 e2, pair2 thr, float sl0) {
    float r0, r1, s0, s1, e0, e1;
    upk(rho, r0, r1);
    upk(thr, s0, s1);
    upk(e2, e0, e1);
    return pk(e0 <= 0.f ? 0.f : r0 < -s0 ? sl0 : r0 > s0 ? -sl0 : -r0 / e0, e1 <= 0.f ? 0.f : r1 < -s1 ? sl0 : r1 > s1 ? -sl0 : -r1 / e1);
}

// Whether a pixel pair's |e|^2 is outside the quotient's range; of such a pair, whether it has no data at all: its step
// moves nothing, whatever t, as long as It is finite, so that with a zero reciprocal it is inside after all.
__device__ __forceinline__ bool prox_unusual(pair2 e2) {
    float a, b;
    upk(e2, a, b);
    return !(fminf(a, b) > 0x1p-100f && fmaxf(a, b) < 0x1p40f);
}
__device__ __forceinline__ bool prox_empty(pair2 e2, pair2 ix, pair2 iy, pair2 it, float beta) {
    auto one = [&](float e, float x, float y, float t) {
        return (e > 0x1p-100f && e < 0x1p40f) || (e == 0.f && x == 0.f && y == 0.f && beta == 0.f && fabsf(t) < INFINITY);
    };
    return one(lo2(e2), lo2(ix), lo2(iy), lo2(it)) && one(hi2(e2), hi2(ix), hi2(iy), hi2(it));
}
__device__ __forceinline__ float prox_rcp(float e) { return e > 0.f ? __frcp_rn(e) : 0.f; }
__device__ __forceinline__ pair2 prox_rcp2(pair2 e2) { return pk(prox_rcp(lo2(e2)), prox_rcp(hi2(e2))); }

}  // namespace tvl1
