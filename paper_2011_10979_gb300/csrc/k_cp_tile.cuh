// k_cp_tile.cuh -- several ALG1 iterations (Sec. 4: Chambolle-Pock with constant steps on
// eq. primal-dual:optical:o) in one launch, the state in registers, for the single-pair levels that
// run on the per-iteration engine.
//
// The frame layout is that of the ADMM tile kernel (k_admm_tile.cuh): a block of TILE_WARPS warps holds
// 64 columns by TILE_WARPS R rows, each lane two neighbouring columns (a register pair per plane) in R
// rows; east and west neighbours travel by shuffle, south and north ones in registers and, between
// the warps' bands, through shared memory.  One iteration at a pixel needs y^{k+1} there and one pixel
// west and north (the divergence in the primal step), and y^{k+1} at a pixel needs Xbar^k there and
// one pixel east and south (the forward differences in the dual step), so ni iterations need a halo of
// ni pixels on every side.
// The per-pixel arithmetic is that of the per-iteration kernel (k_cp.cu, k_cp_math.cuh) in the same
// order, and the state between the iterations is rounded to the flow storage type where that kernel's
// stores round it (y^{k+1} when read as y, X and Xbar when written), so ni iterations here are bitwise
// ni launches of k_cp.
//
// The primal step divides by |e|^2, a constant of the pixel: -rho / |e|^2 is formed from the correctly
// rounded reciprocal with two remainder steps, the first of which makes the quotient faithful and the
// second correctly rounded (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", IBM J. Res. Dev. 34, 1990), as long as neither the remainders nor the
// quotient underflow: |e|^2 in (2^-100, 2^40) and |rho| = 0 or at least 2^-80, else the warp's
// iteration divides.  So that this costs one branch per iteration and not one per row (a branch in a
// row keeps the rows from overlapping: 2.8 against 1.5 us per iteration at R = 4), the primal step
// first forms Z and rho of all rows, Z in the registers of the spent Xbar.
//
// Bound by latency and issue with three warps per SM quarter (some 240 clocks per row and warp), beside
// 4 to 6 us per launch for instruction fetch and the state's loads and stores.  Measured per iteration,
// and in brackets with the frame in shared memory and scalar instructions, which this replaced:
// 640x480 2.83 us (4.51), 320x240 1.30 (1.87), 160x120 1.09 (1.32), 3840x2160 75 (114).
#pragma once
#include <math.h>

#include <type_traits>

#include "k_cp_math.cuh"
#include "k_pack2.cuh"

namespace tvl1 {

void cp_tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s);
void cp_tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s);

namespace cptile {

constexpr int NW = TILE_WARPS;
constexpr unsigned FULL = 0xffffffffu;

template <int R> struct Shared {
    pair2 top[NW][3][32];   // Xbar of the top rows, read by the warp above
    pair2 bot[NW][3][32];   // y2 components of the bottom rows, read by the warp below
    pair2 ix[NW * R][32], iy[NW * R][32], it[NW * R][32], rc[NW * R][32];  // data and 1 / |e|^2 (each thread its own)
    double red[32];
};

template <typename T, typename TF, bool HAS_W, int R> struct Kernel {
    static constexpr int C0 = HAS_W ? 0 : 1;
    using SH = Shared<R>;

    // BX, BY: as the ADMM tile kernel's.
    template <int BX, bool BY>
    static __device__ __forceinline__ void body(const TileArgs &A, SH &G, int bx, int by, int lane, int wid) {
        const int H = A.a.g.H, W = A.a.g.W, P = A.a.g.pitch;
        const int c = bx * A.ow - A.offx + 2 * lane, ib = by * A.oh - A.offy + wid * R;
        const unsigned me0 = mask_of(c >= 0 && c < W - 1), me1 = mask_of(c + 1 >= 0 && c + 1 < W - 1);
        const int rlast = __shfl_sync(FULL, H - 1 - ib, 0), rfirst = __shfl_sync(FULL, -ib, 0);
        pair2 y[R][6], X[R][3], B[R][3];
        const float beta = A.a.k.beta, lam = A.a.k.lambda, sg = A.a.k.cp_sigma, sl0 = sg * lam;
        const pair2 tau2 = bc2(A.a.k.cp_tau), sg2 = bc2(sg), beta2 = bc2(beta), bb2 = bc2(beta * beta), sl02 = bc2(sl0);
        bool odd = !(sl0 < 0x1p20f);  // quotients outside the fast division's range
        {
            const int c0 = BX ? min(max(c, 0), W - 1) : c, c1 = BX ? min(max(c + 1, 0), W - 1) : c + 1;
            auto load = [&](auto VEC_) {
                constexpr bool VEC = decltype(VEC_)::value;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = ib + r;
                    const unsigned m0 = mask_of(i >= 0 && i < H && c >= 0 && c < W);
                    const unsigned m1 = mask_of(i >= 0 && i < H && c + 1 >= 0 && c + 1 < W);
                    const size_t row = (size_t)(BY ? min(max(i, 0), H - 1) : i) * P;
                    const size_t o0 = row + (VEC ? c0 & ~1 : c0), o1 = row + c1;
                    auto mask = [&](pair2 q) -> pair2 {
                        if (!BX && !BY) return q;
                        float a, b;
                        upk(q, a, b);
                        return pk(keep(a, m0), keep(b, m1));
                    };
                    // outside the image the data are 1: |e|^2 > 0 and rho != 0 there, for the fast quotient
                    auto fill = [&](pair2 q) -> pair2 {
                        if (!BX && !BY) return q;
                        float a, b;
                        upk(q, a, b);
                        return pk(__uint_as_float((__float_as_uint(a) & m0) | (0x3f800000u & ~m0)),
                                  __uint_as_float((__float_as_uint(b) & m1) | (0x3f800000u & ~m1)));
                    };
                    auto LT = [&](const void *p) { return fill(VEC ? ld_pair<T>(p, o0) : pk(ldT<T>(p, o0), ldT<T>(p, o1))); };
                    auto LF = [&](const void *p) { return mask(VEC ? ld_pair<TF>(p, o0) : pk(ldT<TF>(p, o0), ldT<TF>(p, o1))); };
#pragma unroll
                    for (int k = 2 * C0; k < 6; ++k) y[r][k] = LF(A.a.in.f[F_P1 + k]);
#pragma unroll
                    for (int k = C0; k < 3; ++k) {
                        X[r][k] = LF(A.a.in.f[F_W + k]);
                        B[r][k] = LF(A.a.in.f[F_WB + k]);
                    }
                    const pair2 ix = LT(A.a.Ix), iy = LT(A.a.Iy);
                    G.ix[wid * R + r][lane] = ix;
                    G.iy[wid * R + r][lane] = iy;
                    G.it[wid * R + r][lane] = LT(A.a.It);
                    float e0, e1;
                    upk(fma2(iy, iy, fma2(ix, ix, bb2)), e0, e1);
                    odd = odd || !(fminf(e0, e1) > 0x1p-100f && fmaxf(e0, e1) < 0x1p40f);
                    G.rc[wid * R + r][lane] = pk(__frcp_rn(e0), __frcp_rn(e1));
                }
            };
            if (BX < 2 || A.vec) load(std::true_type{});
            else load(std::false_type{});
        }
        auto put_top = [&]() {
            if (wid > 0)
#pragma unroll
                for (int k = C0; k < 3; ++k) G.top[wid][k][lane] = B[0][k];
        };
        put_top();
        odd = __syncthreads_or(odd);
        float res = 0.f;
#pragma unroll 1
        for (int kk = 0; kk < A.ni; ++kk) {
            const bool last = kk == A.ni - 1;
            // ---- the dual step, top row first (the last row needs the warp below)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                pair2 g[6];
#pragma unroll
                for (int k = C0; k < 3; ++k) {
                    float a, b;
                    upk(B[r][k], a, b);
                    const float e = __shfl_down_sync(FULL, a, 1);
                    g[2 * k] = pk(BX == 2 ? keep(b - a, me0) : b - a, BX ? keep(e - b, me1) : e - b);
                }
                if (r == R - 1) {
                    __syncthreads();
#pragma unroll
                    for (int k = C0; k < 3; ++k) g[2 * k + 1] = sub2(wid < NW - 1 ? G.top[wid < NW - 1 ? wid + 1 : 0][k][lane] : 0ull, B[r][k]);
                } else {
#pragma unroll
                    for (int k = C0; k < 3; ++k) g[2 * k + 1] = sub2(B[r + 1 < R ? r + 1 : r][k], B[r][k]);
                }
                if (BY && (r < rfirst || r == rlast)) {
                    asm volatile("");
#pragma unroll
                    for (int k = C0; k < 3; ++k) g[2 * k + 1] = 0ull;
                }
                if (!std::is_same<TF, float>::value)
#pragma unroll
                    for (int k = 2 * C0; k < 6; ++k) y[r][k] = round2<TF>(y[r][k]);
                if (HAS_W) {
                    const pair2 t1 = fma2(tau2, g[0], y[r][0]), t2 = fma2(tau2, g[1], y[r][1]);
                    const pair2 f = ball_scale2(fma2(t1, t1, mul2(t2, t2)));
                    y[r][0] = mul2(t1, f);
                    y[r][1] = mul2(t2, f);
                }
                const pair2 t11 = fma2(tau2, g[2], y[r][2]), t12 = fma2(tau2, g[3], y[r][3]);
                const pair2 t21 = fma2(tau2, g[4], y[r][4]), t22 = fma2(tau2, g[5], y[r][5]);
                const pair2 f = ball_scale2(fma2(t11, t11, fma2(t12, t12, fma2(t21, t21, mul2(t22, t22)))));
                y[r][2] = mul2(t11, f);
                y[r][3] = mul2(t12, f);
                y[r][4] = mul2(t21, f);
                y[r][5] = mul2(t22, f);
            }
            if (wid < NW - 1)
#pragma unroll
                for (int k = C0; k < 3; ++k) G.bot[wid][k][lane] = y[R - 1][2 * k + 1];
            // ---- the primal step, bottom row first (row 0 needs the warp above): Z = X + sigma div y' in
            // place of Xbar, and rho(Z).  y is zero where its difference crosses the image's border and one pixel
            // outside on the west and north: it starts at zero and those differences are zero.
            pair2 rho[R];
            unsigned small = ~0u;  // least (2 |rho| - 1) as integers: zero wraps around
#pragma unroll
            for (int r = R - 1; r >= 0; --r) {
                if (r == 0) __syncthreads();
#pragma unroll
                for (int k = C0; k < 3; ++k) {
                    const pair2 n = r > 0 ? y[r > 0 ? r - 1 : 0][2 * k + 1] : wid > 0 ? G.bot[wid > 0 ? wid - 1 : 0][k][lane] : 0ull;
                    float a, b;
                    upk(y[r][2 * k], a, b);
                    const float wv = __shfl_up_sync(FULL, b, 1);
                    B[r][k] = fma2(sg2, sub2(add2(pk(a - wv, b - a), y[r][2 * k + 1]), n), X[r][k]);
                }
                pair2 q = G.it[wid * R + r][lane];
                if (HAS_W) q = fma2(beta2, B[r][0], q);
                rho[r] = fma2(G.iy[wid * R + r][lane], B[r][2], fma2(G.ix[wid * R + r][lane], B[r][1], q));
                float r0, r1;
                upk(rho[r], r0, r1);
                small = min(small, min(2 * __float_as_uint(r0) - 1, 2 * __float_as_uint(r1) - 1));
            }
            // ---- X' = Z + t e, t = -rho / |e|^2, or -+ sigma lambda where |rho| > sigma lambda |e|^2
            auto finish = [&](auto SLOW_) {
                constexpr bool SLOW = decltype(SLOW_)::value;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const pair2 ix = G.ix[wid * R + r][lane], iy = G.iy[wid * R + r][lane];
                    const pair2 e2 = fma2(iy, iy, fma2(ix, ix, bb2));
                    float r0, r1, s0, s1, q0, q1;
                    upk(rho[r], r0, r1);
                    upk(mul2(sl02, e2), s0, s1);
                    if (SLOW) {
                        float e0, e1;
                        upk(e2, e0, e1);
                        q0 = e0 <= 0.f ? 0.f : r0 < -s0 ? sl0 : r0 > s0 ? -sl0 : -r0 / e0;
                        q1 = e1 <= 0.f ? 0.f : r1 < -s1 ? sl0 : r1 > s1 ? -sl0 : -r1 / e1;
                    } else {  // |t| first, then the sign of -rho
                        const pair2 rc = G.rc[wid * R + r][lane], ne = neg2(e2);
                        pair2 q = mul2(rho[r], rc);
                        q = fma2(fma2(ne, q, rho[r]), rc, q);
                        q = fma2(fma2(ne, q, rho[r]), rc, q);
                        upk(q, q0, q1);
                        auto sgn = [](float m, float x) {
                            return __uint_as_float((__float_as_uint(m) & 0x7fffffffu) | (~__float_as_uint(x) & 0x80000000u));
                        };
                        q0 = sgn(fabsf(r0) > s0 ? sl0 : q0, r0);
                        q1 = sgn(fabsf(r1) > s1 ? sl0 : q1, r1);
                    }
                    const pair2 t = pk(q0, q1);
                    pair2 z[3] = {0ull, fma2(t, ix, B[r][1]), fma2(t, iy, B[r][2])};
                    if (HAS_W) z[0] = fma2(t, beta2, B[r][0]);
                    if (last && A.a.partials) {
                        const int fr = wid * R + r;
                        const pair2 dw = HAS_W ? sub2(z[0], X[r][0]) : 0ull, du = sub2(z[1], X[r][1]), dd = sub2(z[2], X[r][2]);
                        float p0, p1;
                        upk(fma2(dd, dd, fma2(du, du, mul2(dw, dw))), p0, p1);
                        if (fr >= A.offy && fr < A.offy + A.oh && ib + r < H && 2 * lane >= A.offx && 2 * lane < A.offx + A.ow) {
                            if (c < W) res += p0;
                            if (c + 1 < W) res += p1;
                        }
                    }
#pragma unroll
                    for (int k = C0; k < 3; ++k) {
                        B[r][k] = round2<TF>(sub2(add2(z[k], z[k]), X[r][k]));
                        X[r][k] = round2<TF>(z[k]);
                    }
                }
            };
            if (__any_sync(FULL, odd || small < 2 * 0x17800000u)) finish(std::true_type{});  // |rho| < 2^-80
            else finish(std::false_type{});
            if (!last) put_top();
        }
        // ---- store the tile
        const bool inx = 2 * lane >= A.offx && 2 * lane < A.offx + A.ow;
        const bool ok0 = inx && (!BX || c < W), ok1 = inx && (!BX || c + 1 < W);
        auto store = [&](auto f) {
            auto plane = [&](void *p, auto val) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int fr = wid * R + r, i = ib + r;
                    if (fr >= A.offy && fr < A.offy + A.oh && i < H) f(p, (size_t)i * P + c, val(r));
                }
            };
#pragma unroll
            for (int k = 2 * C0; k < 6; ++k) plane(A.a.out.f[F_P1 + k], [&](int r) { return y[r][k]; });
#pragma unroll
            for (int k = C0; k < 3; ++k) {
                plane(A.a.out.f[F_W + k], [&](int r) { return X[r][k]; });
                plane(A.a.out.f[F_WB + k], [&](int r) { return B[r][k]; });
            }
        };
        if (ok0 && ok1 && (BX < 2 || A.vec)) {
            store([](void *p, size_t o, pair2 q) { st_pair<TF>(p, o, q); });
        } else if (BX && (ok0 || ok1)) {
            store([&](void *p, size_t o, pair2 q) {
                if (ok0) stT<TF>(p, o, lo2(q));
                if (ok1) stT<TF>(p, o + 1, hi2(q));
            });
        }
        if (A.a.partials) {
            const double tot = block_sum((double)res, G.red);
            if (threadIdx.x == 0) A.a.partials[blockIdx.x] = tot;
        }
    }

    static __device__ __forceinline__ void run(const TileArgs &A) {
        extern __shared__ __align__(16) char smem_[];
        SH &G = *reinterpret_cast<SH *>(smem_);
        if (A.a.done && *A.a.done) return;  // the pair's warp met its stopping test
        const int lane = threadIdx.x & 31, wid = __shfl_sync(FULL, threadIdx.x >> 5, 0);
        const int bx = blockIdx.x % A.gx, by = blockIdx.x / A.gx;
        const int fj = bx * A.ow - A.offx, fi = by * A.oh - A.offy;
        if (fj >= 1 && fj + 64 <= A.a.g.W - 1 && A.vec) {
            if (fi >= 1 && fi + R * NW <= A.a.g.H - 1) body<0, false>(A, G, bx, by, lane, wid);
            else body<0, true>(A, G, bx, by, lane, wid);
        } else if (A.a.g.W % 2 == 0 && A.vec) {
            body<1, true>(A, G, bx, by, lane, wid);
        } else {
            body<2, true>(A, G, bx, by, lane, wid);
        }
    }
};

template <typename T, typename TF, bool HAS_W, int R>
__global__ void __launch_bounds__(NW * 32, 1) k_cp_tile(const __grid_constant__ TileArgs A) {
    Kernel<T, TF, HAS_W, R>::run(A);
}

template <typename T, typename TF, bool HAS_W, int R> void launch_r(const TileArgs &a, cudaStream_t s) {
    constexpr int SMEM = (int)sizeof(Shared<R>);
    static DeviceOnce once;
    once.run(current_device(), [] {
        return cudaFuncSetAttribute(k_cp_tile<T, TF, HAS_W, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    });
    k_cp_tile<T, TF, HAS_W, R><<<a.ntiles, NW * 32, SMEM, s>>>(a);
}

template <typename T, typename TF> void launch_m(const TileArgs &a, cudaStream_t s) {
    const bool has_w = a.a.k.beta != 0.f;
    switch (a.R) {
    case 2: return has_w ? launch_r<T, TF, true, 2>(a, s) : launch_r<T, TF, false, 2>(a, s);
    case 3: return has_w ? launch_r<T, TF, true, 3>(a, s) : launch_r<T, TF, false, 3>(a, s);
    default: return has_w ? launch_r<T, TF, true, 4>(a, s) : launch_r<T, TF, false, 4>(a, s);
    }
}

}  // namespace cptile
}  // namespace tvl1
