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
// The primal step divides by |e|^2, a constant of the pixel: by its reciprocal and remainder steps
// (k_quot2.cuh).  A warp that holds a pixel whose |e|^2 is outside (2^-100, 2^40), or a numerator below 2^-80,
// divides, and sets a flag by which the pair's later launches take a body of its own, whose quotients take any
// numerator and pixels without data (beta = 0 on a flat region): images with flat regions have such numerators
// wherever the illumination and the flow decay into them, and a launch is as slow as its slowest tile.  Measured
// over a solve (three warps of 40 iterations, four levels), in brackets where every such warp divided, and the
// kernel before this one: 640x480 with one half flat 1.20 ms (2.08, 1.73), textured 0.97 (0.97, 1.51); 1920x1080
// without beta, one half flat, 2.94 (2.64, 3.50).  So that this costs one branch per iteration and not one per
// row (a branch in a row keeps the rows from overlapping: 2.8 against 1.5 us per iteration at R = 4), the primal
// step first forms Z and rho of all rows, Z in the registers of the spent Xbar.
//
// Bound by latency and issue with three warps per SM quarter (some 240 clocks per row and warp), beside
// 4 to 6 us per launch for instruction fetch and the state's loads and stores.  Measured per iteration,
// and in brackets with the frame in shared memory and scalar instructions, which this replaced:
// 640x480 2.65 us (4.54), 320x240 1.22 (1.87), 160x120 1.07 (1.32), 3840x2160 76 (115).
#pragma once
#include <math.h>

#include <type_traits>

#include "k_cp_math.cuh"
#include "k_pack2.cuh"
#include "k_quot2.cuh"

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
    int any, met;           // the pair takes the quotients' form for any numerator; the usual form had to divide
};

template <typename T, typename TF, bool HAS_W, int R> struct Kernel {
    static constexpr int C0 = HAS_W ? 0 : 1;
    using SH = Shared<R>;

    // BX, BY: as the ADMM tile kernel's.  ANY: the quotients' form for any numerator, with divisions where the divisors
    // need them.  False (the usual form only): the pair takes the other form; nothing is stored.
    template <int BX, bool BY, bool ANY>
    static __device__ __forceinline__ bool body(const TileArgs &A, SH &G, int bx, int by, int lane, int wid) {
        const int H = A.a.g.H, W = A.a.g.W, P = A.a.g.pitch;
        const int c = bx * A.ow - A.offx + 2 * lane, ib = by * A.oh - A.offy + wid * R;
        const unsigned me0 = mask_of(c >= 0 && c < W - 1), me1 = mask_of(c + 1 >= 0 && c + 1 < W - 1);
        const int rlast = __shfl_sync(FULL, H - 1 - ib, 0), rfirst = __shfl_sync(FULL, -ib, 0);
        pair2 y[R][6], X[R][3], B[R][3];
        const float beta = A.a.k.beta, lam = A.a.k.lambda, sg = A.a.k.cp_sigma, sl0 = sg * lam;
        const pair2 tau2 = bc2(A.a.k.cp_tau), sg2 = bc2(sg), beta2 = bc2(beta), bb2 = bc2(beta * beta), sl02 = bc2(sl0);
        // (set by another block of this launch, either will do; stored behind the frame's loads)
        const int any = !ANY && threadIdx.x == 0 && A.tiny ? *(const volatile int *)A.tiny : 0;
        bool odd = !(sl0 < 0x1p20f);  // quotients outside the range of the reciprocal's
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
                    const pair2 it = LT(A.a.It), e2 = fma2(iy, iy, fma2(ix, ix, bb2));
                    G.it[wid * R + r][lane] = it;
                    odd = odd || prox_unusual(e2);
                    G.rc[wid * R + r][lane] = pk(__frcp_rn(lo2(e2)), __frcp_rn(hi2(e2)));
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
        if (threadIdx.x == 0) {
            G.met = 0;
            G.any = any;
        }
        odd = __syncthreads_or(odd);
        if (!ANY && G.any) return false;
        float res = 0.f;
        if (ANY && odd) {  // by what: a pixel without data takes a zero reciprocal
            bool bad = !(sl0 < 0x1p20f);
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const pair2 ix = G.ix[wid * R + r][lane], iy = G.iy[wid * R + r][lane], e2 = fma2(iy, iy, fma2(ix, ix, bb2));
                bad = bad || !prox_empty(e2, ix, iy, G.it[wid * R + r][lane], beta);
                G.rc[wid * R + r][lane] = prox_rcp2(e2);
            }
            odd = __any_sync(FULL, bad);
        }
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
                    const pair2 thr = mul2(sl02, e2);
                    const pair2 t = SLOW ? prox_div2(rho[r], e2, thr, sl0)
                                         : prox_quot2<ANY>(rho[r], e2, G.rc[wid * R + r][lane], thr, sl0);
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
            if (__any_sync(FULL, odd || (!ANY && small < QUOT_SMALL_BITS))) {
                if (!ANY) G.met = 1;
                finish(std::true_type{});
            } else {
                finish(std::false_type{});
            }
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
        return true;
    }

    static __device__ __forceinline__ void run(const TileArgs &A) {
        extern __shared__ __align__(16) char smem_[];
        SH &G = *reinterpret_cast<SH *>(smem_);
        if (A.a.done && *A.a.done) return;  // the pair's warp met its stopping test
        const int lane = threadIdx.x & 31, wid = __shfl_sync(FULL, threadIdx.x >> 5, 0);
        const int bx = blockIdx.x % A.gx, by = blockIdx.x / A.gx;
        const int fj = bx * A.ow - A.offx, fi = by * A.oh - A.offy;
        bool ok;
        if (fj >= 1 && fj + 64 <= A.a.g.W - 1 && A.vec) {
            if (fi >= 1 && fi + R * NW <= A.a.g.H - 1) ok = body<0, false, false>(A, G, bx, by, lane, wid);
            else ok = body<0, true, false>(A, G, bx, by, lane, wid);
        } else if (A.a.g.W % 2 == 0 && A.vec) {
            ok = body<1, true, false>(A, G, bx, by, lane, wid);
        } else {
            ok = body<2, true, false>(A, G, bx, by, lane, wid);
        }
        // (a second body of the other form, for tiles inside the image, made the usual one 1% slower)
        if (!ok) body<2, true, true>(A, G, bx, by, lane, wid);
        else if (lane == 0 && *(volatile int *)&G.met && A.tiny) *A.tiny = 1;  // the pair's next launches take the other form
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
