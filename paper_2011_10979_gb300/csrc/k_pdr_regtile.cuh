// k_pdr_regtile.cuh -- several pDR iterations with one symmetric Gauss-Seidel sweep (Sec. 3.1.2, eq. pDR: red,
// black, red) in one launch, the state in registers, for a single pair's larger levels.
//
// A block of TILE_WARPS warps holds a frame of 64 columns by 48 rows: each lane two neighbouring columns (a
// register pair per plane of X, ybar and the right-hand side b) in four rows; Xbar and the data stay in
// the shared memory that the copies (TMA, zeros outside the image) leave them in.  East and west
// neighbours travel by shuffle, south and north ones in registers and, between the warps' bands, through
// shared memory, across four block barriers per iteration (the rows that need no other band come first).
// The frames start at even rows and columns, so a pair's even (odd) column is red in the band's even
// (odd) rows whatever the warp, and a half-sweep updates one half of each pair in place.
// An iteration at a pixel needs the state three pixels around it and X one more on the east and south
// (ybar' needs X' there; X' two half-sweeps of black and red neighbours, which need X and b; b the
// ybar one pixel west and north), so ni iterations take halos of 3 ni and 3 ni + 1 pixels.
//
// The divisor of a Gauss-Seidel update, 1 + sigma tau n, depends on the number n of neighbours only: the
// quotient is formed from the reciprocal and its error (one FMA more exact than the reciprocal alone, so
// faithful) with one remainder step, which makes it correctly rounded, and the quotient by |e|^2 as in the ALG1
// tile kernel (k_quot2.cuh).  So every stage rounds as the kernels of k_pdr.cu do, X to its storage type after every
// half-sweep, and ni iterations here are ni launches of k_pdr_tile, value for value.  The usual form of the body
// needs divisors in (2^-100, 2^40), state below 2^60 and numerators that are zero or at least 2^-80.  A block whose
// tile breaks that starts over with a body whose quotients take any numerator (and which divides where
// the divisors or the state are to blame), and sets a flag by which the pair's later launches take that body at
// once: images with regions without data have such numerators wherever the flow decays into them, and pixels
// without a divisor with beta = 0.  Measured at 640x480 (three warps of 40 iterations, four levels), in brackets
// where every warp that met one divided in place, and k_pdr_tile: textured 2.71 ms (2.81, 3.58), one half
// flat 3.41 (6.81, 3.84), a textured box on an empty background 3.35 (7.28, 3.86).
//
// What bounds it: with one iteration per launch, the state's traffic through L2 (184 KB in and 147 KB out
// per SM) and the fetch of straight-line code, most of a launch's 9.0 us at 640x480, and per iteration issue and
// latency with three warps per SM quarter (some 330 instructions per row of a warp).  A tile on the image's border costs
// no more than the others, since a launch of one round is as slow as its slowest tile: pixels outside
// have a zero reciprocal, which keeps X zero there, and ybar is zero across the border (masks and
// branches instead: 1.0 us more at 640x480).  Pairs of rows in packed arithmetic took more moves than it saved.
// Measured per iteration, in brackets k_pdr_tile: 240x180 3.8 us (5.6), 320x240 3.9 (5.8), 640x480 9.0
// (13.4), 1024x436 10.5 (19.3), 3840x2160 188 (335).
#pragma once
#include <cuda.h>
#include <math.h>

#include <type_traits>

#include "k_mbar.cuh"
#include "k_pack2.cuh"
#include "k_pdr_math.cuh"
#include "k_quot2.cuh"

namespace tvl1 {

void pdr_tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s);
void pdr_tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s);

namespace pdrtile {

constexpr unsigned FULL = 0xffffffffu;

constexpr int NW = TILE_WARPS, R = 4, FH = NW * R;
static_assert(FH == TILE_STAGED_HEIGHT, "the tensor maps' boxes");

struct Shared {
    float top[NW][2][3][32], bot[NW][2][3][32];  // X of the bands' first and last rows, per column of the pair
    pair2 yb[NW][3][32];                         // the y-components of ybar of the last rows
    // per frame row and number of horizontal neighbours (3: a column outside the image): the divisor 1 + sigma tau n,
    // its reciprocal and the reciprocal's error; the latter two zero outside the image
    float4 gs[FH][4];
    double red[32];
    unsigned long long full;                     // the mbarrier the copies complete on
    // the pair takes the quotients' form for any numerator; numerators that need it were met; a wait ran out
    int any, met, dead;
};

// The frame in shared memory, as the copies leave it: Xbar and the data, which stay there, then X and ybar,
// which go to registers; their place then holds each thread's own X and b (where a warp divides, below) and
// 1 / |e|^2.  A copy must start on a 16-byte boundary, i.e. at a multiple of 4 FP32 or 8 16-bit columns;
// frames start at multiples of 4, so rows of 16-bit planes are 8 columns wider and start up to 4 early.
template <typename T, typename TF> struct Stage {
    static constexpr int wid_of(int bytes) { return bytes == 4 ? 64 : 72; }
    static constexpr int WT = wid_of(sizeof(T)), WTF = wid_of(sizeof(TF));
    static constexpr int up(int x) { return (x + 127) / 128 * 128; }
    static constexpr int mx(int a, int b) { return a > b ? a : b; }
    static constexpr int pt = FH * WT * (int)sizeof(T), ptf = FH * WTF * (int)sizeof(TF);
    static constexpr int xbar = 0, data = up(3 * ptf), x = data + up(3 * pt), y = x + up(3 * ptf),
                         bytes = mx(y + up(6 * pt), x + 7 * FH * 256);
    static constexpr int own = x, own_b = x + 3 * FH * 256, own_rc = x + 6 * FH * 256;
};

template <typename T, typename TF, bool HAS_W> struct Kernel {
    static_assert(R % 2 == 0, "a row's colours must not depend on the warp");
    static constexpr int C0 = HAS_W ? 0 : 1;
    using ST = Stage<T, TF>;
    static constexpr int NF = HAS_W ? 3 : 2, ND = HAS_W ? 6 : 4;  // planes copied of X, Xbar and of ybar

    // ANY: the quotients' form for any numerator, with divisions where the divisors need them.  False (the usual form
    // only): the tile holds what needs the other form; nothing is stored.
    template <int BX, bool BY, bool ANY>
    static __device__ __forceinline__ bool body(const TileArgs &A, Shared &G, char *stage, int bx, int by, int lane, int wid, float sg,
                                                float ta, unsigned phase) {
        const int H = A.a.g.H, W = A.a.g.W, P = A.a.g.pitch;
        const int c = bx * A.ow - A.offx + 2 * lane, ib = by * A.oh - A.offy + wid * R;  // both even
        const unsigned me0 = mask_of(c >= 0 && c < W - 1), me1 = mask_of(c + 1 >= 0 && c + 1 < W - 1);
        const bool in0 = !BX || (c >= 0 && c < W), in1 = !BX || (c + 1 >= 0 && c + 1 < W);
        const int rlast = __shfl_sync(FULL, H - 1 - ib, 0), rfirst = __shfl_sync(FULL, -ib, 0);  // the image's rows in the band
        const float beta = A.a.k.beta, st = sg * ta, sl0 = sg * A.a.k.lambda;
        const pair2 sg2 = bc2(sg), beta2 = bc2(beta), bb2 = bc2(beta * beta), sl02 = bc2(sl0), t22 = bc2(2.f * ta), nta2 = bc2(-ta);
        pair2 y[R][6], X[R][3], b[R][3];
        // quotients outside the range of the reciprocal's: in the usual form of any kind, in the other those of the
        // half-sweeps (odd) and of the proximal step (oddp)
        bool odd = !(st < 0x1p37f && (ANY || sl0 < 0x1p20f)), oddp = ANY && !(sl0 < 0x1p20f), unusual = false;
        float big = 0.f;
        // this thread's pixel pairs in the stage
        const int x0 = c - 2 * lane, at = 2 * lane + (sizeof(T) == 4 ? 0 : x0 & 7), af = 2 * lane + (sizeof(TF) == 4 ? 0 : x0 & 7);
        auto dat = [&](int k, int r) { return ld_pair<T>(stage + ST::data, (k * FH + wid * R + r) * ST::WT + at); };
        auto xb_at = [&](int k, int r) { return ((k - C0) * FH + wid * R + r) * ST::WTF + af; };
        auto xb = [&](int k, int r) { return ld_pair<TF>(stage + ST::xbar, xb_at(k, r)); };
        auto own = [&](int base, int k, int r) -> pair2 & {
            return *reinterpret_cast<pair2 *>(stage + base + ((k * FH + wid * R + r) * 32 + lane) * 8);
        };
        if (!mbar_wait(&G.full, phase, A.wait_ns, A.timeout)) {  // reported; the copies in flight have the same time again
            G.dead = 1;
            if (A.timeout) *A.timeout = 1;
            mbar_wait(&G.full, phase, A.wait_ns, nullptr);
        }
        pair2 rcp[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int fr = wid * R + r;
#pragma unroll
            for (int k = 2 * C0; k < 6; ++k) y[r][k] = ld_pair<T>(stage + ST::y, ((k - 2 * C0) * FH + fr) * ST::WT + at);
#pragma unroll
            for (int k = C0; k < 3; ++k) {
                X[r][k] = ld_pair<TF>(stage + ST::x, xb_at(k, r));
                float x0, x1, q0, q1;
                upk(X[r][k], x0, x1);
                upk(xb(k, r), q0, q1);
                big = fmaxf(fmaxf(big, fmaxf(fabsf(x0), fabsf(x1))), fmaxf(fabsf(q0), fabsf(q1)));
            }
            const pair2 ix = dat(0, r), iy = dat(1, r);
            const pair2 e2 = fma2(iy, iy, fma2(ix, ix, bb2));
            auto usual = [](float e) { return e > 0x1p-100f && e < 0x1p40f; };
            const bool in = !BY || (ib + r >= 0 && ib + r < H);
            unusual = unusual || (in && ((in0 && !usual(lo2(e2))) || (in1 && !usual(hi2(e2)))));
            rcp[r] = prox_rcp2(e2);  // (zero outside the image without beta)
        }
        odd = odd || big > 0x1p60f || (!ANY && unusual);
        if (threadIdx.x < FH * 4) {
            const int fr = threadIdx.x / 4, n = threadIdx.x & 3, i = by * A.oh - A.offy + fr;
            const bool in = i >= 0 && i < H && n < 3;
            const float dv = fmaf(st, (float)(n + (i > 0) + (i < H - 1)), 1.f), q = __frcp_rn(dv);
            G.gs[fr][n] = in ? make_float4(dv, q, fmaf(-dv, q, 1.f) * q, 0.f) : make_float4(1.f, 0.f, 0.f, 0.f);
        }
        // Row 0 of a band is even and row R - 1 odd: their red (black) pixels are the pairs' even and odd
        // (odd and even) columns.
        auto put = [&](auto COL_) {
            constexpr int col = decltype(COL_)::value;
#pragma unroll
            for (int k = C0; k < 3; ++k) {
                G.top[wid][col][k][lane] = col ? hi2(X[0][k]) : lo2(X[0][k]);
                G.bot[wid][col ^ 1][k][lane] = col ? lo2(X[R - 1][k]) : hi2(X[R - 1][k]);
            }
        };
        auto put_y = [&]() {
            if (wid < NW - 1)
#pragma unroll
                for (int k = C0; k < 3; ++k) G.yb[wid][k][lane] = y[R - 1][2 * k + 1];
        };
        put(std::integral_constant<int, 1>{});
        put_y();
        odd = __syncthreads_or(odd);  // the places of X and ybar in the stage are free
        if (!ANY && odd) return false;
#pragma unroll
        for (int r = 0; r < R; ++r) own(ST::own_rc, 0, r) = rcp[r];
        if (ANY) {
            oddp = oddp || odd;
            if (__any_sync(FULL, unusual))
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    const pair2 ix = dat(0, r), iy = dat(1, r);
                    oddp = oddp || !prox_empty(fma2(iy, iy, fma2(ix, ix, bb2)), ix, iy, dat(2, r), beta);
                }
            oddp = __any_sync(FULL, oddp);
        }
        // the columns' entries in a row of the table
        const int nx0 = !BX ? 2 : !in0 ? 3 : (c > 0) + (c < W - 1), nx1 = !BX ? 2 : !in1 ? 3 : (c + 1 > 0) + (c + 1 < W - 1);
        const float4 mid = G.gs[wid * R][2];
        // One Gauss-Seidel update of the pixels of a colour in row r, from its rows above and below
        unsigned small;  // least (2 |numerator| - 1) as integers since it was reset: zero wraps around
        auto update = [&](bool odd_col, int quot, float4 t, pair2 x, pair2 n, pair2 s, pair2 bb) -> pair2 {
            float x0, x1, acc;
            upk(x, x0, x1);
            if (odd_col) acc = x0 + __shfl_down_sync(FULL, x0, 1);
            else acc = __shfl_up_sync(FULL, x1, 1) + x1;
            acc = (acc + (odd_col ? hi2(n) : lo2(n))) + (odd_col ? hi2(s) : lo2(s));
            const float num = fmaf(st, acc, odd_col ? hi2(bb) : lo2(bb));
            float q;
            if (quot == 2) {
                q = t.y == 0.f ? 0.f : num / t.x;
            } else {  // a zero reciprocal keeps X zero outside the image
                const QuotScale sc = quot == 1 ? quot_scale(num) : QuotScale{1.f, 1.f};
                if (!ANY) small = min(small, 2 * __float_as_uint(num) - 1);
                const float m = quot == 1 ? num * sc.up : num;
                q = fmaf(m, t.y, m * t.z);
                q = fmaf(fmaf(-t.x, q, m), t.y, q);
                if (quot == 1) q = quot_unscale(q, m, t.x, sc);
            }
            q = storage_round<TF>(q);
            return odd_col ? pk(x0, q) : pk(q, x1);
        };
        auto edge = [&](float (*p)[3][32], int k, bool odd_col) -> pair2 { return bc2(p[odd_col][k][lane]); };
        const int up = wid > 0 ? wid - 1 : 0, dn = wid < NW - 1 ? wid + 1 : 0;
        auto sweep = [&](auto COL_, int r0, int r1) {
            constexpr int col = decltype(COL_)::value;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r < r0 || r >= r1) continue;
                const bool odd_col = (r & 1) ^ col;  // the pair's odd column has the colour
                const float4 t = BX || BY ? G.gs[wid * R + r][odd_col ? nx1 : nx0] : mid;
#pragma unroll
                for (int k = C0; k < 3; ++k)
                    X[r][k] = update(odd_col, ANY ? 1 : 0, t, X[r][k],
                                     r > 0 ? X[r > 0 ? r - 1 : 0][k] : wid > 0 ? edge(G.bot[up], k, odd_col) : 0ull,
                                     r < R - 1 ? X[r < R - 1 ? r + 1 : r][k] : wid < NW - 1 ? edge(G.top[dn], k, odd_col) : 0ull,
                                     b[r][k]);
            }
        };
        // the same with divisions, for all rows: rolled, through shared memory, since it runs seldom
        auto sweep_slow = [&](int col) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int k = C0; k < 3; ++k) {
                    own(ST::own, k, r) = X[r][k];
                    own(ST::own_b, k, r) = b[r][k];
                }
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const bool odd_col = (r & 1) ^ col;
                const float4 t = G.gs[wid * R + r][odd_col ? nx1 : nx0];
#pragma unroll 1
                for (int k = C0; k < 3; ++k) {
                    const pair2 n = r > 0 ? own(ST::own, k, r - 1) : wid > 0 ? edge(G.bot[up], k, odd_col) : 0ull;
                    const pair2 s = r < R - 1 ? own(ST::own, k, r + 1) : wid < NW - 1 ? edge(G.top[dn], k, odd_col) : 0ull;
                    own(ST::own, k, r) = update(odd_col, 2, t, own(ST::own, k, r), n, s, own(ST::own_b, k, r));
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int k = C0; k < 3; ++k) X[r][k] = own(ST::own, k, r);
        };
        auto half_sweep = [&](auto COL_, bool wait) {
            small = ~0u;
            sweep(COL_, 1, R - 1);
            if (wait) __syncthreads();
            sweep(COL_, 0, 1);
            sweep(COL_, R - 1, R);
            if (ANY) {
                if (odd) sweep_slow(decltype(COL_)::value);
            } else if (small < QUOT_SMALL_BITS) {
                G.met = 1;
            }
            put(COL_);
        };
        using RED = std::integral_constant<int, 0>;
        using BLACK = std::integral_constant<int, 1>;
        double res = 0.0;
#pragma unroll 1
        for (int kk = 0; kk < A.ni; ++kk) {
            const bool last = kk == A.ni - 1;
            // ---- b = Xbar + sigma div ybar.  ybar is zero where its difference crosses the image's border and
            // outside: it starts at zero and those differences are zero.
#pragma unroll
            for (int r = R - 1; r >= 0; --r) {
                if (r == 0 && kk > 0) __syncthreads();
#pragma unroll
                for (int k = C0; k < 3; ++k) {
                    const pair2 n = r > 0 ? y[r > 0 ? r - 1 : 0][2 * k + 1] : wid > 0 ? G.yb[wid > 0 ? wid - 1 : 0][k][lane] : 0ull;
                    float a, e;
                    upk(y[r][2 * k], a, e);
                    const float wv = __shfl_up_sync(FULL, e, 1);
                    b[r][k] = fma2(sg2, sub2(add2(pk(a - wv, e - a), y[r][2 * k + 1]), n), xb(k, r));
                }
            }
            half_sweep(RED{}, false);
            half_sweep(BLACK{}, true);
            half_sweep(RED{}, true);
            // ---- Z = 2 X - Xbar and rho(Z), Z in the registers of b
            pair2 rho[R];
            small = ~0u;
#pragma unroll
            for (int r = 0; r < R; ++r) {
#pragma unroll
                for (int k = C0; k < 3; ++k) b[r][k] = sub2(add2(X[r][k], X[r][k]), xb(k, r));
                pair2 q = dat(2, r);
                if (HAS_W) q = fma2(beta2, b[r][0], q);
                rho[r] = fma2(dat(1, r), b[r][2], fma2(dat(0, r), b[r][1], q));
                float r0, r1;
                upk(rho[r], r0, r1);
                small = min(small, min(2 * __float_as_uint(r0) - 1, 2 * __float_as_uint(r1) - 1));
            }
            // ---- Xbar' = Xbar + (Z + t e) - X, t = -rho / |e|^2, or -+ sigma lambda where |rho| > sigma lambda |e|^2
            auto xbar = [&](auto SLOW_, int r, pair2 rho, const pair2 *x, const pair2 *zr) {
                constexpr bool SLOW = decltype(SLOW_)::value;
                const pair2 ix = dat(0, r), iy = dat(1, r);
                const pair2 e2 = fma2(iy, iy, fma2(ix, ix, bb2)), thr = mul2(sl02, e2);
                const pair2 t = SLOW ? prox_div2(rho, e2, thr, sl0) : prox_quot2<ANY>(rho, e2, own(ST::own_rc, 0, r), thr, sl0);
                pair2 z[3] = {0ull, fma2(t, ix, zr[1]), fma2(t, iy, zr[2])};
                if (HAS_W) z[0] = fma2(t, beta2, zr[0]);
#pragma unroll
                for (int k = C0; k < 3; ++k) st_pair<TF>(stage + ST::xbar, xb_at(k, r), sub2(add2(xb(k, r), z[k]), x[k]));
            };
            if (!ANY && small < QUOT_SMALL_BITS) G.met = 1;
            if (ANY && oddp) {
                // (the place of rho: that of 1 / |e|^2, which is formed again)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    own(ST::own_rc, 0, r) = rho[r];
#pragma unroll
                    for (int k = C0; k < 3; ++k) {
                        own(ST::own, k, r) = X[r][k];
                        own(ST::own_b, k, r) = b[r][k];
                    }
                }
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    pair2 x[3] = {0ull, 0ull, 0ull}, z[3] = {0ull, 0ull, 0ull};
#pragma unroll
                    for (int k = C0; k < 3; ++k) x[k] = own(ST::own, k, r), z[k] = own(ST::own_b, k, r);
                    xbar(std::true_type{}, r, own(ST::own_rc, 0, r), x, z);
                    const pair2 e2 = fma2(dat(1, r), dat(1, r), fma2(dat(0, r), dat(0, r), bb2));
                    own(ST::own_rc, 0, r) = prox_rcp2(e2);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) xbar(std::false_type{}, r, rho[r], X[r], b[r]);
            }
            // ---- ybar' = P(ybar + 2 tau grad X) - tau grad X
#pragma unroll
            for (int r = 0; r < R; ++r) {
                pair2 g[6];
                if (r == R - 1) __syncthreads();
#pragma unroll
                for (int k = C0; k < 3; ++k) {
                    float a, e;
                    upk(X[r][k], a, e);
                    const float ev = __shfl_down_sync(FULL, a, 1);
                    g[2 * k] = pk(BX ? keep(e - a, me0) : e - a, BX ? keep(ev - e, me1) : ev - e);
                    pair2 s;
                    if (r < R - 1) s = X[r < R - 1 ? r + 1 : r][k];
                    else s = wid < NW - 1 ? pk(G.top[wid < NW - 1 ? wid + 1 : 0][0][k][lane], G.top[wid < NW - 1 ? wid + 1 : 0][1][k][lane]) : 0ull;
                    g[2 * k + 1] = sub2(s, X[r][k]);
                }
                if (BY && (r < rfirst || r >= rlast)) {
                    asm volatile("");
#pragma unroll
                    for (int k = C0; k < 3; ++k) g[2 * k + 1] = 0ull;
                }
                if (HAS_W) {
                    const pair2 a1 = fma2(t22, g[0], y[r][0]), a2 = fma2(t22, g[1], y[r][1]);
                    const pair2 f = ball_scale2(fma2(a1, a1, mul2(a2, a2)));
                    y[r][0] = round2<T>(fma2(nta2, g[0], mul2(a1, f)));
                    y[r][1] = round2<T>(fma2(nta2, g[1], mul2(a2, f)));
                }
                const pair2 b11 = fma2(t22, g[2], y[r][2]), b12 = fma2(t22, g[3], y[r][3]);
                const pair2 b21 = fma2(t22, g[4], y[r][4]), b22 = fma2(t22, g[5], y[r][5]);
                const pair2 f = ball_scale2(fma2(b11, b11, fma2(b12, b12, fma2(b21, b21, mul2(b22, b22)))));
                y[r][2] = round2<T>(fma2(nta2, g[2], mul2(b11, f)));
                y[r][3] = round2<T>(fma2(nta2, g[3], mul2(b12, f)));
                y[r][4] = round2<T>(fma2(nta2, g[4], mul2(b21, f)));
                y[r][5] = round2<T>(fma2(nta2, g[5], mul2(b22, f)));
                if (A.a.partials) {  // one iteration: X^k is the input
                    const int fr = wid * R + r;
                    if (fr >= A.offy && fr < A.offy + A.oh && ib + r < H && 2 * lane >= A.offx && 2 * lane < A.offx + A.ow) {
#pragma unroll
                        for (int k = C0; k < 3; ++k) {
                            float d0, d1;
                            upk(X[r][k], d0, d1);
                            const size_t o = (size_t)(ib + r) * P + c;
                            if (c < W) res += (double)(d0 -= ldT<TF>(A.a.in.f[F_W + k], o)) * d0;
                            if (c + 1 < W) res += (double)(d1 -= ldT<TF>(A.a.in.f[F_W + k], o + 1)) * d1;
                        }
                    }
                }
            }
            if (!last) put_y();
        }
        // (set before the last barrier)
        if (!ANY && *(volatile int *)&G.met) return false;
        // ---- store the tile
        const bool inx = 2 * lane >= A.offx && 2 * lane < A.offx + A.ow;
        const bool ok0 = inx && (!BX || c < W), ok1 = inx && (!BX || c + 1 < W);
        auto store = [&](auto ST_, auto SF_) {
            auto plane = [&](auto f, void *p, auto val) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int fr = wid * R + r, i = ib + r;
                    if (fr >= A.offy && fr < A.offy + A.oh && i < H) f(p, (size_t)i * P + c, val(r));
                }
            };
#pragma unroll
            for (int k = 2 * C0; k < 6; ++k) plane(ST_, A.a.out.f[F_P1 + k], [&](int r) { return y[r][k]; });
#pragma unroll
            for (int k = C0; k < 3; ++k) {
                plane(SF_, A.a.out.f[F_W + k], [&](int r) { return X[r][k]; });
                plane(SF_, A.a.out.f[F_WB + k], [&](int r) { return xb(k, r); });
            }
        };
        if (ok0 && ok1) {
            store([](void *p, size_t o, pair2 q) { st_pair<T>(p, o, q); },
                  [](void *p, size_t o, pair2 q) { st_pair<TF>(p, o, q); });
        } else if (BX && (ok0 || ok1)) {
            store(
                [&](void *p, size_t o, pair2 q) {
                    if (ok0) stT<T>(p, o, lo2(q));
                    if (ok1) stT<T>(p, o + 1, hi2(q));
                },
                [&](void *p, size_t o, pair2 q) {
                    if (ok0) stT<TF>(p, o, lo2(q));
                    if (ok1) stT<TF>(p, o + 1, hi2(q));
                });
        }
        if (A.a.partials) {
            const double tot = block_sum(res, G.red);
            if (threadIdx.x == 0) A.a.partials[blockIdx.x] = tot;
        }
        return true;
    }

    static __device__ __forceinline__ void run(const TileArgs &A) {
        extern __shared__ __align__(128) char smem_[];
        char *stage = smem_;
        Shared &G = *reinterpret_cast<Shared *>(smem_ + ST::bytes);
        if (A.a.done && *A.a.done) return;  // the pair's warp met its stopping test
        const int lane = threadIdx.x & 31, wid = __shfl_sync(FULL, threadIdx.x >> 5, 0);
        const int bx = blockIdx.x % A.gx, by = blockIdx.x / A.gx;
        const int fj = bx * A.ow - A.offx, fi = by * A.oh - A.offy;
        auto copy = [&]() {
            mbar_expect(&G.full, 2 * NF * ST::ptf + (ND + 3) * ST::pt);
            const int xf = sizeof(TF) == 4 ? fj : fj & ~7, xt = sizeof(T) == 4 ? fj : fj & ~7;
            if (blockIdx.x != A.withhold) {
                tma_load(stage + ST::x, A.maps, xf, fi, &G.full);
                tma_load(stage + ST::y, A.maps + 1, xt, fi, &G.full);
                tma_load(stage + ST::data, A.maps + 2, xt, fi, &G.full);
                tma_load(stage + ST::xbar, A.maps + 3, xf, fi, &G.full);
            }
        };
        if (threadIdx.x == 0) {
            mbar_init(&G.full, 1);
            mbar_init_fence();
            copy();
        }
        // the launch's scalars, while the copies are on their way
        float sg, ta;
        pdr_steps(A.a.k, A.a.ms_max, sg, ta);
        if (threadIdx.x == 0) {
            G.met = G.dead = 0;
            G.any = A.tiny ? *(const volatile int *)A.tiny : 0;  // (set by another block of this launch, either will do)
        }
        __syncthreads();
        unsigned phase = 0;
        if (!G.any) {
            bool ok;
            if (fj >= 1 && fj + 64 <= A.a.g.W - 1) {
                if (fi >= 1 && fi + FH <= A.a.g.H - 1) ok = body<0, false, false>(A, G, stage, bx, by, lane, wid, sg, ta, 0);
                else ok = body<0, true, false>(A, G, stage, bx, by, lane, wid, sg, ta, 0);
            } else if (A.a.g.W % 2 == 0) {
                ok = body<1, true, false>(A, G, stage, bx, by, lane, wid, sg, ta, 0);
            } else {
                ok = body<2, true, false>(A, G, stage, bx, by, lane, wid, sg, ta, 0);
            }
            if (ok || *(volatile int *)&G.dead) return;
            // the frame once more; the pair's next launches start with the other form
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (threadIdx.x == 0) {
                copy();
                if (A.tiny) *A.tiny = 1;
            }
            phase = 1;
        }
        body<2, true, true>(A, G, stage, bx, by, lane, wid, sg, ta, phase);
    }
};

template <typename T, typename TF, bool HAS_W>
__global__ void __launch_bounds__(NW * 32, 1) k_pdr_regtile(const __grid_constant__ TileArgs A) {
    Kernel<T, TF, HAS_W>::run(A);
}

template <typename T, typename TF, bool HAS_W> void launch_w(const TileArgs &a, cudaStream_t s) {
    constexpr int SMEM = (int)sizeof(Shared) + Stage<T, TF>::bytes;
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static DeviceOnce once;
    once.run(current_device(), [] {
        return cudaFuncSetAttribute(k_pdr_regtile<T, TF, HAS_W>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    });
    k_pdr_regtile<T, TF, HAS_W><<<a.ntiles, NW * 32, SMEM, s>>>(a);
}

template <typename T, typename TF> void launch_m(const TileArgs &a, cudaStream_t s) {
    a.a.k.beta != 0.f ? launch_w<T, TF, true>(a, s) : launch_w<T, TF, false>(a, s);
}

}  // namespace pdrtile
}  // namespace tvl1
