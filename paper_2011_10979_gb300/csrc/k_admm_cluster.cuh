// k_admm_cluster.cuh -- level-resident engine of the ADMM methods on small levels (Sec. 3.1.1, eq.
// rpADMMI / rpADMMII / Zach-pADMM): one thread-block cluster keeps the whole level in registers and
// runs every inner iteration of one warp, with the stopping test, in a single launch.
//
// The level is cut into gx x gy tiles of ow x oh pixels, one per CTA; a CTA's frame is its tile and a
// halo of HALO pixels on the sides where the image goes on, one or two frame rows per warp, two
// neighbouring columns per lane (one 64-bit register pair per plane).  The state of an iteration at a
// pixel, div y among it, is a function of the state one pixel around it, so HALO iterations run on a
// frame without anything from outside; then every CTA sends the pixels that its neighbours hold in
// their halos straight into the neighbours' shared memory (st.async, counted by the receiver's
// mbarrier), and the warps with halo pixels wait for theirs.  The inbox is doubled: what arrives for
// the exchange after the next was sent by neighbours that have this CTA's next one, which it
// sends after reading its inbox.
// Within the CTA east and west neighbours travel by shuffle and north and south ones through shared
// memory, ordered between each two neighbouring warps by named barriers.
//
// What bounds it: the chain of one iteration (some 700 clocks with one warp per SM quarter: exchange of
// rows, two reductions to the unit ball, the projection of s), and with it the number of rows per SM
// quarter (0.33 us per iteration with 4 rows, 0.44 with 8, 0.70 with 16 in two rows per warp), hence few
// rows and a small halo; and the exchange, paid every second iteration (0.5 us: distributed shared memory
// takes some 20 bytes per clock and CTA).  A cluster barrier in place of the mbarriers waits for the
// stores' completion: 0.82 us per iteration at 64x48 against 0.73.  Measured per iteration, in brackets
// the engine that keeps the level in shared memory with two cluster barriers per iteration
// (k_resident.cu), which this replaced: 40x30 0.63 us (1.04), 64x48 0.72 (1.06), 80x60 1.02 (1.34),
// 128x55 1.11 (1.58 on the tile kernel), 120x90 1.12 (1.36 on it).  Sending the duals before the rest,
// as soon as they are final, was slower (1.18 at 80x60).
// The per-pixel arithmetic is that of the row-streaming kernel (k_admm_math.cuh) in the same order,
// rounded to the storage types where its stores round, so the results are bitwise the same.
#pragma once
#include <cooperative_groups.h>

#include "k_admm_math.cuh"
#include "k_mbar.cuh"
#include "k_pack2.cuh"

namespace tvl1 {

namespace cluster {

constexpr unsigned FULL = 0xffffffffu;
constexpr int HALO = 2, MAXWARPS = 8, MAXROWS = 16;
constexpr int NQ = 7;  // quads of an exchanged pixel pair: y (3), s w, u v, div y q1 q2, div y p
enum { G_D = 0, G_S = 3, G_W = 4, G_U = 5, G_V = 6, G_SIX = 7, G_SIY = 8, NG = 9 };

struct Shared {
    ulonglong2 inbox[2][MAXROWS][NQ][32];
    pair2 top[MAXWARPS][NG][32], bot[MAXWARPS][3][32];
    double red[32], part[2], total;  // part: alternating, a CTA may still read the last one's
    unsigned long long full[2];      // the mbarrier an inbox completes on
    unsigned expect;                 // bytes an inbox receives
    int leader;                      // the first warp that waits for them
    int dead;                        // set when a wait of this CTA ran out
};

__device__ __forceinline__ unsigned remote(unsigned p, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(p), "r"(rank));
    return a;
}
// 16 bytes into another CTA's shared memory, counted by its mbarrier
__device__ __forceinline__ void st_remote(unsigned a, pair2 v, pair2 w, unsigned bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(a), "l"(v), "l"(w), "r"(bar)
                 : "memory");
}
template <typename T, typename TF, bool HAS_W, bool II, int R> __device__ __forceinline__ void run(const ResArgs &A) {
    constexpr int C0 = HAS_W ? 0 : 1;
    constexpr unsigned PIXEL = 16 * (HAS_W ? NQ : NQ - 2), SOUTH = 16 * (HAS_W ? 4 : 3);  // bytes sent of a pixel pair
    extern __shared__ __align__(16) char smem_[];
    Shared &G = *reinterpret_cast<Shared *>(smem_);
    auto cl = cooperative_groups::this_cluster();
    const int rank = (int)cl.block_rank(), nc = (int)cl.num_blocks();
    const int lane = threadIdx.x & 31, wid = __shfl_sync(FULL, threadIdx.x >> 5, 0), nw = blockDim.x >> 5;
    const int H = A.g.H, W = A.g.W, P = A.g.pitch, gx = A.gx, ow = A.ow, oh = A.oh;
    const int by = rank / gx, bx = rank - by * gx;
    const int l0 = gx > 1 ? HALO / 2 : 0, l1 = l0 + ow / 2;  // the lanes of the tile's own columns
    const int c = bx * ow + 2 * (lane - l0);                 // this thread's columns c and c + 1
    const int q0 = wid * R - HALO, i0 = by * oh + q0;        // its first row, in the tile and in the image
    const unsigned me0 = mask_of(c < W - 1), me1 = mask_of(c + 1 < W - 1), mw0 = mask_of(c > 0);
    const int rlast = __shfl_sync(FULL, H - 1 - i0, 0), rfirst = __shfl_sync(FULL, -i0, 0);
    auto own = [&](int r) { return q0 + r >= 0 && q0 + r < oh && i0 + r < H && lane >= l0 && lane < l1; };

    // ---- the frame (pixels outside the image: zero)
    pair2 y[R][6], s[R], w[R], u[R], v[R], d[R][3], ix[R], iy[R], it[R], kf[R], inv_atc[R];
    const StepK SK = step_coefs(A.k, a_tilde_of(A.k, A.ms_max), c_of(A.k, A.ms_max));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = i0 + r;
        const bool row = i >= 0 && i < H;
        const unsigned m0 = mask_of(row && c >= 0 && c < W), m1 = mask_of(row && c + 1 >= 0 && c + 1 < W);
        const int cc = min(max(c, 0), W - 1) & ~1;
        const size_t ro = (size_t)min(max(i, 0), H - 1) * P, o = ro + cc;
        const size_t on = (size_t)min(max(i - 1, 0), H - 1) * P + cc, west = ro + min(max(c - 1, 0), W - 1);
        auto mask = [&](pair2 q) {
            float a, b;
            upk(q, a, b);
            return pk(keep(a, m0), keep(b, m1));
        };
        auto LT = [&](const void *p) { return mask(ld_pair<T>(p, o)); };
#pragma unroll
        for (int k = 2 * C0; k < 6; ++k) y[r][k] = LT(A.in.f[F_P1 + k]);
        s[r] = LT(A.in.f[F_S]);
        w[r] = HAS_W ? mask(ld_pair<TF>(A.in.f[F_W], o)) : 0ull;
        u[r] = mask(ld_pair<TF>(A.in.f[F_U], o));
        v[r] = mask(ld_pair<TF>(A.in.f[F_V], o));
        ix[r] = LT(A.Ix);
        iy[r] = LT(A.Iy);
        it[r] = LT(A.It);
        // div y, its west and north neighbours read here
#pragma unroll
        for (int k = C0; k < 3; ++k) {
            float a, b;
            upk(y[r][2 * k], a, b);
            const float wv = ldT<T>(A.in.f[F_P1 + 2 * k], west);
            const pair2 n = i > 0 ? ld_pair<T>(A.in.f[F_P1 + 2 * k + 1], on) : 0ull, ys = i < H - 1 ? y[r][2 * k + 1] : 0ull;
            d[r][k] = sub2(add2(pk(keep(a, me0) - keep(wv, mw0), keep(b, me1) - a), ys), n);
        }
        const pair2 ms = fma2(iy[r], iy[r], fma2(ix[r], ix[r], bc2(SK.beta * SK.beta)));
        pair2 inv_at = bc2(SK.inv_at);
        inv_atc[r] = bc2(SK.inv_atc);
        if (SK.per_pixel) {
            float e0, e1;
            upk(ms, e0, e1);
            e0 = fmaxf(e0, 1e-12f);
            e1 = fmaxf(e1, 1e-12f);
            inv_at = pk(__frcp_rn(e0), __frcp_rn(e1));
            inv_atc[r] = pk(__frcp_rn(e0 * SK.cc), __frcp_rn(e1 * SK.cc));
        }
        kf[r] = fma2(II ? mul2(bc2(-SK.rho), ms) : neg2(ms), inv_at, bc2(1.f));
    }
    const pair2 inv_a = bc2(SK.inv_a), inv_c = bc2(SK.inv_c), nbeta = bc2(-SK.beta), beta = bc2(SK.beta);
    const pair2 ccp = bc2(II ? SK.cc * SK.rho : SK.cc), rc = bc2(SK.rc);

    // ---- which of this thread's pixels arrive from neighbours, and how many bytes in all
    auto arrives = [&](int r) {
        const int q = q0 + r;
        const bool rows = q < 0 ? by > 0 && by * oh < H : i0 + r < H && q < oh + HALO && by * oh < H;
        const bool cols = lane < l0 ? bx > 0 : lane < l1 ? q < 0 || q >= oh : lane < l1 + l0 && bx + 1 < gx;
        return rows && cols;
    };
    if (threadIdx.x == 0) {
        G.expect = 0;
        G.leader = MAXWARPS;
        G.dead = 0;
        for (int b = 0; b < 2; ++b) mbar_init(&G.full[b], 1);
        mbar_init_fence();
    }
    cl.sync();
    bool halo = false;  // whether the warp waits for its neighbours' pixels
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (arrives(r)) {
            halo = true;
            atomicAdd(&G.expect, q0 + r == oh + HALO - 1 ? SOUTH : PIXEL);
        }
    halo = __any_sync(FULL, halo);
    if (halo && lane == 0) atomicMin(&G.leader, wid);
    __syncthreads();
    const bool leader = wid == G.leader && lane == 0;

    auto dx2 = [&](pair2 q) -> pair2 {  // east neighbour differences (zero across the image border)
        float a, b;
        upk(q, a, b);
        const float e = __shfl_down_sync(FULL, a, 1);
        return pk(keep(b - a, me0), keep(e - b, me1));
    };
    // div y without the north neighbours' part
    auto div_ = [&](int r, pair2 *out) {
        pair2 ys[3] = {y[r][1], y[r][3], y[r][5]};
        if (r == rlast) {
            asm volatile("");  // a branch, not selects
            ys[0] = ys[1] = ys[2] = 0ull;
        }
#pragma unroll
        for (int k = C0; k < 3; ++k) {
            float a, b;
            upk(y[r][2 * k], a, b);
            const float wv = __shfl_up_sync(FULL, b, 1);
            out[k] = add2(pk(keep(a, me0) - keep(wv, mw0), keep(b, me1) - a), ys[k]);
        }
    };

    // The exchange between neighbouring warps: the warp below gives its first row's values before this one's
    // last row, the warp above its last row's duals before this one's first.  Each direction of a pair has a
    // named barrier (the hardware has sixteen), on which the giving warp does not wait; a slot is
    // rewritten only after the pair's other barrier.
    float res = 0.f;
    auto iteration = [&](bool resid) {
        pair2 six[R], siy[R], ex[R][3];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            six[r] = mul2(s[r], ix[r]);
            siy[r] = mul2(s[r], iy[r]);
        }
        if (wid > 0) {
#pragma unroll
            for (int k = C0; k < 3; ++k) G.top[wid][G_D + k][lane] = d[0][k];
            if (HAS_W) {
                G.top[wid][G_S][lane] = s[0];
                G.top[wid][G_W][lane] = w[0];
            }
            G.top[wid][G_U][lane] = u[0];
            G.top[wid][G_V][lane] = v[0];
            G.top[wid][G_SIX][lane] = six[0];
            G.top[wid][G_SIY][lane] = siy[0];
            bar_arrive(wid, 64);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (HAS_W) ex[r][0] = fma2(nbeta, dx2(s[r]), fma2(dx2(w[r]), inv_c, dx2(d[r][0])));
            ex[r][1] = sub2(fma2(dx2(u[r]), inv_c, dx2(d[r][1])), dx2(six[r]));
            ex[r][2] = sub2(fma2(dx2(v[r]), inv_c, dx2(d[r][2])), dx2(siy[r]));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            pair2 so[NG];
            if (r < R - 1) {
                constexpr int n = R - 1;  // R <= 2
#pragma unroll
                for (int k = C0; k < 3; ++k) so[G_D + k] = d[n][k];
                so[G_S] = s[n];
                so[G_W] = w[n];
                so[G_U] = u[n];
                so[G_V] = v[n];
                so[G_SIX] = six[n];
                so[G_SIY] = siy[n];
            } else {
                const int below = min(wid + 1, MAXWARPS - 1);
                if (wid < nw - 1) bar_wait(wid + 1, 64);
#pragma unroll
                for (int k = HAS_W ? 0 : 1; k < NG; ++k)
                    if (HAS_W || (k != G_S && k != G_W)) so[k] = G.top[below][k][lane];
            }
            pair2 ey[NG];
#pragma unroll
            for (int k = C0; k < 3; ++k) ey[G_D + k] = sub2(so[G_D + k], d[r][k]);
            if (HAS_W) {
                ey[G_S] = sub2(so[G_S], s[r]);
                ey[G_W] = sub2(so[G_W], w[r]);
            }
            ey[G_U] = sub2(so[G_U], u[r]);
            ey[G_V] = sub2(so[G_V], v[r]);
            ey[G_SIX] = sub2(so[G_SIX], six[r]);
            ey[G_SIY] = sub2(so[G_SIY], siy[r]);
            if (r == rlast) {
                asm volatile("");
#pragma unroll
                for (int k = 0; k < NG; ++k) ey[k] = 0ull;
            }
            if (HAS_W) {
                const pair2 a1 = fma2(ex[r][0], inv_a, y[r][0]);
                const pair2 a2 = fma2(fma2(nbeta, ey[G_S], fma2(ey[G_W], inv_c, ey[G_D])), inv_a, y[r][1]);
                const pair2 f = ball_scale2(fma2(a1, a1, mul2(a2, a2)));
                y[r][0] = mul2(a1, f);
                y[r][1] = mul2(a2, f);
            }
            const pair2 b11 = fma2(ex[r][1], inv_a, y[r][2]), b21 = fma2(ex[r][2], inv_a, y[r][4]);
            const pair2 b12 = fma2(sub2(fma2(ey[G_U], inv_c, ey[G_D + 1]), ey[G_SIX]), inv_a, y[r][3]);
            const pair2 b22 = fma2(sub2(fma2(ey[G_V], inv_c, ey[G_D + 2]), ey[G_SIY]), inv_a, y[r][5]);
            const pair2 f = ball_scale2(fma2(b11, b11, fma2(b12, b12, fma2(b21, b21, mul2(b22, b22)))));
            y[r][2] = mul2(b11, f);
            y[r][3] = mul2(b12, f);
            y[r][4] = mul2(b21, f);
            y[r][5] = mul2(b22, f);
        }
        if (wid < nw - 1) {
#pragma unroll
            for (int k = C0; k < 3; ++k) G.bot[wid][k][lane] = y[R - 1][2 * k + 1];
            bar_arrive(MAXWARPS + wid, 64);
        }
        if (resid) res = 0.f;
#pragma unroll
        for (int r = R - 1; r >= 0; --r) {
            pair2 lin = fma2(iy[r], v[r], fma2(ix[r], u[r], it[r]));
            if (HAS_W) lin = fma2(beta, w[r], lin);
            pair2 n[3], dn[3];
            div_(r, dn);
            if (r > 0) {
#pragma unroll
                for (int k = C0; k < 3; ++k) n[k] = y[0][2 * k + 1];
            } else {
                const int above = max(wid - 1, 0);
                if (wid > 0) bar_wait(MAXWARPS + wid - 1, 64);
#pragma unroll
                for (int k = C0; k < 3; ++k) n[k] = G.bot[above][k][lane];
            }
            if (r == rfirst) {
                asm volatile("");
                n[0] = n[1] = n[2] = 0ull;
            }
#pragma unroll
            for (int k = C0; k < 3; ++k) dn[k] = sub2(dn[k], n[k]);
            pair2 divt = fma2(iy[r], dn[2], mul2(ix[r], dn[1]));
            if (HAS_W) divt = fma2(beta, dn[0], divt);
            const pair2 so = s[r];
            float s0, s1;
            upk(fma2(fma2(ccp, divt, lin), inv_atc[r], mul2(kf[r], so)), s0, s1);
            s0 = fminf(fmaxf(s0, -SK.lam), SK.lam);
            s1 = fminf(fmaxf(s1, -SK.lam), SK.lam);
            const pair2 sn = pk(s0, s1), ns = pk(-s0, -s1);
            // minus the constraint residual A s^{k+1} - div y^{k+1}
            const pair2 ncw = HAS_W ? fma2(nbeta, sn, dn[0]) : 0ull;
            const pair2 ncu = fma2(ix[r], ns, dn[1]), ncv = fma2(iy[r], ns, dn[2]);
            if (!II) {
                if (HAS_W) w[r] = fma2(rc, ncw, w[r]);
                u[r] = fma2(rc, ncu, u[r]);
                v[r] = fma2(rc, ncv, v[r]);
            } else {
                const pair2 nrho = bc2(-SK.rho), nomr = bc2(-SK.omr), ncc = bc2(-SK.cc);
                if (HAS_W) w[r] = fma2(ncc, fma2(bc2(-SK.omr * SK.beta), so, fma2(nrho, dn[0], mul2(beta, sn))), w[r]);
                u[r] = fma2(ncc, fma2(mul2(nomr, ix[r]), so, fma2(nrho, dn[1], mul2(ix[r], sn))), u[r]);
                v[r] = fma2(ncc, fma2(mul2(nomr, iy[r]), so, fma2(nrho, dn[2], mul2(iy[r], sn))), v[r]);
            }
            if (resid && own(r)) {
                float p0, p1;
                upk(fma2(ncv, ncv, fma2(ncu, ncu, mul2(ncw, ncw))), p0, p1);
                if (c < W) res += p0;
                if (c + 1 < W) res += p1;
            }
            s[r] = round2<T>(sn);
            if (HAS_W) w[r] = round2<TF>(w[r]);
            u[r] = round2<TF>(u[r]);
            v[r] = round2<TF>(v[r]);
            if (!std::is_same<T, float>::value) {  // the next iteration reads y as stored
#pragma unroll
                for (int k = 2 * C0; k < 6; ++k) y[r][k] = round2<T>(y[r][k]);
                div_(r, dn);
#pragma unroll
                for (int k = C0; k < 3; ++k) dn[k] = sub2(dn[k], round2<T>(n[k]));
            }
#pragma unroll
            for (int k = C0; k < 3; ++k) d[r][k] = dn[k];
        }
    };

    // ---- the exchange between CTAs: the tile's rows within HALO of the north / south edge, its columns within
    // HALO of the west / east edge
    const bool to_w = bx > 0 && lane < l0 + HALO / 2, to_e = bx + 1 < gx && lane >= l1 - HALO / 2;
    auto send = [&](int par, int r, int dv, int dh) {
        const int to = rank + dv * gx + dh;
        const unsigned a = remote(smem_u32(&G.inbox[par][wid * R + r - dv * oh][0][lane - dh * (ow / 2)]), to);
        const unsigned b = remote(smem_u32(&G.full[par]), to);
        if (dv >= 0 || q0 + r < HALO - 1) {  // the frame's last row gives its south differences only
            if (HAS_W) st_remote(a, y[r][0], y[r][1], b);
            st_remote(a + 512, y[r][2], y[r][3], b);
            st_remote(a + 1024, y[r][4], y[r][5], b);
        }
        st_remote(a + 1536, s[r], w[r], b);
        st_remote(a + 2048, u[r], v[r], b);
        st_remote(a + 2560, d[r][1], d[r][2], b);
        if (HAS_W) st_remote(a + 3072, d[r][0], 0ull, b);
    };
    auto push = [&](int par) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!own(r)) continue;
            const bool to_n = by > 0 && q0 + r < HALO, to_s = (by + 1) * oh < H && q0 + r >= oh - HALO;
            if (to_n) send(par, r, -1, 0);
            if (to_s) send(par, r, 1, 0);
            // west and east columns at once: they are different lanes but in tiles two pixels wide
            if (to_w || to_e) {
                const int dh = to_w ? -1 : 1;
                send(par, r, 0, dh);
                if (to_n) send(par, r, -1, dh);
                if (to_s) send(par, r, 1, dh);
            }
            if (to_w && to_e) {
                send(par, r, 0, 1);
                if (to_n) send(par, r, -1, 1);
                if (to_s) send(par, r, 1, 1);
            }
        }
    };
    auto pull = [&](int par) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!arrives(r) || c < 0 || c >= W) continue;
            const ulonglong2 *b = &G.inbox[par][wid * R + r][0][lane];
            auto get = [&](int k, pair2 &p0, pair2 &p1) {
                const ulonglong2 t = b[32 * k];
                p0 = t.x;
                p1 = t.y;
            };
            pair2 none;
            if (HAS_W) get(0, y[r][0], y[r][1]);
            get(1, y[r][2], y[r][3]);
            get(2, y[r][4], y[r][5]);
            if (HAS_W) get(3, s[r], w[r]);
            else get(3, s[r], none);
            get(4, u[r], v[r]);
            get(5, d[r][1], d[r][2]);
            if (HAS_W) get(6, d[r][0], none);
        }
    };

    int run = 0, par = 0, pp = 0;
    unsigned ph = 0;   // the inboxes' phase
    bool have_tot = false, dead = false;
    double tot = 0.0;
    while (run < A.iters) {
        const bool quit = *(volatile int *)&G.dead != 0;
        const int n = min(HALO, A.iters - run);
        const bool check = A.check && (run + n) % 10 == 0, fin = A.final_res && run + n == A.iters;
        for (int k = 1; k <= n; ++k) iteration(k == n && (check || fin));
        run += n;
        if (check || fin) {  // uniform over the cluster
            const double b = block_sum((double)res, G.red);
            if (threadIdx.x == 0) G.part[pp] = b;
            cl.sync();
            if (threadIdx.x == 0) {
                double t = 0.0;
                for (int r = 0; r < nc; ++r) t += *cl.map_shared_rank(&G.part[pp], r);
                G.total = t;
            }
            __syncthreads();
            tot = G.total;
            have_tot = true;
            pp ^= 1;
            if (check) {
                const bool met = A.tol > 0.0 && sqrt(tot / A.sc.rows) < A.tol;
                if (rank == 0 && threadIdx.x == 0) {
                    *A.sc.res_check = tot;
                    if (met) *A.sc.done = 1;
                }
                if (met) break;
            }
        }
        if (run >= A.iters) break;
        // the leader has waited for this inbox's last phase, so the arrival counts for the next (a warp without
        // halo may be iterations ahead)
        // After a wait that ran out, the CTA goes on without sending or waiting (its neighbours' waits then run
        // out too), and the result is reported as a timeout.
        dead |= __any_sync(FULL, quit);
        if (leader && !dead) mbar_expect(&G.full[par], G.expect);
        if (!dead && rank != A.withhold) push(par);
        if (halo && !dead) {
            const bool here = mbar_wait<true>(&G.full[par], ph, A.wait_ns, A.timeout);
            if (__all_sync(FULL, here)) {
                pull(par);
            } else {
                dead = true;
                G.dead = 1;
                if (lane == 0 && A.timeout) *A.timeout = 1;
            }
        }
        __syncwarp();
        par ^= 1;
        if (!par) ph ^= 1;
    }
    if (rank == 0 && threadIdx.x == 0) {
        *A.sc.iters += run;
        if (A.final_res && have_tot) *A.sc.res_final = tot;
    }
    // out may be in: no CTA stores while another still loads; nor leaves while another uses its shared memory
    cl.sync();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (!own(r)) continue;
        const size_t o = (size_t)(i0 + r) * P + c;
        auto ST = [&](auto tag, void *p, pair2 val) {
            using S = decltype(tag);
            if (c + 1 < W) st_pair<S>(p, o, val);
            else if (c < W) stT<S>(p, o, lo2(val));
        };
#pragma unroll
        for (int k = 2 * C0; k < 6; ++k) ST(T{}, A.out.f[F_P1 + k], y[r][k]);
        ST(T{}, A.out.f[F_S], s[r]);
        if (HAS_W) ST(TF{}, A.out.f[F_W], w[r]);
        ST(TF{}, A.out.f[F_U], u[r]);
        ST(TF{}, A.out.f[F_V], v[r]);
    }
}

template <typename T, typename TF, bool HAS_W, bool II, int R>
__global__ void __launch_bounds__(MAXWARPS * 32, 1) k_admm_cluster(const __grid_constant__ ResArgs A) {
    run<T, TF, HAS_W, II, R>(A);
}

}  // namespace cluster
}  // namespace tvl1
