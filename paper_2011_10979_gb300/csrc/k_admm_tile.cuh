// k_admm_tile.cuh -- several ADMM inner iterations (Sec. 3.1.1, eq. rpADMMI / rpADMMII /
// Zach-pADMM) in one launch, the state in registers.
//
// A block of NW warps (12, or 8 in the FP32 looping form) holds a frame of 64 columns by NW R rows: each
// lane the pixels of two
// neighbouring columns (one 64-bit register pair per plane, so that the packed FP32 instructions
// serve both) in R consecutive rows.  One iteration at a pixel needs y^{k+1} one pixel west and
// north (div y^{k+1}), y^{k+1} at a pixel needs div y^k, s, Lambda and the data one pixel east and
// south, and div y^k needs y^k one pixel west and north; ni iterations chain that ni times, so a
// frame whose outermost ni + 1 pixels (west, north) and ni pixels (east, south) are halo yields ni
// iterations on the ow x oh pixels inside.  The whole frame is computed in every iteration; what
// the halo's pixels compute beyond their valid region is never read.
// East and west neighbours travel by shuffle, south and north ones in the thread's own registers
// and, between the warps' bands, through shared memory: a warp leaves its top row's values for the
// warp above and its bottom row's duals for the warp below, read after a barrier at the last row of the
// y phase and the last row of the finish phase, so most of a phase's work needs no neighbour.
// What bounds it: the FMA pipe and, with three warps per SM quarter, latency.  One pixel-iteration
// takes 77 FP32 operations; the packed form issues some 65 instructions for them, 6 shuffles and 3
// shared-memory accesses, against some 200 instructions and 96 shared-memory wavefronts per 32
// pixels of a kernel that keeps the frame in shared memory (the one this replaced: 5.41 us per
// iteration at 640x480, 145 at 3840x2160; now 3.5 and 60).  Measured on 64 x 48 frames: 1.05 us per
// iteration with 8 warps of 6 rows, 1.35 with 12 of 4, and 4 to 6 us per tile beside the iterations
// (L2 reads and writes of the state, instruction fetch).  One tile per block: 12 x 4 takes 10.5 us
// per three-iteration launch at 640x480, 8 x 6 13.1, 16 x 3 10.7.
//
// Levels with more tiles than SMs run the staged form: one block per SM loops over the tiles, and the
// next tile's planes are copied to shared memory by TMA while the current one iterates (3840x2160,
// four iterations: 239 us per launch against 301 with one tile per block).
// Every expression is that of the row-streaming kernel (k_admm_math.cuh, k_admm_roll.cuh) in the
// same order, each packed instruction rounds its halves as the scalar one does, and the state
// between the iterations is rounded to its storage type where that kernel's stores round it, so ni
// iterations here are bitwise ni launches of it.  The launch reads one state buffer and writes the
// other; the residual's partial sums are those of the last iteration, grouped per tile.
//
// Instantiated per storage type in k_admm_tile_{f32,f16,bf16}.cu, launch policy in k_admm_tile.cu.
#pragma once
#include <cuda.h>
#include <math.h>

#include <type_traits>

#include "k_admm_math.cuh"
#include "k_mbar.cuh"
#include "k_pack2.cuh"

namespace tvl1 {

void tile_launch_f32(const TileArgs &a, cudaStream_t s);
void tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s);
void tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s);

namespace tile {

constexpr int FW = 64;           // frame columns: two per lane
constexpr unsigned FULL = 0xffffffffu;

// The planes of a tile: duals and data in storage type T, multipliers in TF.
enum { L_Y = 0, L_S = 6, L_W = 7, L_U = 8, L_V = 9, L_IX = 10, L_IY = 11, L_IT = 12, NL = 13 };

// What a warp's top row gives the warp above: div y (p, q1, q2), s, w, u, v, s Ix, s Iy.
enum { G_D = 0, G_S = 3, G_W = 4, G_U = 5, G_V = 6, G_SIX = 7, G_SIY = 8, NG = 9 };

template <int NW, int R> struct Shared {
    pair2 top[NW][NG][32];                 // top rows, read by the warp above
    pair2 bot[NW][3][32];                  // p2, q12, q22 of the bottom rows, read by the warp below
    pair2 it[NW * R][32], kf[NW * R][32];  // It and 1 - M_s / a~ per pixel (each thread its own)
    // batched form: the descriptors of the current and the next two tiles' pairs and the work-list
    // entries of the next three tiles, copied ahead by cp.async
    PairIter pi[3];
    int4 tr[4];
    double red[32];
    int dead;                              // staged form: the first thread's wait for copies ran out
    unsigned long long full;               // staged form: the mbarrier the copies complete on
};

// How the frame reaches the registers: straight from global memory, one tile per block (DIRECT), or
// through a stage in shared memory that the next tile's TMA copies fill while the current one
// iterates, blocks looping over the tiles of a pair (STAGED) or of a batch's work-list (BATCHED).
enum Mode { DIRECT, STAGED, BATCHED };

// The stage of one frame: three planes of TF, ten of T, each 8 R rows of WT columns.  A copy must
// start on a 16-byte boundary, i.e. at a multiple of 4 FP32 or 8 16-bit columns; frames start at
// multiples of 4, so rows of 16-bit planes are 8 columns wider and start up to 4 columns early.
template <typename T, typename TF, int FH_> struct Stage {
    static constexpr int FH = FH_;
    static constexpr int wid_of(int bytes) { return bytes == 4 ? FW : FW + 8; }
    static constexpr int WT = wid_of(sizeof(T)), WTF = wid_of(sizeof(TF));
    static constexpr int up(int x) { return (x + 127) / 128 * 128; }
    static constexpr int flow = 0, dual = up(3 * FH * WTF * (int)sizeof(TF)), data = dual + up(7 * FH * WT * (int)sizeof(T)),
                         bytes = data + up(3 * FH * WT * (int)sizeof(T));
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Makes a tensor map in global memory, which the host wrote before the launch, visible to this thread's
// copies: without it they may use what an earlier launch's map at the same address left in a cache.
__device__ __forceinline__ void map_acquire(const CUtensorMap *map) {
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

// Step constants as pairs.
struct PairK {
    pair2 inv_a, inv_c, nbeta, beta, cc, inv_atc, rc;
    float lam;
};

// The tile in hand.
struct Tile {
    int H, W, P, bx, by, id;
};

template <typename T, typename TF, bool HAS_W, int VARIANT, int NW, int R, Mode MODE> struct Kernel {
    // VARIANT bit 0: rpADMMII; bit 1: the per-pixel a~ (a template choice: its reciprocals behind a run-time
    // branch made every iteration 70% slower)
    static constexpr bool II = VARIANT & 1, PP = VARIANT & 2;
    // few warps order the exchange between neighbours by a pair of named barriers each (the hardware has
    // sixteen), more by the block barrier
    static constexpr bool PAIRED = NW <= 8;
    static constexpr int C0 = HAS_W ? 0 : 1;
    static constexpr bool STAGE = MODE != DIRECT;
    using SH = Shared<NW, R>;
    using ST = Stage<T, TF, NW * R>;
    static constexpr int NF = HAS_W ? 3 : 2, ND = HAS_W ? 7 : 5;   // flow and dual planes copied

    static __device__ __forceinline__ Tile tile_at(const TileArgs &A, const SH &G, int t, int n) {
        Tile D;
        D.id = t;
        if (MODE == BATCHED) {
            const int4 tr = G.tr[n & 3];
            const Geom g = G.pi[n % 3].g;
            D.H = g.H;
            D.W = g.W;
            D.P = g.pitch;
            D.bx = tr.y;
            D.by = tr.z;
        } else {
            D.H = A.a.g.H;
            D.W = A.a.g.W;
            D.P = A.a.g.pitch;
            D.bx = t % A.gx;
            D.by = t / A.gx;
        }
        return D;
    }

    // After a wait that ran out: reports the pair (what the block makes of the tile is void).  The first thread starts
    // no more copies, so it reports the pairs of all the block's later tiles, and gives the copies in flight the
    // same time again.
    static __device__ __noinline__ void missed(const TileArgs &A, SH &G, int t, int n) {
        if (MODE == BATCHED) *G.pi[n % 3].timeout = 1;
        else if (A.timeout) *A.timeout = 1;
        if (threadIdx.x != 0) return;
        G.dead = 1;
        if (MODE == BATCHED)
            for (t += gridDim.x; t < A.ntiles; t += gridDim.x) *A.a.pairs[A.a.tiles[t].pair].timeout = 1;
        mbar_wait(&G.full, n & 1, A.wait_ns, nullptr);
    }

    // Batched form: a pair's three tensor maps.
    static __device__ __forceinline__ const CUtensorMap *maps_of(const TileArgs &A, int pair) {
        return A.table + 6 * pair + 3 * A.a.parity;
    }
    // Batched form, first warp: acquires the tensor maps of the block's tiles n to n + m - 1, a map per lane, but those
    // of the tile before (a single pair's maps are parameters of the kernel, which need no fence).
    static constexpr int ACQUIRED = 10;
    static __device__ __forceinline__ void acquire_maps(const TileArgs &A, int n, int m, int lane) {
        const int q = n + lane / 3, t = blockIdx.x + q * gridDim.x;
        if (lane < 3 * m && t < A.ntiles) {
            const int pair = A.a.tiles[t].pair;
            if (lane < 3 || A.a.tiles[t - gridDim.x].pair != pair) map_acquire(maps_of(A, pair) + lane % 3);
        }
        __syncwarp();
    }

    // Starts the copies of a tile's frame into the stage (one thread); zeros outside the image.
    static __device__ __forceinline__ void prefetch(const TileArgs &A, SH &G, char *stage, int t, int n) {
        const Tile D = tile_at(A, G, t, n);
        const CUtensorMap *maps =
            MODE == BATCHED ? maps_of(A, G.tr[n & 3].x) : A.maps;
        const int x = D.bx * A.ow - A.offx, y = D.by * A.oh - A.offy;
        mbar_expect(&G.full, ST::FH * (NF * ST::WTF * (int)sizeof(TF) + (ND + 3) * ST::WT * (int)sizeof(T)));
        if (t == A.withhold) return;
        tma_load(stage + ST::flow, maps, sizeof(TF) == 4 ? x : x & ~7, y, &G.full);
        tma_load(stage + ST::dual, maps + 1, sizeof(T) == 4 ? x : x & ~7, y, &G.full);
        tma_load(stage + ST::data, maps + 2, sizeof(T) == 4 ? x : x & ~7, y, &G.full);
    }

    // Batched form, first warp: starts the copy of tile n's pair descriptor (its work-list entry is here).
    static __device__ __forceinline__ void fetch_pair(const TileArgs &A, SH &G, int n, int lane) {
        static_assert(sizeof(PairIter) % 16 == 0 && sizeof(PairIter) <= 512, "copied in 16-byte words by one warp");
        if (lane < (int)sizeof(PairIter) / 16)
            cp_async16((char *)&G.pi[n % 3] + 16 * lane, (const char *)(A.a.pairs + G.tr[n & 3].x) + 16 * lane);
    }
    static __device__ __forceinline__ void fetch_ref(const TileArgs &A, SH &G, int t, int n, int lane) {
        if (lane == 0) cp_async16(&G.tr[n & 3], reinterpret_cast<const int4 *>(A.a.tiles) + min(t, A.ntiles - 1));
    }

    // BX: 0, the frame lies between the image's left and right borders; 1, it touches one of them and the
    // width is even (the border is then the odd column of a pair); 2, any width, and rows that are not
    // aligned.  Column borders mask (logic instructions: floating-point selects cost the FMA pipe), row
    // borders branch (masks in every row made a tile with both borders 20% slower).
    // BY: it touches the top or bottom one.
    template <int BX, bool BY>
    static __device__ __forceinline__ void body(const TileArgs &A, SH &G, char *stage, const Tile &D, int n, int lane,
                                                int wid) {
        const int H = D.H, W = D.W, P = D.P;
        const int c = D.bx * A.ow - A.offx + 2 * lane;   // this lane's even column
        const int ib = D.by * A.oh - A.offy + wid * R;   // this warp's first row
        const float *ms_max = MODE == BATCHED ? G.pi[n % 3].ms_max : A.a.ms_max;
        const float at = a_tilde_of(A.a.k, ms_max), cs = c_of(A.a.k, ms_max);
        const int *donep = MODE == BATCHED ? G.pi[n % 3].done : nullptr;
        const int done = donep ? *donep : 0;
        // ~0 where the even / odd column has an east neighbour in the image, and the even one a west one
        const unsigned me0 = mask_of(c < W - 1), me1 = mask_of(c + 1 < W - 1), mw0 = mask_of(c > 0);
        // this warp's row that is the image's last / first, if any (uniform: the rows are tested by branches
        // that one warp per tile column takes)
        const int rlast = __shfl_sync(FULL, H - 1 - ib, 0), rfirst = __shfl_sync(FULL, -ib, 0);
        pair2 y[R][6], s[R], w[R], u[R], v[R], ix[R], iy[R], d[R][3];
        // ---- the frame, zero outside the image
        pair2 it[R];
        if constexpr (STAGE) {
            if (!mbar_wait(&G.full, n & 1, A.wait_ns, MODE == BATCHED ? G.pi[n % 3].timeout : A.timeout)) missed(A, G, D.id, n);
            const int x = c - 2 * lane;
            const int at_ = sizeof(T) == 4 ? 2 * lane : 2 * lane + (x & 7), af_ = sizeof(TF) == 4 ? 2 * lane : 2 * lane + (x & 7);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int fr = wid * R + r;
                auto LD = [&](int k) { return ld_pair<T>(stage + ST::dual, ((k - 2 * C0) * ST::FH + fr) * ST::WT + at_); };
                auto LI = [&](int k) { return ld_pair<T>(stage + ST::data, (k * ST::FH + fr) * ST::WT + at_); };
                auto LF = [&](int k) { return ld_pair<TF>(stage + ST::flow, ((k - C0) * ST::FH + fr) * ST::WTF + af_); };
#pragma unroll
                for (int k = 2 * C0; k < 6; ++k) y[r][k] = LD(k);
                s[r] = LD(6);
                if (HAS_W) w[r] = LF(0);
                u[r] = LF(1);
                v[r] = LF(2);
                ix[r] = LI(0);
                iy[r] = LI(1);
                it[r] = LI(2);
            }
            // the stage is free for the next tile, whose descriptor the first warp has by now
            if (MODE == BATCHED && wid == 0) cp_async_wait();
            const bool dead = threadIdx.x == 0 && *(volatile int *)&G.dead;
            __syncthreads();
            const int t1 = D.id + gridDim.x;
            if (t1 < A.ntiles) {
                if (MODE == BATCHED && wid == 0 && (n + 1) % ACQUIRED == 0) acquire_maps(A, n + 1, ACQUIRED, lane);
                if (threadIdx.x == 0 && !dead) prefetch(A, G, stage, t1, n + 1);
                if (MODE == BATCHED && wid == 0) {
                    fetch_pair(A, G, n + 2, lane);
                    fetch_ref(A, G, t1 + 2 * gridDim.x, n + 3, lane);
                }
            }
            if (done) return;  // the pair's warp met its stopping test
        } else {
            // pixels outside are read at the nearest pixel inside
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
                    auto LT = [&](const void *p) { return mask(VEC ? ld_pair<T>(p, o0) : pk(ldT<T>(p, o0), ldT<T>(p, o1))); };
                    auto LF = [&](const void *p) { return mask(VEC ? ld_pair<TF>(p, o0) : pk(ldT<TF>(p, o0), ldT<TF>(p, o1))); };
#pragma unroll
                    for (int k = 2 * C0; k < 6; ++k) y[r][k] = LT(A.a.in.f[F_P1 + k]);
                    s[r] = LT(A.a.in.f[F_S]);
                    if (HAS_W) w[r] = LF(A.a.in.f[F_W]);
                    u[r] = LF(A.a.in.f[F_U]);
                    v[r] = LF(A.a.in.f[F_V]);
                    ix[r] = LT(A.a.Ix);
                    iy[r] = LT(A.a.Iy);
                    it[r] = LT(A.a.It);
                }
            };
            if (BX < 2 || A.vec) load(std::true_type{});
            else load(std::false_type{});
        }
        const StepK SK = step_coefs(A.a.k, at, cs);
        PairK K;
        K.inv_a = bc2(SK.inv_a);
        K.inv_c = bc2(SK.inv_c);
        K.nbeta = bc2(-SK.beta);
        K.beta = bc2(SK.beta);
        K.cc = bc2(II ? SK.cc * SK.rho : SK.cc);
        K.inv_atc = bc2(SK.inv_atc);
        K.rc = bc2(SK.rc);
        K.lam = SK.lam;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            G.it[wid * R + r][lane] = it[r];
            const pair2 ms = fma2(iy[r], iy[r], fma2(ix[r], ix[r], bc2(SK.beta * SK.beta)));
            pair2 inv_at = bc2(SK.inv_at);
            if (PP) {
                float q0, q1;
                upk(ms, q0, q1);
                inv_at = pk(__frcp_rn(fmaxf(q0, 1e-12f)), __frcp_rn(fmaxf(q1, 1e-12f)));
            }
            const pair2 nms = II ? mul2(bc2(-SK.rho), ms) : neg2(ms);
            G.kf[wid * R + r][lane] = fma2(nms, inv_at, bc2(1.f));
        }

        auto shdn = [](float x) { return __shfl_down_sync(FULL, x, 1); };
        auto shup = [](float x) { return __shfl_up_sync(FULL, x, 1); };
        // east neighbour differences of a pair (zero across the image border)
        auto dx2 = [&](pair2 q) -> pair2 {
            float a, b;
            upk(q, a, b);
            const float e = shdn(a);
            return pk(BX == 2 ? keep(b - a, me0) : b - a, BX ? keep(e - b, me1) : e - b);
        };
        // div y on row r: north values n (p2, q12, q22 of the row above)
        auto divr = [&](int r, const pair2 *yy, const pair2 *n, pair2 *out) {
            pair2 ys[3] = {yy[1], yy[3], yy[5]}, nn[3] = {n[0], n[1], n[2]};
            if (BY && r == rlast) {
                asm volatile("");  // a branch, not selects
                ys[0] = ys[1] = ys[2] = 0ull;
            }
            if (BY && r == rfirst) {
                asm volatile("");
                nn[0] = nn[1] = nn[2] = 0ull;
            }
#pragma unroll
            for (int k = C0; k < 3; ++k) {
                float a, b;
                upk(yy[2 * k], a, b);
                const float wv = shup(b);
                const pair2 x = pk((BX == 2 ? keep(a, me0) : a) - (BX ? keep(wv, mw0) : wv), (BX ? keep(b, me1) : b) - a);
                out[k] = sub2(add2(x, ys[k]), nn[k]);
            }
        };
        // the exchange between neighbouring warps.  A slot is rewritten only after the barrier that
        // follows its last reading.
        // the barrier before the last row of the y phase; whether there is a warp below
        auto below = [&]() -> bool {
            if (!PAIRED) __syncthreads();
            else if (wid < NW - 1) bar_wait(wid + 1, 64);
            return wid < NW - 1;
        };
        auto put_bot = [&]() {
            if (wid < NW - 1) {
#pragma unroll
                for (int k = C0; k < 3; ++k) G.bot[wid][k][lane] = y[R - 1][2 * k + 1];
                if (PAIRED) bar_arrive(NW + wid, 64);
            }
        };
        auto get_bot = [&](pair2 *n) {
            n[0] = n[1] = n[2] = 0ull;
            if (!PAIRED) __syncthreads();
            if (wid > 0) {
                if (PAIRED) bar_wait(NW + wid - 1, 64);
#pragma unroll
                for (int k = C0; k < 3; ++k) n[k] = G.bot[wid - 1][k][lane];
            }
        };
        auto put_top = [&]() {
            if (wid > 0) {
#pragma unroll
                for (int k = C0; k < 3; ++k) G.top[wid][G_D + k][lane] = d[0][k];
                G.top[wid][G_S][lane] = s[0];
                if (HAS_W) G.top[wid][G_W][lane] = w[0];
                G.top[wid][G_U][lane] = u[0];
                G.top[wid][G_V][lane] = v[0];
                G.top[wid][G_SIX][lane] = mul2(s[0], ix[0]);
                G.top[wid][G_SIY][lane] = mul2(s[0], iy[0]);
                if (PAIRED) bar_arrive(wid, 64);
            }
        };
        // ---- div y^k of the frame
        put_bot();
#pragma unroll
        for (int r = R - 1; r >= 0; --r) {
            pair2 n[3];
            if (r > 0) {
#pragma unroll
                for (int k = 0; k < 3; ++k) n[k] = y[r - 1][2 * k + 1];
            } else {
                get_bot(n);
            }
            divr(r, y[r], n, d[r]);
        }
        put_top();
        float res = 0.f;
#pragma unroll 1
        for (int kk = 0; kk < A.ni; ++kk) {
            const bool last = kk == A.ni - 1;
            // ---- y^{k+1}, top row first (the last row needs the warp below)
            pair2 six = mul2(s[0], ix[0]), siy = mul2(s[0], iy[0]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                pair2 sd[3], ss, sw, su, sv, ssix, ssiy;
                if (r < R - 1) {
#pragma unroll
                    for (int k = C0; k < 3; ++k) sd[k] = d[r + 1][k];
                    ss = s[r + 1];
                    sw = w[r + 1];
                    su = u[r + 1];
                    sv = v[r + 1];
                    ssix = mul2(ss, ix[r + 1]);
                    ssiy = mul2(ss, iy[r + 1]);
                } else if (below()) {
#pragma unroll
                    for (int k = C0; k < 3; ++k) sd[k] = G.top[wid + 1][G_D + k][lane];
                    ss = G.top[wid + 1][G_S][lane];
                    if (HAS_W) sw = G.top[wid + 1][G_W][lane];
                    su = G.top[wid + 1][G_U][lane];
                    sv = G.top[wid + 1][G_V][lane];
                    ssix = G.top[wid + 1][G_SIX][lane];
                    ssiy = G.top[wid + 1][G_SIY][lane];
                } else {
                    sd[0] = sd[1] = sd[2] = ss = sw = su = sv = ssix = ssiy = 0ull;
                }
                pair2 ey[9];  // south differences: div y, s, w, u, v, s Ix, s Iy
#pragma unroll
                for (int k = C0; k < 3; ++k) ey[G_D + k] = sub2(sd[k], d[r][k]);
                if (HAS_W) {
                    ey[G_S] = sub2(ss, s[r]);
                    ey[G_W] = sub2(sw, w[r]);
                }
                ey[G_U] = sub2(su, u[r]);
                ey[G_V] = sub2(sv, v[r]);
                ey[G_SIX] = sub2(ssix, six);
                ey[G_SIY] = sub2(ssiy, siy);
                if (BY && r == rlast) {
                    asm volatile("");
#pragma unroll
                    for (int k = 0; k < 9; ++k) ey[k] = 0ull;
                }
                if (HAS_W) {
                    const pair2 a1 = fma2(fma2(K.nbeta, dx2(s[r]), fma2(dx2(w[r]), K.inv_c, dx2(d[r][0]))), K.inv_a, y[r][0]);
                    const pair2 a2 = fma2(fma2(K.nbeta, ey[G_S], fma2(ey[G_W], K.inv_c, ey[G_D])), K.inv_a, y[r][1]);
                    const pair2 f = ball_scale2(fma2(a1, a1, mul2(a2, a2)));
                    y[r][0] = mul2(a1, f);
                    y[r][1] = mul2(a2, f);
                }
                const pair2 b11 = fma2(sub2(fma2(dx2(u[r]), K.inv_c, dx2(d[r][1])), dx2(six)), K.inv_a, y[r][2]);
                const pair2 b12 = fma2(sub2(fma2(ey[G_U], K.inv_c, ey[G_D + 1]), ey[G_SIX]), K.inv_a, y[r][3]);
                const pair2 b21 = fma2(sub2(fma2(dx2(v[r]), K.inv_c, dx2(d[r][2])), dx2(siy)), K.inv_a, y[r][4]);
                const pair2 b22 = fma2(sub2(fma2(ey[G_V], K.inv_c, ey[G_D + 2]), ey[G_SIY]), K.inv_a, y[r][5]);
                const pair2 f = ball_scale2(fma2(b11, b11, fma2(b12, b12, fma2(b21, b21, mul2(b22, b22)))));
                y[r][2] = mul2(b11, f);
                y[r][3] = mul2(b12, f);
                y[r][4] = mul2(b21, f);
                y[r][5] = mul2(b22, f);
                six = ssix;
                siy = ssiy;
            }
            put_bot();
            // ---- div y^{k+1}, s^{k+1}, Lambda^{k+1}, bottom row first (row 0 needs the warp above)
#pragma unroll
            for (int r = R - 1; r >= 0; --r) {
                pair2 n[3], dn[3];
                if (r > 0) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) n[k] = y[r - 1][2 * k + 1];
                } else {
                    get_bot(n);
                }
                divr(r, y[r], n, dn);
                pair2 lin = fma2(iy[r], v[r], fma2(ix[r], u[r], G.it[wid * R + r][lane]));
                pair2 divt = fma2(iy[r], dn[2], mul2(ix[r], dn[1]));
                if (HAS_W) {
                    lin = fma2(K.beta, w[r], lin);
                    divt = fma2(K.beta, dn[0], divt);
                }
                pair2 inv_atc = K.inv_atc;
                if (PP) {
                    const pair2 ms = fma2(iy[r], iy[r], fma2(ix[r], ix[r], bc2(SK.beta * SK.beta)));
                    float m0, m1;
                    upk(ms, m0, m1);
                    inv_atc = pk(__frcp_rn(fmaxf(m0, 1e-12f) * SK.cc), __frcp_rn(fmaxf(m1, 1e-12f) * SK.cc));
                }
                const pair2 so = s[r];
                const pair2 sr = fma2(fma2(K.cc, divt, lin), inv_atc, mul2(G.kf[wid * R + r][lane], so));
                float s0, s1;
                upk(sr, s0, s1);
                s0 = fminf(fmaxf(s0, -K.lam), K.lam);
                s1 = fminf(fmaxf(s1, -K.lam), K.lam);
                const pair2 sn = pk(s0, s1), ns = pk(-s0, -s1);
                // minus the constraint residual A s^{k+1} - div y^{k+1}
                const pair2 ncw = HAS_W ? fma2(K.nbeta, sn, dn[0]) : 0ull;
                const pair2 ncu = fma2(ix[r], ns, dn[1]), ncv = fma2(iy[r], ns, dn[2]);
                if (!II) {
                    if (HAS_W) w[r] = fma2(K.rc, ncw, w[r]);
                    u[r] = fma2(K.rc, ncu, u[r]);
                    v[r] = fma2(K.rc, ncv, v[r]);
                } else {
                    const pair2 nrho = bc2(-SK.rho), nomr = bc2(-SK.omr), ncc = bc2(-SK.cc);
                    if (HAS_W)
                        w[r] = fma2(ncc, fma2(bc2(-SK.omr * SK.beta), so, fma2(nrho, dn[0], mul2(K.beta, sn))), w[r]);
                    u[r] = fma2(ncc, fma2(mul2(nomr, ix[r]), so, fma2(nrho, dn[1], mul2(ix[r], sn))), u[r]);
                    v[r] = fma2(ncc, fma2(mul2(nomr, iy[r]), so, fma2(nrho, dn[2], mul2(iy[r], sn))), v[r]);
                }
                if (last && A.a.partials) {
                    const int fr = wid * R + r;
                    const pair2 q = fma2(ncv, ncv, fma2(ncu, ncu, mul2(ncw, ncw)));
                    float q0, q1;
                    upk(q, q0, q1);
                    if (fr >= A.offy && fr < A.offy + A.oh && ib + r < H && 2 * lane >= A.offx && 2 * lane < A.offx + A.ow) {
                        if (c < W) res += q0;
                        if (c + 1 < W) res += q1;
                    }
                }
                s[r] = round2<T>(sn);
                if (HAS_W) w[r] = round2<TF>(w[r]);
                u[r] = round2<TF>(u[r]);
                v[r] = round2<TF>(v[r]);
                if (!std::is_same<T, float>::value) {  // the next iteration reads y as stored
#pragma unroll
                    for (int k = 2 * C0; k < 6; ++k) y[r][k] = round2<T>(y[r][k]);
#pragma unroll
                    for (int k = C0; k < 3; ++k) n[k] = round2<T>(n[k]);
                    divr(r, y[r], n, dn);
                }
#pragma unroll
                for (int k = C0; k < 3; ++k) d[r][k] = dn[k];
            }
            if (!last) put_top();
        }
        // ---- store the tile
        const bool inx = 2 * lane >= A.offx && 2 * lane < A.offx + A.ow;
        const bool ok0 = inx && (!BX || c < W), ok1 = inx && (!BX || c + 1 < W);
        const Fields &out = MODE == BATCHED ? G.pi[n % 3].buf[A.a.parity ^ 1] : A.a.out;
        auto store = [&](auto ST_, auto SF_) {
            auto plane = [&](auto f, void *p, auto val) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int fr = wid * R + r, i = ib + r;
                    if (fr >= A.offy && fr < A.offy + A.oh && i < H) f(p, (size_t)i * P + c, val(r));
                }
            };
#pragma unroll
            for (int k = 2 * C0; k < 6; ++k) plane(ST_, out.f[F_P1 + k], [&](int r) { return y[r][k]; });
            plane(ST_, out.f[F_S], [&](int r) { return s[r]; });
            if (HAS_W) plane(SF_, out.f[F_W], [&](int r) { return w[r]; });
            plane(SF_, out.f[F_U], [&](int r) { return u[r]; });
            plane(SF_, out.f[F_V], [&](int r) { return v[r]; });
        };
        if (ok0 && ok1 && (BX < 2 || A.vec)) {
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
            const double tot = block_sum((double)res, G.red);
            if (threadIdx.x == 0) A.a.partials[D.id] = tot;
        }
    }

    static __device__ __forceinline__ void run(const TileArgs &A) {
        extern __shared__ __align__(128) char smem_[];
        char *stage = smem_;
        SH &G = *reinterpret_cast<SH *>(smem_ + (STAGE ? ST::bytes : 0));
        const int lane = threadIdx.x & 31, wid = __shfl_sync(FULL, threadIdx.x >> 5, 0);
        if (MODE != BATCHED && A.a.done && *A.a.done) return;  // the pair's warp met its stopping test
        if (STAGE) {
            if (threadIdx.x == 0) {
                G.dead = 0;
                mbar_init(&G.full, 1);
                mbar_init_fence();
            }
            if (MODE == BATCHED && wid == 0) {
                for (int k = 0; k < 3; ++k) fetch_ref(A, G, blockIdx.x + k * gridDim.x, k, lane);
                cp_async_wait();
                __syncwarp();
                fetch_pair(A, G, 0, lane);
                fetch_pair(A, G, 1, lane);
                acquire_maps(A, 0, 1, lane);
                cp_async_wait();
            }
            __syncthreads();
            if (threadIdx.x == 0) prefetch(A, G, stage, blockIdx.x, 0);
            if (MODE == BATCHED && wid == 0) acquire_maps(A, 1, ACQUIRED - 1, lane);  // while the first copies arrive
        }
        int n = 0;
#pragma unroll 1
        for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x, ++n) {
            const Tile D = tile_at(A, G, t, n);
            const int fj = D.bx * A.ow - A.offx;
            if (fj >= 1 && fj + FW <= D.W - 1 && A.vec) {
                const int fi = D.by * A.oh - A.offy;
                if (fi >= 1 && fi + R * NW <= D.H - 1) body<0, false>(A, G, stage, D, n, lane, wid);
                else body<0, true>(A, G, stage, D, n, lane, wid);
            } else if (D.W % 2 == 0 && A.vec) {
                body<1, true>(A, G, stage, D, n, lane, wid);
            } else {
                body<2, true>(A, G, stage, D, n, lane, wid);
            }
        }
    }
};

template <typename T, typename TF, bool HAS_W, int VARIANT, int NW, int R, Mode MODE>
__global__ void __launch_bounds__(NW * 32, 1) k_admm_tile(const __grid_constant__ TileArgs A) {
    Kernel<T, TF, HAS_W, VARIANT, NW, R, MODE>::run(A);
}

template <typename T, typename TF, bool HAS_W, int VARIANT, int NW, int R, Mode MODE>
void launch_r(const TileArgs &a, cudaStream_t s) {
    constexpr int SMEM = (int)sizeof(Shared<NW, R>) + (MODE != DIRECT ? Stage<T, TF, NW * R>::bytes : 0);
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static DeviceOnce once;
    once.run(current_device(), [] {
        return cudaFuncSetAttribute(k_admm_tile<T, TF, HAS_W, VARIANT, NW, R, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    });
    const int blocks = MODE != DIRECT && a.ntiles > TILE_SMS ? TILE_SMS : a.ntiles;
    k_admm_tile<T, TF, HAS_W, VARIANT, NW, R, MODE><<<blocks, NW * 32, SMEM, s>>>(a);
}

// Blocks of TILE_WARPS warps where one tile per block is staged by its own loads; the looping forms
// run 8 warps of 6 rows with FP32 storage, which iterate faster (1.05 against 1.35 us for 48 rows: fewer
// rows are exchanged, and 255 registers hold the state without spills) but start more slowly (more
// straight-line code).  With 16-bit storage the roundings want the registers: 12 warps of 4 rows
// (a batch of 32 pairs with BF16 duals 151 against 155 ms).
template <typename T, typename TF, bool HAS_W, bool II> void launch_v(const TileArgs &a, cudaStream_t s) {
    constexpr int NW = TILE_WARPS, SW = sizeof(T) == 4 ? 8 : 12, SR = TILE_STAGED_HEIGHT / SW;
    if (a.a.k.a_tilde_mode == 1) {  // per-pixel a~: single pairs, one frame height
        if (a.staged) launch_r<T, TF, HAS_W, II | 2, SW, SR, STAGED>(a, s);
        else launch_r<T, TF, HAS_W, II | 2, NW, 4, DIRECT>(a, s);
        return;
    }
    if (a.a.tiles) return launch_r<T, TF, HAS_W, II, SW, SR, BATCHED>(a, s);
    if (a.staged) return launch_r<T, TF, HAS_W, II, SW, SR, STAGED>(a, s);
    switch (a.R) {
    case 2: return launch_r<T, TF, HAS_W, II, NW, 2, DIRECT>(a, s);
    case 3: return launch_r<T, TF, HAS_W, II, NW, 3, DIRECT>(a, s);
    default: return launch_r<T, TF, HAS_W, II, NW, 4, DIRECT>(a, s);
    }
}

template <typename T, typename TF> void launch_m(const TileArgs &a, cudaStream_t s) {
    const bool has_w = a.a.k.beta != 0.f;
    if (a.a.k.method == 1) has_w ? launch_v<T, TF, true, true>(a, s) : launch_v<T, TF, false, true>(a, s);
    else has_w ? launch_v<T, TF, true, false>(a, s) : launch_v<T, TF, false, false>(a, s);
}

}  // namespace tile
}  // namespace tvl1
