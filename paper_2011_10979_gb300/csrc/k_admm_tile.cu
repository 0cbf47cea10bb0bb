// k_admm_tile.cu -- launch policy of the ADMM tile kernel (k_admm_tile.cuh): the frame height and
// iterations per launch of a level, the tensor maps of its staged form, storage-type dispatch.
#include <cudaTypedefs.h>

#include <algorithm>

#include "tvl1_internal.h"

namespace tvl1 {

void tile_launch_f32(const TileArgs &a, cudaStream_t s);
void tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s);
void tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s);

namespace {

// The tiling of a level into frames of 64 x TILE_WARPS R (staged: 64 x 48) with ni iterations of halo.
// Staged frames start at multiples of 4 columns (16-byte aligned copies), the others at even ones.
TilePlan plan_of(Geom g, int R, int ni, bool staged) {
    TilePlan p;
    p.R = R;
    p.ni = ni;
    p.staged = staged;
    const int al = staged ? 4 : 2;
    p.offx = (ni + 1 + al - 1) / al * al;
    p.offy = ni + 1;
    p.ow = (64 - p.offx - ni) / al * al;
    p.oh = (staged ? TILE_STAGED_HEIGHT : TILE_WARPS * R) - 2 * ni - 1;
    p.gx = (g.W + p.ow - 1) / p.ow;
    p.gy = (g.H + p.oh - 1) / p.oh;
    return p;
}

// Microseconds of one launch of the plan, fitted to launches inside a CUDA graph (per round of tiles
// over the SMs: a part per tile and one per iteration; FP32, beta > 0).  Measured against it: 320x240,
// R = 2, five iterations 8.4 us; 640x480, R = 4, three 10.6 and R = 3, six 20.7; 1024x436 staged, six
// 27.1 and R = 3, three 14.5; 3840x2160 staged, four 239.
float plan_us(const TilePlan &p, int R, int ni) {
    static const float per_iter[5] = {0.f, 0.f, 0.95f, 1.2f, 1.7f}, per_tile[5] = {0.f, 0.f, 3.2f, 3.7f, 4.9f};
    const int n = p.gx * p.gy, rounds = (n + TILE_SMS - 1) / TILE_SMS;
    return p.staged ? 3.4f + rounds * (3.8f + 1.25f * ni) : 0.4f + rounds * (per_tile[R] + ni * per_iter[R]);
}
float plan_us(const TilePlan &p) { return plan_us(p, p.R, p.ni); }

}  // namespace

TilePlan admm_tile_plan(Geom g, int ni, bool direct) {
    TilePlan best;
    float us = 0.f;
    for (int k = ni ? ni : 1; k <= (ni ? ni : TILE_MAX_ITERS); ++k)
        for (int R = 2; R <= (direct ? 4 : 5); ++R) {  // 5: staged
            const TilePlan p = plan_of(g, R, k, R == 5);
            if (p.oh < 1) continue;
            const float t = plan_us(p) / k;
            if (us == 0.f || t < us) {
                us = t;
                best = p;
            }
        }
    return best;
}

TilePlan admm_tile_plan_tested(Geom g, bool direct) {
    const TilePlan a = admm_tile_plan(g, TILE_ITERS, direct), b = admm_tile_plan(g, TILE_TEST_ITERS, direct);
    return 2 * plan_us(b) < 3 * plan_us(a) + plan_us(a, a.R, 1) ? b : a;
}

// Batches run the staged form; the iterations per launch that cost the least over all pairs' tiles.
TilePlan admm_tile_plan_batch(const Geom *g, int n, int ni) {
    TilePlan best;
    float us = 0.f;
    for (int k = ni ? ni : 1; k <= (ni ? ni : TILE_MAX_ITERS); ++k) {
        TilePlan p;
        int tiles = 0;
        for (int q = 0; q < n; ++q) {
            p = plan_of(g[q], 5, k, true);
            tiles += p.gx * p.gy;
        }
        p.gx = tiles;
        p.gy = 1;
        const float t = plan_us(p) / k;
        if (us == 0.f || t < us) {
            us = t;
            best = p;
        }
    }
    return best;
}

float admm_tile_us(const TilePlan &p, int ni, bool per_pixel) { return plan_us(p, per_pixel ? 4 : p.R, ni); }

int admm_tile_blocks(const TilePlan &p) { return p.gx * p.gy; }

void tile_set_plan(TileArgs &t, const TilePlan &p, int ni) {
    t.R = p.R;
    t.ni = ni;
    t.offx = p.offx;
    t.offy = p.offy;
    t.ow = p.ow;
    t.oh = p.oh;
    t.gx = p.gx;
    t.ntiles = p.gx * p.gy;
    t.staged = p.staged;
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 map_encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 enc = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }();
    return enc;
}

}  // namespace

bool tile_maps_available() { return map_encoder() != nullptr; }

bool tile_encode_maps(CUtensorMap *maps, const Fields &f, const void *Ix, const void *Iy, Geom g, int prec,
                      int prec_flow, bool has_w, bool pdr) {
    const PFN_cuTensorMapEncodeTiled_v12000 enc = map_encoder();
    if (!enc) return false;
    auto one = [&](CUtensorMap *m, const void *base, size_t plane, int n, int pr) {
        const int eb = (int)prec_bytes(pr);
        const cuuint64_t dim[3] = {(cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)n};
        const cuuint64_t stride[2] = {(cuuint64_t)g.pitch * eb, (cuuint64_t)plane};
        const cuuint32_t box[3] = {eb == 4 ? 64u : 72u, (cuuint32_t)TILE_STAGED_HEIGHT, (cuuint32_t)n}, es[3] = {1, 1, 1};
        const CUtensorMapDataType dt = pr == PREC_F32   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                       : pr == PREC_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                        : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
        return enc(m, dt, 3, const_cast<void *>(base), dim, stride, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    const size_t ps = (size_t)((const char *)f.f[1] - (const char *)f.f[0]), pd = (size_t)((const char *)Iy - (const char *)Ix);
    return one(&maps[0], f.f[has_w ? F_W : F_U], ps, has_w ? 3 : 2, prec_flow) &&
           one(&maps[1], f.f[has_w ? F_P1 : F_Q11], ps, (has_w ? 7 : 5) - pdr, prec) && one(&maps[2], Ix, pd, 3, prec) &&
           (!pdr || one(&maps[3], f.f[has_w ? F_WB : F_UB], ps, has_w ? 3 : 2, prec_flow));
}

void launch_admm_tile(const TileArgs &a, int prec, int prec_flow, cudaStream_t s) {
    if (prec == PREC_F32) tile_launch_f32(a, s);
    else if (prec == PREC_F16) tile_launch_f16(a, prec_flow == PREC_F32, s);
    else tile_launch_bf16(a, prec_flow == PREC_F32, s);
}

}  // namespace tvl1
