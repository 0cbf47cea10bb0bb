// k_cp_tile.cu -- launch policy of the ALG1 tile kernel (k_cp_tile.cuh): the frame height and
// iterations per launch of a level, storage-type dispatch.
#include "k_cp_tile.cuh"

namespace tvl1 {

// Estimated microseconds of a launch of k iterations, fitted to launches inside a CUDA graph (per round of tiles over the
// SMs a part per tile and one per iteration; FP32, beta > 0).  Measured against it: 320x240, R = 2, six
// iterations 8.2 us; 640x480, R = 4, three 10.4 and four 11.9, R = 3, six 20.4; 3840x2160, R = 4, six 414.
float cp_tile_us(const TilePlan &p, int k) {
    static const float per_iter[5] = {0.f, 0.f, 0.72f, 1.12f, 1.5f}, per_tile[5] = {0.f, 0.f, 3.5f, 3.9f, 5.4f};
    const int rounds = (p.gx * p.gy + TILE_SMS - 1) / TILE_SMS;
    return 0.4f + rounds * (per_tile[p.R] + k * per_iter[p.R]);
}

// Ten tested iterations as 3, 3, 3 and one on k_cp (some 2.8 us, 9 at 640x480), or as 5 and 5.
TilePlan cp_tile_plan_tested(Geom g) {
    const TilePlan a = cp_tile_plan(g, TILE_ITERS), b = cp_tile_plan(g, TILE_TEST_ITERS);
    return 2 * cp_tile_us(b, 5) < 3 * cp_tile_us(a, 3) + 2.8f + 2e-5f * (float)g.H * (float)g.W ? b : a;
}

// The tiling of a level into frames of 64 x TILE_WARPS R whose outermost ni pixels are halo (the west
// side rounded up to the even columns that frames start at), with the least estimated time per
// iteration.
TilePlan cp_tile_plan(Geom g, int ni) {
    TilePlan best;
    float us = 0.f;
    for (int k = ni ? ni : 1; k <= (ni ? ni : TILE_MAX_ITERS); ++k)
        for (int R = 2; R <= 4; ++R) {
            TilePlan p;
            p.R = R;
            p.ni = k;
            p.offx = (k + 1) / 2 * 2;
            p.offy = k;
            p.ow = (64 - p.offx - k) / 2 * 2;
            p.oh = TILE_WARPS * R - 2 * k;
            p.gx = (g.W + p.ow - 1) / p.ow;
            p.gy = (g.H + p.oh - 1) / p.oh;
            const float t = cp_tile_us(p, k) / k;
            if (us == 0.f || t < us) {
                us = t;
                best = p;
            }
        }
    return best;
}

void launch_cp_tile(const TileArgs &a, int prec, int prec_flow, cudaStream_t s) {
    if (prec == PREC_F32) cptile::launch_m<float, float>(a, s);
    else if (prec == PREC_F16) cp_tile_launch_f16(a, prec_flow == PREC_F32, s);
    else cp_tile_launch_bf16(a, prec_flow == PREC_F32, s);
}

}  // namespace tvl1
