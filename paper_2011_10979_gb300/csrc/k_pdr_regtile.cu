// k_pdr_regtile.cu -- launch policy of the pDR register tile kernel (k_pdr_regtile.cuh): the iterations per
// launch of a level, storage-type dispatch.
#include "k_pdr_regtile.cuh"

namespace tvl1 {

// Microseconds of a launch of k iterations, fitted to launches of one round before the divisions left the usual body
// (640x480, one iteration, 10.8 us; 320x240, five, 21.6; now 9.0 and 19.4, both a tenth or so less).
float pdr_regtile_us(const TilePlan &p, int k) {
    const int rounds = (p.gx * p.gy + TILE_SMS - 1) / TILE_SMS;
    return 0.4f + rounds * (7.7f + 2.7f * k);
}

// The tiling of a level into frames of 64 x TILE_STAGED_HEIGHT with the least estimated time per iteration:
// an iteration takes three pixels of halo on every side and one more on the east and south.  Frames
// start at multiples of four columns (16-byte aligned copies) and of two rows (a row's colours).
TilePlan pdr_regtile_plan(Geom g, int max_ni) {
    TilePlan best;
    float us = 0.f;
    for (int k = 1; k <= max_ni && k <= 5; ++k) {
        TilePlan p;
        p.ni = k;
        p.staged = true;
        p.offx = (3 * k + 3) / 4 * 4;
        p.offy = (3 * k + 1) / 2 * 2;
        p.ow = (64 - p.offx - (3 * k + 1)) / 4 * 4;
        p.oh = (TILE_STAGED_HEIGHT - p.offy - (3 * k + 1)) / 2 * 2;
        p.gx = (g.W + p.ow - 1) / p.ow;
        p.gy = (g.H + p.oh - 1) / p.oh;
        const float t = pdr_regtile_us(p, k) / k;
        if (us == 0.f || t < us) {
            us = t;
            best = p;
        }
    }
    return best;
}

void launch_pdr_regtile(const TileArgs &a, int prec, int prec_flow, cudaStream_t s) {
    if (prec == PREC_F32) pdrtile::launch_m<float, float>(a, s);
    else if (prec == PREC_F16) pdr_tile_launch_f16(a, prec_flow == PREC_F32, s);
    else pdr_tile_launch_bf16(a, prec_flow == PREC_F32, s);
}

}  // namespace tvl1
