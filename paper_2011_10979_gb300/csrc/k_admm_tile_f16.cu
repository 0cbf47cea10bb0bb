// k_admm_tile_f16.cu -- instantiations of the ADMM tile kernel (k_admm_tile.cuh) with F16 duals and
// data, the flow in FP32.
#include "k_admm_tile.cuh"

namespace tvl1 {

void tile_launch_f16_all(const TileArgs &a, cudaStream_t s);

void tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s) {
    if (flow32) tile::launch_m<__half, float>(a, s);
    else tile_launch_f16_all(a, s);
}

}  // namespace tvl1
