// k_admm_tile_f16_all.cu -- instantiations of the ADMM tile kernel (k_admm_tile.cuh) with every plane
// in F16.
#include "k_admm_tile.cuh"

namespace tvl1 {

void tile_launch_f16_all(const TileArgs &a, cudaStream_t s) { tile::launch_m<__half, __half>(a, s); }

}  // namespace tvl1
