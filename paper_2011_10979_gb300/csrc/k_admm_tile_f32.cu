// k_admm_tile_f32.cu -- FP32 instantiations of the ADMM tile kernel (k_admm_tile.cuh).
#include "k_admm_tile.cuh"

namespace tvl1 {

void tile_launch_f32(const TileArgs &a, cudaStream_t s) { tile::launch_m<float, float>(a, s); }

}  // namespace tvl1
