// k_admm_tile_bf16_all.cu -- instantiations of the ADMM tile kernel (k_admm_tile.cuh) with every plane
// in BF16.
#include "k_admm_tile.cuh"

namespace tvl1 {

void tile_launch_bf16_all(const TileArgs &a, cudaStream_t s) { tile::launch_m<__nv_bfloat16, __nv_bfloat16>(a, s); }

}  // namespace tvl1
