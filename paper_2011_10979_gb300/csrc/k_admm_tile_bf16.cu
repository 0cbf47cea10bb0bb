// k_admm_tile_bf16.cu -- instantiations of the ADMM tile kernel (k_admm_tile.cuh) with BF16 duals and
// data, the flow in FP32.
#include "k_admm_tile.cuh"

namespace tvl1 {

void tile_launch_bf16_all(const TileArgs &a, cudaStream_t s);

void tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s) {
    if (flow32) tile::launch_m<__nv_bfloat16, float>(a, s);
    else tile_launch_bf16_all(a, s);
}

}  // namespace tvl1
