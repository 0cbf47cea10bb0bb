// k_cp_tile_bf16.cu -- the ALG1 tile kernel with BF16 data (k_cp_tile.cuh).
#include "k_cp_tile.cuh"

namespace tvl1 {

void cp_tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s) {
    flow32 ? cptile::launch_m<__nv_bfloat16, float>(a, s) : cptile::launch_m<__nv_bfloat16, __nv_bfloat16>(a, s);
}

}  // namespace tvl1
