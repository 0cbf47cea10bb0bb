// k_cp_tile_f16.cu -- the ALG1 tile kernel with FP16 data (k_cp_tile.cuh).
#include "k_cp_tile.cuh"

namespace tvl1 {

void cp_tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s) {
    flow32 ? cptile::launch_m<__half, float>(a, s) : cptile::launch_m<__half, __half>(a, s);
}

}  // namespace tvl1
