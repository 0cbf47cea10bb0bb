// k_pdr_regtile_f16.cu -- the pDR register tile kernel with FP16 duals and data (k_pdr_regtile.cuh).
#include "k_pdr_regtile.cuh"

namespace tvl1 {

void pdr_tile_launch_f16(const TileArgs &a, bool flow32, cudaStream_t s) {
    flow32 ? pdrtile::launch_m<__half, float>(a, s) : pdrtile::launch_m<__half, __half>(a, s);
}

}  // namespace tvl1
