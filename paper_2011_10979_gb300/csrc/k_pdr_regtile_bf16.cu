// k_pdr_regtile_bf16.cu -- the pDR register tile kernel with BF16 duals and data (k_pdr_regtile.cuh).
#include "k_pdr_regtile.cuh"

namespace tvl1 {

void pdr_tile_launch_bf16(const TileArgs &a, bool flow32, cudaStream_t s) {
    flow32 ? pdrtile::launch_m<__nv_bfloat16, float>(a, s) : pdrtile::launch_m<__nv_bfloat16, __nv_bfloat16>(a, s);
}

}  // namespace tvl1
