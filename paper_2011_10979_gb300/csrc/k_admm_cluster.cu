// k_admm_cluster.cu -- launch policy of the ADMM methods' register-resident cluster engine
// (k_admm_cluster.cuh): the tiling of a level over one cluster, storage-type dispatch.
#include "k_admm_cluster.cuh"

#include <algorithm>

namespace tvl1 {

namespace {

template <typename T, typename TF, bool HAS_W, bool II, int R> cudaError_t launch_r(const ResArgs &a, int nc, cudaStream_t s) {
    auto kern = cluster::k_admm_cluster<T, TF, HAS_W, II, R>;
    static DeviceOnce once;
    const int prep = once.run(current_device(), [&] {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(cluster::Shared));
        return e != cudaSuccess ? e : cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
    if (prep != cudaSuccess) return (cudaError_t)prep;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3((a.oh + 2 * cluster::HALO + R - 1) / R * 32);
    cfg.dynamicSmemBytes = sizeof(cluster::Shared);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// One row per warp while eight warps hold the frame, else two.
template <typename T, typename TF, bool HAS_W, bool II> cudaError_t launch(const ResArgs &a, int nc, cudaStream_t s) {
    return a.oh + 2 * cluster::HALO <= cluster::MAXWARPS ? launch_r<T, TF, HAS_W, II, 1>(a, nc, s)
                                                         : launch_r<T, TF, HAS_W, II, 2>(a, nc, s);
}

template <typename T, typename TF> cudaError_t launch_m(const ResArgs &a, int nc, cudaStream_t s) {
    const bool has_w = a.k.beta != 0.f;
    if (a.k.method == 1) return has_w ? launch<T, TF, true, true>(a, nc, s) : launch<T, TF, false, true>(a, nc, s);
    return has_w ? launch<T, TF, true, false>(a, nc, s) : launch<T, TF, false, false>(a, nc, s);
}

}  // namespace

// The tiling with the fewest rows per CTA: gx columns of tiles, at most nc / gx rows of them.  A tile is as
// high as a halo at least, and with more than one column its frame has a lane's two columns on either side.
bool admm_cluster_plan(Geom g, int nc, ResArgs *a) {
    int best = 0;
    for (int n = 1; n <= nc; ++n) {
        const int ow = ((g.W + n - 1) / n + 1) / 2 * 2, gx = (g.W + ow - 1) / ow;
        if (gx != n || ow > (gx > 1 ? 64 - 2 * cluster::HALO : 64)) continue;
        const int gy = nc / gx, oh = std::max((g.H + gy - 1) / gy, cluster::HALO);
        if (oh + 2 * cluster::HALO > cluster::MAXROWS || (best && oh >= best)) continue;
        best = oh;
        if (a) {
            a->gx = gx;
            a->ow = ow;
            a->oh = oh;
        }
    }
    return best > 0;
}

cudaError_t launch_admm_cluster(const ResArgs &a, int nc, int prec, int prec_flow, cudaStream_t s) {
    if (prec == PREC_F32) return launch_m<float, float>(a, nc, s);
    if (prec == PREC_F16)
        return prec_flow == PREC_F32 ? launch_m<__half, float>(a, nc, s) : launch_m<__half, __half>(a, nc, s);
    return prec_flow == PREC_F32 ? launch_m<__nv_bfloat16, float>(a, nc, s) : launch_m<__nv_bfloat16, __nv_bfloat16>(a, nc, s);
}

}  // namespace tvl1
