// plane_relax_inst.cu -- instantiates the FP64 plane-relaxation kernels for one x-line chunk size
// K = SMG_K (rows per lane; nx <= 32 K).  The build compiles this unit once per K so the
// instantiations compile in parallel.
#include "plane_lean.cuh"
#include "plane_relax.cuh"

#if !defined(SMG_K)
#error "compile with -DSMG_K=<rows per lane>"
#endif

namespace smg {

#define SMG_CAT2(a, b) a##b
#define SMG_NAME(base, k) SMG_CAT2(base, k)

// a.R > 1: one thread-block cluster of a.R CTAs per plane.
cudaError_t SMG_NAME(launch_plane_relax_k, SMG_K)(int nplanes, int nb, int threads, const PlaneRelaxArgs &a, size_t smem,
                                                  cudaStream_t st) {
    return a.R > 1 ? launch_pr<double, double, SMG_K, true>(nplanes, nb, threads, a, smem, st)
                   : launch_pr<double, double, SMG_K, false>(nplanes, nb, threads, a, smem, st);
}

int SMG_NAME(set_plane_relax_smem_k, SMG_K)(bool cl, size_t smem) {
    return cl ? set_smem_attr<double, double, SMG_K, true>(smem) : set_smem_attr<double, double, SMG_K, false>(smem);
}

bool SMG_NAME(cluster_resident_k, SMG_K)(int R, int threads, size_t smem) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(R, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = R;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, plane_relax_kernel<double, double, SMG_K, true>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

#if SMG_K <= 8
// The shortened-step plane cycle (plane_lean.cuh) on one CTA or a cluster (a.R > 1) per plane.
cudaError_t SMG_NAME(launch_plane_lean_k, SMG_K)(int nplanes, int nb, int threads, const PlaneRelaxArgs &a, size_t smem,
                                                 cudaStream_t st) {
    return a.R > 1 ? launch_lean<double, double, SMG_K, true>(nplanes, nb, threads, a, smem, st)
                   : launch_lean<double, double, SMG_K, false>(nplanes, nb, threads, a, smem, st);
}
int SMG_NAME(set_plane_lean_smem_k, SMG_K)(bool cl, size_t smem) {
    return cl ? set_lean_smem_attr<double, double, SMG_K, true>(smem) : set_lean_smem_attr<double, double, SMG_K, false>(smem);
}
bool SMG_NAME(lean_cluster_resident_k, SMG_K)(int R, int threads, size_t smem) {
    return lean_cluster_resident<double, double, SMG_K>(R, threads, smem);
}
#endif

}  // namespace smg
