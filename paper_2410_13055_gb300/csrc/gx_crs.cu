// Launches of the cluster-resident solver (kernel: gx_crs.cuh).
#include "gx_internal.cuh"

namespace gx {

CrsFn crs_pick_fwd1(int kw, int hpl, int reg);
CrsFn crs_pick_fwd4(int kw, int hpl, int reg);
CrsFn crs_pick_adj1(int kw, int hpl, int reg);
CrsFn crs_pick_adj4(int kw, int hpl, int reg);

namespace {

CrsFn crs_kernel(int adj, const CrsShape& p) {
    if (adj) return p.V == 4 ? crs_pick_adj4(p.kw, p.hpl, p.reg) : crs_pick_adj1(p.kw, p.hpl, p.reg);
    return p.V == 4 ? crs_pick_fwd4(p.kw, p.hpl, p.reg) : crs_pick_fwd1(p.kw, p.hpl, p.reg);
}

void crs_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int nclusters, int C, int threads, size_t smem,
                cudaStream_t st) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(nclusters * C));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

}  // namespace

// Launch groups share instantiations with different image sizes, so each instantiation is
// opened to the largest image and to non-portable cluster sizes; a launch states its own size.
cudaError_t crs_prepare(int adj, const CrsShape& p) {
    const void* f = reinterpret_cast<const void*>(crs_kernel(adj, p));
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCrsSmemMax);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

int crs_max_clusters(int adj, const CrsShape& p, size_t smem) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    crs_config(cfg, at, 1, p.C, p.threads, smem, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(crs_kernel(adj, p)), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

int launch_crs(const Ctx& c, const CrsTables& tab, int adj, const int4* runs, int n, const CrsShape& p, double tol, cudaStream_t st) {
    if (n <= 0) return 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    crs_config(cfg, at, n, p.C, p.threads, p.smem[adj], st);
    cudaLaunchKernelEx(&cfg, crs_kernel(adj, p), c, tab, runs, p.C, p.bat_smem[adj], tol);
    return 1;
}

}  // namespace gx
