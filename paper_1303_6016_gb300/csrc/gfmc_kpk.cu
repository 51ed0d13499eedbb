// Launch of the packed cluster engine (gfmc_packed.cuh), FP64 and FP32-mixed.
#include "gfmc_packed.cuh"

namespace gfmc {

namespace {

template <class R> cudaError_t pk_config(int C)
{
    cudaError_t e = allow_dynamic_smem((const void*)gfmc_packed_cluster<R>);
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(gfmc_packed_cluster<R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <class R>
cudaLaunchConfig_t pk_launch_config(int njobs, int C, int smem, cudaStream_t s, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C * njobs));
    cfg.blockDim = dim3(pk_threads<R>());
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <class R> cudaError_t pk_launch(const TeamJob* d_jobs, int njobs, int C, int smem, cudaStream_t s)
{
    cudaError_t e = pk_config<R>(C);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = pk_launch_config<R>(njobs, C, smem, s, attr);
    return cudaLaunchKernelEx(&cfg, gfmc_packed_cluster<R>, d_jobs);
}

template <class R> cudaError_t pk_max_active(int C, int smem, int* out)
{
    cudaError_t e = pk_config<R>(C);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = pk_launch_config<R>(1, C, smem, nullptr, attr);
    return cudaOccupancyMaxActiveClusters(out, gfmc_packed_cluster<R>, &cfg);
}

template <class R> cudaError_t pk_static_smem(int* out)
{
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, gfmc_packed_cluster<R>);
    if (e == cudaSuccess) *out = (int)a.sharedSizeBytes;
    return e;
}

}  // namespace

cudaError_t launch_packed(int precision, const TeamJob* d_jobs, int njobs, int C, int smem, cudaStream_t s)
{
    return precision == 0 ? pk_launch<double>(d_jobs, njobs, C, smem, s) : pk_launch<float>(d_jobs, njobs, C, smem, s);
}

cudaError_t packed_max_active(int precision, int C, int smem, int* out)
{
    return precision == 0 ? pk_max_active<double>(C, smem, out) : pk_max_active<float>(C, smem, out);
}

cudaError_t packed_static_smem(int precision, int* out)
{
    return precision == 0 ? pk_static_smem<double>(out) : pk_static_smem<float>(out);
}

}  // namespace gfmc
