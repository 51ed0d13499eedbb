// Launch of the packed engines: clusters FP32-mixed and FP64 (gfmc_packed.cuh),
// FP64 small tiles on a cluster or on the whole grid (gfmc_packed64.cuh), chains on
// one CTA (gfmc_team.cuh).
#include "gfmc_packed64.cuh"
#include "gfmc_team.cuh"

namespace gfmc {

namespace {

using PkKernel = void (*)(const TeamJob*);

// engine: 0 FP64 and 1 FP32-mixed clusters, 2 FP64 clusters with small tiles
PkKernel pk_kernel(int engine)
{
    return engine == 0 ? gfmc_packed_cluster<double> : engine == 1 ? gfmc_packed_cluster<float> : gfmc_packed64_cluster;
}
int pk_block(int engine) { return engine == 0 ? kPkThreads64 : engine == 1 ? kPkThreads32 : kPk64Threads; }

cudaError_t pk_config(int engine, int njobs, int C, int smem, cudaStream_t s, cudaLaunchConfig_t* cfg,
                      cudaLaunchAttribute* attr)
{
    cudaError_t e = allow_dynamic_smem((const void*)pk_kernel(engine));
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute((const void*)pk_kernel(engine), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    *cfg = {};
    cfg->gridDim = dim3((unsigned)(C * njobs));
    cfg->blockDim = dim3((unsigned)pk_block(engine));
    cfg->dynamicSmemBytes = (size_t)smem;
    cfg->stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
}

}  // namespace

cudaError_t launch_packed(int engine, const TeamJob* d_jobs, int njobs, int C, int smem, cudaStream_t s)
{
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    cudaError_t e = pk_config(engine, njobs, C, smem, s, &cfg, attr);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, pk_kernel(engine), d_jobs);
}

cudaError_t launch_packed_single(int engine, const Params& p, int smem, cudaStream_t s)
{
    const auto fn = engine == 1 ? gfmc_packed_single<float> : gfmc_packed_single<double>;
    cudaError_t e = allow_dynamic_smem((const void*)fn);
    if (e == cudaSuccess && p.ncta > 8)
        e = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    if (e == cudaSuccess) e = pk_config(engine, 1, p.ncta, smem, s, &cfg, attr);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, fn, p);
}

// six clusters of p.ncta CTAs
cudaError_t launch_packed64_moments(const Params& p, int smem, cudaStream_t s)
{
    cudaError_t e = allow_dynamic_smem((const void*)gfmc_packed64_moments);
    if (e == cudaSuccess && p.ncta > 8)
        e = cudaFuncSetAttribute((const void*)gfmc_packed64_moments, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    if (e == cudaSuccess) e = pk_config(2, 6, p.ncta, smem, s, &cfg, attr);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, gfmc_packed64_moments, p);
}

cudaError_t packed_max_active(int engine, int C, int smem, int* out)
{
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    cudaError_t e = pk_config(engine, 1, C, smem, nullptr, &cfg, attr);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveClusters(out, pk_kernel(engine), &cfg);
}

cudaError_t packed_static_smem(int engine, int* out)
{
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, (const void*)pk_kernel(engine));
    if (e == cudaSuccess) *out = (int)a.sharedSizeBytes;
    return e;
}

cudaError_t launch_packed64_grid(const Params& p, int smem, cudaStream_t s)
{
    cudaError_t e = allow_dynamic_smem((const void*)gfmc_packed64_grid);
    if (e != cudaSuccess) return e;
    Params q = p;
    void* args[] = {(void*)&q};
    return cudaLaunchCooperativeKernel((void*)gfmc_packed64_grid, dim3((unsigned)p.ncta), dim3(kPk64Threads), args,
                                       (size_t)smem, s);
}

cudaError_t packed64_grid_max_ctas(int smem, int* out)
{
    cudaError_t e = allow_dynamic_smem((const void*)gfmc_packed64_grid);
    int per_sm = 0, dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gfmc_packed64_grid, kPk64Threads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *out = per_sm > 0 ? sms : 0;  // one CTA per SM
    return e;
}

using OneCtaKernel = void (*)(const Params, int);
static OneCtaKernel one_cta_kernel(int precision, int N)
{
    if (precision == 0) return gfmc_one_cta<double, 2 * kThreads>;
    return one_cta_threads(precision, N) == kThreads ? gfmc_one_cta<float, kThreads> : gfmc_one_cta<float, 2 * kThreads>;
}

cudaError_t launch_one_cta(int precision, const Params& p, int smem, cudaStream_t s)
{
    const OneCtaKernel fn = one_cta_kernel(precision, p.N);
    const cudaError_t e = allow_dynamic_smem((const void*)fn);
    if (e != cudaSuccess) return e;
    fn<<<1, one_cta_threads(precision, p.N), smem, s>>>(p, smem / (int)sizeof(double2));
    return cudaGetLastError();
}

bool one_cta_fits(int precision, int N, int smem)
{
    const OneCtaKernel fn = one_cta_kernel(precision, N);
    int n = 0;
    const bool ok = allow_dynamic_smem((const void*)fn) == cudaSuccess &&
                    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, one_cta_threads(precision, N), smem) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

}  // namespace gfmc
