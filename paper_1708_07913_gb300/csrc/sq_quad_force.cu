// sq_quad_force.cu -- instantiations and launches of the quad force kernels.
#include "sq_quad_force.cuh"

namespace sq {

template <int M>
static int config_m(int ccap, int lb, int npl, size_t* smem)
{
    const size_t bytes = quad_smem_bytes<M>(true, ccap, lb, quad_force_npl(npl));
    const void* fn = (const void*)quad_force_kernel<M>;
    cudaFuncAttributes fa;                       // the limit only ever grows (see sq_region_dispatch.cuh)
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
        cudaGetLastError();
        return SQ_ECUDA;
    }
    if (bytes > 232448 - fa.sharedSizeBytes) return SQ_EUNSUPPORTED;
    if ((int)bytes > fa.maxDynamicSharedSizeBytes &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) {
        cudaGetLastError();
        return SQ_EUNSUPPORTED;
    }
    *smem = bytes;
    return SQ_OK;
}

template <int M>
static int launch_m(const QuadForceArgs& f, size_t smem, int blocks, cudaStream_t st)
{
    quad_force_kernel<M><<<blocks, QD_NT, smem, st>>>(f);
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

int quad_force_config(int m, int ccap, int lb, int npl, size_t* smem)
{
    switch (m) {
#define C(M) case M: return config_m<M>(ccap, lb, npl, smem);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

int quad_force_launch(int m, const QuadForceArgs& f, size_t smem, int blocks, cudaStream_t st)
{
    switch (m) {
#define C(M) case M: return launch_m<M>(f, smem, blocks, st);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

// cos(j pi (k + 1/2) / (n_pl + 1)), j and k from 0 to n_pl.
__global__ void chebyshev_table_kernel(int npl, double* tab)
{
    const int n = npl + 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * n; i += gridDim.x * blockDim.x)
        tab[i] = cos((i / n) * (M_PI * (i % n + 0.5) / n));
}

int launch_chebyshev_table(int npl, double* tab, cudaStream_t st)
{
    chebyshev_table_kernel<<<((npl + 1) * (npl + 1) + 127) / 128, 128, 0, st>>>(npl, tab);
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

}  // namespace sq
