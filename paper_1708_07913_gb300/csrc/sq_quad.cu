// sq_quad.cu -- instantiations and launches of the FP32 quad kernels.
#include "sq_quad.cuh"

namespace sq {

template <int M>
static int config_m(int which, bool has_nl, int ccap, int lb, int npl, size_t* smem)
{
    const size_t bytes = quad_smem_bytes<M>(has_nl, ccap, lb, which == 0 ? npl : 0);
    const void* fn = nullptr;
    if (which == 0) fn = (const void*)quad_kernel<M, false>;
    else if constexpr (quad_has_lanczos(M)) fn = (const void*)quad_kernel<M, true>;
    if (!fn) return SQ_EUNSUPPORTED;
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
static int launch_m(int which, const QuadArgs& a, size_t smem, int blocks, cudaStream_t st)
{
    if (which == 0) quad_kernel<M, false><<<blocks, QD_NT, smem, st>>>(a);
    else if constexpr (quad_has_lanczos(M)) quad_kernel<M, true><<<blocks, QD_NT, smem, st>>>(a);
    else return SQ_EUNSUPPORTED;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

// Shared memory of the quad kernel `which` (0 moments, 1 Lanczos) for regions
// of half-width m and a context's projector tables; SQ_EUNSUPPORTED: none, or
// the tables do not fit.
int quad_config(int m, int which, bool has_nl, int ccap, int lb, int npl, size_t* smem)
{
    switch (m) {
#define C(M) case M: return config_m<M>(which, has_nl, ccap, lb, npl, smem);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

int quad_launch(int m, int which, const QuadArgs& a, size_t smem, int blocks, cudaStream_t st)
{
    switch (m) {
#define C(M) case M: return launch_m<M>(which, a, smem, blocks, st);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

}  // namespace sq
