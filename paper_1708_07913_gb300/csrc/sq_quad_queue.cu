// sq_quad_queue.cu -- instantiations and launches of the quad kernels that a
// batch's queue feeds.
#include "sq_quad.cuh"

namespace sq {

template <int M>
static int launch_m(int which, const QuadQueueArgs& q, size_t smem, int blocks, cudaStream_t st)
{
    if (which == 0) quad_queue_kernel<M, false><<<blocks, QD_NT, smem, st>>>(q);
    else if constexpr (quad_has_lanczos(M)) quad_queue_kernel<M, true><<<blocks, QD_NT, smem, st>>>(q);
    else return SQ_EUNSUPPORTED;
    return cudaGetLastError() == cudaSuccess ? SQ_OK : SQ_ECUDA;
}

template <int M>
static int config_m(int which, size_t smem)
{
    const void* fn = nullptr;
    if (which == 0) fn = (const void*)quad_queue_kernel<M, false>;
    else if constexpr (quad_has_lanczos(M)) fn = (const void*)quad_queue_kernel<M, true>;
    if (!fn) return SQ_EUNSUPPORTED;
    cudaFuncAttributes fa;                       // the limit only ever grows (see sq_region_dispatch.cuh)
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
        cudaGetLastError();
        return SQ_ECUDA;
    }
    if (smem > 232448 - fa.sharedSizeBytes) return SQ_EUNSUPPORTED;
    if ((int)smem > fa.maxDynamicSharedSizeBytes &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return SQ_EUNSUPPORTED;
    }
    return SQ_OK;
}

int quad_queue_config(int m, int which, size_t smem)
{
    switch (m) {
#define C(M) case M: return config_m<M>(which, smem);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

int quad_queue_launch(int m, int which, const QuadQueueArgs& q, size_t smem, int blocks, cudaStream_t st)
{
    switch (m) {
#define C(M) case M: return launch_m<M>(which, q, smem, blocks, st);
        QUAD_CASES
#undef C
    }
    return SQ_EUNSUPPORTED;
}

}  // namespace sq
