// ann_search_grp.cu -- the kernels that walk indexes with the c2 group level
// (Algorithm 1, Sec. 4.2), instantiated in their own translation unit so that
// the kernels of indexes without groups keep their own register allocation and
// both compile in parallel.
#include "ann_search_dev.cuh"

namespace ann {

// the function's dynamic shared-memory limit is raised once to the opt-in
// maximum (a captured graph may hold nodes of one kernel with different sizes)
template <class F>
static cudaError_t config_one(F kernel, bool &raised, size_t smem, int threads, int *blocks_per_sm) {
    if (!raised) {
        int dev = 0, optin = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (e != cudaSuccess) return e;
        raised = true;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kernel, threads, smem);
}

cudaError_t config_grouped(int dtype, bool sp, size_t smem, int threads, int *blocks) {
    static bool raised[4] = {};
    if (dtype == ANN_U8)
        return sp ? config_one(resume_kernel<ANN_U8, true, true>, raised[0], smem, threads, blocks)
                  : config_one(resume_kernel<ANN_U8, false, true>, raised[1], smem, threads, blocks);
    return sp ? config_one(resume_kernel<ANN_F32, true, true>, raised[2], smem, threads, blocks)
              : config_one(resume_kernel<ANN_F32, false, true>, raised[3], smem, threads, blocks);
}

cudaError_t config_grouped_prologue(int dtype, size_t smem, int threads, int *blocks) {
    static bool raised[2] = {};
    return dtype == ANN_U8 ? config_one(prologue_kernel<ANN_U8, true>, raised[0], smem, threads, blocks)
                           : config_one(prologue_kernel<ANN_F32, true>, raised[1], smem, threads, blocks);
}

void launch_grouped(int dtype, bool sp, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const SearchArgs &A) {
    if (dtype == ANN_U8) {
        if (sp) resume_kernel<ANN_U8, true, true><<<grid, block, smem, s>>>(A);
        else resume_kernel<ANN_U8, false, true><<<grid, block, smem, s>>>(A);
    } else {
        if (sp) resume_kernel<ANN_F32, true, true><<<grid, block, smem, s>>>(A);
        else resume_kernel<ANN_F32, false, true><<<grid, block, smem, s>>>(A);
    }
}

void launch_grouped_prologue(int dtype, dim3 grid, dim3 block, size_t smem, cudaStream_t s, const SearchArgs &A) {
    if (dtype == ANN_U8) prologue_kernel<ANN_U8, true><<<grid, block, smem, s>>>(A);
    else prologue_kernel<ANN_F32, true><<<grid, block, smem, s>>>(A);
}

}  // namespace ann
