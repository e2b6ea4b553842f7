// pat_mx_row_f32_3d.cu -- the mixed-radix row kernels instantiated for float fields, 3-D.
#include "pat_mx.cuh"

namespace pat {

template <typename T, int D>
cudaError_t mx_row_launch_d(const cudaLaunchConfig_t* lc, int kind, const DevPlan<T>& P, const MxAxis& x,
                            const cplx<T>* tw, int R, int flag, T* data_row, const T* h_row, T* qrow, T* gc2,
                            const T* p0c) {
    switch (kind) {
        case R2_FWD_U: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_FWD_U>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        case R2_FWD_RHO: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_FWD_RHO>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        case R2_FWD_P: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_FWD_P>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        case R2_ADJ_RHO: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_ADJ_RHO>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        case R2_ADJ_U: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_ADJ_U>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        case R2_ADJ_P: return cudaLaunchKernelEx(lc, k_mx_row<T, D, R2_ADJ_P>, P, x, tw, R, flag, data_row, h_row, qrow, gc2, p0c);
        default: return cudaErrorInvalidValue;
    }
}
template <typename T, int D> cudaError_t mx_row_attrs_d(int bytes) {
    const void* ks[] = {(const void*)k_mx_row<T, D, R2_FWD_U>, (const void*)k_mx_row<T, D, R2_FWD_RHO>, (const void*)k_mx_row<T, D, R2_FWD_P>, (const void*)k_mx_row<T, D, R2_ADJ_RHO>, (const void*)k_mx_row<T, D, R2_ADJ_U>, (const void*)k_mx_row<T, D, R2_ADJ_P>};
    for (const void* k : ks) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
template cudaError_t mx_row_launch_d<float, 3>(const cudaLaunchConfig_t*, int, const DevPlan<float>&, const MxAxis&,
                                              const cplx<float>*, int, int, float*, const float*, float*, float*, const float*);
template cudaError_t mx_row_attrs_d<float, 3>(int);

}  // namespace pat
