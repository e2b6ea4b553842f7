// pat_pmx_f64.cu -- the any-length persistent kernel instantiated for double fields.
#include "pat_pmx.cuh"

namespace pat {

template <> const void* pmx_kernel<double>(bool adjoint) {
    return adjoint ? (const void*)k_pmx<double, true> : (const void*)k_pmx<double, false>;
}
template <> size_t pmx_smem<double>(const MxAxis& x, const MxAxis& y, const PersistCfg& c, int lossy) {
    return pmx_smem_bytes<double>(x, y, c, lossy);
}
template <>
cudaError_t pmx_launch<double>(bool adjoint, const cudaLaunchConfig_t* lc, const DevPlan<double>& P, const PersistCfg& C,
                           const MxAxis& x, const MxAxis& y, const cplx<double>* twx, const cplx<double>* twy, const double* kap,
                           const double* abs, unsigned* gbar) {
    if (adjoint) return cudaLaunchKernelEx(lc, k_pmx<double, true>, P, C, x, y, twx, twy, kap, abs, gbar);
    return cudaLaunchKernelEx(lc, k_pmx<double, false>, P, C, x, y, twx, twy, kap, abs, gbar);
}

}  // namespace pat
