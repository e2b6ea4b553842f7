// pat_pmx_f32.cu -- the any-length persistent kernel instantiated for float fields.
#include "pat_pmx.cuh"

namespace pat {

template <> const void* pmx_kernel<float>(bool adjoint) {
    return adjoint ? (const void*)k_pmx<float, true> : (const void*)k_pmx<float, false>;
}
template <> size_t pmx_smem<float>(const MxAxis& x, const MxAxis& y, const PersistCfg& c, int lossy) {
    return pmx_smem_bytes<float>(x, y, c, lossy);
}
template <>
cudaError_t pmx_launch<float>(bool adjoint, const cudaLaunchConfig_t* lc, const DevPlan<float>& P, const PersistCfg& C,
                           const MxAxis& x, const MxAxis& y, const cplx<float>* twx, const cplx<float>* twy, const float* kap,
                           const float* abs, unsigned* gbar) {
    if (adjoint) return cudaLaunchKernelEx(lc, k_pmx<float, true>, P, C, x, y, twx, twy, kap, abs, gbar);
    return cudaLaunchKernelEx(lc, k_pmx<float, false>, P, C, x, y, twx, twy, kap, abs, gbar);
}

}  // namespace pat
