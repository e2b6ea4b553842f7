// pat_mx_spec_f32.cu -- the mixed-radix spectral kernels instantiated for float fields.
#include "pat_mx.cuh"

namespace pat {

template <typename T, int D>
static cudaError_t spec_d(const cudaLaunchConfig_t* lc, int mode, const DevPlan<T>& P, const MxAxis& a, const cplx<T>* tw,
                          int W, int lgW, int lax, const T* mt) {
    switch (mode) {
        case SPEC_PLAIN_FWD: return cudaLaunchKernelEx(lc, k_mx_spec<T, 3, SPEC_PLAIN_FWD>, P, a, tw, W, lgW, lax, mt);
        case SPEC_PLAIN_INV: return cudaLaunchKernelEx(lc, k_mx_spec<T, 3, SPEC_PLAIN_INV>, P, a, tw, W, lgW, lax, mt);
        case SPEC_GRAD: return cudaLaunchKernelEx(lc, k_mx_spec<T, D, SPEC_GRAD>, P, a, tw, W, lgW, lax, mt);
        case SPEC_DIV: return cudaLaunchKernelEx(lc, k_mx_spec<T, D, SPEC_DIV>, P, a, tw, W, lgW, lax, mt);
        case SPEC_ABS: return cudaLaunchKernelEx(lc, k_mx_spec<T, D, SPEC_ABS>, P, a, tw, W, lgW, lax, mt);
        case SPEC_DIVT: return cudaLaunchKernelEx(lc, k_mx_spec<T, D, SPEC_DIVT>, P, a, tw, W, lgW, lax, mt);
        case SPEC_GRADT: return cudaLaunchKernelEx(lc, k_mx_spec<T, D, SPEC_GRADT>, P, a, tw, W, lgW, lax, mt);
        default: return cudaErrorInvalidValue;
    }
}

template <>
cudaError_t mx_spec_launch<float>(const cudaLaunchConfig_t* lc, int D, int mode, const DevPlan<float>& P, const MxAxis& a,
                               const cplx<float>* tw, int W, int lax, const float* mt) {
    int lgW = 0;
    while ((1 << lgW) < W) ++lgW;
    return D == 2 ? spec_d<float, 2>(lc, mode, P, a, tw, W, lgW, lax, mt) : spec_d<float, 3>(lc, mode, P, a, tw, W, lgW, lax, mt);
}

template <> cudaError_t mx_spec_attrs<float>(int bytes) {
    const void* ks[] = {
        (const void*)k_mx_spec<float, 3, SPEC_PLAIN_FWD>,
        (const void*)k_mx_spec<float, 3, SPEC_PLAIN_INV>,
        (const void*)k_mx_spec<float, 3, SPEC_GRAD>,
        (const void*)k_mx_spec<float, 3, SPEC_DIV>,
        (const void*)k_mx_spec<float, 3, SPEC_ABS>,
        (const void*)k_mx_spec<float, 3, SPEC_DIVT>,
        (const void*)k_mx_spec<float, 3, SPEC_GRADT>,
        (const void*)k_mx_spec<float, 2, SPEC_GRAD>,
        (const void*)k_mx_spec<float, 2, SPEC_DIV>,
        (const void*)k_mx_spec<float, 2, SPEC_ABS>,
        (const void*)k_mx_spec<float, 2, SPEC_DIVT>,
        (const void*)k_mx_spec<float, 2, SPEC_GRADT>,
    };
    for (const void* k : ks) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <> cudaError_t mx_tables<float>(const MxTableArgs& A, float* kap, float* abs, cudaStream_t s) {
    const size_t n = (size_t)A.ny * A.nz * A.ldh;
    const int blocks = (int)std::min<size_t>((n + 255) / 256, 4096);
    k_mx_kap<float><<<blocks, 256, 0, s>>>(A, kap, abs);
    return cudaGetLastError();
}

}  // namespace pat
