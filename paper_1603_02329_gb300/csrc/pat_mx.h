// pat_mx.h -- host-side view of the mixed-radix per-phase kernels (pat_mx.cuh): the transform
// schedule of an axis, its twiddle tables, shared-memory sizes and the launch entries, compiled in a
// translation unit per precision.
#pragma once

#include <complex>
#include <vector>

#include <algorithm>
#include <cmath>

#include "pat_p2.h"

namespace pat {

// Two or three stages n = R0 RL or R0 R1 RL (R1 = 1 for two).  Forward: stage 0 of radix R0 on elements
// j + m0 r (m0 = n / R0), the middle stage of radix R1, the last stage of radix RL, whose butterfly q
// (M = n / RL of them) yields the spectrum at q + M k; the inverse runs them backwards.  Every butterfly
// writes the slots it read: output k0 of stage-0 butterfly j at slot P0 k0 + j.
struct MxAxis {
    int n, R0, R1, RL;
    int m0;      // n / R0
    int M;       // n / RL
    int P0;      // slot pitch of the stage-0 outputs: odd, so that lanes along q hit distinct banks
    int LS;      // slots of a line (even: lines start on 16 bytes)
    unsigned dn, dm0, dM, dR0, dRL, dB, dU;   // mx_magic of n, m0, M, R0, RL, R0 RL, (M + 1) / 2
};

// radices with a butterfly: R0 even and at most 10, RL at most 10, R1 any
constexpr bool mx_radix(int r) { return (r >= 2 && r <= 10) || r == 12 || r == 14 || r == 15 || r == 16; }

// ceil(2^32 / d), 0 for d = 1: floor(t / d) = (t * magic) >> 32 for t d < 2^32 (t and d here stay below 2^16)
inline unsigned mx_magic(int d) { return d == 1 ? 0u : (unsigned)(((1ull << 32) + d - 1) / d); }

// The schedule of an even length; false when there is none.  r1max: 16, or 10 in double (registers).
//   stage = 0 (the FP32 per-phase kernels): two stages where the radices allow it, else three, with the
//   smallest largest radix.  Radices stay small on purpose: the outer stages are unrolled code that every warp
//   runs once per launch, and with radices up to 16 (two stages for most lines up to 256) the kernels waited
//   for instructions (4 to 9 stall cycles per issue, 128 registers).
//   stage > 0 (the persistent kernel, and the per-phase kernels in double): the least work of one thread over
//   all stages, where the last stage counts twice (its threads run two butterflies) and a third stage costs
//   `stage`.  With a butterfly or less per thread a phase takes as long as its longest threads, the more so in
//   double, where an instruction holds its pipe for 64 clocks (30 x 50 x 70 FP64, us a step: 318 against 450
//   with the two-stage schedules of radices up to 10 and 350 in the generic kernels; 54^2: 71, 118, 80).
inline bool mx_axis(int n, int r1max, int stage, MxAxis* out) {
    int best = 1 << 30;
    MxAxis a{};
    auto take = [&](int r0, int r1, int rl) {
        const int last = stage ? 2 * rl : rl, mx = std::max(std::max(r0, r1), last);
        const int three = r1 > 1 ? (stage ? stage : 1000) : 0, sum = r0 + (r1 > 1 ? r1 : 0) + last;
        const int cost = stage ? (sum + three) * 64 + mx : three * 64 + mx * 64 + sum + (r0 >= rl ? 0 : 8);
        if (cost >= best) return;
        best = cost;
        a.R0 = r0;
        a.R1 = r1;
        a.RL = rl;
    };
    for (int r0 = 2; r0 <= 10; r0 += 2) {
        if (n % r0) continue;
        const int m = n / r0;
        if (m >= 2 && m <= 10) take(r0, 1, m);
        for (int r1 = 2; r1 <= r1max; ++r1)
            if (mx_radix(r1) && m % r1 == 0 && m / r1 >= 2 && m / r1 <= 10) take(r0, r1, m / r1);
    }
    if (best == 1 << 30) return false;
    a.n = n;
    a.m0 = n / a.R0;
    a.M = n / a.RL;
    a.P0 = a.m0 | 1;
    a.LS = a.R0 * a.P0;
    // lines of a CTA start m0 slots apart modulo the 16 banks of 8 bytes (8 when m0 is a multiple of 16)
    const int want = (a.m0 % 16) ? (a.m0 % 16) & ~1 : 8;
    while (a.LS % 16 != want) ++a.LS;
    a.dn = mx_magic(n);
    a.dm0 = mx_magic(a.m0);
    a.dM = mx_magic(a.M);
    a.dR0 = mx_magic(a.R0);
    a.dRL = mx_magic(a.RL);
    a.dB = mx_magic(a.R0 * a.RL);
    a.dU = mx_magic((a.M + 1) / 2);
    *out = a;
    return true;
}

// twiddles of the last stage [RL - 1][M], then of the middle stage [R1][R0 RL]; values of the full
// table tw[m] = exp(-2 pi i m / n)
inline std::vector<std::complex<double>> mx_table(const std::vector<std::complex<double>>& tw, const MxAxis& a) {
    std::vector<std::complex<double>> t;
    for (int r = 1; r < a.RL; ++r)
        for (int q = 0; q < a.M; ++q) t.push_back(tw[(size_t)(a.R1 == 1 ? q * r : a.R0 * r * (q / a.R0)) % a.n]);
    if (a.R1 > 1)
        for (int r = 0; r < a.R1; ++r)
            for (int b = 0; b < a.R0 * a.RL; ++b)
                t.push_back(tw[(size_t)((b % a.RL) + a.RL * r) * (b / a.RL) % a.n]);
    return t;
}

// Mean gain, less 1, of a forward and an inverse transform of an axis whose twiddles and butterfly constants
// are rounded to T: the mean of |fl(w)|^2 - 1 over the factors that an element meets.  It is the same for
// every step (a few 1e-8 in FP32), so kappa / N is divided by it.
template <typename T> double mx_unit(std::complex<double> w) {
    const double c = (double)(T)w.real(), s = (double)(T)w.imag();
    return c * c + s * s - 1.0;
}
template <typename T> double mx_radix_gain(int R) {
    const auto w = [](int m, int n) { return std::polar(1.0, 2.0 * M_PI * m / n); };
    switch (R) {
        case 8: case 16: {   // even / odd split: the odd half meets the twiddles
            double g = 0.0;
            for (int k = 0; k < R / 2; ++k) g += mx_unit<T>(w(k, R)) / R;
            return g + (R == 16 ? mx_radix_gain<T>(8) : 0.0);
        }
        case 9: {
            double g = 0.0;
            for (int k = 0; k < 9; ++k) g += mx_unit<T>(w((k / 3) * (k % 3), 9)) / 9.0;
            return g + 2.0 * mx_radix_gain<T>(3);
        }
        case 6: case 12: return mx_radix_gain<T>(3);
        case 10: return mx_radix_gain<T>(5);
        case 14: return mx_radix_gain<T>(7);
        case 15: return mx_radix_gain<T>(3) + mx_radix_gain<T>(5);
        case 3: case 5: case 7: {
            double g = 0.0;
            for (int k = 0; k < R; ++k)
                for (int r = 0; r < R; ++r) g += mx_unit<T>(w(k * r % R, R)) / (R * R);
            return g;
        }
        default: return 0.0;   // 2, 4: exact
    }
}
template <typename T> double mx_gain(const MxAxis& a, const std::vector<std::complex<double>>& table) {
    double last = 0.0, mid = 0.0;
    const size_t nl = (size_t)(a.RL - 1) * a.M;
    for (size_t i = 0; i < table.size(); ++i) (i < nl ? last : mid) += mx_unit<T>(table[i]);
    return (last + mid) / a.n + mx_radix_gain<T>(a.R0) + (a.R1 > 1 ? mx_radix_gain<T>(a.R1) : 0.0) + mx_radix_gain<T>(a.RL);
}

template <typename T> constexpr int mx_r1max() { return sizeof(T) == 4 ? 16 : 10; }

// ---- row kernels ----
// line buffers [NB][np LS] (complex) | staged real rows [nrow][R][nx] | pml [nx + (D - 1) R] (real)
struct MxRowDims {
    int nb, nrow;
};
inline __host__ __device__ MxRowDims mx_row_dims(int D, int kind, int lossy, int atd) {
    switch (kind) {
        case R2_FWD_U: case R2_ADJ_U: return {1, 2};                       // one component: b, u
        case R2_FWD_RHO: return {D, 2 + D + (atd ? 1 : 0)};                // rho0, c2, rho_xi (, source)
        case R2_FWD_P: return {2, 4};                                      // c2, c2 tau, c2 eta, r
        case R2_ADJ_RHO: return {D, 3 + D};                                // c2, rho0, p_bar, rho_xi
        default: return {lossy ? 2 : D, 3 + D};                            // two of the medium, M^T h, rho_xi
    }
}
template <typename T> size_t mx_row_smem(int D, int kind, int lossy, int atd, const MxAxis& x, int R) {
    const MxRowDims d = mx_row_dims(D, kind, lossy, atd);
    return (size_t)d.nb * (R / 2) * x.LS * sizeof(cplx<T>) +
           ((size_t)d.nrow * R * x.n + x.n + (((D - 1) * R + 3) & ~3)) * sizeof(T);
}
// threads of a row kernel: one per stage-0 butterfly of its lines, at most 256
inline int mx_row_threads(const MxAxis& x, int nb, int R) {
    const int t = nb * (R / 2) * std::max(x.m0, x.M);
    return std::max(32, std::min(256, (t + 31) / 32 * 32));
}
template <typename T, int D>
cudaError_t mx_row_launch_d(const cudaLaunchConfig_t* lc, int kind, const DevPlan<T>& P, const MxAxis& x,
                            const cplx<T>* tw, int R, int flag, T* data_row, const T* h_row, T* qrow, T* gc2,
                            const T* p0c);
template <typename T, int D> cudaError_t mx_row_attrs_d(int bytes);

// ---- spectral kernels ----
// tile buffers [slots][W] (complex): GRADT holds its D inputs at once, GRAD the spectrum and one output
template <typename T> size_t mx_spec_smem(int D, int mode, const MxAxis& a, int W) {
    return (size_t)(mode == SPEC_GRADT ? D : (mode == SPEC_GRAD ? 2 : 1)) * a.R0 * a.P0 * W * sizeof(cplx<T>);
}
inline int mx_spec_threads(const MxAxis& a, int W) {
    const int b = std::max(a.m0, std::max(a.M, a.R1 > 1 ? a.R0 * a.RL : 0));
    return std::max(32, std::min(256, (b * W + 31) / 32 * 32));
}
// mt: kappa / N ([outer][line][ldh]) for the derivative modes, the two absorption tables for SPEC_ABS
template <typename T>
cudaError_t mx_spec_launch(const cudaLaunchConfig_t* lc, int D, int mode, const DevPlan<T>& P, const MxAxis& a,
                           const cplx<T>* tw, int W, int lax, const T* mt);
template <typename T> cudaError_t mx_spec_attrs(int bytes);
// fill multiplier tables of the plan (kappa / N; |k|^(y-2) / N and |k|^(y-1) / N; either may be nullptr)
struct MxTableArgs {
    int d, ny, nz, nxh, ldh;
    const double* kv[3];   // wavenumbers per axis (device)
    double kap_a, pha, phb, invN;
    double scale;          // of kappa: takes out mean rounding errors (k_mx_kap)
    double tr_kc2;         // > 0: |k|^(y-2) / N reversed and windowed at 1 / sqrt(tr_kc2) (time reversal)
};
template <typename T> cudaError_t mx_tables(const MxTableArgs& A, T* kap, T* abs, cudaStream_t s);

// ---- the persistent 2-D solve on these stages (pat_pmx.cuh) ----
template <typename T> const void* pmx_kernel(bool adjoint);
template <typename T> size_t pmx_smem(const MxAxis& x, const MxAxis& y, const PersistCfg& c, int lossy);
template <typename T>
cudaError_t pmx_launch(bool adjoint, const cudaLaunchConfig_t* lc, const DevPlan<T>& P, const PersistCfg& C,
                       const MxAxis& x, const MxAxis& y, const cplx<T>* twx, const cplx<T>* twy, const T* kap,
                       const T* abs, unsigned* gbar);
// threads: a stage-0 butterfly of its line pairs or columns each
inline int pmx_threads(const MxAxis& x, const MxAxis& y, int ppc, int W) {
    const int rowt = 2 * ppc * std::max(x.m0, x.M);
    const int colt = 2 * W * std::max(y.m0, y.M);
    return std::min(256, std::max(128, (std::max(rowt, colt) + 31) / 32 * 32));
}

}  // namespace pat
