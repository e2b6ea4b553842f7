// pat_mx.cuh -- per-phase row and spectral kernels for line lengths with factors 2, 3, 5, 7: two or
// three register stages, one buffer.
//
// The work of the generic kernels of pat_kernels.cuh (the x transforms of a step fused with its
// pointwise physics; the y / z transforms with the k-space multiply; Sec. II.A, Sec. III).  Those run
// one shared-memory pass per radix (up to 8) plus staging, packing, pointwise, unpacking and storing
// passes, each with its barrier, and divide an index per element.  Here
//   * a stage is one butterfly in registers (radix up to 10 first and last), so lines take two or three;
//   * the outermost stages load from and store to global memory themselves (the C2R packing and R2C
//     unpacking of two real lines happen on the loaded and computed values: butterflies q and M - q of
//     the last stage hold X[k] and X[n - k]);
//   * the k-space multiply runs in registers between the last forward and the first inverse stage of the
//     y / z lines (q + M k); the pointwise step of a row kernel is one pass over the line buffer, lanes
//     along x, so that its fields move in whole cache lines and its code does not depend on the radix;
//   * every butterfly writes the slots it read, so one buffer serves; with two-stage lines a spectral
//     kernel has two CTA barriers, a row kernel four.
// Radices are chosen at run time (MxAxis): a butterfly is unrolled code behind one switch per stage,
// its addresses are one base plus a running stride.
#pragma once

#include "pat_kernels.cuh"
#include "pat_mx.h"

namespace pat {

// lambdas of these kernels are inlined whatever their size: one that is not keeps what it captures in
// local memory
#define PAT_INLINE __attribute__((always_inline))

// ---- register transforms beyond radices 2, 3, 4, 5, 7, 8, 16 ----
// N = A B with A, B coprime, no twiddles (prime-factor map): input (B a + A b) mod N, output k with
// k mod A = ka, k mod B = kb
constexpr int mx_inv(int a, int m) {   // a^-1 mod m
    for (int x = 1; x < m; ++x)
        if (a * x % m == 1) return x;
    return 1;
}
template <typename T, int R, bool INV> __device__ __forceinline__ void mx_dft(cplx<T>* v);
template <typename T, int A, int B, bool INV> __device__ __forceinline__ void mx_pfa(cplx<T>* v) {
    constexpr int N = A * B, EA = B * mx_inv(B % A, A), EB = A * mx_inv(A % B, B);
    cplx<T> w[N];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        cplx<T> x[A];
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = v[(B * a + A * b) % N];
        mx_dft<T, A, INV>(x);
#pragma unroll
        for (int a = 0; a < A; ++a) w[a * B + b] = x[a];
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
        mx_dft<T, B, INV>(w + a * B);
#pragma unroll
        for (int b = 0; b < B; ++b) v[(a * EA + b * EB) % N] = w[a * B + b];
    }
}
// 9 = 3 x 3: X[ka + 3 kb] = sum_b W9^(b ka) W3^(b kb) sum_a W3^(a ka) x[3 a + b]
template <typename T, bool INV> __device__ __forceinline__ void mx_dft9(cplx<T>* v) {
    const T c[5] = {(T)1, (T)0.7660444431189780352024, (T)0.1736481776669303488517, (T)-0.5, (T)-0.9396926207859083840541};
    const T s[5] = {(T)0, (T)0.6427876096865393263226, (T)0.9848077530122080593667, (T)0.8660254037844386467637,
                    (T)0.3420201433256687330441};   // cos, sin of 2 pi m / 9
    cplx<T> w[9];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        cplx<T> x[3] = {v[b], v[3 + b], v[6 + b]};
        dft<T, 3, INV>(x);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int m = b * k;
            const T sn = INV ? s[m] : -s[m];
            w[k * 3 + b] = m == 0 ? x[k] : mkc<T>(x[k].x * c[m] - x[k].y * sn, x[k].x * sn + x[k].y * c[m]);
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dft<T, 3, INV>(w + 3 * k);
#pragma unroll
        for (int b = 0; b < 3; ++b) v[k + 3 * b] = w[3 * k + b];
    }
}
template <typename T, int R, bool INV> __device__ __forceinline__ void mx_dft(cplx<T>* v) {
    if constexpr (R == 6) mx_pfa<T, 2, 3, INV>(v);
    else if constexpr (R == 9) mx_dft9<T, INV>(v);
    else if constexpr (R == 10) mx_pfa<T, 2, 5, INV>(v);
    else if constexpr (R == 12) mx_pfa<T, 4, 3, INV>(v);
    else if constexpr (R == 14) mx_pfa<T, 2, 7, INV>(v);
    else if constexpr (R == 15) mx_pfa<T, 3, 5, INV>(v);
    else if constexpr (R >= 2) dft<T, R, INV>(v);
}

// fn(integral constant) for the run-time radix r of stage 0 (S = 0), the middle (1) or the last stage (2)
template <int S, class Fn> __device__ __forceinline__ void with_mx(int r, Fn&& fn) {   // S = 3: 1, in double
#define PAT_MX(v) case v: fn(std::integral_constant<int, v>{}); break;
    if constexpr (S == 0) {
        switch (r) { PAT_MX(2) PAT_MX(4) PAT_MX(6) PAT_MX(8) default: fn(std::integral_constant<int, 10>{}); }
    } else if constexpr (S == 2 || S == 3) {
        switch (r) { PAT_MX(2) PAT_MX(3) PAT_MX(4) PAT_MX(5) PAT_MX(6) PAT_MX(7) PAT_MX(8) PAT_MX(9)
                     default: fn(std::integral_constant<int, 10>{}); }
    } else {
        switch (r) { PAT_MX(2) PAT_MX(3) PAT_MX(4) PAT_MX(5) PAT_MX(6) PAT_MX(7) PAT_MX(8) PAT_MX(9) PAT_MX(10)
                     PAT_MX(12) PAT_MX(14) PAT_MX(15) default: fn(std::integral_constant<int, 16>{}); }
    }
#undef PAT_MX
}

// t / d by the precomputed multiplier of d (mx_magic; 0 stands for d = 1)
__device__ __forceinline__ int mx_div(int t, unsigned magic) { return magic ? (int)__umulhi((unsigned)t, magic) : t; }

// first slot of the last-stage butterfly q (its elements are consecutive)
__device__ __forceinline__ int mx_base(const MxAxis& x, int q) {
    if (x.R1 == 1) return x.P0 * q;
    const int k1 = mx_div(q, x.dR0);
    return x.P0 * (q - k1 * x.R0) + x.RL * k1;
}

// the middle stage of `lines` lines with `es` elements between slots and `ls` between lines, lanes
// stepping over `lanes` interleaved lines (1 for contiguous lines)
template <typename T, bool INV>
__device__ __forceinline__ void mx_mid(cplx<T>* buf, const MxAxis& x, const cplx<T>* tab1, int lines, int ls, int W,
                                       int lgW) {
    const int nb = x.R0 * x.RL;
    with_mx<sizeof(T) == 4 ? 1 : 3>(x.R1, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value;
        for (int t = threadIdx.x; t < ((lines * nb) << lgW); t += blockDim.x) {
            const int c = t & (W - 1), q = t >> lgW;
            const int line = mx_div(q, x.dB), b = q - line * nb;
            const int k0 = mx_div(b, x.dRL), j = b - k0 * x.RL;
            cplx<T>* p = buf + (size_t)line * ls + ((x.P0 * k0 + j) << lgW) + c;
            const int st = x.RL << lgW;
            cplx<T> v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = p[r * st];
            if constexpr (!INV) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = cmul(v[r], __ldg(tab1 + r * nb + b));
                mx_dft<T, R, false>(v);
            } else {
                mx_dft<T, R, true>(v);
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = cmulc(v[r], __ldg(tab1 + r * nb + b));
            }
#pragma unroll
            for (int r = 0; r < R; ++r) p[r * st] = v[r];
        }
    });
}

// ---------------------------------------------------------------------------------------------
// row kernels: R x-lines per CTA, packed in pairs (line 2p real, 2p + 1 imaginary)
// ---------------------------------------------------------------------------------------------
// (the sign of v flipped when neg; integer operations, where a product would cost a double multiply)
__device__ __forceinline__ float mx_flip(float v, bool neg) { return __int_as_float(__float_as_int(v) ^ (neg ? 0x80000000 : 0)); }
__device__ __forceinline__ double mx_flip(double v, bool neg) {
    return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}
template <typename T> __device__ __forceinline__ cplx<T> mx_shfl(cplx<T> v, int lane) {
    v.x = __shfl_sync(0xffffffffu, v.x, lane);
    v.y = __shfl_sync(0xffffffffu, v.y, lane);
    return v;
}

// inverse last stage, a butterfly per thread: C2R packing of the half spectra of FI fields (an element
// past n / 2 is the conjugate of its mirror image, read by that one's thread as well), radix RL, twiddles
template <typename T>
__device__ __forceinline__ void mx_row_in(cplx<T>* buf, const MxAxis& x, const cplx<T>* tabL, cplx<T>* const* spec,
                                          int FI, int np, int line0, int ldh) {
    const int n = x.n, M = x.M, half = n >> 1;
    with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value;
        for (int t = threadIdx.x; t < FI * np * M; t += blockDim.x) {
            const int line = mx_div(t, x.dM), q = t - line * M;
            const int f = (line >= np) + (line >= 2 * np), p = line - f * np;
            const cplx<T>* a = spec[f] + (size_t)(line0 + 2 * p) * ldh;
            const cplx<T>* b = a + ldh;
            cplx<T> v[R], w[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = q + M * r, kk = k <= half ? k : n - k;
                v[r] = __ldcg(a + kk);
                w[r] = __ldcg(b + kk);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = q + M * r;
                const bool real = k == 0 || k == half;
                const T ay = real ? (T)0 : mx_flip(v[r].y, k > half), by = real ? (T)0 : mx_flip(w[r].y, k > half);
                v[r] = mkc<T>(v[r].x - by, ay + w[r].x);   // A + i B
            }
            mx_dft<T, R, true>(v);
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = cmulc(v[r], __ldg(tabL + (r - 1) * M + q));
            cplx<T>* s = buf + line * x.LS + mx_base(x, q);
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = v[r];
        }
    });
}

// forward last stage, R2C unpacking, half spectra of FO fields to global memory.  Lanes 2 u and 2 u + 1 run
// the butterflies u and M - u (u = 0: 0 and, when M is even, M / 2), which hold every X[k] with its
// X[n - k], element j of one against R - 1 - j of the other; each stores half of the pairs.  HALF = false
// leaves out the factor 1/2 (a power of two: the caller's multipliers carry it without a rounding).
template <typename T, bool HALF>
__device__ __forceinline__ void mx_row_out(const cplx<T>* buf, const MxAxis& x, const cplx<T>* tabL,
                                           cplx<T>* const* spec, int FO, int np, int line0, int ldh) {
    const int n = x.n, M = x.M, half = n >> 1, U = (M + 1) >> 1, lane = threadIdx.x & 31;
    with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value, J = (R - 1) / 2;
        const int total = 2 * FO * np * U;
        for (int t0 = 0; t0 < total; t0 += blockDim.x) {   // uniform trip count: whole warps shuffle
            const int t = t0 + (int)threadIdx.x, h = t & 1;
            const int line = mx_div(t >> 1, x.dU), u = (t >> 1) - line * U;
            const bool u0 = u == 0;
            const int q = h ? (u0 ? M >> 1 : M - u) : u;
            const bool ok = t < total && !(u0 && h && (M & 1));
            cplx<T> v[R];
            if (ok) {
                const cplx<T>* s = buf + line * x.LS + mx_base(x, q);
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = s[r];
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(tabL + (r - 1) * M + q));
                mx_dft<T, R, false>(v);
            }
            const int f = (line >= np) + (line >= 2 * np), p = line - f * np;
            cplx<T>* a = spec[ok ? f : 0] + (size_t)(line0 + 2 * p) * ldh;
            cplx<T>* b = a + ldh;
            auto put = [&](int k, cplx<T> zk, cplx<T> zm) PAT_INLINE {   // X[k] with X[n - k], either k
                const bool up = k > half;
                const int kk = up ? n - k : k;
                cplx<T> A = mkc<T>(zk.x + zm.x, mx_flip(zk.y - zm.y, up)), B = mkc<T>(zk.y + zm.y, mx_flip(zm.x - zk.x, up));
                if constexpr (HALF) {
                    A = cscale(A, (T)0.5);
                    B = cscale(B, (T)0.5);
                }
                a[kk] = A;
                b[kk] = B;
            };
            const int from = u0 ? lane : lane ^ 1;   // unit 0's butterflies are their own mirror images
#pragma unroll
            for (int j = 0; j <= J; ++j) {
                cplx<T> zm = mx_shfl<T>(v[R - 1 - j], from);
                if (u0 && !h) zm = v[(R - j) % R];
                // odd R: the middle element once per pair
                if (ok && !(R % 2 == 1 && j == J && h && !u0)) put(q + M * j, v[j], zm);
            }
            if (R % 2 == 0 && ok && u0 && !h) put(half, v[R / 2], v[R / 2]);
        }
    });
}

// stage 0 (radix R0, no twiddles) of `lines` lines, forward or inverse: elements j + m0 r, slots P0 r + j
template <typename T, bool INV> __device__ __forceinline__ void mx_row_s0(cplx<T>* buf, const MxAxis& x, int lines) {
    with_mx<0>(x.R0, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value;
        for (int t = threadIdx.x; t < lines * x.m0; t += blockDim.x) {
            const int line = mx_div(t, x.dm0), j = t - line * x.m0;
            cplx<T>* b = buf + line * x.LS + j;
            cplx<T> v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = b[r * x.P0];
            mx_dft<T, R, INV>(v);
#pragma unroll
            for (int r = 0; r < R; ++r) b[r * x.P0] = v[r];
        }
    });
}

// One row kernel of a step (Row2Kind); grid nlines / R, or (nlines / R, D) for the u update and its
// transpose, whose CTAs hold one velocity component.
template <typename T, int D, int KIND>
__global__ void __launch_bounds__(256) k_mx_row(DevPlan<T> P, MxAxis x, const cplx<T>* __restrict__ tw, int R, int flag,
                                                T* data_row, const T* h_row, T* qrow, T* gc2, const T* p0c) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool U = (KIND == R2_FWD_U || KIND == R2_ADJ_U);
    const int nx = x.n, np = R >> 1, line0 = blockIdx.x * R;
    const bool lossy = P.lossy != 0;
    const MxRowDims dims = mx_row_dims(D, KIND, lossy, P.atd);
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
    T* rows = reinterpret_cast<T*>(buf + (size_t)dims.nb * np * x.LS);
    T* pmlx = rows + (size_t)dims.nrow * R * nx;
    T* pmlr = pmlx + nx;
    const cplx<T>* tabL = tw;
    const cplx<T>* tab1 = tw + (x.RL - 1) * x.M;
    auto row = [&](int k) PAT_INLINE { return rows + k * R * nx; };
    const T dt = P.dt;
    const int xi0 = U ? blockIdx.y : 0;
    cplx<T>* const* spec = P.spec + xi0;

    // ---- prologue: constants of the plan ----
    int FI = D, FO = D, inj = -1;
    bool fwd = true, gath = false;
    const T* const* pml_tab = P.a;
    if constexpr (U) {
        FI = FO = 1;
        pml_tab = P.au;
        stage_rows(row(0), P.b[xi0], line0, R, nx);
    } else if constexpr (KIND == R2_FWD_RHO) {
        stage_rows(row(0), P.rho0, line0, R, nx);
        if (!lossy) stage_rows(row(1), P.c2, line0, R, nx);
        FO = lossy ? 2 : 1;
        fwd = lossy || !flag;
        gath = !lossy && !P.atd;
        if (P.atd) inj = 2 + D;
    } else if constexpr (KIND == R2_FWD_P) {
        stage_rows(row(0), P.c2, line0, R, nx);
        stage_rows(row(1), P.c2tau, line0, R, nx);
        stage_rows(row(2), P.c2eta, line0, R, nx);
        FI = 2;
        FO = 1;
        fwd = !flag;
        gath = true;
    } else if constexpr (KIND == R2_ADJ_RHO) {
        stage_rows(row(0), P.c2, line0, R, nx);
        stage_rows(row(1), P.rho0, line0, R, nx);
        FI = 2;
    } else {
        if (lossy && !flag) {
            stage_rows(row(0), P.c2tau, line0, R, nx);
            stage_rows(row(1), P.c2eta, line0, R, nx);
        } else {
            stage_rows(row(0), P.c2, line0, R, nx);
            stage_rows(row(1), P.rho0, line0, R, nx);
        }
        FI = 1;
        FO = lossy ? 2 : D;
        fwd = !flag;
        inj = 2;
    }
    stage_elems(pmlx, pml_tab[0], nx);
    for (int t = threadIdx.x; t < (D - 1) * R; t += blockDim.x) {
        const int a = 1 + t / R, r = t - (a - 1) * R;
        const int line = line0 + r;
        pmlr[t] = pml_tab[a][(a == 1) ? line % P.ny : line / P.ny];
    }
    cp_commit();
    const DevSensors<T>& S = P.sens;
    if (inj >= 0) {   // M^T of the record's row into a zeroed row buffer (segments are distinct points)
        T* g = row(inj);
        const T* hr = (KIND == R2_FWD_RHO) ? P.atd_row : h_row;
        for (int t = threadIdx.x; t < R * nx; t += blockDim.x) g[t] = 0;
        __syncthreads();
        const int s0 = S.s_lineptr[line0], s1 = S.s_lineptr[line0 + R];
        for (int q = s0 + threadIdx.x; q < s1; q += blockDim.x) {
            T acc = 0;
            for (int e = S.s_seg_e0[q]; e < S.s_seg_e0[q + 1]; ++e) acc += S.s_ent_w[e] * hr[S.s_ent_sensor[e]];
            g[(S.s_seg_line[q] - line0) * nx + S.s_seg_x[q]] += acc;
        }
    }
    pdl_trigger();
    pdl_wait();

    // ---- state rows, asynchronously; the spectra go to registers in the first stage ----
    if constexpr (U) {
        if (KIND == R2_ADJ_U || !flag) stage_rows(row(1), P.u[xi0], line0, R, nx);
    } else if constexpr (KIND == R2_FWD_RHO) {
#pragma unroll
        for (int xi = 0; xi < D; ++xi) stage_rows(row(2 + xi), P.rh[xi], line0, R, nx);
    } else if constexpr (KIND == R2_FWD_P) {
        stage_rows(row(3), P.rsum, line0, R, nx);
    } else if constexpr (KIND == R2_ADJ_RHO) {
        stage_rows(row(2), P.pbar, line0, R, nx);
#pragma unroll
        for (int xi = 0; xi < D; ++xi) stage_rows(row(3 + xi), P.rh[xi], line0, R, nx);
    } else {
        if (!(lossy && !flag)) {
#pragma unroll
            for (int xi = 0; xi < D; ++xi) stage_rows(row(3 + xi), P.rh[xi], line0, R, nx);
        }
    }
    cp_commit();

    mx_row_in<T>(buf, x, tabL, spec, FI, np, line0, P.ldh);
    cp_wait_all();
    __syncthreads();
    if (x.R1 > 1) {
        mx_mid<T, true>(buf, x, tab1, FI * np, x.LS, 1, 0);
        __syncthreads();
    }

    auto pml = [&](int xi, int r, int i) PAT_INLINE { return xi == 0 ? pmlx[i] : pmlr[(xi - 1) * R + r]; };
    // ---- inverse stage 0, the pointwise step on the real rows, forward stage 0 ----
    mx_row_s0<T, true>(buf, x, FI * np);
    __syncthreads();
    const int fs = np * x.LS, pad = x.P0 - x.m0;   // slots between the fields of a line pair
    for (int e = threadIdx.x; e < np * nx; e += blockDim.x) {
        const int p = mx_div(e, x.dn), xx = e - p * nx;
        cplx<T>* bp = buf + p * x.LS + xx + pad * mx_div(xx, x.dm0);
        cplx<T> z[D], w[D];
#pragma unroll
        for (int f = 0; f < D; ++f)
            if (f < FI) z[f] = bp[f * fs];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int rr = 2 * p + h, tt = rr * nx + xx;
            const size_t idx = (size_t)line0 * nx + tt;
            auto in = [&](int f) PAT_INLINE { return h ? z[f].y : z[f].x; };
            T out[D] = {};
            if constexpr (KIND == R2_FWD_U) {
                const T g = in(0);
                const T bq = row(0)[tt];
                const T au = pml(xi0, rr, xx);
                const T uo = flag ? (T)0.5 * dt * bq * g : row(1)[tt];
                const T un = au * (au * uo - dt * bq * g);
                P.u[xi0][idx] = un;
                out[0] = un;
                if (P.hk_g[0]) P.hk_g[xi0][idx] = g;
            } else if constexpr (KIND == R2_ADJ_U) {
                const T bq = row(0)[tt];
                const T au = pml(xi0, rr, xx);
                T ub = row(1)[tt] + in(0);
                T g = -dt * bq * au * ub;
                const T ubn = ub;
                ub = au * au * ub;
                if (flag) g += (T)0.5 * dt * bq * ub;
                P.u[xi0][idx] = ub;
                out[0] = g;
                if (P.hk_gb[0]) {
                    const T gv = P.hk_gin[xi0][idx];
                    T add = ubn * (-dt * au * gv);
                    if (flag) add += ub * (T)0.5 * dt * gv;
                    P.hk_gb[xi0][idx] += add;
                }
            } else if constexpr (KIND == R2_FWD_RHO) {
                const T rho0 = row(0)[tt];
                const T src = P.atd ? row(inj)[tt] : (T)0;
                const int trj = P.tr_node ? P.tr_node[idx] : -1;
                T rs = 0, es = 0;
#pragma unroll
                for (int xi = 0; xi < D; ++xi) {
                    const T ev = in(xi);
                    const T a = pml(xi, rr, xx);
                    const T rh = P.atd ? a * (a * row(2 + xi)[tt] - dt * rho0 * ev + dt * rho0 * src / T(D))
                                       : a * (a * row(2 + xi)[tt] - dt * rho0 * ev);
                    P.rh[xi][idx] = (trj >= 0) ? P.tr_row[trj] / (T(D) * P.c2[idx]) : rh;
                    rs += rh;
                    es += ev;
                    if (P.hk_e[0]) P.hk_e[xi][idx] = ev;
                }
                if (lossy) {
                    P.rsum[idx] = rs;
                    out[0] = P.atd ? P.c2tau[idx] * (src - es) : rho0 * es;
                    out[1] = P.atd ? P.c2eta[idx] * rs / rho0 : rs;
                } else {
                    T pv = row(1)[tt] * rs;
                    if (trj >= 0) pv = P.tr_row[trj];
                    if (P.tr_img && flag) P.tr_img[idx] = pv;
                    if (qrow) qrow[idx] = rs;   // d p / d c0^2 (lossless)
                    row(0)[tt] = pv;            // for the sensors
                    out[0] = pv;
                }
            } else if constexpr (KIND == R2_FWD_P) {
                const T c2 = row(0)[tt], rs = row(3)[tt];
                T pv;
                if (P.atd) {
                    const T rho0 = P.rho0[idx];
                    pv = c2 * rs - rho0 * in(0) - rho0 * in(1);
                } else {
                    pv = c2 * rs + row(1)[tt] * in(0) - row(2)[tt] * in(1);
                }
                if (P.tr_node) {
                    const int trj = P.tr_node[idx];
                    if (trj >= 0) pv = P.tr_row[trj];
                }
                if (P.tr_img && flag) P.tr_img[idx] = pv;
                if (qrow)   // d p / d c0^2 with tau, eta following c0 (Eq. (Twelve))
                    qrow[idx] = rs + ((P.phb + (T)1) * row(1)[tt] * in(0) - (P.pha + (T)2) * row(2)[tt] * in(1)) / c2;
                row(0)[tt] = pv;   // for the sensors
                out[0] = pv;
            } else if constexpr (KIND == R2_ADJ_RHO) {
                const T ddbar = in(0);
                const T rbar = row(0)[tt] * row(2)[tt] - in(1);
                const T rho0 = row(1)[tt];
                T gr = 0;
#pragma unroll
                for (int xi = 0; xi < D; ++xi) {
                    const T a = pml(xi, rr, xx);
                    const T rb = row(3 + xi)[tt] + rbar;
                    out[xi] = rho0 * ddbar - dt * rho0 * a * rb;
                    P.rh[xi][idx] = a * a * rb;
                    if (P.hk_grho) gr += P.hk_ein[xi][idx] * (ddbar - dt * a * rb);
                }
                if (P.hk_grho) P.hk_grho[idx] += gr;
            } else {   // R2_ADJ_P
                const T pv = in(0) + row(inj)[tt];
                if (flag) {   // final level: the transpose of the initial state
                    T sum = 0;
#pragma unroll
                    for (int xi = 0; xi < D; ++xi) sum += row(3 + xi)[tt];
                    const T c2 = row(0)[tt];
                    P.img[idx] = pv + sum / (T(D) * c2);
                    if (gc2) gc2[idx] -= sum * p0c[idx] / (T(D) * c2 * c2);
                } else {
                    if (gc2) gc2[idx] += pv * qrow[idx];
                    if (lossy) {
                        P.pbar[idx] = pv;
                        out[0] = row(0)[tt] * pv;
                        out[1] = row(1)[tt] * pv;
                    } else {
                        const T rbar = row(0)[tt] * pv;
                        const T rho0 = row(1)[tt];
                        T gr = 0;
#pragma unroll
                        for (int xi = 0; xi < D; ++xi) {
                            const T a = pml(xi, rr, xx);
                            const T rb = row(3 + xi)[tt] + rbar;
                            out[xi] = -dt * rho0 * a * rb;
                            P.rh[xi][idx] = a * a * rb;
                            if (P.hk_grho) gr += P.hk_ein[xi][idx] * (-dt * a * rb);
                        }
                        if (P.hk_grho) P.hk_grho[idx] += gr;
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < D; ++g) {
                if (h) w[g].y = out[g];
                else w[g].x = out[g];
            }
        }
#pragma unroll
        for (int g = 0; g < D; ++g)
            if (g < FO) bp[g * fs] = w[g];
    }
    __syncthreads();
    if (gath) {   // s_j += this CTA's part of sensor j (one atomic add per (line, sensor) segment)
        const int s0 = S.g_lineptr[line0], s1 = S.g_lineptr[line0 + R];
        for (int q = s0 + threadIdx.x; q < s1; q += blockDim.x) {
            const int j = S.g_seg_sensor[q];
            const T* pr = row(0) + (S.g_seg_line[q] - line0) * nx + S.g_seg_x0[q];
            const T w0 = S.g_seg_w0[q], w1 = S.g_seg_w1[q];
            T acc = w0 * pr[0];
            if (w1 != (T)0) acc += w1 * pr[1];
            atomicAdd(&data_row[j], acc);
        }
    }
    if (!fwd) return;
    mx_row_s0<T, false>(buf, x, FO * np);
    __syncthreads();
    if (x.R1 > 1) {
        mx_mid<T, false>(buf, x, tab1, FO * np, x.LS, 1, 0);
        __syncthreads();
    }
    mx_row_out<T, true>(buf, x, tabL, spec, FO, np, line0, P.ldh);
}

// ---------------------------------------------------------------------------------------------
// spectral kernels: lines along y (lax = 1) or z (lax = 2), W half-spectrum columns per CTA
// ---------------------------------------------------------------------------------------------
// Multipliers on the half spectrum, [outer][line][ldh]: (1, ny) in 2-D, (ny, nz) in 3-D (padding columns:
// the last valid kx): kappa / N and, where abs, |k|^(y-2) / N and |k|^(y-1) / N.  Formed in double and
// rounded once: 1 / N rounded by itself would scale every mode of every step by the same few 1e-8, an
// error that grows with the number of steps.  In FP32 kappa / N carries `scale` for errors of the same kind:
// dt and the medium rounded (every derivative meets them later), and the transforms' mean gain (mx_gain).
// The fractional Laplacians take D- u without dt, where 6e-8 once is nothing.  Relative error of the
// gradient of 40 x 160 x 160, 200 steps: 2.2e-6 with `scale`, 3.7e-6 without the gain, 5.6e-6 without dt;
// of the batch of eight 2-D instances, 300 steps: 1.6e-6 to 1.8e-6 against 2e-6 to 6e-6.
template <typename T> __global__ void k_mx_kap(MxTableArgs A, T* kap, T* abs) {
    const int L = A.d == 2 ? A.ny : A.nz, la = A.d - 1;
    const size_t n = (size_t)A.ny * A.nz * A.ldh;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int kx = (int)(i % A.ldh);
        const size_t q = i / A.ldh;
        const int kl = (int)(q % L), ko = (int)(q / L);
        const double kxv = A.kv[0][min(kx, A.nxh - 1)], klv = A.kv[la][kl];
        double k2 = kxv * kxv + klv * klv;
        if (A.d == 3) k2 += A.kv[1][ko] * A.kv[1][ko];
        if (kap) kap[i] = (T)(sinc_sq(A.kap_a * A.kap_a * k2) * A.invN * A.scale);
        if (abs) {
            double win = 1.0;
            if (A.tr_kc2 > 0.0) {   // time reversal: reversed and windowed
                const double q2 = k2 * A.tr_kc2, q = sqrt(q2);
                win = q2 < 1.0 ? -(0.42 + 0.5 * cospi(q) + 0.08 * cospi(2.0 * q)) : 0.0;
            }
            abs[i] = (k2 > 0.0) ? (T)(win * pow(k2, A.pha) * A.invN) : (T)0;
            abs[n + i] = (k2 > 0.0) ? (T)(pow(k2, A.phb) * A.invN) : (T)0;
        }
    }
}

// grid (fields or 1, column tiles, outer lines): one field per CTA for the plain and field-wise modes.  The
// register bound (80 in FP32, 128 in double) keeps three and two CTAs of 256 threads per SM; only GRADT, which
// holds two spectra, spills under it (FP32 444 bytes stored, 464 loaded in 3-D; double 496 and 496).
template <typename T, int D, int MODE>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2) k_mx_spec(DevPlan<T> P, MxAxis x, const cplx<T>* __restrict__ tw, int W, int lgW,
                                                 int lax, const T* __restrict__ mt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool MUL = (MODE != SPEC_PLAIN_FWD && MODE != SPEC_PLAIN_INV);
    constexpr bool plus = (MODE == SPEC_GRAD || MODE == SPEC_DIVT);
    constexpr int NT = (MODE == SPEC_GRADT) ? D : 1;
    cplx<T>* S = reinterpret_cast<cplx<T>*>(smem_raw);
    const int tile = (x.R0 * x.P0) << lgW;
    const cplx<T>* tabL = tw;
    const cplx<T>* tab1 = tw + (x.RL - 1) * x.M;
    const int f0 = blockIdx.x, kx0 = blockIdx.y * W, outer = blockIdx.z;
    const int c = threadIdx.x & (W - 1);
    const bool ok = kx0 + c < P.nxh;
    const size_t es = (lax == 1) ? (size_t)P.ldh : (size_t)P.ny * P.ldh;
    const size_t base = ((lax == 1) ? (size_t)outer * P.ny * P.ldh : (size_t)outer * P.ldh) + kx0 + c;
    const int M = x.M, m0 = x.m0;

    // the multiply's constants (padding columns take the last valid kx; their data are zero)
    const int kx = min(kx0 + c, P.nxh - 1);
    cplx<T> mx = mkc<T>(0, 0), mo = mkc<T>(0, 0);
    const cplx<T>* ml = nullptr;
    if constexpr (MUL) {
        mx = plus ? P.dp[0][kx] : P.dm[0][kx];
        ml = plus ? P.dp[lax] : P.dm[lax];
        if (D == 3) mo = plus ? P.dp[1][outer] : P.dm[1][outer];
    }
    pdl_trigger();
    pdl_wait();

    // forward stage 0 of field f into buffer b
    auto fwd0 = [&](int f, int b) PAT_INLINE {
        with_mx<0>(x.R0, [&](auto RC) PAT_INLINE {
            constexpr int R = decltype(RC)::value;
            const cplx<T>* src = P.spec[f] + base;
            cplx<T>* d = S + b * tile + c;
            for (int t = threadIdx.x; t < (m0 << lgW); t += blockDim.x) {
                const int j = t >> lgW;
                cplx<T> v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = ok ? src[(size_t)(j + m0 * r) * es] : mkc<T>(0, 0);
                mx_dft<T, R, false>(v);
#pragma unroll
                for (int r = 0; r < R; ++r) d[(x.P0 * r + j) << lgW] = v[r];
            }
        });
    };
    // inverse stage 0 of buffer b into field f
    auto inv0 = [&](int b, int f) PAT_INLINE {
        with_mx<0>(x.R0, [&](auto RC) PAT_INLINE {
            constexpr int R = decltype(RC)::value;
            cplx<T>* dst = P.spec[f] + base;
            const cplx<T>* s = S + b * tile + c;
            for (int t = threadIdx.x; t < (m0 << lgW); t += blockDim.x) {
                const int j = t >> lgW;
                cplx<T> v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = s[(x.P0 * r + j) << lgW];
                mx_dft<T, R, true>(v);
                if (ok) {
#pragma unroll
                    for (int r = 0; r < R; ++r) dst[(size_t)(j + m0 * r) * es] = v[r];
                }
            }
        });
    };
    auto mid_f = [&](int b) PAT_INLINE {
        if (x.R1 > 1) {
            mx_mid<T, false>(S + b * tile, x, tab1, 1, 0, W, lgW);
            __syncthreads();
        }
    };
    auto mid_i = [&](int b) PAT_INLINE {
        if (x.R1 > 1) {
            mx_mid<T, true>(S + b * tile, x, tab1, 1, 0, W, lgW);
            __syncthreads();
        }
    };

    if constexpr (MODE == SPEC_PLAIN_FWD) {
        fwd0(f0, 0);
        __syncthreads();
        mid_f(0);
        with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
            constexpr int R = decltype(RC)::value;
            cplx<T>* dst = P.spec[f0] + base;
            for (int t = threadIdx.x; t < (M << lgW); t += blockDim.x) {
                const int q = t >> lgW;
                const cplx<T>* s = S + (mx_base(x, q) << lgW) + c;
                cplx<T> v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = s[r << lgW];
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(tabL + (r - 1) * M + q));
                mx_dft<T, R, false>(v);
                if (ok) {
#pragma unroll
                    for (int r = 0; r < R; ++r) dst[(size_t)(q + M * r) * es] = v[r];
                }
            }
        });
    } else if constexpr (MODE == SPEC_PLAIN_INV) {
        with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
            constexpr int R = decltype(RC)::value;
            const cplx<T>* src = P.spec[f0] + base;
            for (int t = threadIdx.x; t < (M << lgW); t += blockDim.x) {
                const int q = t >> lgW;
                cplx<T> v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = ok ? src[(size_t)(q + M * r) * es] : mkc<T>(0, 0);
                mx_dft<T, R, true>(v);
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmulc(v[r], __ldg(tabL + (r - 1) * M + q));
                cplx<T>* s = S + (mx_base(x, q) << lgW) + c;
#pragma unroll
                for (int r = 0; r < R; ++r) s[r << lgW] = v[r];
            }
        });
        __syncthreads();
        mid_i(0);
        inv0(0, f0);
    } else {
        // shift symbol of output (input) field f at line index k
        auto shift = [&](int f, int k) PAT_INLINE { return f == 0 ? mx : (D == 3 && f == 1 ? mo : __ldg(ml + k)); };
        if constexpr (MODE == SPEC_GRADT) {
#pragma unroll
            for (int f = 0; f < D; ++f) fwd0(f, f);
        } else {
            fwd0((MODE == SPEC_GRAD) ? 0 : f0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < NT; ++b) mid_f(b);
        // last forward stage of butterfly q of buffer b: the spectrum at q + M r
        const size_t L = x.n;
        const T* mrow = mt + ((MODE == SPEC_ABS) ? (size_t)f0 * gridDim.z * L * P.ldh : 0) + (size_t)outer * L * P.ldh + kx0 + c;
        auto mult = [&](int k) -> T { return ok ? __ldg(mrow + (size_t)k * P.ldh) : (T)0; };
        const int nf = (MODE == SPEC_GRAD) ? D : 1;
        for (int fo = 0; fo < nf; ++fo) {
            with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
                constexpr int R = decltype(RC)::value;
                for (int t = threadIdx.x; t < (M << lgW); t += blockDim.x) {
                    const int q = t >> lgW;
                    cplx<T>* s = S + (mx_base(x, q) << lgW) + c;
                    auto spectrum = [&](cplx<T>(&v)[R], int b) {
#pragma unroll
                        for (int r = 0; r < R; ++r) v[r] = s[b * tile + (r << lgW)];
#pragma unroll
                        for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(tabL + (r - 1) * M + q));
                        mx_dft<T, R, false>(v);
                    };
                    cplx<T> v[R];
                    if constexpr (MODE == SPEC_GRADT) {
#pragma unroll
                        for (int r = 0; r < R; ++r) v[r] = mkc<T>(0, 0);
#pragma unroll
                        for (int b = 0; b < D; ++b) {
                            cplx<T> w[R];
                            spectrum(w, b);
#pragma unroll
                            for (int r = 0; r < R; ++r) v[r] = cadd(v[r], cmul(w[r], shift(b, q + M * r)));
                        }
#pragma unroll
                        for (int r = 0; r < R; ++r) v[r] = cscale(v[r], -mult(q + M * r));
                    } else if constexpr (MODE == SPEC_GRAD) {
                        // the scaled spectrum stays in buffer 0 for the outputs after the first; the
                        // inverse runs in buffer 1
                        if (fo == 0) {
                            spectrum(v, 0);
#pragma unroll
                            for (int r = 0; r < R; ++r) v[r] = cscale(v[r], mult(q + M * r));
#pragma unroll
                            for (int r = 0; r < R; ++r) s[r << lgW] = v[r];
                        } else {
#pragma unroll
                            for (int r = 0; r < R; ++r) v[r] = s[r << lgW];
                        }
#pragma unroll
                        for (int r = 0; r < R; ++r) v[r] = cmul(v[r], shift(fo, q + M * r));
                    } else {
                        spectrum(v, 0);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const int k = q + M * r;
                            if constexpr (MODE == SPEC_ABS) {
                                v[r] = cscale(v[r], mult(k));
                            } else {
                                const T sc = mult(k);
                                v[r] = cscale(cmul(v[r], shift(f0, k)), (MODE == SPEC_DIVT) ? -sc : sc);
                            }
                        }
                    }
                    mx_dft<T, R, true>(v);
#pragma unroll
                    for (int r = 1; r < R; ++r) v[r] = cmulc(v[r], __ldg(tabL + (r - 1) * M + q));
                    cplx<T>* d = s + (MODE == SPEC_GRAD ? tile : 0);
#pragma unroll
                    for (int r = 0; r < R; ++r) d[r << lgW] = v[r];
                }
            });
            __syncthreads();
            mid_i(MODE == SPEC_GRAD ? 1 : 0);
            inv0(MODE == SPEC_GRAD ? 1 : 0, (MODE == SPEC_GRAD) ? fo : (MODE == SPEC_GRADT ? 0 : f0));
            if (fo + 1 < nf) __syncthreads();   // buffer 1 is read before the next output overwrites it
        }
    }
}

}  // namespace pat
