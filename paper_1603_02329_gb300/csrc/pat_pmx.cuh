// pat_pmx.cuh -- the whole Nt-step solve of a 2-D grid of any supported line lengths as one persistent
// cooperative kernel, on the mixed-radix stages of pat_mx.cuh.
//
// The scheme of k_persist (pat_persist.cuh): each CTA keeps the state and medium of its own x-lines in
// shared memory for all steps, only the half spectra cross L2 between phases, phases are separated by
// the bounded grid barrier, and the phase schedule is that of k_persist2 (p2_phase).  Against k_persist:
//   * transforms run in two or three register stages (k_persist: one shared-memory pass per radix plus
//     staging, packing and unpacking passes); the half spectra go straight to and from registers;
//   * the multipliers of the CTA's columns (kappa / N, |k|^(y-2) / N, |k|^(y-1) / N) are resident: in
//     double, forming them anew cost as much as the transforms;
//   * every phase kind has one call site (the row phase's pointwise step is one short loop per phase).
// It also runs the time-reversal solve (Sec. II.B.1): after each step the state at the sensors' nodes is
// overwritten with the next reversed datum, and the last pressure is stored as the image.
#pragma once

#include "pat_mx.cuh"
#include "pat_persist2.cuh"

namespace pat {

// work buffer: 2 fields of ppc line pairs, or 3 tiles of W columns (GRAD: the spectrum and two outputs)
template <typename T> __host__ __device__ size_t pmx_work_elems(const MxAxis& x, const MxAxis& y, int ppc, int W) {
    const size_t rowp = (size_t)2 * ppc * x.LS, colp = (size_t)3 * y.R0 * y.P0 * W;
    return ((rowp > colp ? rowp : colp) + 1) & ~(size_t)1;
}
__host__ __device__ inline int pmx_nres(int lossy) { return lossy ? 11 : 9; }
// work (complex) | resident rows [nres + 1][rmax][nx] (the last: sensor buffer) | a, au along x [nx] and
// of the CTA's lines | multipliers [1 or 3][ny W] (real) | flag
template <typename T> size_t pmx_smem_bytes(const MxAxis& x, const MxAxis& y, const PersistCfg& c, int lossy) {
    const size_t rows = (size_t)(pmx_nres(lossy) + 1) * c.rmax * x.n;
    const size_t mul = (size_t)(lossy ? 3 : 1) * ((y.n * c.W + 3) & ~3);
    return pmx_work_elems<T>(x, y, c.ppc, c.W) * sizeof(cplx<T>) +
           (rows + 2 * ((x.n + 3) & ~3) + 2 * ((c.rmax + 3) & ~3) + mul) * sizeof(T) + 16;
}

template <typename C> __device__ __forceinline__ C mx_sel(bool p, C a, C b) {
    a.x = p ? a.x : b.x;
    a.y = p ? a.y : b.y;
    return a;
}

// The last stage of a line pair runs in units of two butterflies that hold every X[k] with its X[n - k]:
// unit u > 0 has butterflies u and M - u (elements r of one and R - 1 - r of the other), unit 0 has
// butterflies 0 and, when M is even, M / 2, each its own mirror image.  Unit 0 takes the same code, with
// its elements exchanged by selects, so that no warp runs two versions.  FP32: half the loads of
// mx_row_in and no shuffles; with mx_row_in and mx_row_out the kernel spills and 168^2 takes 34.8 us a
// step instead of 27.9.  In double they lose (78.2 against 74.5 us lossless): a butterfly per thread
// halves the double instructions of the longest thread, although the double instances spill as they are
// (255 registers; 1916 bytes stored and 2536 loaded per thread forward, 1832 and 1620 adjoint).

// inverse last stage: C2R packing of the half spectra of FI fields, radix RL, twiddles
template <typename T>
__device__ __forceinline__ void pmx_row_in_units(cplx<T>* buf, const MxAxis& x, const cplx<T>* tabL, cplx<T>* const* spec,
                                          int FI, int np, int line0, int ldh) {
    const int n = x.n, M = x.M, half = n >> 1, U = (M + 1) >> 1;
    with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value, H = R / 2, E = (R - 1) / 2;
        for (int t = threadIdx.x; t < FI * np * U; t += blockDim.x) {
            const int line = mx_div(t, x.dU), u = t - line * U;
            const int f = (line >= np) + (line >= 2 * np), p = line - f * np;
            const bool u0 = u == 0;
            const int q2 = u0 ? M >> 1 : M - u;
            const cplx<T>* a = spec[f] + (size_t)(line0 + 2 * p) * ldh;
            const cplx<T>* b = a + ldh;
            cplx<T> v1[R], v2[R], ea, eb;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                // unit 0: M r up to n / 2, then M / 2 + M r' downwards
                const int k = u0 ? (r <= H ? M * r : (M >> 1) + M * (R - 1 - r)) : u + M * r;
                const int kk = k <= half ? k : n - k;
                v1[r] = __ldcg(a + kk);
                v2[R - 1 - r] = __ldcg(b + kk);
            }
            {
                const int kk = (M >> 1) + M * E;   // unit 0's last element
                ea = u0 ? __ldcg(a + kk) : v1[0];
                eb = u0 ? __ldcg(b + kk) : v2[R - 1];
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool up = !u0 && u + M * r > half;
                T ay = mx_flip(v1[r].y, up), by = mx_flip(v2[R - 1 - r].y, up);
                if (r == 0 || (R % 2 == 0 && r == H)) {   // the real elements k = 0 and n / 2 of unit 0
                    ay = u0 ? (T)0 : ay;
                    by = u0 ? (T)0 : by;
                }
                const T ax = v1[r].x, bx = v2[R - 1 - r].x;
                v1[r] = mkc<T>(ax - by, ay + bx);              // A + i B
                v2[R - 1 - r] = mkc<T>(ax + by, bx - ay);      // conj(A) + i conj(B)
            }
            {
                const T ay = (R % 2) ? (T)0 : ea.y, by = (R % 2) ? (T)0 : eb.y;   // odd R: k = n / 2
                const cplx<T> A = ea, B = eb;
                ea = mkc<T>(A.x - by, ay + B.x);
                eb = mkc<T>(A.x + by, B.x - ay);
                cplx<T> w1[R], w2[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    w1[r] = r <= H ? v1[r] : mx_sel(u0, v2[r - 1], v1[r]);
                    if (r < R - 1 - H) w2[r] = mx_sel(u0, v1[R - 1 - r], v2[r]);
                    else if (r == E) w2[r] = mx_sel(u0, ea, v2[r]);
                    else if (r == R - 1 - E) w2[r] = mx_sel(u0, eb, v2[r]);
                    else w2[r] = mx_sel(u0, v2[R - 1 - r], v2[r]);
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    v1[r] = w1[r];
                    v2[r] = w2[r];
                }
            }
            mx_dft<T, R, true>(v1);
#pragma unroll
            for (int r = 1; r < R; ++r) v1[r] = cmulc(v1[r], __ldg(tabL + (r - 1) * M + u));
            cplx<T>* s = buf + line * x.LS;
            cplx<T>* s1 = s + mx_base(x, u);
#pragma unroll
            for (int r = 0; r < R; ++r) s1[r] = v1[r];
            mx_dft<T, R, true>(v2);
#pragma unroll
            for (int r = 1; r < R; ++r) v2[r] = cmulc(v2[r], __ldg(tabL + (r - 1) * M + q2));
            cplx<T>* s2 = s + mx_base(x, q2);
            if (!u0 || !(M & 1)) {
#pragma unroll
                for (int r = 0; r < R; ++r) s2[r] = v2[r];
            }
        }
    });
}

// forward last stage, R2C unpacking (without its factor 1/2, which the multipliers carry), half spectra of
// FO fields to global memory
template <typename T>
__device__ __forceinline__ void pmx_row_out_units(const cplx<T>* buf, const MxAxis& x, const cplx<T>* tabL,
                                           cplx<T>* const* spec, int FO, int np, int line0, int ldh) {
    const int n = x.n, M = x.M, half = n >> 1, U = (M + 1) >> 1;
    with_mx<2>(x.RL, [&](auto RC) PAT_INLINE {
        constexpr int R = decltype(RC)::value, H = R / 2, E = (R - 1) / 2;
        for (int t = threadIdx.x; t < FO * np * U; t += blockDim.x) {
            const int line = mx_div(t, x.dU), u = t - line * U;
            const int f = (line >= np) + (line >= 2 * np), p = line - f * np;
            const bool u0 = u == 0;
            const int q2 = u0 ? M >> 1 : M - u;
            const cplx<T>* s = buf + line * x.LS;
            cplx<T> v1[R], v2[R];
            const cplx<T>* s1 = s + mx_base(x, u);
            const cplx<T>* s2 = s + mx_base(x, q2);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v1[r] = s1[r];
                v2[r] = s2[r];
            }
#pragma unroll
            for (int r = 1; r < R; ++r) {
                v1[r] = cmul(v1[r], __ldg(tabL + (r - 1) * M + u));
                v2[r] = cmul(v2[r], __ldg(tabL + (r - 1) * M + q2));
            }
            mx_dft<T, R, false>(v1);
            mx_dft<T, R, false>(v2);
            cplx<T>* a = spec[f] + (size_t)(line0 + 2 * p) * ldh;
            cplx<T>* b = a + ldh;
            auto put = [&](int k, cplx<T> zk, cplx<T> zm) PAT_INLINE {   // X[k] with X[n - k], either k
                const bool up = k > half;
                const int kk = up ? n - k : k;
                cplx<T> A = mkc<T>(zk.x + zm.x, mx_flip(zk.y - zm.y, up)), B = mkc<T>(zk.y + zm.y, mx_flip(zm.x - zk.x, up));
                a[kk] = A;
                b[kk] = B;
            };
            const bool two = !(M & 1);   // unit 0 has its second butterfly
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r <= H) {
                    // R odd: element H of unit 0 lies at M H <= n / 2 as well
                    put(u + M * r, v1[r], mx_sel(u0, v1[(R - r) % R], v2[R - 1 - r]));
                } else if (!u0 || two) {
                    put(u0 ? (M >> 1) + M * (R - 1 - r) : u + M * r, mx_sel(u0, v2[R - 1 - r], v1[r]),
                        mx_sel(u0, v2[r], v2[R - 1 - r]));
                }
            }
            if (u0 && two) put((M >> 1) + M * E, v2[E], v2[R - 1 - E]);
        }
    });
}

template <typename T, bool ADJ>
__global__ void __launch_bounds__(256) k_pmx(const __grid_constant__ DevPlan<T> P, const __grid_constant__ PersistCfg C,
                                             const __grid_constant__ MxAxis x, const __grid_constant__ MxAxis y,
                                             const cplx<T>* __restrict__ twx, const cplx<T>* __restrict__ twy,
                                             const T* __restrict__ kap, const T* __restrict__ abs, unsigned* gbar) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = x.n, ny = y.n, b = blockIdx.x, W = C.W, lgW = C.lgW;
    const bool lossy = P.lossy != 0;
    cplx<T>* const buf = reinterpret_cast<cplx<T>*>(smem_raw);
    T* const res = reinterpret_cast<T*>(buf + pmx_work_elems<T>(x, y, C.ppc, W));
    const int rstride = C.rmax * nx;
    T* const gb = res + pmx_nres(lossy) * rstride;
    T* const ax = gb + rstride;
    T* const aux = ax + ((nx + 3) & ~3);
    T* const ay = aux + ((nx + 3) & ~3);
    T* const auy = ay + ((C.rmax + 3) & ~3);
    T* const kapt = auy + ((C.rmax + 3) & ~3);
    const int tl = (ny * W + 3) & ~3;
    T* const s0t = kapt + tl;
    T* const s1t = s0t + tl;
    int* const flag = reinterpret_cast<int*>(kapt + (lossy ? 3 : 1) * tl);
    auto row = [&](int k) PAT_INLINE { return res + k * rstride; };

    const unsigned G = gridDim.x;
    const int pair0 = b * C.ppc;
    const int np = max(0, min(ny / 2 - pair0, C.ppc));
    const int R = 2 * np, line0 = 2 * pair0;
    const bool rows = R > 0, tile = b < C.ntiles;
    const int kx0 = b * W;
    const T dt = P.dt;
    const int Nt = P.Nt, Ns = P.sens.Ns;
    unsigned kbar = 0;
    const TraceRef TR{P.trace, P.trace_k0, P.trace_nk};
    const cplx<T>* const xL = twx;
    const cplx<T>* const x1 = twx + (x.RL - 1) * x.M;
    const cplx<T>* const yL = twy;
    const cplx<T>* const y1 = twy + (y.RL - 1) * y.M;
    const bool rev = !ADJ && P.tr_node != nullptr;   // time reversal
    const DevSensors<T>& S = P.sens;
    // sub-phase mark j of the trace
    auto mark = [&](int j) PAT_INLINE {
        if (!TR.buf || threadIdx.x != 0) return;
        const int kt = (int)kbar - TR.k0;
        if (kt >= 0 && kt < TR.nk) TR.buf[((size_t)b * TR.nk + kt) * kTraceStride + 2 + j] = globaltimer_ns();
    };

    // ---- setup: multipliers of the tile, resident medium and state ----
    stage_elems(ax, P.a[0], nx);
    stage_elems(aux, P.au[0], nx);
    if (tile) {
        for (int t = threadIdx.x; t < ny * W; t += blockDim.x) {
            const int i = t >> lgW, c = t & (W - 1);
            // from the plan's tables, with the factor 1/2 of the R2C unpacking (exact in binary)
            const size_t at = (size_t)i * P.ldh + min(kx0 + c, P.nxh - 1);
            kapt[t] = (T)0.5 * kap[at];
            if (lossy) {
                s0t[t] = (T)0.5 * abs[at];
                s1t[t] = (T)0.5 * abs[(size_t)ny * P.ldh + at];
                if (P.tr_kc2 > (T)0) {   // time reversal: reversed and windowed
                    const T kx = P.kv[0][min(kx0 + c, P.nxh - 1)], ky = P.kv[1][i];
                    s0t[t] = (T)0.5 * abs_mult0(P, kx * kx + ky * ky);
                }
            }
        }
    }
    int s0 = 0, s1 = 0;   // this CTA's sensor segments
    if (rows) {
        for (int r = threadIdx.x; r < R; r += blockDim.x) {
            ay[r] = P.a[1][line0 + r];
            auy[r] = P.au[1][line0 + r];
        }
        stage_rows(row(PS_C2), P.c2, line0, R, nx);
        stage_rows(row(PS_RHO0), P.rho0, line0, R, nx);
        stage_rows(row(PS_B0), P.b[0], line0, R, nx);
        stage_rows(row(PS_B1), P.b[1], line0, R, nx);
        if (lossy) {
            stage_rows(row(PS_C2TAU), P.c2tau, line0, R, nx);
            stage_rows(row(PS_C2ETA), P.c2eta, line0, R, nx);
        }
        if (!ADJ) stage_rows(row(PS_RS), P.img, line0, R, nx);   // p0 (consumed by the init)
        s0 = ADJ ? S.s_lineptr[line0] : S.g_lineptr[line0];
        s1 = ADJ ? S.s_lineptr[line0 + R] : S.g_lineptr[line0 + R];
        for (int t = threadIdx.x; t < R * nx; t += blockDim.x) gb[t] = 0;
        if (ADJ || rev)   // the state starts at zero (time reversal: u^{-1/2} = 0)
            for (int j = 0; j < (ADJ ? 4 : 2); ++j)
                for (int t = threadIdx.x; t < R * nx; t += blockDim.x) row(PS_U0 + j)[t] = 0;
    }
    cp_commit();
    cp_wait_all();
    __syncthreads();

    auto pml_a = [&](int xi, int r, int i) PAT_INLINE { return xi == 0 ? ax[i] : ay[r]; };
    auto pml_au = [&](int xi, int r, int i) PAT_INLINE { return xi == 0 ? aux[i] : auy[r]; };
    // adjoint: M^T h is added into gb, which stays zero between uses
    auto take_inj = [&](int t) PAT_INLINE {
        const T v = gb[t];
        gb[t] = (T)0;
        return v;
    };
    // adjoint: p_bar of the current level -> the gradient (final level), else the inputs of the next
    // x transforms
    auto tail = [&](int r, int i, int t, T pv, bool final_, T* out) PAT_INLINE {
        if (final_) {
            const T sr = row(PS_R0)[t] + row(PS_R1)[t];
            P.img[(size_t)line0 * nx + t] = pv + sr / ((T)2 * row(PS_C2)[t]);
            return;
        }
        if (lossy) {
            row(PS_RS)[t] = pv;
            out[0] = row(PS_C2TAU)[t] * pv;
            out[1] = row(PS_C2ETA)[t] * pv;
        } else {
            const T rbar = row(PS_C2)[t] * pv;
            const T rho0 = row(PS_RHO0)[t];
#pragma unroll
            for (int xi = 0; xi < 2; ++xi) {
                const T a = pml_a(xi, r, i);
                const T rb = row(PS_R0 + xi)[t] + rbar;
                out[xi] = -dt * rho0 * a * rb;
                row(PS_R0 + xi)[t] = a * a * rb;
            }
        }
    };
    // forward: rho update from e = D- u; returns rho0, sets sum_xi rho_xi and sum_xi e_xi
    auto rho_upd = [&](int r, int i, int t, const T* in, T& rs, T& es) PAT_INLINE {
        const T rho0 = row(PS_RHO0)[t];
        rs = 0;
        es = 0;
#pragma unroll
        for (int xi = 0; xi < 2; ++xi) {
            const T e = in[xi];
            const T a = pml_a(xi, r, i);
            const T rh = a * (a * row(PS_R0 + xi)[t] - dt * rho0 * e);
            row(PS_R0 + xi)[t] = rh;
            rs += rh;
            es += e;
        }
        return rho0;
    };

    // one row phase: inverse x transform of FI spectra, the pointwise step of `pid`, forward x transform
    // of its FO outputs (unless it ends the solve)
    auto row_phase = [&](int pid, int n, bool lastph) PAT_INLINE {
        int FI = 2, FO = 2;
        bool fwd = true, gath = false, scat = false;
        switch (pid) {
            case R_F_INIT: FI = 0; FO = 1; fwd = !lastph; gath = true; break;
            case R_F_RHO_LOSSLESS:
            case R_F_P: FO = 1; fwd = !lastph; gath = true; break;
            case R_A_INIT: FI = 0; fwd = !lastph; scat = true; break;
            case R_A_GRADT: FI = 1; fwd = !lastph; scat = true; break;
            default: break;
        }
        const bool first = (n == 0) && !rev;
        const int level = ADJ ? n : (pid == R_F_INIT ? 0 : n + 1);
        T* drow = P.data + (size_t)(rev ? Nt - 1 - level : level) * Ns;
        if (scat)
            for (int q = s0 + threadIdx.x; q < s1; q += blockDim.x) {
                T v = 0;
                for (int e = S.s_seg_e0[q]; e < S.s_seg_e0[q + 1]; ++e) v += S.s_ent_w[e] * drow[S.s_ent_sensor[e]];
                gb[(S.s_seg_line[q] - line0) * nx + S.s_seg_x[q]] += v;
            }
        if (FI > 0) {
            if constexpr (sizeof(T) == 4) pmx_row_in_units<T>(buf, x, xL, P.spec, FI, np, line0, P.ldh);
            else mx_row_in<T>(buf, x, xL, P.spec, FI, np, line0, P.ldh);
            __syncthreads();
            mark(0);
            if (x.R1 > 1) {
                mx_mid<T, true>(buf, x, x1, FI * np, x.LS, 1, 0);
                __syncthreads();
            }
            mark(1);
            mx_row_s0<T, true>(buf, x, FI * np);
        }
        __syncthreads();
        mark(2);
        const int fs = np * x.LS, pad = x.P0 - x.m0;
        // fn(row r, x index i, element t of the resident rows, in[2], out[2]) over the CTA's points, two rows
        // of a line pair at a time; one loop per phase, so each is short code with no branch inside
        auto each = [&](auto FIc, auto FOc, auto&& fn) PAT_INLINE {
            constexpr int NI = decltype(FIc)::value, NO = decltype(FOc)::value;
            for (int e = threadIdx.x; e < np * nx; e += blockDim.x) {
                const int p = mx_div(e, x.dn), i = e - p * nx;
                cplx<T>* bp = buf + p * x.LS + i + pad * mx_div(i, x.dm0);
                cplx<T> z[2] = {mkc<T>(0, 0), mkc<T>(0, 0)};
                if (NI > 0) z[0] = bp[0];
                if (NI > 1) z[1] = bp[fs];
                T i0[2] = {z[0].x, z[1].x}, i1[2] = {z[0].y, z[1].y}, o0[2] = {0, 0}, o1[2] = {0, 0};
                const int t = 2 * p * nx + i;
                fn(2 * p, i, t, i0, o0);
                fn(2 * p + 1, i, t + nx, i1, o1);
                if (fwd) {
                    bp[0] = mkc<T>(o0[0], o1[0]);
                    if (NO > 1) bp[fs] = mkc<T>(o0[1], o1[1]);
                }
            }
        };
        const std::integral_constant<int, 0> c0;
        const std::integral_constant<int, 1> c1;
        const std::integral_constant<int, 2> c2;
        switch (pid) {
            case R_F_INIT:
                each(c0, c1, [&](int, int, int t, const T*, T* out) PAT_INLINE {
                    const T pv = row(PS_RS)[t];
                    const T rh = pv / ((T)2 * row(PS_C2)[t]);
                    row(PS_R0)[t] = rh;
                    row(PS_R1)[t] = rh;
                    gb[t] = pv;
                    out[0] = pv;
                });
                break;
            case R_F_U:
                each(c2, c2, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
#pragma unroll
                    for (int xi = 0; xi < 2; ++xi) {
                        const T g = in[xi];
                        const T bq = row(PS_B0 + xi)[t];
                        const T au = pml_au(xi, r, i);
                        const T uo = first ? (T)0.5 * dt * bq * g : row(PS_U0 + xi)[t];
                        const T un = au * (au * uo - dt * bq * g);
                        row(PS_U0 + xi)[t] = un;
                        out[xi] = un;
                    }
                });
                break;
            case R_F_RHO_LOSSY:
                each(c2, c2, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
                    T rs, es;
                    const T rho0 = rho_upd(r, i, t, in, rs, es);
                    row(PS_RS)[t] = rs;
                    out[0] = rho0 * es;
                    out[1] = rs;
                });
                break;
            case R_F_RHO_LOSSLESS:
                each(c2, c1, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
                    T rs, es;
                    rho_upd(r, i, t, in, rs, es);
                    const T pv = row(PS_C2)[t] * rs;
                    gb[t] = pv;
                    out[0] = pv;
                });
                break;
            case R_F_P:
                each(c2, c1, [&](int, int, int t, const T* in, T* out) PAT_INLINE {
                    const T pv = row(PS_C2)[t] * row(PS_RS)[t] + row(PS_C2TAU)[t] * in[0] - row(PS_C2ETA)[t] * in[1];
                    gb[t] = pv;
                    out[0] = pv;
                });
                break;
            case R_A_INIT:
                each(c0, c2, [&](int r, int i, int t, const T*, T* out) PAT_INLINE { tail(r, i, t, take_inj(t), lastph, out); });
                break;
            case R_A_ABS:
                each(c2, c2, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
                    const T ddbar = in[0];
                    const T rbar = row(PS_C2)[t] * row(PS_RS)[t] - in[1];
                    const T rho0 = row(PS_RHO0)[t];
#pragma unroll
                    for (int xi = 0; xi < 2; ++xi) {
                        const T a = pml_a(xi, r, i);
                        const T rb = row(PS_R0 + xi)[t] + rbar;
                        out[xi] = rho0 * ddbar - dt * rho0 * a * rb;
                        row(PS_R0 + xi)[t] = a * a * rb;
                    }
                });
                break;
            case R_A_DIVT:
                each(c2, c2, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
#pragma unroll
                    for (int xi = 0; xi < 2; ++xi) {
                        const T bq = row(PS_B0 + xi)[t];
                        const T au = pml_au(xi, r, i);
                        T ub = row(PS_U0 + xi)[t] + in[xi];
                        T g = -dt * bq * au * ub;
                        ub = au * au * ub;
                        if (first) g += (T)0.5 * dt * bq * ub;
                        row(PS_U0 + xi)[t] = ub;
                        out[xi] = g;
                    }
                });
                break;
            default:   // R_A_GRADT
                each(c1, c2, [&](int r, int i, int t, const T* in, T* out) PAT_INLINE {
                    tail(r, i, t, in[0] + take_inj(t), lastph, out);
                });
                break;
        }
        __syncthreads();
        mark(3);
        if (gath && !rev) {   // s_j += this CTA's part of sensor j
            for (int q = s0 + threadIdx.x; q < s1; q += blockDim.x) {
                const T* pr = gb + (S.g_seg_line[q] - line0) * nx + S.g_seg_x0[q];
                const T w0 = S.g_seg_w0[q], w1 = S.g_seg_w1[q];
                T acc = w0 * pr[0];
                if (w1 != (T)0) acc += w1 * pr[1];
                atomicAdd(&drow[S.g_seg_sensor[q]], acc);
            }
        } else if (rev && pid != R_F_INIT && pid != R_F_U) {
            // the split densities and the pressure at the sensors' nodes take the reversed datum of the
            // new level (a node lies in one pair's slot: two nodes of a slot are its two components)
            const bool rho = pid != R_F_P, pr = pid != R_F_RHO_LOSSY;
            for (int q = s0 + threadIdx.x; q < s1; q += blockDim.x) {
                if (S.g_seg_w0[q] == (T)0) continue;
                const int r = S.g_seg_line[q] - line0, i = S.g_seg_x0[q], t = r * nx + i;
                const T v = drow[S.g_seg_sensor[q]];
                if (rho) {
                    const T rh = v / ((T)2 * row(PS_C2)[t]);
                    row(PS_R0)[t] = rh;
                    row(PS_R1)[t] = rh;
                }
                if (pr) {
                    gb[t] = v;
                    cplx<T>& z = buf[(r >> 1) * x.LS + i + pad * mx_div(i, x.dm0)];
                    if (r & 1) z.y = v;
                    else z.x = v;
                }
            }
            __syncthreads();
            if (pr && lastph)
                for (int t = threadIdx.x; t < R * nx; t += blockDim.x) P.img[(size_t)line0 * nx + t] = gb[t];
        }
        if (!fwd) return;
        mx_row_s0<T, false>(buf, x, FO * np);
        __syncthreads();
        if (x.R1 > 1) {
            mx_mid<T, false>(buf, x, x1, FO * np, x.LS, 1, 0);
            __syncthreads();
        }
        mark(4);
        if constexpr (sizeof(T) == 4) pmx_row_out_units<T>(buf, x, xL, P.spec, FO, np, line0, P.ldh);
        else mx_row_out<T, false>(buf, x, xL, P.spec, FO, np, line0, P.ldh);
        mark(5);
    };

    // one column phase: y transform, the multiply of `mode`, inverse y transform of the CTA's columns
    auto col_phase = [&](int mode) PAT_INLINE {
        const int fi = (mode == SPEC_GRAD) ? 1 : 2, fo = (mode == SPEC_GRADT) ? 1 : 2;
        const int tile_sz = (y.R0 * y.P0) << lgW;
        const int o0 = (mode == SPEC_GRAD) ? 1 : 0;   // GRAD: outputs in tiles 1 and 2
        const int c = threadIdx.x & (W - 1);
        const bool ok = kx0 + c < P.nxh;
        const int ldh = P.ldh, m0 = y.m0, M = y.M;
        with_mx<0>(y.R0, [&](auto RC) PAT_INLINE {
            constexpr int Q = decltype(RC)::value;
            for (int t = threadIdx.x; t < ((fi * m0) << lgW); t += blockDim.x) {
                const int u = t >> lgW, f = (u >= m0) ? 1 : 0, j = u - f * m0;
                const cplx<T>* src = P.spec[f] + kx0 + c;
                cplx<T>* d = buf + f * tile_sz + c;
                cplx<T> v[Q];
#pragma unroll
                for (int r = 0; r < Q; ++r) v[r] = ok ? __ldcg(src + (size_t)(j + m0 * r) * ldh) : mkc<T>(0, 0);
                mx_dft<T, Q, false>(v);
#pragma unroll
                for (int r = 0; r < Q; ++r) d[(y.P0 * r + j) << lgW] = v[r];
            }
        });
        __syncthreads();
        mark(0);
        if (y.R1 > 1) {
            mx_mid<T, false>(buf, y, y1, fi, tile_sz, W, lgW);
            __syncthreads();
        }
        mark(1);
        const bool plus = (mode == SPEC_GRAD || mode == SPEC_DIVT);
        const int kx = min(kx0 + c, P.nxh - 1);
        const cplx<T> mx0 = plus ? __ldg(P.dp[0] + kx) : __ldg(P.dm[0] + kx);
        const cplx<T>* ml = plus ? P.dp[1] : P.dm[1];
        with_mx<2>(y.RL, [&](auto RC) PAT_INLINE {
            constexpr int Q = decltype(RC)::value;
            for (int t = threadIdx.x; t < ((fo * M) << lgW); t += blockDim.x) {
                const int u = t >> lgW, f = (u >= M) ? 1 : 0, q = u - f * M;
                const cplx<T>* s = buf + (mx_base(y, q) << lgW) + c;
                cplx<T> v[Q], w[Q];
                // GRADT: both inputs; GRAD: the one input for either output; else its own field
                const int nin = (mode == SPEC_GRADT) ? 2 : 1;
                for (int g = 0; g < nin; ++g) {
                    const cplx<T>* sg = s + ((mode == SPEC_GRAD) ? 0 : (mode == SPEC_GRADT ? g : f)) * tile_sz;
#pragma unroll
                    for (int r = 0; r < Q; ++r) w[r] = sg[r << lgW];
#pragma unroll
                    for (int r = 1; r < Q; ++r) w[r] = cmul(w[r], __ldg(yL + (r - 1) * M + q));
                    mx_dft<T, Q, false>(w);
                    if (mode == SPEC_ABS) {
                        const T* sc = f ? s1t : s0t;
#pragma unroll
                        for (int r = 0; r < Q; ++r) v[r] = cscale(w[r], sc[((q + M * r) << lgW) + c]);
                    } else {
                        const int sf = (mode == SPEC_GRADT) ? g : f;   // the derivative's axis
#pragma unroll
                        for (int r = 0; r < Q; ++r) {
                            const cplx<T> m = cmul(w[r], sf ? __ldg(ml + q + M * r) : mx0);
                            v[r] = (g == 0) ? m : cadd(v[r], m);
                        }
                    }
                }
                if (mode != SPEC_ABS) {
                    const bool neg = mode == SPEC_DIVT || mode == SPEC_GRADT;
#pragma unroll
                    for (int r = 0; r < Q; ++r) v[r] = cscale(v[r], mx_flip(kapt[((q + M * r) << lgW) + c], neg));
                }
                mx_dft<T, Q, true>(v);
#pragma unroll
                for (int r = 1; r < Q; ++r) v[r] = cmulc(v[r], __ldg(yL + (r - 1) * M + q));
                cplx<T>* d = buf + (o0 + f) * tile_sz + (mx_base(y, q) << lgW) + c;
#pragma unroll
                for (int r = 0; r < Q; ++r) d[r << lgW] = v[r];
            }
        });
        __syncthreads();
        mark(2);
        cplx<T>* ob = buf + o0 * tile_sz;
        if (y.R1 > 1) {
            mx_mid<T, true>(ob, y, y1, fo, tile_sz, W, lgW);
            __syncthreads();
        }
        mark(3);
        with_mx<0>(y.R0, [&](auto RC) PAT_INLINE {
            constexpr int Q = decltype(RC)::value;
            for (int t = threadIdx.x; t < ((fo * m0) << lgW); t += blockDim.x) {
                const int u = t >> lgW, f = (u >= m0) ? 1 : 0, j = u - f * m0;
                cplx<T>* dst = P.spec[f] + kx0 + c;
                const cplx<T>* s = ob + f * tile_sz + c;
                cplx<T> v[Q];
#pragma unroll
                for (int r = 0; r < Q; ++r) v[r] = s[(y.P0 * r + j) << lgW];
                mx_dft<T, Q, true>(v);
                if (ok) {
#pragma unroll
                    for (int r = 0; r < Q; ++r) dst[(size_t)(j + m0 * r) * ldh] = v[r];
                }
            }
        });
        mark(4);
    };

    const int nph = (Nt > 1) ? 1 + (Nt - 1) * (lossy ? 6 : 4) : 1;
    for (int k = 0; k < nph; ++k) {
        const P2Phase d = p2_phase<ADJ>(k, Nt, lossy);
        const bool lastph = (k == nph - 1);
        if (d.col) {
            if (tile) col_phase(d.id);
        } else if (rows) {
            row_phase(d.id, d.n, lastph);
        }
        if (!lastph && !grid_barrier(gbar, G, kbar, flag, TR, P.bar_extra, P.bar_limit_ns)) return;
    }
}

}  // namespace pat
