// pat_optim.cu -- image-space kernels of the optimisation shell (Sec. IV, Sec. V):
//   isotropic TV and its proximal map by the dual fast-gradient-projection iteration
//   (Sec. IV Eq. (proxmal)), smoothed TV and its gradient (Sec. V.B Eqs. (Thirty-two),
//   (Twentyone)), the transfer operators I_h^{h-1} = 2^-d P^T and I_{h-1}^h = P (Sec. V.A), the
//   restricted bound (Sec. V.C Eq. (constraint)), FP64 reductions and FISTA vector updates.
// Conventions: image [Nz][Ny][Nx], x fastest; D = forward differences with a zero difference at
// the last index of each axis; D^T its exact transpose.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "pat_host.h"
#include "pat_optim.h"

namespace pat {

struct ImgDims {
    int d, n[3];
    long long N;
    long long s[3];   // strides
};

static ImgDims img_dims(const pat_grid& g) {
    ImgDims D;
    D.d = g.ndim;
    D.n[0] = g.n[0];
    D.n[1] = g.n[1];
    D.n[2] = (g.ndim == 3) ? g.n[2] : 1;
    D.N = (long long)D.n[0] * D.n[1] * D.n[2];
    D.s[0] = 1;
    D.s[1] = D.n[0];
    D.s[2] = (long long)D.n[0] * D.n[1];
    return D;
}

__device__ __forceinline__ void unflat(long long i, const ImgDims& D, int* c) {
    c[0] = (int)(i % D.n[0]);
    const long long r = i / D.n[0];
    c[1] = (int)(r % D.n[1]);
    c[2] = (int)(r / D.n[1]);
}

// ------------------------------------------------------------------------------------------
// TV pieces
// ------------------------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ T dfwd(const T* x, long long i, const int* c, const ImgDims& D, int a) {
    return (c[a] < D.n[a] - 1) ? x[i + D.s[a]] - x[i] : (T)0;
}
// One FGP iteration (dual of the TV prox, Sec. IV): r = q + w (q - q_prev), then
// q_new = Pi_{|q|<=1}(r + step D x(r)) with x(r) = P_C(z - lam D^T r).
//
// A CTA takes a tile of (x, y) and marches along z over `chunk` planes.  Each plane's x(r) goes once through
// shared memory with a halo of one column and one row; the next plane's is formed before the barrier, so its
// loads are in flight there, and r is formed where it is read and kept in registers for the plane's update.
// FP32 is bound by memory: z and the last two duals read, the new one written, 1 + 3 d fields per iteration,
// each fetched from DRAM about once (256^3, 20 iterations: 3.65 ms, 3.7 TB/s; 4.25 ms with the next plane after
// the barrier; 20 ms for one thread per point over flat indices, which formed x(r) d + 1 times from global
// memory).  Its 64 x 8 tile is compiled in: run-time sides cost a quarter (256^3: 5.9 against 4.8 ms).  Images of at most 32 columns would leave half of its lanes idle, and
// double is bound by its pipes, where an idle lane costs as much as a busy one: both take a run-time tile whose
// points fill the CTA's lanes (fgp_tile).  20 iterations, flat / 64 x 8 tiles / run-time tiles, in us:
// 1000 x 1000 x 4 FP32 4220 / 8260 / 1360; 256 x 256 x 8 FP32 740 / 790 / 290; double 1000 x 1000 x 4 10800 /
// 58400 / 8200, 64^3 1040 / 1330 / 800, 256^2 376 / 439 / 323, 256^3 44400 / 32800 / 31900.
constexpr int kFgpX = 64, kFgpY = 8;
constexpr int kFgpThreads = 512;   // tile points, and threads, of a CTA
constexpr int kFgpRows = 256;      // rows of a tile

template <typename T> struct FgpArgs {
    int nx, ny, nz, chunk;   // chunk: planes per CTA (3-D)
    int tw, th;              // points of a tile along x and y
    unsigned gx, gy;         // tiles along x and y (the grid is one-dimensional: no limit on a side)
    const T* z;
    const T* q[3];           // q_k
    const T* qp[3];          // q_{k-1}
    T* qn[3];                // q_{k+1}
    T lam, step, w;
    int nonneg, first;       // first: q_k = q_{k-1} = 0 (not read)
};

template <typename T, int D, bool FIXED>
__global__ void __launch_bounds__(kFgpThreads) k_fgp_iter(FgpArgs<T> A) {
    // (tw + 1)(th + 1), at most kFgpThreads + kFgpRows + 3
    __shared__ T sx[2][FIXED ? (kFgpX + 1) * (kFgpY + 1) : kFgpThreads + kFgpRows + 4];
    const int tw = FIXED ? kFgpX : A.tw, th = FIXED ? kFgpY : A.th, ld = tw + 1;
    const int tid = threadIdx.x, ty = tid / tw, tx = tid - ty * tw;
    const unsigned bx = blockIdx.x % A.gx, byz = blockIdx.x / A.gx, by = byz % A.gy, bz = byz / A.gy;
    const int x0 = bx * tw, y0 = by * th;
    const int k0 = (D == 3) ? bz * A.chunk : 0;
    const int k1 = (D == 3) ? min(k0 + A.chunk, A.nz) : 1;
    const int nx = A.nx, ny = A.ny;
    const size_t sy = (size_t)nx, sz = (size_t)nx * ny;
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");

    auto r_at = [&](int a, size_t i) {
        const T q = A.q[a][i];
        return q + A.w * (q - A.qp[a][i]);
    };
    // x(r) at (x, y, k); r[] receives r_a there (0 where D_a is zero is kept by the projection), rzm
    // is r_z of the plane below
    auto prox = [&](int x, int y, int k, size_t i, T rzm, T* r) {
        T v = 0;
        if (!A.first) {
            r[0] = r_at(0, i);
            r[1] = r_at(1, i);
            if (x >= 1) v += r_at(0, i - 1);
            if (x <= nx - 2) v -= r[0];
            if (y >= 1) v += r_at(1, i - sy);
            if (y <= ny - 2) v -= r[1];
            if constexpr (D == 3) {
                r[2] = r_at(2, i);
                if (k >= 1) v += rzm;
                if (k <= A.nz - 2) v -= r[2];
            }
        } else {
#pragma unroll
            for (int a = 0; a < D; ++a) r[a] = 0;
        }
        v = A.z[i] - A.lam * v;
        return A.nonneg ? fmax(v, (T)0) : v;
    };

    const int x = x0 + tx, y = y0 + ty;
    const bool in = ty < th && x < nx && y < ny;
    // this thread's halo point, if any: the column x0 + tw (rows 0 .. th - 1), the row y0 + th
    int hx = -1, hy = 0;
    if (FIXED) {
        if (tid < th) {
            hx = tw;
            hy = tid;
        } else if (tid >= 32 && tid < 32 + tw) {
            hx = tid - 32;
            hy = th;
        }
    } else if (tid < th) {
        hx = tw;
        hy = tid;
    } else if (tid < th + tw) {
        hx = tid - th;
        hy = th;
    }
    const bool hin = hx >= 0 && x0 + hx < nx && y0 + hy < ny;
    const size_t i0 = (size_t)y * sy + x, h0 = (size_t)(y0 + hy) * sy + (x0 + (hx < 0 ? 0 : hx));
    const int at = ty * ld + tx;
    T r[3] = {0, 0, 0}, xk = 0, rzm = 0, hrzm = 0;
    if (D == 3 && k0 >= 1 && !A.first) {
        if (in) rzm = r_at(2, i0 + (size_t)(k0 - 1) * sz);
        if (hin) hrzm = r_at(2, h0 + (size_t)(k0 - 1) * sz);
    }
    if (in) xk = prox(x, y, k0, i0 + (size_t)k0 * sz, rzm, r);
    for (int k = k0; k < k1; ++k) {
        T* s = sx[(k - k0) & 1];
        if (in) s[at] = xk;
        if (hin) {
            T hr[3];
            s[hy * ld + hx] = prox(x0 + hx, y0 + hy, k, h0 + (size_t)k * sz, hrzm, hr);
            if constexpr (D == 3) hrzm = hr[2];
        }
        // the next plane's x(r), for this plane's difference along z; its loads are in flight at the barrier
        const bool up = D == 3 && k + 1 < A.nz;
        T rn[3] = {0, 0, 0}, xn = 0;
        if (in && up) xn = prox(x, y, k + 1, i0 + (size_t)(k + 1) * sz, r[2], rn);
        __syncthreads();
        if (in) {
            T q[3] = {r[0] + A.step * ((x < nx - 1) ? s[at + 1] - xk : (T)0),
                      r[1] + A.step * ((y < ny - 1) ? s[at + ld] - xk : (T)0),
                      (D == 3) ? r[2] + A.step * (up ? xn - xk : (T)0) : (T)0};
            T nrm2 = 0;
#pragma unroll
            for (int a = 0; a < D; ++a) nrm2 += q[a] * q[a];
            T sc = (T)1;   // of |q| <= 1 and of NaN: in double the branch saves a division and a root
            if (sizeof(T) == 4 || nrm2 > (T)1) sc = (T)1 / fmax((T)1, sqrt(nrm2));
#pragma unroll
            for (int a = 0; a < D; ++a) A.qn[a][i0 + (size_t)k * sz] = q[a] * sc;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) r[a] = rn[a];
        xk = xn;
    }
}

// x = P_C(z - lam D^T q): z and the duals read once, x written once
template <typename T, int D>
__global__ void __launch_bounds__(256) k_fgp_final(FgpArgs<T> A, T* x) {
    const unsigned bx = blockIdx.x % A.gx, byz = blockIdx.x / A.gx;
    const int ty = threadIdx.x / A.tw, i = bx * A.tw + (threadIdx.x - ty * A.tw);
    const int j = (byz % A.gy) * A.th + ty, k = byz / A.gy;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (ty >= A.th || i >= A.nx || j >= A.ny) return;
    const size_t sy = (size_t)A.nx, sz = sy * A.ny, p = (size_t)k * sz + (size_t)j * sy + i;
    T v = 0;
    if (i >= 1) v += A.q[0][p - 1];
    if (i <= A.nx - 2) v -= A.q[0][p];
    if (j >= 1) v += A.q[1][p - sy];
    if (j <= A.ny - 2) v -= A.q[1][p];
    if constexpr (D == 3) {
        if (k >= 1) v += A.q[2][p - sz];
        if (k <= A.nz - 2) v -= A.q[2][p];
    }
    v = A.z[p] - A.lam * v;
    x[p] = A.nonneg ? fmax(v, (T)0) : v;
}

// v_a(j) = D_a y(j) / sqrt(|D y(j)|^2 + rho^2)
template <typename T>
__device__ __forceinline__ T vsm(const T* y, long long j, const int* c, const ImgDims& D, int a, T rho) {
    T g[3] = {0, 0, 0};
    T s = rho * rho;
    for (int b = 0; b < D.d; ++b) {
        g[b] = dfwd(y, j, c, D, b);
        s += g[b] * g[b];
    }
    return g[a] / sqrt(s);
}

// gradient of J_rho: D^T v (Sec. V.B Eq. (Twentyone)); out = beta * out + alpha * grad
template <typename T>
__global__ void k_tv_smooth_grad(ImgDims D, const T* y, T rho, T* out, T alpha, T beta) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < D.N; i += (long long)gridDim.x * blockDim.x) {
        int c[3];
        unflat(i, D, c);
        T g = 0;
        for (int a = 0; a < D.d; ++a) {
            if (c[a] >= 1) {
                int cm[3] = {c[0], c[1], c[2]};
                cm[a] -= 1;
                g += vsm(y, i - D.s[a], cm, D, a, rho);
            }
            if (c[a] <= D.n[a] - 2) g -= vsm(y, i, c, D, a, rho);
        }
        out[i] = (beta == (T)0 ? (T)0 : beta * out[i]) + alpha * g;
    }
}

// ------------------------------------------------------------------------------------------
// FP64 reductions (two passes, fixed order: deterministic)
// ------------------------------------------------------------------------------------------
enum RedOp : int { RED_DOT = 0, RED_TV = 1, RED_TVS = 2, RED_SQDIFF = 3 };

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)((blockDim.x + 31) >> 5); ++k) s += sh[k];
    return s;
}

template <typename T>
__global__ void k_reduce(int op, ImgDims D, long long n, const T* a, const T* b, T rho, double* partial) {
    __shared__ double sh[32];
    double acc = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (op == RED_DOT) {
            acc += (double)a[i] * (double)b[i];
        } else if (op == RED_SQDIFF) {
            const double d = (double)a[i] - (double)b[i];
            acc += d * d;
        } else {
            int c[3];
            unflat(i, D, c);
            double s = 0;
            for (int k = 0; k < D.d; ++k) {
                const double g = (double)dfwd(a, i, c, D, k);
                s += g * g;
            }
            if (op == RED_TV) acc += sqrt(s);
            else acc += sqrt(s + (double)rho * (double)rho) - (double)rho;
        }
    }
    const double s = block_sum(acc, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void k_reduce_final(const double* partial, int nb, double* out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0;
        for (int k = 0; k < nb; ++k) s += partial[k];
        *out = s;
    }
}

// ------------------------------------------------------------------------------------------
// grid transfer and the restricted bound
// ------------------------------------------------------------------------------------------
// R = 2^-d P^T: coarse i gathers fine 2i-1 (1/2, i >= 1), 2i (1), 2i+1 (1/2; 1 at the last
// coarse index, where P clamps) per axis.
template <typename T>
__global__ void k_restrict(ImgDims F, ImgDims C, const T* xf, T* xc) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < C.N; i += (long long)gridDim.x * blockDim.x) {
        int c[3];
        unflat(i, C, c);
        int fi[3][3];
        T fw[3][3];
        int cnt[3];
        for (int a = 0; a < 3; ++a) {
            if (a >= C.d) {
                fi[a][0] = 0;
                fw[a][0] = 1;
                cnt[a] = 1;
                continue;
            }
            int k = 0;
            if (c[a] >= 1) {
                fi[a][k] = 2 * c[a] - 1;
                fw[a][k++] = (T)0.5;
            }
            fi[a][k] = 2 * c[a];
            fw[a][k++] = (T)1;
            fi[a][k] = 2 * c[a] + 1;
            fw[a][k++] = (c[a] == C.n[a] - 1) ? (T)1 : (T)0.5;
            cnt[a] = k;
        }
        T acc = 0;
        for (int kz = 0; kz < cnt[2]; ++kz)
            for (int ky = 0; ky < cnt[1]; ++ky)
                for (int kx = 0; kx < cnt[0]; ++kx) {
                    const long long j = fi[0][kx] + F.s[1] * fi[1][ky] + F.s[2] * fi[2][kz];
                    acc += fw[0][kx] * fw[1][ky] * fw[2][kz] * xf[j];
                }
        xc[i] = acc / (T)(1 << C.d);
    }
}

// P: fine 2i <- coarse i; fine 2i+1 <- (coarse i + coarse min(i+1, nc-1)) / 2, per axis.
// out = beta * out + alpha * P xc (beta = 0 overwrites).
template <typename T>
__global__ void k_prolong(ImgDims F, ImgDims C, const T* xc, T* xf, T alpha, T beta) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < F.N; i += (long long)gridDim.x * blockDim.x) {
        int f[3];
        unflat(i, F, f);
        int ci[3][2];
        T cw[3][2];
        int cnt[3];
        for (int a = 0; a < 3; ++a) {
            if (a >= F.d) {
                ci[a][0] = 0;
                cw[a][0] = 1;
                cnt[a] = 1;
                continue;
            }
            const int k = f[a] >> 1;
            if ((f[a] & 1) == 0) {
                ci[a][0] = k;
                cw[a][0] = 1;
                cnt[a] = 1;
            } else {
                ci[a][0] = k;
                ci[a][1] = min(k + 1, C.n[a] - 1);
                cw[a][0] = cw[a][1] = (T)0.5;
                cnt[a] = 2;
            }
        }
        T acc = 0;
        for (int kz = 0; kz < cnt[2]; ++kz)
            for (int ky = 0; ky < cnt[1]; ++ky)
                for (int kx = 0; kx < cnt[0]; ++kx)
                    acc += cw[0][kx] * cw[1][ky] * cw[2][kz] * xc[ci[0][kx] + C.s[1] * ci[1][ky] + C.s[2] * ci[2][kz]];
        xf[i] = (beta == (T)0 ? (T)0 : beta * xf[i]) + alpha * acc;
    }
}

// phi_i = (R y)_i - min over fine {2i-1, 2i, 2i+1}^d (clamped) of y  (Sec. V.C)
template <typename T>
__global__ void k_coarse_bound(ImgDims F, ImgDims C, const T* y, const T* Ry, const T* b, T* phi) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < C.N; i += (long long)gridDim.x * blockDim.x) {
        int c[3];
        unflat(i, C, c);
        T m = (T)INFINITY;
        const int oz = (C.d == 3) ? 1 : 0;
        for (int dz = -oz; dz <= oz; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                    const int fx = min(max(2 * c[0] + dx, 0), F.n[0] - 1);
                    const int fy = min(max(2 * c[1] + dy, 0), F.n[1] - 1);
                    const int fz = (C.d == 3) ? min(max(2 * c[2] + dz, 0), F.n[2] - 1) : 0;
                    const long long f = fx + F.s[1] * fy + F.s[2] * fz;
                    m = fmin(m, b ? y[f] - b[f] : y[f]);
                }
        phi[i] = Ry[i] - m;
    }
}

// ------------------------------------------------------------------------------------------
// vector updates: out = a x + b y (+ c w); optional lower bound
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void k_lincomb(long long n, T* out, T a, const T* x, T b, const T* y, T c, const T* w, const T* lower,
                          int nonneg) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        T v = a * x[i];
        if (y) v += b * y[i];
        if (w) v += c * w[i];
        if (lower) v = fmax(v, lower[i]);
        else if (nonneg) v = fmax(v, (T)0);
        out[i] = v;
    }
}

// decimate the data record in time: out[m] = in[2 m] (rows of Ns)
template <typename T> __global__ void k_decimate_rows(const T* in, T* out, int Ntc, int Ns) {
    const long long n = (long long)Ntc * Ns;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long m = i / Ns, j = i - m * Ns;
        out[i] = in[2 * m * Ns + j];
    }
}

// ------------------------------------------------------------------------------------------
// host-side launchers (internal API, pat_optim.h)
// ------------------------------------------------------------------------------------------
static int grid_for(long long n) {
    long long b = (n + 255) / 256;
    if (b > 4 * 152) b = 4 * 152;
    return (int)(b < 1 ? 1 : b);
}

template <typename T>
pat_status Ops<T>::reduce(int op, const pat_grid* g, long long n, const T* a, const T* b, double rho, double* out,
                          cudaStream_t s) {
    ImgDims D{};
    if (g) D = img_dims(*g);
    const int nb = grid_for(n);
    double* part = nullptr;
    cudaError_t e = cudaMallocAsync(&part, (nb + 1) * sizeof(double), s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync (reduction)");
    k_reduce<T><<<nb, 256, 0, s>>>(op, D, n, a, b, (T)rho, part);
    k_reduce_final<<<1, 32, 0, s>>>(part, nb, part + nb);
    e = cudaMemcpyAsync(out, part + nb, sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(part, s);
    if (e != cudaSuccess) return cuda_fail(e, "reduction result");
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize (reduction)");
    return PAT_OK;
}

// tile and planes per CTA of k_fgp_iter; true: the tile compiled in
template <typename T, int D> static bool fgp_tile(FgpArgs<T>& A) {
    const auto up = [](int a, int b) { return (a + b - 1) / b; };
    const int nsm = 152;
    if (sizeof(T) == 4 && A.nx > 32) {
        A.tw = kFgpX;
        A.th = kFgpY;
        A.gx = up(A.nx, A.tw);
        A.gy = up(A.ny, A.th);
        // a CTA reads one plane more than it writes, so long chunks save traffic as long as about four
        // rounds of 4 CTAs per SM remain (13 planes at 256^3); at least 3 planes, or 2 where 3 would leave two
        // CTAs per SM or less (128^3: 633 us with 3, 671 with 4, 708 with 2; 64^3: 270, 294, 247)
        const long long planes = (long long)A.gx * A.gy * A.nz;
        A.chunk = (int)std::max<long long>(planes < 6 * nsm ? 2 : 3, std::min<long long>(64, planes / (16 * nsm)));
        return true;
    }
    // planes: the plane that is read but not written is dear where there are few (100^3 double: 2390 us with
    // 4, 2560 with 2), CTAs are where the image is small (50 x 60 x 30: 460 us with 1, 740 with 2)
    const double load = (double)A.nx * A.ny * A.nz / (nsm * 1024);   // points per SM, in 1024
    A.chunk = D == 3 ? std::max(1, std::min({16, A.nz, (int)(load + 0.5), std::max(2, (int)(load / 2 + 0.5))})) : 1;
    // sides: warps of the main tile count three times (x(r) and the update), those of its halo once, times the
    // rounds of CTAs over the SMs.  Of all sides tried at 17 images in double this choice is on average 5 %
    // slower than the best one, at most 20 % (40^3)
    long long best = -1;
    for (int tw : {up(A.nx, up(A.nx, 64)), std::min(A.nx, 32)})
        for (int th = std::min({A.ny, kFgpRows, kFgpThreads / tw}); th >= 1 && (tw * th >= 64 || best < 0); --th) {
            const int main = up(tw * th, 32), halo = up(tw + th, 32);   // warps
            const long long n = (long long)up(A.nx, tw) * up(A.ny, th) * up(A.nz, A.chunk);
            const long long cost = (n + nsm - 1) / nsm * (A.chunk * (3 * main + halo) + (D == 3 ? main : 0));
            if (best >= 0 && cost >= best) continue;
            best = cost;
            A.tw = tw;
            A.th = th;
        }
    A.gx = up(A.nx, A.tw);
    A.gy = up(A.ny, A.th);
    return false;
}

// the FGP loop: three rotating dual fields; every launch may start (programmatic dependent launch) while
// its predecessor drains
template <typename T, int D>
static pat_status fgp(const ImgDims& M, const T* z, T* x, double lam, int n_inner, int nonneg, cudaStream_t s) {
    T* buf = nullptr;
    const size_t N = (size_t)M.N;
    cudaError_t e = cudaMallocAsync(&buf, (size_t)3 * D * N * sizeof(T), s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync (TV prox)");
    FgpArgs<T> A{};
    A.nx = M.n[0];
    A.ny = M.n[1];
    A.nz = M.n[2];
    A.z = z;
    A.lam = (T)lam;
    A.step = (T)(1.0 / (4.0 * D * lam));
    A.nonneg = nonneg;
    const bool fixed = fgp_tile<T, D>(A);
    const unsigned gz = (D == 3) ? (A.nz + A.chunk - 1) / A.chunk : 1;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.stream = s;
    lc.attrs = attr;
    auto field = [&](int k, int a) { return buf + (size_t)(k * D + a) * N; };
    double t = 1.0, w = 0.0;   // the first iteration starts from r = q = 0
    for (int it = 0; it < n_inner && e == cudaSuccess; ++it) {
        for (int a = 0; a < D; ++a) {
            A.q[a] = field(it % 3, a);
            A.qp[a] = field((it + 2) % 3, a);
            A.qn[a] = field((it + 1) % 3, a);
        }
        A.first = it == 0;
        // after the first iteration q_0 = 0 and its extrapolation weight is (t_0 - 1) / t_1 = 0
        if (it == 1)
            for (int a = 0; a < D; ++a) A.qp[a] = A.q[a];
        A.w = (T)w;
        lc.gridDim = dim3(A.gx * A.gy * gz);
        lc.blockDim = dim3((std::max(A.tw * A.th, A.tw + A.th) + 31) / 32 * 32);   // a thread per halo point as well
        lc.numAttrs = it == 0 ? 0 : 1;   // the first launch follows the allocation and the caller's work
        e = fixed ? cudaLaunchKernelEx(&lc, k_fgp_iter<T, D, true>, A) : cudaLaunchKernelEx(&lc, k_fgp_iter<T, D, false>, A);
        const double tn = 0.5 * (1.0 + std::sqrt(1.0 + 4.0 * t * t));
        w = (t - 1.0) / tn;
        t = tn;
    }
    if (e == cudaSuccess) {
        for (int a = 0; a < D; ++a) A.q[a] = field(n_inner % 3, a);
        A.tw = std::min(A.nx, 64);
        A.th = std::min(A.ny, 256 / A.tw);
        A.gx = (A.nx + A.tw - 1) / A.tw;
        A.gy = (A.ny + A.th - 1) / A.th;
        lc.gridDim = dim3(A.gx * A.gy * (D == 3 ? A.nz : 1));
        lc.blockDim = dim3((A.tw * A.th + 31) / 32 * 32);
        lc.numAttrs = 1;
        e = cudaLaunchKernelEx(&lc, k_fgp_final<T, D>, A, x);
    }
    cudaFreeAsync(buf, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "TV prox kernels");
    return PAT_OK;
}

template <typename T>
pat_status Ops<T>::tv_prox(const pat_grid* g, const T* z, T* x, double lam, int n_inner, int nonneg, cudaStream_t s) {
    const ImgDims D = img_dims(*g);
    const int nb = grid_for(D.N);
    if (!(lam > 0.0) || n_inner <= 0) {
        k_lincomb<T><<<nb, 256, 0, s>>>(D.N, x, (T)1, z, (T)0, nullptr, (T)0, nullptr, nullptr, nonneg);
        return PAT_OK;
    }
    return D.d == 2 ? fgp<T, 2>(D, z, x, lam, n_inner, nonneg, s) : fgp<T, 3>(D, z, x, lam, n_inner, nonneg, s);
}

template <typename T>
pat_status Ops<T>::tv_smooth_grad(const pat_grid* g, const T* y, double rho, T* out, double alpha, double beta,
                                  cudaStream_t s) {
    const ImgDims D = img_dims(*g);
    k_tv_smooth_grad<T><<<grid_for(D.N), 256, 0, s>>>(D, y, (T)rho, out, (T)alpha, (T)beta);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "smoothed TV gradient");
}

static pat_grid coarse_of(const pat_grid& f) {
    pat_grid c = f;
    for (int a = 0; a < f.ndim; ++a) c.n[a] = f.n[a] / 2;
    return c;
}

template <typename T> pat_status Ops<T>::restrict_(const pat_grid* fine, const T* xf, T* xc, cudaStream_t s) {
    const ImgDims F = img_dims(*fine), C = img_dims(coarse_of(*fine));
    k_restrict<T><<<grid_for(C.N), 256, 0, s>>>(F, C, xf, xc);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "restriction");
}

template <typename T>
pat_status Ops<T>::prolong(const pat_grid* fine, const T* xc, T* xf, double alpha, double beta, cudaStream_t s) {
    const ImgDims F = img_dims(*fine), C = img_dims(coarse_of(*fine));
    k_prolong<T><<<grid_for(F.N), 256, 0, s>>>(F, C, xc, xf, (T)alpha, (T)beta);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "prolongation");
}

template <typename T>
pat_status Ops<T>::coarse_bound(const pat_grid* fine, const T* y, T* phi, T* tmp, cudaStream_t s, const T* b) {
    const ImgDims F = img_dims(*fine), C = img_dims(coarse_of(*fine));
    k_restrict<T><<<grid_for(C.N), 256, 0, s>>>(F, C, y, tmp);
    k_coarse_bound<T><<<grid_for(C.N), 256, 0, s>>>(F, C, y, tmp, b, phi);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "coarse bound");
}

template <typename T>
pat_status Ops<T>::lincomb(long long n, T* out, double a, const T* x, double b, const T* y, double c, const T* w,
                           const T* lower, int nonneg, cudaStream_t s) {
    k_lincomb<T><<<grid_for(n), 256, 0, s>>>(n, out, (T)a, x, (T)b, y, (T)c, w, lower, nonneg);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "vector update");
}

template <typename T> pat_status Ops<T>::decimate_rows(const T* in, T* out, int Ntc, int Ns, cudaStream_t s) {
    k_decimate_rows<T><<<grid_for((long long)Ntc * Ns), 256, 0, s>>>(in, out, Ntc, Ns);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "data decimation");
}

template struct Ops<float>;
template struct Ops<double>;

static pat_status check_img_grid(const pat_grid* g) {
    if (!g || (g->ndim != 2 && g->ndim != 3)) {
        set_error("bad grid");
        return PAT_EINVAL;
    }
    for (int a = 0; a < g->ndim; ++a)
        if (g->n[a] < 1) {
            set_error("bad grid size");
            return PAT_EINVAL;
        }
    return PAT_OK;
}

static long long img_count(const pat_grid* g) {
    long long n = 1;
    for (int a = 0; a < g->ndim; ++a) n *= g->n[a];
    return n;
}

}  // namespace pat

using namespace pat;

extern "C" {

pat_status pat_tv_prox(const pat_grid* grid, const void* z, void* x, double weight, int n_inner, int nonneg,
                       pat_precision prec, void* stream) {
    set_error("");
    pat_status st = check_img_grid(grid);
    if (st != PAT_OK) return st;
    if (!z || !x || n_inner < 0) {
        set_error("bad arguments");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PAT_F32) return Ops<float>::tv_prox(grid, (const float*)z, (float*)x, weight, n_inner, nonneg, s);
    return Ops<double>::tv_prox(grid, (const double*)z, (double*)x, weight, n_inner, nonneg, s);
}

pat_status pat_tv(const pat_grid* grid, const void* x, double rho, double* value, pat_precision prec, void* stream) {
    set_error("");
    pat_status st = check_img_grid(grid);
    if (st != PAT_OK) return st;
    if (!x || !value) {
        set_error("bad arguments");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int op = (rho > 0.0) ? RED_TVS : RED_TV;
    if (prec == PAT_F32) return Ops<float>::reduce(op, grid, img_count(grid), (const float*)x, nullptr, rho, value, s);
    return Ops<double>::reduce(op, grid, img_count(grid), (const double*)x, nullptr, rho, value, s);
}

pat_status pat_tv_smooth_grad(const pat_grid* grid, const void* y, double rho, void* grad, pat_precision prec,
                              void* stream) {
    set_error("");
    pat_status st = check_img_grid(grid);
    if (st != PAT_OK) return st;
    if (!y || !grad || !(rho > 0.0)) {
        set_error("bad arguments");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PAT_F32) return Ops<float>::tv_smooth_grad(grid, (const float*)y, rho, (float*)grad, 1.0, 0.0, s);
    return Ops<double>::tv_smooth_grad(grid, (const double*)y, rho, (double*)grad, 1.0, 0.0, s);
}

static pat_status check_even(const pat_grid* g) {
    for (int a = 0; a < g->ndim; ++a)
        if (g->n[a] < 2 || (g->n[a] & 1)) {
            set_error("fine grid sizes must be even");
            return PAT_EINVAL;
        }
    return PAT_OK;
}

pat_status pat_restrict(const pat_grid* fine, const void* xf, void* xc, pat_precision prec, void* stream) {
    set_error("");
    pat_status st = check_img_grid(fine);
    if (st == PAT_OK) st = check_even(fine);
    if (st != PAT_OK) return st;
    if (!xf || !xc) {
        set_error("NULL argument");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PAT_F32) return Ops<float>::restrict_(fine, (const float*)xf, (float*)xc, s);
    return Ops<double>::restrict_(fine, (const double*)xf, (double*)xc, s);
}

pat_status pat_prolong(const pat_grid* fine, const void* xc, void* xf, pat_precision prec, void* stream) {
    set_error("");
    pat_status st = check_img_grid(fine);
    if (st == PAT_OK) st = check_even(fine);
    if (st != PAT_OK) return st;
    if (!xf || !xc) {
        set_error("NULL argument");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PAT_F32) return Ops<float>::prolong(fine, (const float*)xc, (float*)xf, 1.0, 0.0, s);
    return Ops<double>::prolong(fine, (const double*)xc, (double*)xf, 1.0, 0.0, s);
}

pat_status pat_coarse_bound(const pat_grid* fine, const void* y, void* phi, pat_precision prec, void* stream) {
    set_error("");
    pat_status st = check_img_grid(fine);
    if (st == PAT_OK) st = check_even(fine);
    if (st != PAT_OK) return st;
    if (!y || !phi) {
        set_error("NULL argument");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const long long nc = img_count(fine) >> fine->ndim;
    const size_t eb = (prec == PAT_F32) ? 4 : 8;
    void* tmp = nullptr;
    cudaError_t e = cudaMallocAsync(&tmp, nc * eb, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync (bound)");
    if (prec == PAT_F32) st = Ops<float>::coarse_bound(fine, (const float*)y, (float*)phi, (float*)tmp, s);
    else st = Ops<double>::coarse_bound(fine, (const double*)y, (double*)phi, (double*)tmp, s);
    cudaFreeAsync(tmp, s);
    return st;
}

pat_status pat_dot(const void* a, const void* b, int64_t n, pat_precision prec, double* out, void* stream) {
    set_error("");
    if (!a || !b || !out || n < 0) {
        set_error("bad arguments");
        return PAT_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PAT_F32) return Ops<float>::reduce(RED_DOT, nullptr, n, (const float*)a, (const float*)b, 0.0, out, s);
    return Ops<double>::reduce(RED_DOT, nullptr, n, (const double*)a, (const double*)b, 0.0, out, s);
}

}  // extern "C"
