"""The mixed-radix schedules of every line length, on the CPU: a small program compiled from pat_mx.h prints
each axis (radices, slots, multipliers) and its twiddle table, and numpy runs the stages by them, with the
kernels' slots, pairings and divisions.  Tolerance: a transform of up to 1024 points in double with
products of table values, 1e-12 of the largest input."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")

# (largest middle radix, stage cost): per-phase FP32, persistent FP32, both in double
KINDS = ((16, 0), (16, 8), (10, 4))
NO_SCHEDULE = {16: {2, 686, 882, 972},
               10: {2, 588, 672, 686, 750, 756, 768, 784, 840, 864, 882, 896, 960, 972, 980, 1008, 1024}}
FIELDS = ("n", "R0", "R1", "RL", "m0", "M", "P0", "LS", "dn", "dm0", "dM", "dR0", "dRL", "dB", "dU")

SRC = r"""
#include <cmath>
#include <cstdio>
#include "pat_mx.h"
int main() {
    const int kinds[3][2] = {{16, 0}, {16, 8}, {10, 4}};
    for (auto& k : kinds)
        for (int n = 2; n <= 1024; n += 2) {
            pat::MxAxis a{};
            if (!pat::mx_axis(n, k[0], k[1], &a)) continue;
            std::vector<std::complex<double>> tw(n);
            for (int m = 0; m < n; ++m) tw[m] = std::polar(1.0, -2.0 * M_PI * m / n);
            const auto t = pat::mx_table(tw, a);
            std::printf("%d %d %d %d %d %d %d %d %d %d %u %u %u %u %u %u %u", k[0], k[1], a.n, a.R0, a.R1, a.RL, a.m0, a.M, a.P0,
                        a.LS, a.dn, a.dm0, a.dM, a.dR0, a.dRL, a.dB, a.dU);
            for (auto v : t) std::printf(" %.17g %.17g", v.real(), v.imag());
            std::printf("\n");
        }
}
"""


def _smooth(n):
    for f in (2, 3, 5, 7):
        while n % f == 0:
            n //= f
    return n == 1


@pytest.fixture(scope="module")
def axes(tmp_path_factory):
    d = tmp_path_factory.mktemp("mx")
    (d / "dump.cu").write_text(SRC)
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1603_02329_gb300", "csrc"), "-o",
                    str(d / "dump"), str(d / "dump.cu")], check=True, capture_output=True)
    out = {}
    for line in subprocess.run([str(d / "dump")], check=True, capture_output=True, text=True).stdout.splitlines():
        w = line.split()
        v = np.array(w[17:], dtype=float)
        x = dict(zip(FIELDS, map(int, w[2:17])), table=v[::2] + 1j * v[1::2])
        out.setdefault((int(w[0]), int(w[1])), {})[x["n"]] = x
    return out


def _base(x, q):
    return x["P0"] * q if x["R1"] == 1 else x["P0"] * (q % x["R0"]) + x["RL"] * (q // x["R0"])


def _forward(x, v):
    R0, R1, RL, m0, M, P0 = (x[k] for k in ("R0", "R1", "RL", "m0", "M", "P0"))
    tab_l = x["table"][:(RL - 1) * M].reshape(RL - 1, M)
    buf = np.full(x["LS"], np.nan, complex)
    slots = np.array([[P0 * r + j for r in range(R0)] for j in range(m0)])
    assert slots.max() < x["LS"] and np.unique(slots).size == x["n"]
    buf[slots] = np.fft.fft(v[np.array([[j + m0 * r for r in range(R0)] for j in range(m0)])], axis=1)
    if R1 > 1:
        tab_1 = x["table"][(RL - 1) * M:].reshape(R1, R0 * RL)
        mid = np.array([[P0 * (b // RL) + b % RL + RL * r for r in range(R1)] for b in range(R0 * RL)])
        assert set(mid.ravel()) == set(slots.ravel())
        buf[mid] = np.fft.fft(buf[mid] * tab_1.T, axis=1)
    last = np.array([[_base(x, q) + r for r in range(RL)] for q in range(M)])
    assert set(last.ravel()) == set(slots.ravel())
    t = np.vstack([np.ones(M), tab_l]).T
    out = np.empty(x["n"], complex)
    out[np.array([[q + M * r for r in range(RL)] for q in range(M)])] = np.fft.fft(buf[last] * t, axis=1)
    return out


def test_every_length_has_its_schedule_and_transforms(axes):
    rng = np.random.default_rng(1)
    for kind in KINDS:
        have = axes[kind]
        lengths = {n for n in range(2, 1025, 2) if _smooth(n)}
        assert lengths - set(have) == NO_SCHEDULE[kind[0]]
        for n, x in have.items():
            assert x["R0"] * x["R1"] * x["RL"] == n and x["R0"] % 2 == 0 and x["LS"] % 2 == 0
            assert x["m0"] == n // x["R0"] and x["M"] == n // x["RL"]
            v = rng.standard_normal(n) + 1j * rng.standard_normal(n)
            assert np.abs(_forward(x, v) - np.fft.fft(v)).max() <= 1e-12 * np.abs(v).max() * n ** 0.5


def test_divisions_by_multiplier(axes):
    # every divisor of every schedule, over the range of numerators the kernels form (below 2^16)
    t = np.arange(1 << 16, dtype=np.uint64)
    pairs = set()
    for have in axes.values():
        for x in have.values():
            pairs |= {(x["n"], x["dn"]), (x["m0"], x["dm0"]), (x["M"], x["dM"]), (x["R0"], x["dR0"]), (x["RL"], x["dRL"]),
                      (x["R0"] * x["RL"], x["dB"]), ((x["M"] + 1) // 2, x["dU"])}
    for d, magic in pairs:
        q = (t * np.uint64(magic)) >> np.uint64(32) if magic else t
        assert (q == t // np.uint64(d)).all()


# (last radix RL, butterflies M): every pair that a schedule has
def _pairs(axes):
    return sorted({(x["RL"], x["M"]) for have in axes.values() for x in have.values()})


def test_lane_pair_unpacking_covers_the_half_spectrum(axes):
    # mx_row_out: lanes 2 u, 2 u + 1 run butterflies u and M - u, each stores half of the pairs (k, n - k)
    for R, M in _pairs(axes):
        n, half, J = M * R, M * R // 2, (R - 1) // 2
        cnt = np.zeros(half + 1, int)
        for u in range((M + 1) // 2):
            u0 = u == 0
            qs = [u, (M >> 1) if u0 else M - u]
            v = [[qs[h] + M * r for r in range(R)] for h in (0, 1)]
            for h in (0, 1):
                ok = not (u0 and h and M & 1)
                src = v[h] if u0 else v[1 - h]
                puts = []
                for j in range(J + 1):
                    zm = v[0][(R - j) % R] if u0 and not h else src[R - 1 - j]
                    if ok and not (R % 2 == 1 and j == J and h and not u0):
                        puts.append((qs[h] + M * j, v[h][j], zm))
                if R % 2 == 0 and ok and u0 and not h:
                    puts.append((half, v[0][R // 2], v[0][R // 2]))
                for k, zk, zm in puts:
                    assert k < n and zk == k and (zk + zm) % n == 0
                    cnt[n - k if k > half else k] += 1
        assert (cnt == 1).all(), (R, M)


def test_two_butterfly_units_pack_and_unpack(axes):
    # pmx_row_in_units / pmx_row_out_units: unit u holds butterflies u and M - u, unit 0 butterflies 0 and M / 2
    rng = np.random.default_rng(2)
    for R, M in _pairs(axes):
        n, half, H, E = M * R, M * R // 2, R // 2, (R - 1) // 2
        A, B = (rng.standard_normal(half + 1) + 1j * rng.standard_normal(half + 1) for _ in range(2))
        A[[0, half]], B[[0, half]] = A[[0, half]].real, B[[0, half]].real
        Z = np.array([A[k] + 1j * B[k] if k <= half else np.conj(A[n - k]) + 1j * np.conj(B[n - k]) for k in range(n)])
        got = np.full(n, np.nan, complex)
        for u in range((M + 1) // 2):
            u0, q2 = u == 0, (M >> 1 if u == 0 else M - u)
            v1, v2 = [None] * R, [None] * R
            for r in range(R):
                k = (M * r if r <= H else (M >> 1) + M * (R - 1 - r)) if u0 else u + M * r
                kk = k if k <= half else n - k
                assert 0 <= kk <= half
                a, b = (np.conj(A[kk]), np.conj(B[kk])) if not u0 and k > half else (A[kk], B[kk])
                if u0 and (r == 0 or (R % 2 == 0 and r == H)):
                    a, b = a.real, b.real
                v1[r], v2[R - 1 - r] = a + 1j * b, np.conj(a) + 1j * np.conj(b)
            w1, w2 = list(v1), list(v2)
            if u0:
                kk = (M >> 1) + M * E
                assert kk <= half
                a, b = (A[kk].real, B[kk].real) if R % 2 else (A[kk], B[kk])
                for r in range(R):
                    w1[r] = v1[r] if r <= H else v2[r - 1]
                    w2[r] = (v1[R - 1 - r] if r < R - 1 - H else a + 1j * b if r == E else
                             np.conj(a) + 1j * np.conj(b) if r == R - 1 - E else v2[R - 1 - r])
            for r in range(R):
                got[u + M * r] = w1[r]
                if not u0 or M % 2 == 0:
                    got[q2 + M * r] = w2[r]
        assert np.allclose(got, Z), (R, M)
        cnt, OA, OB = np.zeros(half + 1, int), np.full(half + 1, np.nan, complex), np.full(half + 1, np.nan, complex)

        def put(k, zk, zm):
            up = k > half
            kk = n - k if up else k
            cnt[kk] += 1
            OA[kk] = complex(zk.real + zm.real, (zm.imag - zk.imag) if up else (zk.imag - zm.imag)) / 2
            OB[kk] = complex(zk.imag + zm.imag, (zk.real - zm.real) if up else (zm.real - zk.real)) / 2

        for u in range((M + 1) // 2):
            u0, q2, two = u == 0, (M >> 1 if u == 0 else M - u), M % 2 == 0
            v1, v2 = [Z[u + M * r] for r in range(R)], [Z[(q2 + M * r) % n] for r in range(R)]
            for r in range(R):
                if r <= H:
                    put(u + M * r, v1[r], v1[(R - r) % R] if u0 else v2[R - 1 - r])
                elif not u0 or two:
                    put((M >> 1) + M * (R - 1 - r) if u0 else u + M * r, v2[R - 1 - r] if u0 else v1[r],
                        v2[r] if u0 else v2[R - 1 - r])
            if u0 and two:
                put((M >> 1) + M * E, v2[E], v2[R - 1 - E])
        assert (cnt == 1).all() and np.allclose(OA, A) and np.allclose(OB, B), (R, M)


def test_gpu_parity_lists_hold_every_radix(axes):
    pytest.importorskip("torch")
    import test_gpu_mixed_radix as a
    import test_gpu_mixed_radix_stages as b

    for kind in KINDS:
        have = axes[kind]
        for axis in (0, 1):   # y, x
            # a double plan's x lines stop at F64_X_MAX, and its persistent kernel's y lines below 1000
            top = 1024 if kind[0] == 16 else (1000, b.F64_X_MAX)[axis]
            every = {(s, x[s]) for n, x in have.items() if n <= top for s in ("R0", "R1", "RL")}
            got = set()
            for shape in a.SHAPES_2D + b.SHAPES_2D:
                if all(n in have for n in shape) and shape[axis] <= top:
                    got |= {(s, have[shape[axis]][s]) for s in ("R0", "R1", "RL")}
            assert got == every, (kind, axis, every - got)
    assert [n for n, x in axes[(10, 4)].items() if x["RL"] == 10] == [1000] and b.F64_PER_PHASE == ((1000, 10),)
