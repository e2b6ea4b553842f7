"""The mixed-radix kernels on line lengths taken from the schedules themselves, so that every radix a
schedule holds (first 2 4 6 8 10, middle 3 .. 10 and in FP32 12 14 15 16, last 2 .. 10) runs along x and
along y, in the per-phase kernels and in the persistent kernel, FP32 and FP64, against the FP64 oracle
(test_mixed_radix_schedule.py asserts that the lists are complete).  Tolerances are the library's parity
bounds, relative L2 1e-5 (FP32) and 1e-11 (FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu

# the last radices 2 6 8 9 10, the middle ones 3 4 6 8 9 10 12 14 16, lines of 1024 points (FP32)
LINES = (4, 8, 36, 54, 64, 72, 80, 96, 100, 108, 128, 160, 162, 240, 252, 300, 486, 512, 672, 784, 1000, 1024)
SHAPES_2D = [(n, 10) for n in LINES] + [(10, n) for n in LINES]
SHAPES_3D = [(8, 36, 54), (36, 54, 8), (54, 8, 36), (100, 10, 8), (8, 100, 10), (10, 8, 100), (108, 6, 12), (6, 108, 12),
             (12, 6, 108), (6, 6, 240), (6, 240, 6), (240, 6, 6), (6, 300, 6), (300, 6, 6), (6, 6, 300)]
F64_NONE = (672, 784, 1024)   # no schedule in double
F64_X_MAX = 810                 # longer x lines in double: refused, the initial state's rows do not fit on chip
F64_PER_PHASE = ((1000, 10),)   # four line pairs per CTA and more: the columns' buffers do not fit on chip


def _check(pb, prec, path=None):
    from paper_1603_02329_gb300.api import PATOperator

    ref = Operator.from_problem(pb)
    h = np.random.default_rng(3).standard_normal((pb.Nt, ref.Ns))
    d_ref, g_ref = ref.forward(pb.p0), ref.adjoint(h)
    op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
    assert path is None or op.info.path == path
    dt, tol = (torch.float32, 1e-5) if prec == "f32" else (torch.float64, 1e-11)
    d = op.forward(torch.tensor(pb.p0, dtype=dt, device="cuda")).cpu().numpy()
    g = op.adjoint(torch.tensor(h, dtype=dt, device="cuda")).cpu().numpy()
    op.close()
    assert np.linalg.norm(d - d_ref) <= tol * np.linalg.norm(d_ref)
    assert np.linalg.norm(g - g_ref) <= tol * np.linalg.norm(g_ref)


@pytest.mark.parametrize("persist", ["0", "1"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES_2D, ids=lambda s: "x".join(map(str, s)))
def test_2d(monkeypatch, shape, prec, persist):
    if prec == "f64" and (max(shape) in F64_NONE or shape[1] > F64_X_MAX):
        pytest.skip("no double plan, or none with a mixed-radix schedule")
    monkeypatch.setenv("PAT_PERSIST", persist)
    monkeypatch.setenv("PAT_MX", "2")   # lengths that are a power of two as well
    alpha0 = 0.0 if shape[1] in (36, 128) else 0.75
    _check(synth.small_lossy_2d(shape=shape, pml=1, Nt=21, n_sensors=5, alpha0=alpha0, sensor_radius_frac=0.2), prec,
           0 if prec == "f64" and shape in F64_PER_PHASE else int(persist))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES_3D, ids=lambda s: "x".join(map(str, s)))
def test_3d(monkeypatch, shape, prec):
    monkeypatch.setenv("PAT_MX", "2")
    monkeypatch.setenv("PAT_AUTOTUNE", "0")
    _check(synth.small_lossy_3d(shape=shape, pml=1, Nt=12, alpha0=0.0 if shape[2] == 36 else 0.75), prec)
