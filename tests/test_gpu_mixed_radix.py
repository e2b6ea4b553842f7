"""The mixed-radix kernels on line lengths that cover every radix of every stage (first 2 4 6 8 10, last
2 .. 10, middle up to 16 in FP32), two and three stages, odd and even numbers of last-stage butterflies,
short and long lines, against the FP64 oracle: H and H^T in 2-D and 3-D, FP32 and FP64, absorbing and
lossless.  Tolerances are the library's parity bounds, relative L2 1e-5 (FP32) and 1e-11 (FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu

# (ny, nx): 12 = 4.3 or 6.2, 14 = 2.7, 18 = 2.9 or 6.3, 20 = 4.5 ..., 42 = 6.7, 50 = 10.5, 98 = 2.7.7,
# 126 = 2.9.7 ..., 150, 200, 250 = 10.5.5, 270, 350 = 10.5.7, 490 = 10.7.7, 750 = 10.15.5, 784 = 8.14.7, 840
SHAPES_2D = [(12, 14), (14, 18), (18, 12), (20, 42), (42, 20), (50, 98), (98, 50), (126, 24), (24, 126), (150, 20),
             (20, 200), (250, 16), (16, 270), (350, 12), (12, 490), (750, 10), (10, 750), (784, 10), (10, 840)]
SHAPES_3D = [(12, 14, 18), (18, 20, 12), (14, 12, 50), (10, 98, 12), (98, 10, 12), (16, 20, 126), (20, 16, 64)]


def _check(pb, prec):
    from paper_1603_02329_gb300.api import PATOperator

    ref = Operator.from_problem(pb)
    h = np.random.default_rng(3).standard_normal((pb.Nt, ref.Ns))
    d_ref, g_ref = ref.forward(pb.p0), ref.adjoint(h)
    op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
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
    monkeypatch.setenv("PAT_PERSIST", persist)
    lossless = shape[0] == 98 or shape[1] == 12
    _check(synth.small_lossy_2d(shape=shape, pml=2, Nt=25, n_sensors=7, alpha0=0.0 if lossless else 0.75,
                                sensor_radius_frac=0.25), prec)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES_3D, ids=lambda s: "x".join(map(str, s)))
def test_3d(shape, prec):
    _check(synth.small_lossy_3d(shape=shape, pml=2, Nt=15, alpha0=0.0 if shape[0] == 98 else 0.75), prec)


@pytest.mark.parametrize("lines,width", [(2, 1), (4, 8), (16, 16)])
def test_layouts(monkeypatch, lines, width):
    monkeypatch.setenv("PAT_ROW_LINES", str(lines))
    monkeypatch.setenv("PAT_COL_W", str(width))
    monkeypatch.setenv("PAT_PERSIST", "0")
    _check(synth.small_lossy_2d(shape=(48, 90), pml=3, Nt=25, n_sensors=7, sensor_radius_frac=0.25), "f32")
    _check(synth.small_lossy_3d(shape=(12, 24, 36), pml=2, Nt=15), "f32")
