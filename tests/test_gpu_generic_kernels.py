"""The generic kernels (one shared-memory pass per radix) and, in 2-D, the register-fused per-phase ones
behind PAT_MX=0, and the line lengths that have no mixed-radix schedule (2, 686, 882, 972; in double also
588 and others): H and H^T against the FP64 oracle.  Tolerances are the library's parity bounds, relative
L2 1e-5 (FP32) and 1e-11 (FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("alpha0", [0.75, 0.0], ids=["lossy", "lossless"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("fused", ["1", "0"])
@pytest.mark.parametrize("persist", ["1", "0"])
@pytest.mark.parametrize("shape", [(32, 64), (64, 16), (48, 90), (20, 42), (16, 128, 32), (32, 16, 64), (12, 20, 18)],
                         ids=lambda s: "x".join(map(str, s)))
def test_without_the_mixed_radix_kernels(monkeypatch, shape, persist, fused, prec, alpha0):
    if len(shape) == 3 and persist == "1":
        pytest.skip("3-D plans have no persistent kernel")
    monkeypatch.setenv("PAT_MX", "0")
    monkeypatch.setenv("PAT_PERSIST", persist)
    for k in ("PAT_P2", "PAT_ROW2", "PAT_SPEC2"):
        monkeypatch.setenv(k, fused)
    if len(shape) == 2:
        _check(synth.small_lossy_2d(shape=shape, pml=2, Nt=25, n_sensors=7, alpha0=alpha0, sensor_radius_frac=0.25), prec)
    else:
        _check(synth.small_lossy_3d(shape=shape, pml=2, Nt=14, alpha0=alpha0), prec)


@pytest.mark.parametrize("prec,n", [("f32", 686), ("f32", 882), ("f32", 972), ("f64", 686), ("f64", 588), ("f64", 768)])
@pytest.mark.parametrize("along_x", [True, False])
def test_lengths_without_a_schedule(prec, n, along_x):
    _check(synth.small_lossy_2d(shape=(12, n) if along_x else (n, 12), pml=2, Nt=15, n_sensors=7,
                                sensor_radius_frac=0.25), prec)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_two_point_axis(prec):
    _check(synth.small_lossy_3d(shape=(2, 12, 14), pml=1, Nt=12), prec)
