"""The checkpointed medium gradients where the recomputed forward and the adjoint share the plan's spectra:
128-point y and z lines (FP32: the 16-column passes with tensor copies), absorbing (two spectra put aside
per segment) and lossless (three), and lossless 3-D in FP64, one to several segments, against the FP64
oracle.  Tolerances as for the other medium gradients: 1e-5 (FP32), 1e-10 (FP64) relative L2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import pat_medium as pm  # noqa: E402
from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


def _check(pb, prec, Ks, wide):
    from paper_1603_02329_gb300.api import PATOperator

    ref = Operator.from_problem(pb)
    h = np.random.default_rng(43).standard_normal((pb.Nt, ref.Ns))
    gc_ref, gp_ref = pm.sound_speed_gradient(ref, pb.p0, h, pb.y)
    gr_ref = pm.density_gradient(ref, pb.p0, h)
    dt, tol = (torch.float32, 1e-5) if prec == "f32" else (torch.float64, 1e-10)
    op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
    assert op.info.ywide == op.info.zwide == int(wide)
    x, res = torch.tensor(pb.p0, dtype=dt, device="cuda"), torch.tensor(h, dtype=dt, device="cuda")
    first = None
    for K in Ks:
        out = op.gradient_medium(x, res, checkpoint_every=K)
        for got, want in zip(out, (gr_ref, gc_ref, gp_ref)):
            assert _rel(got, want) <= tol, K
        first = first or out
        assert all(torch.equal(a, b) for a, b in zip(out, first))   # independent of the interval
    op.close()


@pytest.mark.parametrize("alpha0", [0.75, 0.0], ids=["lossy", "lossless"])
def test_wide_passes(monkeypatch, alpha0):
    monkeypatch.setenv("PAT_AUTOTUNE", "0")   # one chunk, the two-stage plain transforms: the wide passes run
    _check(synth.small_lossy_3d(shape=(128, 128, 16), pml=4, Nt=10, alpha0=alpha0, stride=4), "f32", (3, 9), True)


def test_lossless_3d_f64():
    _check(synth.small_lossy_3d(shape=(12, 16, 20), pml=3, Nt=17, alpha0=0.0), "f64", (5, 1, 16), False)
