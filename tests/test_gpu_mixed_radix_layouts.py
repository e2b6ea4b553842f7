"""Plans and launch layouts of the mixed-radix per-phase kernels where shared memory decides: long x lines in
double 3-D (512 points: 4 x-lines per CTA are the most that fit), tuned and untuned; and every pinned width
and line count, up to the tuner's widest.  Against the FP64 oracle; tolerances are the library's parity
bounds, relative L2 1e-5 (FP32) and 1e-11 (FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(pb, prec, layout=None):
    from paper_1603_02329_gb300.api import PATOperator

    ref = Operator.from_problem(pb)
    h = np.random.default_rng(3).standard_normal((pb.Nt, ref.Ns))
    op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
    assert layout is None or (op.info.layout[0], op.info.layout[1]) == layout
    dt, tol = (torch.float32, 1e-5) if prec == "f32" else (torch.float64, 1e-11)
    d = op.forward(torch.tensor(pb.p0, dtype=dt, device="cuda")).cpu().numpy()
    g = op.adjoint(torch.tensor(h, dtype=dt, device="cuda")).cpu().numpy()
    op.close()
    d_ref, g_ref = ref.forward(pb.p0), ref.adjoint(h)
    assert np.linalg.norm(d - d_ref) <= tol * np.linalg.norm(d_ref)
    assert np.linalg.norm(g - g_ref) <= tol * np.linalg.norm(g_ref)


@pytest.mark.parametrize("tune", ["1", "0"])
@pytest.mark.parametrize("shape", [(16, 16, 512), (8, 12, 512), (6, 10, 256)], ids=lambda s: "x".join(map(str, s)))
def test_double_3d_long_x_lines(monkeypatch, shape, tune):
    monkeypatch.setenv("PAT_AUTOTUNE", tune)
    _check(synth.small_lossy_3d(shape=shape, pml=2, Nt=12), "f64")


@pytest.mark.parametrize("tune", ["1", "0"])
@pytest.mark.parametrize("prec,width,lines", [("f32", 1, 2), ("f32", 2, 4), ("f32", 4, 8), ("f32", 8, 16), ("f32", 16, 16),
                                              ("f64", 1, 2), ("f64", 2, 4), ("f64", 4, 8), ("f64", 8, 8)])
def test_pinned_layouts(monkeypatch, prec, width, lines, tune):
    for k, v in (("PAT_COL_W", width), ("PAT_ROW_LINES", lines), ("PAT_PERSIST", 0), ("PAT_AUTOTUNE", tune)):
        monkeypatch.setenv(k, str(v))
    _check(synth.small_lossy_2d(shape=(48, 54), pml=3, Nt=25, n_sensors=7, sensor_radius_frac=0.25), prec, (width, lines))
    _check(synth.small_lossy_3d(shape=(12, 24, 36), pml=2, Nt=15), prec, (width, lines))
