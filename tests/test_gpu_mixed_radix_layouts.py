"""Plans and launch layouts of the mixed-radix per-phase kernels where shared memory decides: long x lines in
double 3-D (512 points: 4 x-lines per CTA are the most that fit), tuned and untuned, against the FP64 oracle.
Tolerance: the library's parity bound, relative L2 1e-11 in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tune", ["1", "0"])
@pytest.mark.parametrize("shape", [(16, 16, 512), (8, 12, 512), (6, 10, 256)], ids=lambda s: "x".join(map(str, s)))
def test_double_3d_long_x_lines(monkeypatch, shape, tune):
    from paper_1603_02329_gb300.api import PATOperator

    monkeypatch.setenv("PAT_AUTOTUNE", tune)
    pb = synth.small_lossy_3d(shape=shape, pml=2, Nt=12)
    ref = Operator.from_problem(pb)
    h = np.random.default_rng(3).standard_normal((pb.Nt, ref.Ns))
    op = PATOperator.from_problem(pb, precision="f64", device=torch.device("cuda", 0))
    d = op.forward(torch.tensor(pb.p0, dtype=torch.float64, device="cuda")).cpu().numpy()
    g = op.adjoint(torch.tensor(h, dtype=torch.float64, device="cuda")).cpu().numpy()
    op.close()
    d_ref, g_ref = ref.forward(pb.p0), ref.adjoint(h)
    assert np.linalg.norm(d - d_ref) <= 1e-11 * np.linalg.norm(d_ref)
    assert np.linalg.norm(g - g_ref) <= 1e-11 * np.linalg.norm(g_ref)
