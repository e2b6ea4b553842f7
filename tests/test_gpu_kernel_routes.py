"""Which kernel a plan's solves run in, as the probe names it: the register-fused power-of-two kernel, the
any-length kernel on the mixed-radix stages, or the generic one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,prec,env,name", [
    ((64, 64), "f32", {}, "k_persist2"),
    ((64, 64), "f64", {}, "k_pmx"),
    ((60, 64), "f32", {}, "k_pmx"),
    ((60, 56), "f64", {}, "k_pmx"),
    ((60, 56), "f32", {"PAT_MX": "0"}, "k_persist"),
    ((64, 64), "f64", {"PAT_MX": "0"}, "k_persist2"),
])
def test_persistent_kernel_is_named(monkeypatch, shape, prec, env, name):
    from paper_1603_02329_gb300.api import PATOperator

    for k, v in env.items():
        monkeypatch.setenv(k, v)
    pb = synth.small_lossy_2d(shape=shape, pml=6, Nt=12, n_sensors=8)
    op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
    op.set_probe(1)
    dt = torch.float32 if prec == "f32" else torch.float64
    op.forward(torch.tensor(pb.p0, dtype=dt, device="cuda"))
    op.adjoint(torch.tensor(np.ones((pb.Nt, op.Ns)), dtype=dt, device="cuda"))
    torch.cuda.synchronize()
    assert [s[0] for s in op.probe(False)] == [name + "_fwd"]
    assert [s[0] for s in op.probe(True)] == [name + "_adj"]
    op.close()
