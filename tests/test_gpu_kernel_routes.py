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
    ((64, 64), "f32", {"PAT_P2": "0"}, "k_persist"),
    ((64, 64), "f64", {"PAT_P2": "0"}, "k_persist"),
    ((60, 56), "f64", {"PAT_P2": "0"}, "k_persist"),
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


# PAT_ROW2=0 and PAT_SPEC2=0 select the generic row and spectral kernels, whatever the mixed-radix kernels
# would take: the same bits as with those kernels off
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(32, 64), (30, 48), (16, 16, 32), (12, 20, 18)], ids=lambda s: "x".join(map(str, s)))
def test_generic_per_phase_kernels_are_selected(monkeypatch, shape, prec):
    from paper_1603_02329_gb300.api import PATOperator

    make = synth.small_lossy_2d if len(shape) == 2 else synth.small_lossy_3d
    pb = make(shape=shape, pml=2, Nt=12)
    for k in ("PAT_PERSIST", "PAT_AUTOTUNE", "PAT_ROW2", "PAT_SPEC2"):
        monkeypatch.setenv(k, "0")
    out = []
    for mx in ("1", "0"):
        monkeypatch.setenv("PAT_MX", mx)
        op = PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))
        assert op.info.path == 0
        h = torch.tensor(np.random.default_rng(3).standard_normal((pb.Nt, op.Ns)), device="cuda",
                         dtype=torch.float32 if prec == "f32" else torch.float64)
        out.append(([int(v) for v in op.info.layout], op.adjoint(h).cpu().numpy()))
        op.close()
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])


# Which family the untuned per-phase kernels are from, as the launch layout shows it: (columns per spectral
# CTA, x-lines per row CTA) are (4 or in double 2-D 2, 8 / 4 / 2) with the mixed-radix kernels, (2 or in
# double 1, 2) with the others
@pytest.mark.parametrize("shape,prec,layout", [
    ((48, 512), "f32", (4, 8)), ((48, 60), "f64", (2, 8)), ((48, 300), "f64", (2, 2)), ((64, 300), "f64", (1, 2)),
    ((540, 100), "f64", (2, 4)),
    ((12, 20, 300), "f64", (4, 8)), ((16, 16, 64), "f64", (4, 8)), ((16, 16, 64), "f32", (2, 2)),
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else v)
def test_untuned_kernel_family(monkeypatch, shape, prec, layout):
    from paper_1603_02329_gb300.api import PATOperator

    monkeypatch.setenv("PAT_PERSIST", "0")
    monkeypatch.setenv("PAT_AUTOTUNE", "0")
    make = synth.small_lossy_2d if len(shape) == 2 else synth.small_lossy_3d
    op = PATOperator.from_problem(make(shape=shape, pml=2, Nt=4), precision=prec, device=torch.device("cuda", 0))
    assert (op.info.layout[0], op.info.layout[1]) == layout
    op.close()
