"""Time reversal on both 2-D routes.  On the persistent one its grid barrier's wait is bounded and reported,
as the solves' is; on the per-phase one (PAT_PERSIST=0) the row kernels enforce the data.  Tolerances:
relative L2 1e-11 (FP64), 1e-5 (FP32), as for the other time-reversal images."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.pat_oracle import Operator  # noqa: E402
from oracle.pat_tr import time_reversal  # noqa: E402
from paper_1603_02329_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _op(pb, prec):
    from paper_1603_02329_gb300.api import PATOperator

    return PATOperator.from_problem(pb, precision=prec, device=torch.device("cuda", 0))


@pytest.mark.parametrize("prec,n", [("f32", 64), ("f32", 60), ("f64", 64)])
def test_barrier_timeout_is_reported_and_recovers(prec, n):
    # the fault hook lets every grid barrier wait for an arrival that never comes; the wait ends after 0.2 s
    from paper_1603_02329_gb300 import _lib

    pb = synth.vessel_phantom_2d(n=n, pml=8, Nt=30, n_vessels=2, n_discs=2)
    op = _op(pb, prec)
    data = torch.tensor(np.random.default_rng(1).standard_normal((pb.Nt, op.Ns)), device="cuda",
                        dtype=torch.float32 if prec == "f32" else torch.float64)
    good = op.time_reversal(data).cpu().numpy()
    L = _lib.lib()
    assert L.pat_plan_status(op._plan) == 0
    assert L.pat_plan_set_fault(op._plan, 1, 0.2) == 0
    t0 = time.perf_counter()
    op.time_reversal(data)
    assert L.pat_plan_status(op._plan) == 5   # PAT_ETIMEOUT
    assert time.perf_counter() - t0 < 5.0
    assert L.pat_plan_set_fault(op._plan, 0, 2.0) == 0
    assert np.array_equal(op.time_reversal(data).cpu().numpy(), good)
    assert L.pat_plan_status(op._plan) == 0
    op.close()


@pytest.mark.parametrize("mx", ["1", "0"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,alpha0", [(64, 0.75), (64, 0.0), (60, 0.75), (48, 0.0)])
def test_per_phase_route_matches_oracle(monkeypatch, n, alpha0, prec, mx):
    monkeypatch.setenv("PAT_PERSIST", "0")
    monkeypatch.setenv("PAT_MX", mx)
    pb = synth.vessel_phantom_2d(n=n, pml=6, Nt=70, alpha0=alpha0, n_vessels=2, n_discs=2)
    ref = Operator.from_problem(pb)
    data = ref.forward(pb.p0)
    op = _op(pb, prec)
    assert op.info.path == 0
    x = torch.tensor(data, dtype=torch.float32 if prec == "f32" else torch.float64, device="cuda")
    for compensate in (True, False):
        want = time_reversal(ref, data, compensate=compensate)
        got = op.time_reversal(x, compensate=compensate).cpu().numpy()
        assert np.linalg.norm(got - want) <= (1e-5 if prec == "f32" else 1e-11) * np.linalg.norm(want)
    op.close()
