"""The TV proximal map's tiles (64 x 8 points, chunks of planes along z): sides below, at and one past a
tile, long in z (several chunks) and flat, against the FP64 oracle.  Tolerances: 20 inner steps of an
O(1) problem, each rounding a handful of operations, stay within 1e-12 (FP64) and 1e-5 (FP32) relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [(8, 64), (9, 65), (7, 63), (1, 130), (130, 1), (2, 2), (4, 8, 64), (5, 9, 65), (70, 3, 5), (9, 17, 66), (3, 1, 2),
          (1, 9, 9)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("n_inner,nonneg", [(1, True), (2, False), (20, True)])
def test_tile_edges(shape, n_inner, nonneg):
    from oracle import pat_optim as po
    from paper_1603_02329_gb300 import api

    z = np.random.default_rng(5).standard_normal(shape) + 0.3
    ref = po.tv_prox(z, 0.2, n_inner, nonneg=nonneg)
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 1e-5)):
        out = api.tv_prox(torch.tensor(z, dtype=dt, device="cuda"), 0.2, n_inner, nonneg=nonneg).cpu().numpy()
        assert np.linalg.norm(out - ref) <= tol * max(np.linalg.norm(ref), 1.0)
