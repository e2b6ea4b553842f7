"""The TV proximal map's run-time tiles: images of few columns (one to 33, where a tile packs many rows; 256
rows at most) in both precisions, and all images in double, up to several planes per CTA, against the FP64
oracle.  Tolerances: a few inner steps of an O(1) problem, each rounding a handful of operations, stay
within 1e-12 (FP64) and 1e-5 (FP32) relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPES = [(300, 2), (257, 1), (256, 1), (130, 33), (129, 32), (64, 100), (2, 256, 2), (2, 257, 2), (3, 600, 4), (70, 8, 3),
          (5, 40, 33), (40, 64, 32), (16, 129, 70), (61, 66, 60), (250, 40, 24)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("n_inner,nonneg", [(1, False), (4, True)])
def test_packed_tiles(shape, n_inner, nonneg):
    from oracle import pat_optim as po
    from paper_1603_02329_gb300 import api

    z = np.random.default_rng(5).standard_normal(shape) + 0.3
    ref = po.tv_prox(z, 0.2, n_inner, nonneg=nonneg)
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 1e-5)):
        out = api.tv_prox(torch.tensor(z, dtype=dt, device="cuda"), 0.2, n_inner, nonneg=nonneg).cpu().numpy()
        assert np.linalg.norm(out - ref) <= tol * max(np.linalg.norm(ref), 1.0)
