"""The FP64 recomputation of flagged candidates in each of its forms: by the flagging block itself (short histories),
in 16 x 16 tiles (short lists), in 64 x 64 tiles (long lists), over several slabs of the workspace and several GPs.
Pools lie on and next to the observations, where the posterior variance is a small difference of large numbers, so that
most candidates are flagged; every element is compared with the oracle."""
import numpy as np
import pytest

from paper_2604_11109_b200 import binding as b
from tests.test_gpu_parity import compare_everything, fit_gpu, rand_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [b.ENGINE_SIMT, b.ENGINE_TENSOR])
@pytest.mark.parametrize("batch,n,m,near", [
    (1, 1, 40, 40),            # a single observation
    (1, 128, 3000, 3000),      # the longest history a block serves itself, more than 16 flagged per slice
    (2, 129, 700, 20),         # one observation more: the list, few entries
    (3, 160, 5000, 5000),      # three lists, 64 x 64 tiles
    (1, 600, 2000, 33),        # 16 x 16 tiles with ragged tails
    (1, 600, 20000, 20000),    # more candidates than one slab of the workspace holds
])
def test_flagged_candidates_are_recomputed(engine, batch, n, m, near):
    g = rand_problem(900 + n, batch, n, 5, m, sn2=1e-4, spread=3.0 if near > 100 else 0.5)
    rng = np.random.default_rng(n)
    for q in range(batch):
        rows = rng.choice(m, size=near, replace=False)
        g["Xcand"][q, rows] = g["X"][q, rng.integers(0, n, near)] + rng.normal(0, 1e-3, (near, 5)).astype(np.float32)
    gp = fit_gpu(g, engine)
    compare_everything(g, gp, min(m, 40), f"rescue n{n} m{m}")
    assert b.r3_gp_last_rescued(gp) >= 0.9 * near * batch
    gp.close()
