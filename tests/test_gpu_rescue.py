"""The FP64 recomputation of flagged candidates in each of its forms: by the flagging block itself (short histories),
in 16 x 16 tiles (short lists), in 64 x 64 tiles (long lists), over several slabs of the workspace and several GPs.
Pools lie on and next to the observations, where the posterior variance is a small difference of large numbers, so that
most candidates are flagged; every element is compared with the oracle."""
import numpy as np
import pytest

from paper_2604_11109_b200 import binding as b
from oracle import gp_oracle as o
from tests.parity import check_scores
from tests.test_gpu_parity import compare_everything, dev, fit_gpu, rand_problem

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


@pytest.mark.parametrize("batch,n,d,m,sn2", [
    (1, 1900, 4, 700, 1e-2),      # a single wave of tiles: scored again with FP16 cross terms
    (1, 2048, 4, 20000, 1e-2),    # more than one wave: the pilot decides
    (2, 1800, 5, 15000, 1e-2),    # the first wave spans both GPs
    (1, 1900, 40, 21000, 1e-3),   # a tame pool: the FP8 form serves it
])
def test_long_histories_on_pools_that_need_fp16_cross_terms(batch, n, d, m, sn2):
    g = rand_problem(77 + n, batch, n, d, m, sn2=sn2, spread=2.0 if d < 10 else 0.4)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    assert b.r3_gp_tensor_info(gp)["f8_cross_terms"] == 1
    rows = np.sort(np.random.default_rng(3).choice(m, size=min(m, 1500), replace=False))
    mu, sd, ei, idx, val = (t.cpu().numpy() for t in b.r3_gp_score_topk(gp, dev(g["Xcand"]), 20))
    b.r3_gp_check(gp)
    for q, f in enumerate(o.fit_batch(g["X"], g["y"], g["ell"], g["sf2"], g["sn2"])):
        mu_r, sd_r, ei_r = o.score(f, g["Xcand"][q][rows])
        check_scores(mu[q][rows], sd[q][rows], ei[q][rows], mu_r, sd_r, ei_r, float(np.abs(g["y"][q]).max()),
                     float(g["sf2"][q]), ei_max=float(ei[q].max()), what=f"n{n} m{m}")
        assert np.array_equal(val[q], ei[q][idx[q]])
        assert np.array_equal(idx[q], o.topk(ei[q], 20)[0])
    gp.close()


@pytest.mark.parametrize("missing", [1, 2])
def test_a_long_history_without_memory_for_both_forms_of_its_operands(missing):
    """The FP16 form's operands are the last two allocations of a fit; without them every pool is scored in the FP8 form."""
    g = rand_problem(1977, 1, 1900, 4, 20000, sn2=1e-2, spread=2.0)
    X, y = dev(g["X"]), dev(g["y"])
    b.r3_test_fail_allocation(-1)
    b.r3_gp_fit(X, y, g["ell"], g["sf2"], g["sn2"]).close()
    b.r3_test_fail_allocation(b.r3_test_fail_allocation(-1) - missing)
    gp = b.r3_gp_fit(X, y, g["ell"], g["sf2"], g["sn2"])
    b.r3_test_fail_allocation(-1)
    assert b.r3_gp_engine(gp) == b.ENGINE_TENSOR and b.r3_gp_tensor_info(gp)["f8_cross_terms"] == 1
    mu, sd, ei, idx, val = (t.cpu().numpy() for t in b.r3_gp_score_topk(gp, dev(g["Xcand"]), 20))
    b.r3_gp_check(gp)
    f = o.fit_batch(g["X"], g["y"], g["ell"], g["sf2"], g["sn2"])[0]
    rows = np.sort(np.random.default_rng(3).choice(20000, size=1000, replace=False))
    mu_r, sd_r, ei_r = o.score(f, g["Xcand"][0][rows])
    check_scores(mu[0][rows], sd[0][rows], ei[0][rows], mu_r, sd_r, ei_r, float(np.abs(g["y"][0]).max()),
                 float(g["sf2"][0]), ei_max=float(ei[0].max()), what="FP8 form only")
    assert np.array_equal(idx[0], o.topk(ei[0], 20)[0])
    gp.close()


@pytest.mark.parametrize("m,k", [(128, 64), (300, 8), (4096, 1), (4096, 128), (4096, 129), (5000, 320), (20000, 321), (70001, 257)])
@pytest.mark.parametrize("kind", ["uniform", "crowded", "equal", "clustered"])
def test_selection_behind_the_guard(m, k, kind):
    """The scoring call's selection must be the oracle's on the EI it returns, on pools whose best values lie spread out,
    side by side, among many equal ones, or almost all below the rest."""
    g = rand_problem(60 + k, 1, 24, 3, m, spread=1.0)
    rng = np.random.default_rng(m + k)
    if kind == "crowded":        # the best candidates side by side (one thread's share of a slice at stride 256)
        best = g["Xcand"][0][:1].repeat(m, axis=0)
        g["Xcand"][0, ::256] = best[::256] + rng.normal(0, 1e-3, (len(best[::256]), 3)).astype(np.float32)
    elif kind == "equal":
        g["Xcand"][0] = g["Xcand"][0][rng.integers(0, 5, m)]
    elif kind == "clustered":
        g["Xcand"][0, k // 2:] = 40.0   # far away: prior mean and variance, one EI value for most of the pool
    gp = fit_gpu(g)
    mu, sd, ei, idx, val = (t.cpu().numpy()[0] for t in b.r3_gp_score_topk(gp, dev(g["Xcand"]), k))
    b.r3_gp_check(gp)
    oidx, oval = o.topk(ei, k)
    assert np.array_equal(idx, oidx) and np.array_equal(val, oval.astype(np.float32))
    gp.close()


@pytest.mark.parametrize("engine,exponent", [
    (b.ENGINE_SIMT, 62), (b.ENGINE_TENSOR, 62),
    (b.ENGINE_TENSOR, 70),   # squares of covariances beyond FP32, in which the other engine forms them
])
def test_large_signal_variances_are_not_taken_for_errors(engine, exponent):
    """Responses in units that make them 2^31 or 2^35 times as large (variances of 5e18 and 1e21): every value scales by a
    power of two, so the same candidates are flagged and the same results come out."""
    g = rand_problem(31, 1, 600, 24, 3000, sn2=0.1, spread=1.5)
    gp = fit_gpu(g, engine)
    want = [t.clone() for t in b.r3_gp_score(gp, dev(g["Xcand"]))]
    few = b.r3_gp_last_rescued(gp)
    assert 2 * few < g["Xcand"].shape[1]   # most of the pool needs no recomputation
    gp.close()
    unit = np.float32(2.0) ** (exponent // 2)
    g["y"], g["sf2"], g["sn2"] = g["y"] * unit, g["sf2"] * unit * unit, g["sn2"] * unit * unit
    gp = fit_gpu(g, engine)
    got = b.r3_gp_score(gp, dev(g["Xcand"]))
    b.r3_gp_check(gp)
    assert b.r3_gp_last_rescued(gp) == few
    for a, c in zip(got, want):
        assert torch.allclose(a / float(unit), c, rtol=1e-6, atol=1e-30)
    gp.close()
