"""Factor and inverse factor at the edges of their 64-row tiles: the whole computation (fit) and its tail (append), for one
GP and for several, against the oracle's factor; the inverse is checked through the scores, which contract with it."""
import numpy as np
import pytest

from oracle import gp_oracle as o
from paper_2604_11109_b200 import binding as b
from tests.test_gpu_append import check_handle, check_scoring, dev, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,n", [(1, 1), (1, 32), (3, 63), (1, 64), (2, 65), (1, 96), (1, 128), (5, 129), (1, 320), (1, 833)])
def test_fit_at_tile_edges(batch, n):
    g = problem(1300 + n, batch, n, 7, 150)
    gp = b.r3_gp_fit(dev(g["X"]), dev(g["y"]), g["ell"], g["sf2"], g["sn2"])
    check_scoring(gp, g, check_handle(gp, g, n))
    gp.close()


@pytest.mark.parametrize("batch,n0,k", [(1, 63, 1), (2, 64, 1), (1, 64, 64), (1, 120, 128), (3, 191, 2), (1, 640, 3)])
def test_append_at_tile_edges(batch, n0, k):
    g = problem(1700 + n0, batch, n0 + k, 7, 150)
    gp = b.r3_gp_fit(dev(g["X"][:, :n0]), dev(g["y"][:, :n0]), g["ell"], g["sf2"], g["sn2"])
    b.r3_gp_append(gp, dev(g["X"][:, n0:]), dev(g["y"][:, n0:]))
    check_scoring(gp, g, check_handle(gp, g, n0 + k))
    # the tail of the computation gives the bits of the whole
    whole = b.r3_gp_fit(dev(g["X"]), dev(g["y"]), g["ell"], g["sf2"], g["sn2"])
    for x, y in zip(b.r3_gp_get_factor(gp), b.r3_gp_get_factor(whole)):
        assert np.array_equal(x, y)
    gp.close()
    whole.close()


@pytest.mark.parametrize("n,twin", [(40, 3), (100, 70), (200, 10)])
def test_duplicated_row_without_noise_is_not_positive_definite(n, twin):
    g = problem(2100 + n, 1, n, 5, 4)
    g["X"][0, -1] = g["X"][0, twin]
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_fit(dev(g["X"]), dev(g["y"]), g["ell"], g["sf2"], np.zeros(1, np.float32))
    assert e.value.status == 3 and f"pivot {n - 1} " in str(e.value)


@pytest.mark.parametrize("batch,n", [(1, 31), (2, 129), (40, 33), (40, 320), (40, 321), (1, 544), (1, 545)])
def test_weights_where_their_split_changes(batch, n):
    """One GP or many, around the history lengths at which W stops fitting the shared memory of two and of eight blocks: the
    weights (check_handle), the norm estimate, and the scores."""
    g = problem(2500 + n, batch, n, 4, 40)
    gp = b.r3_gp_fit(dev(g["X"]), dev(g["y"]), g["ell"], g["sf2"], g["sn2"])
    fits = check_handle(gp, g, n)
    check_norms(gp, fits)
    check_scoring(gp, g, fits)
    gp.close()


def check_norms(gp, fits):
    """1.5 times twelve power iterations on W^T W, which never exceed |W|_2 and reach (c^2)^(1/48) of it if a share c^2 of the
    start vector lies along the leading direction: 0.78 for c^2 = 1e-5.  (W's own error: 1e-4 covers the ill-conditioned.)"""
    for got, f in zip(b.r3_gp_get_norms(gp), fits):
        ratio = got * np.linalg.svd(np.tril(f.L), compute_uv=False)[-1]   # |L^-1|_2 = 1 / smallest singular value
        assert 1.5 * 0.78 <= ratio <= 1.5 * (1 + 1e-4), ratio


@pytest.mark.parametrize("batch,n,spread", [(1, 100, 3.0), (40, 300, 5.0), (1, 500, 5.0), (1, 600, 5.0)])
def test_norm_estimate_of_ill_conditioned_histories(batch, n, spread):
    g = problem(2700 + n, batch, n, 4, 10)
    g["ell"] *= np.float32(spread)
    g["sn2"][:] = 1e-7
    gp = b.r3_gp_fit(dev(g["X"]), dev(g["y"]), g["ell"], g["sf2"], g["sn2"])
    check_norms(gp, o.fit_batch(g["X"], g["y"], g["ell"], g["sf2"], g["sn2"]))
    b.r3_gp_append(gp, dev(g["X"][:, :1] + np.float32(0.5)), dev(g["y"][:, :1]))   # an append makes its own
    X1, y1 = np.concatenate([g["X"], g["X"][:, :1] + np.float32(0.5)], 1), np.concatenate([g["y"], g["y"][:, :1]], 1)
    check_norms(gp, o.fit_batch(X1, y1, g["ell"], g["sf2"], g["sn2"]))
    gp.close()


def test_reciprocal_roots_of_pivots():
    """Relative error at most 2^-52: the last Newton step rounds the product h y (relative 2^-53, which enters halved) and the
    new y (2^-53), and the steps leave 2^-84.  CUDA's own function may be off by one unit in the last place as well."""
    rng = np.random.default_rng(17)
    p = np.concatenate([np.exp(rng.uniform(np.log(1e-290), np.log(1e290), 400000)),   # every exponent
                        rng.uniform(0.25, 4.0, 400000),                               # every mantissa of two binades
                        2.0 ** rng.integers(-200, 200, 1000), 1.0 + np.arange(-64, 65) * 2.0 ** -52])
    p1, s = rng.uniform(0.5, 2.0, 100000), rng.uniform(0.3, 0.7, 100000)
    tail = 10.0 ** rng.uniform(-15, 0, 100000)
    p = np.concatenate([p, p1 * (s * s / p1 + tail) - s * s])   # determinants of nearly singular pairs
    p = p[p > 1e-300]
    y = b.r3_test_rsqrt(dev(p)).cpu().numpy()
    exact = 1.0 / np.sqrt(p.astype(np.longdouble))
    assert float(np.abs(y / exact - 1.0).max()) <= 2.0 ** -52
    assert float(np.abs(y / torch.rsqrt(dev(p)).cpu().numpy() - 1.0).max()) <= 2.0 ** -51
    assert np.isnan(b.r3_test_rsqrt(dev(np.array([0.0, -1.0, np.nan, -np.inf]))).cpu().numpy()).all()


@pytest.mark.parametrize("n", [2, 70])
@pytest.mark.parametrize("gap", [1.9e-8, 2.0e-8, 2.1e-8, 2.2e-8])
def test_a_small_positive_pivot_is_positive(n, gap):
    """Noise-free, all rows far apart but the last, `gap` lengthscales from the first: k = 1 - 5/6 gap^2 = 1 - (3 to 4)e-16,
    computed with an error of at most 2e-16 (three roundings near one), and the last pivot is 1 - k^2 > 0, a few roundings of
    the diagonal."""
    X = (100.0 * np.arange(n, dtype=np.float32))[None, :, None]
    X[0, -1, 0] = gap
    y = np.linspace(-1, 1, n, dtype=np.float32)[None]
    one = np.ones((1, 1), np.float32)
    gp = b.r3_gp_fit(dev(X), dev(y), one, one[0], np.zeros(1, np.float32))
    _, L = b.r3_gp_get_factor(gp)
    assert 0.0 < L[0, -1, -1] ** 2 < 2e-15
    assert L[0, -1, 0] == pytest.approx(1.0, abs=1e-15)
    gp.close()
