"""Failure paths of the CUDA library that can be exercised without faulting a GPU.

* a device-side wait that runs out: the tensor-core kernel's bounded waits, provoked by withholding one stage
  of its operand stream under a short limit; the kernel returns by itself, the status is reported, the handle
  keeps working;
* allocation failures injected on the host; the device-memory cache across fits;
* status bits latched by one call do not leak into the next call's own checks;
* two live handles of different shapes that share a kernel instantiation.
"""
import numpy as np
import pytest

from oracle import gp_oracle as o
from paper_2604_11109_b200 import binding as b
from tests.parity import check_scores
from tests.test_gpu_parity import compare_everything, dev, fit_gpu, rand_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHORT_LIMIT = 2_000_000     # cycles: about a millisecond


def _scores_match(g, gp, what):
    mu, sd, ei = (t.cpu().numpy() for t in b.r3_gp_score(gp, dev(g["Xcand"])))
    b.r3_gp_check(gp)
    for q, f in enumerate(o.fit_batch(g["X"], g["y"], g["ell"], g["sf2"], g["sn2"])):
        mu_r, sd_r, ei_r = o.score(f, g["Xcand"][q])
        check_scores(mu[q], sd[q], ei[q], mu_r, sd_r, ei_r, float(np.abs(g["y"][q]).max()), float(g["sf2"][q]),
                     what=what)


@pytest.mark.parametrize("n,d,m,chunk,pair", [
    (100, 12, 128, 2, False),    # one pass of four chunks, one tile: the third chunk of W never arrives
    (250, 12, 300, 0, False),    # the very first chunk is withheld; three tiles on three thread blocks
    (600, 12, 1000, 11, False),  # three passes; the stream stops inside the second
    (500, 128, 260, 9, False),   # one buffer of scaled candidates, whose next tile comes in before the last strip is read back
    (400, 70, 300, 6, False),    # features in two stages
    (1100, 40, 200, 3, False),   # pairs of strips shared out: no part of a tile arrives
    (140, 20, 148 * 128 * 3 + 5, 6, False),   # several tiles per thread block; both groups of result warps are under way
    (1900, 24, 200, 5, False),   # FP8 cross terms
    (300, 12, 256, 5, True),     # the kernel that runs a tile on a cluster of two thread blocks
])
def test_a_wait_that_runs_out_is_reported_and_the_handle_stays_usable(monkeypatch, n, d, m, chunk, pair):
    if pair:
        monkeypatch.setenv("R3_TC_PAIR", "1")
    g = rand_problem(4000 + n, 1, n, d, m)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    _scores_match(g, gp, "before")
    b.r3_gp_set_wait_limit(gp, SHORT_LIMIT)
    b.r3_gp_test_withhold(gp, chunk)
    b.r3_gp_score(gp, dev(g["Xcand"]))            # returns by itself: every wait is bounded
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_check(gp)
    assert e.value.status == 6                    # R3_ERR_DEVICE_TIMEOUT
    # the latch is cleared, the hook was for one call, and the same handle scores correctly again
    _scores_match(g, gp, "after the timeout")
    b.r3_gp_set_wait_limit(gp, 4_000_000_000)
    _scores_match(g, gp, "default limit")
    gp.close()


@pytest.mark.parametrize("n,d,m,pair", [
    (1500, 20, 148 * 128 * 4 + 3, False),   # two buffers of candidates
    (1000, 128, 148 * 128 * 3, False),      # one buffer, features in two stages
    (2500, 40, 148 * 128 * 2 + 9, False),   # FP8 cross terms
    (900, 24, 300, False),                  # pairs of strips shared out
    (1200, 20, 148 * 64 * 4 + 3, True),     # clusters of two thread blocks, which send each other chunks
])
def test_a_limit_that_runs_out_while_the_pipeline_is_at_work(monkeypatch, n, d, m, pair):
    """The shortest limit there is, less than a tile takes: waits run out in thread blocks whose other warps are still
    handing stages over.  The call returns by itself, with or without a time-out, and the handle keeps working."""
    if pair:
        monkeypatch.setenv("R3_TC_PAIR", "1")
    g = rand_problem(4100 + n, 1, n, d, m)
    gp = fit_gpu(g, b.ENGINE_TENSOR)
    xc = dev(g["Xcand"])
    want = [t.clone() for t in b.r3_gp_score(gp, xc)]
    b.r3_gp_check(gp)
    b.r3_gp_set_wait_limit(gp, 100_000)
    for _ in range(5):
        b.r3_gp_score(gp, xc)
        try:
            b.r3_gp_check(gp)
        except b.R3Error as e:
            assert e.status == 6
    b.r3_gp_set_wait_limit(gp, 4_000_000_000)
    got = b.r3_gp_score(gp, xc)
    b.r3_gp_check(gp)
    # the same kernels on the same operands: only what the FP64 pass recomputes may come in another grouping
    for a, c, scale in zip(got, want, (np.abs(g["y"]).max(), 1.0, float(want[2].max()))):
        assert ((a - c).abs() <= 1e-6 * (c.abs() + scale)).all()
    gp.close()


def test_wait_limit_and_withhold_arguments():
    g = rand_problem(1, 1, 20, 3, 10)
    gp = fit_gpu(g)
    for bad in (0, 99_999, -5):
        with pytest.raises(b.R3Error) as e:
            b.r3_gp_set_wait_limit(gp, bad)
        assert e.value.status == 1
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_test_withhold(gp, -1)
    assert e.value.status == 1
    gp.close()


def test_allocation_failure_in_fit_is_reported_and_leaves_nothing_behind():
    g = rand_problem(2, 2, 150, 10, 64)
    X, y = dev(g["X"]), dev(g["y"])
    b.r3_trim_cache()
    # count the allocations of one successful fit, then fail each of them in turn
    b.r3_test_fail_allocation(-1)
    b.r3_gp_fit(X, y, g["ell"], g["sf2"], g["sn2"]).close()
    total = b.r3_test_fail_allocation(-1)
    assert total >= 15
    for after in range(total):
        b.r3_test_fail_allocation(after)
        try:
            gp = b.r3_gp_fit(X, y, g["ell"], g["sf2"], g["sn2"])
        except b.R3Error as e:
            assert e.status == 4, f"allocation {after}: {e}"       # R3_ERR_ALLOC
            continue
        # allocations of temporaries that the fit can do without (none today) would land here
        gp.close()
    b.r3_test_fail_allocation(-1)
    gp = fit_gpu(g)
    compare_everything(g, gp, 8, "after the injected failures")
    gp.close()


def test_allocation_failure_in_append_leaves_the_handle_unchanged():
    g = rand_problem(3, 1, 200, 6, 500)
    k = 16
    gp = b.r3_gp_fit(dev(g["X"][:, :-k]), dev(g["y"][:, :-k]), g["ell"], g["sf2"], g["sn2"])
    xc = dev(g["Xcand"])
    before = [t.clone() for t in b.r3_gp_score(gp, xc)]
    xn, yn = dev(g["X"][:, -k:]), dev(g["y"][:, -k:])
    for after in (0, 3, 9):
        b.r3_test_fail_allocation(after)
        with pytest.raises(b.R3Error) as e:
            b.r3_gp_append(gp, xn, yn)
        assert e.value.status == 4
        assert b.r3_gp_size(gp) == 200 - k
        for a, c in zip(before, b.r3_gp_score(gp, xc)):
            assert torch.equal(a, c)
    b.r3_test_fail_allocation(-1)
    b.r3_gp_append(gp, xn, yn)
    assert b.r3_gp_size(gp) == 200
    compare_everything(g, gp, 8, "append after the injected failures")
    gp.close()


def test_append_after_an_unchecked_scoring_call_keeps_that_calls_latched_status():
    g = rand_problem(5, 1, 60, 4, 200)
    k = 8
    gp = b.r3_gp_fit(dev(g["X"][:, :-k]), dev(g["y"][:, :-k]), g["ell"], g["sf2"], g["sn2"])
    bad = g["Xcand"].copy()
    bad[0, 17, 2] = np.nan
    b.r3_gp_score(gp, dev(bad))                              # latches "non-finite candidate"; not checked yet
    b.r3_gp_append(gp, dev(g["X"][:, -k:]), dev(g["y"][:, -k:]))   # valid data: must succeed
    assert b.r3_gp_size(gp) == 60
    with pytest.raises(b.R3Error) as e:                      # the scoring call's problem is still reported
        b.r3_gp_check(gp)
    assert e.value.status == 2
    compare_everything(g, gp, 8, "after append")
    gp.close()


def test_freed_blocks_of_every_size_are_kept_and_given_back_on_request():
    """The device-memory cache keeps a closed handle's blocks, the small ones included (a small history's fit is
    two dozen of them), hands them to the next fit of the same shape, and returns everything on r3_trim_cache."""
    b.r3_trim_cache()
    assert b.r3_cached_bytes() == 0
    g = rand_problem(21, 1, 48, 5, 64)
    fit_gpu(g).close()
    kept = b.r3_cached_bytes()
    assert kept > 0
    gp = fit_gpu(g)                       # the same shape again: served from the cache
    assert b.r3_cached_bytes() < kept
    compare_everything(g, gp, 8, "fit from cached blocks")
    gp.close()
    assert b.r3_cached_bytes() >= kept
    big = rand_problem(22, 1, 700, 9, 64)  # blocks above 1 MiB go through the same cache
    fit_gpu(big).close()
    assert b.r3_cached_bytes() > kept + (1 << 20)
    b.r3_trim_cache()
    assert b.r3_cached_bytes() == 0
    gp = fit_gpu(g)
    compare_everything(g, gp, 8, "fit after the cache was emptied")
    gp.close()


def test_two_live_handles_that_share_a_kernel_instantiation():
    """Handles with different feature counts need different amounts of shared memory from the same kernel;
    fitting one must not take away what the other needs."""
    ga = rand_problem(11, 1, 256, 16, 700)
    gb = rand_problem(12, 1, 512, 64, 700)
    a = fit_gpu(ga, b.ENGINE_TENSOR)
    bb = fit_gpu(gb, b.ENGINE_TENSOR)
    for g, gp, what in ((ga, a, "A"), (gb, bb, "B"), (ga, a, "A again")):
        _scores_match(g, gp, what)
    c = fit_gpu(rand_problem(13, 1, 300, 128, 10), b.ENGINE_TENSOR)   # a third shape in between
    _scores_match(ga, a, "A after C")
    _scores_match(gb, bb, "B after C")
    for h in (a, bb, c):
        h.close()


def test_the_cache_makes_room_for_sizes_that_are_still_in_use():
    """A program that changes its sizes must not fill the cache with blocks of sizes it has left: beyond the limit the
    block that has lain there longest goes, and the newest is kept."""
    b.r3_trim_cache()
    for n in (2048, 2304, 2560, 2816, 3072, 3328, 3584, 3840):   # fits of 120 to 420 MB, over 2 GiB together
        g = rand_problem(30, 1, n, 3, 8)
        fit_gpu(g).close()
    full = b.r3_cached_bytes()
    assert (1 << 30) < full <= (2 << 30)
    gp = fit_gpu(g)                       # the last size is served from the cache
    assert b.r3_cached_bytes() < full - (200 << 20)
    gp.close()
    b.r3_trim_cache()
    assert b.r3_cached_bytes() == 0


@pytest.mark.parametrize("where,batch,n", [
    (0, 1, 100), (0, 3, 400),     # the factorisation: the first tile of the first GP is never announced
    (1, 1, 100), (1, 2, 530),     # the weights: a cluster of eight blocks
    (1, 40, 300),                 # a cluster of two
    (1, 1, 700),                  # a team of blocks with a barrier
])
def test_a_wait_of_an_append_that_runs_out_leaves_the_handle_unchanged(where, batch, n):
    g = rand_problem(5000 + n, batch, n, 5, 60)
    k = 70                                        # a whole tile of new rows and more
    gp = b.r3_gp_fit(dev(g["X"][:, :-k]), dev(g["y"][:, :-k]), g["ell"], g["sf2"], g["sn2"])
    xc, xn, yn = dev(g["Xcand"]), dev(g["X"][:, -k:]), dev(g["y"][:, -k:])
    before = [t.clone() for t in b.r3_gp_score(gp, xc)]
    b.r3_gp_test_stall(gp, where, SHORT_LIMIT)
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_append(gp, xn, yn)
    assert e.value.status == 6
    assert b.r3_gp_size(gp) == n - k
    b.r3_gp_check(gp)
    for old, new in zip(before, b.r3_gp_score(gp, xc)):
        assert torch.equal(old, new)
    b.r3_gp_append(gp, xn, yn)                    # the aid was for one launch
    _scores_match(g, gp, "append after a wait that ran out")
    gp.close()


@pytest.mark.parametrize("n,m,k", [
    (40, 600, 16),        # the kernel finishes the selection itself
    (300, 80000, 300),    # its slices' keys go on to the selection's later levels
])
def test_a_guard_barrier_that_runs_out_leaves_indices_inside_the_pool(n, m, k):
    g = rand_problem(6000 + n, 2, n, 5, m)
    gp = fit_gpu(g)
    xc = dev(g["Xcand"])
    b.r3_gp_score_topk(gp, xc, k)                 # the workspace now holds another call's keys
    b.r3_gp_check(gp)
    b.r3_gp_test_stall(gp, 2, SHORT_LIMIT)
    _, _, _, idx, _ = b.r3_gp_score_topk(gp, xc, k)
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_check(gp)
    assert e.value.status == 6
    for row in idx.cpu().numpy():
        assert row.min() >= 0 and row.max() < m and len(set(row.tolist())) == k
    compare_everything(g, gp, 8, "after a guard barrier that ran out")
    gp.close()


@pytest.mark.parametrize("where", [2, 3])
def test_a_proposal_whose_barrier_runs_out_names_rows_of_the_pool(where):
    g = rand_problem(6100, 2, 150, 5, 3000)
    gp = fit_gpu(g)
    xc = dev(g["Xcand"])
    want, _, _ = b.r3_gp_propose(gp, xc, 8)
    b.r3_gp_test_stall(gp, where, SHORT_LIMIT)
    idx, _, _ = b.r3_gp_propose(gp, xc, 8)
    with pytest.raises(b.R3Error) as e:
        b.r3_gp_check(gp)
    assert e.value.status == 6
    for row in np.asarray(idx.cpu()):
        assert row.min() >= 0 and row.max() < 3000 and len(set(row.tolist())) == 8
    again, _, _ = b.r3_gp_propose(gp, xc, 8)
    b.r3_gp_check(gp)
    assert torch.equal(want, again)
    gp.close()


@pytest.mark.parametrize("call", ["optimize", "refit"])
@pytest.mark.parametrize("failure", ["allocation", "wait"])
def test_a_refit_that_fails_keeps_the_previous_fit(call, failure):
    g = rand_problem(7000, 2, 150, 10, 300)
    xc = dev(g["Xcand"])

    def go(gp):
        if call == "optimize":
            b.r3_gp_optimize(gp, max_evals=3, gtol=1e-9)
        else:
            b.r3_gp_refit(gp, 2.0 * g["ell"], g["sf2"], g["sn2"])

    gp = fit_gpu(g)
    before = [t.clone() for t in b.r3_gp_score(gp, xc)]
    factor = b.r3_gp_get_factor(gp)
    spare = fit_gpu(g)
    b.r3_test_fail_allocation(-1)
    go(spare)                                     # how many allocations the call makes
    total = b.r3_test_fail_allocation(-1)
    spare.close()
    for after in range(total) if failure == "allocation" else [None]:
        if after is None:
            b.r3_gp_test_stall(gp, 0, SHORT_LIMIT)
        else:
            b.r3_test_fail_allocation(after)
        with pytest.raises(b.R3Error) as e:
            go(gp)
        assert e.value.status == (6 if after is None else 4) and "were kept" in str(e.value), after
        for old, new in zip(factor, b.r3_gp_get_factor(gp)):
            assert np.array_equal(old, new), after
        for old, new in zip(before, b.r3_gp_score(gp, xc)):
            assert torch.equal(old, new), after
        b.r3_gp_check(gp)
    b.r3_test_fail_allocation(-1)
    go(gp)                                        # and the call goes through afterwards
    gp.close()


def test_an_append_without_memory_for_both_states_operands_keeps_the_tensor_engine():
    """Whichever single allocation fails, the append either leaves the handle as it was or ends on the engine that serves it:
    operands that do not fit beside the old state's are made after those are gone."""
    g = rand_problem(8000, 1, 200, 10, 300)
    k = 16
    xn, yn = dev(g["X"][:, -k:]), dev(g["y"][:, -k:])

    def shorter():
        return b.r3_gp_fit(dev(g["X"][:, :-k]), dev(g["y"][:, :-k]), g["ell"], g["sf2"], g["sn2"])

    gp = shorter()
    b.r3_test_fail_allocation(-1)
    b.r3_gp_append(gp, xn, yn)
    total = b.r3_test_fail_allocation(-1)
    gp.close()
    went_through = 0
    for after in range(total):
        gp = shorter()
        b.r3_test_fail_allocation(after)
        try:
            b.r3_gp_append(gp, xn, yn)
            went_through += 1
        except b.R3Error as e:
            assert e.status == 4 and b.r3_gp_size(gp) == 200 - k
            b.r3_gp_append(gp, xn, yn)
        assert b.r3_gp_engine(gp) == b.ENGINE_TENSOR, after
        _scores_match(g, gp, f"append with allocation {after} failing")
        gp.close()
    b.r3_test_fail_allocation(-1)
    assert went_through >= 5
