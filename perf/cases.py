"""What the speed of this library is judged on: the calls that a tuning program makes, over the range of sizes it
makes them at.

Five kinds of pass, each through the public entry points of the binding:

  score   one proposal round on a fitted handle: r3_gp_score_topk on a pool in device memory, or
          r3_gp_score_topk_host on a pool in pinned host memory
  round   one round of a search that keeps its surrogate: r3_gp_fit of the history, r3_gp_append of the points that
          have just been replayed, r3_gp_propose of the next ones, r3_gp_score of configurations the program watches
  tune    r3_gp_fit and r3_gp_optimize: choosing the hyper-parameters of one or many surrogates
  search  r3_bo_run: the whole inner search with its replay callback
  tpe     one round with the Parzen estimator: r3_tpe_fit, r3_tpe_score, r3_topk

Inputs are made on the GPU from the seed: rows of launch parameters and compiler flags, pass orders or continuous
settings, scaled to [0, 1], with a smooth response and a little noise, standardised as a tuning program would.
"""
import math

import torch

from paper_2604_11109_b200 import binding as r3

# admissible values per launch parameter: block size, grid multiplier, unroll, register cap, carve-out, one switch
_LAUNCH = (32, 8, 4, 224, 5, 2)


def listed():
    return [
        # The smallest search: six launch parameters, a few dozen replays; one proposal is a handful of launches.
        {"name": "score_launch", "kind": "score", "batch": 1, "n": 64, "d": 6, "m": 4096, "k": 8,
         "rows": "launch", "near": 0.0, "host": False},
        # Launch parameters and ten compiler flags: an ordinary single search.
        {"name": "score_flags", "kind": "score", "batch": 1, "n": 256, "d": 16, "m": 262144, "k": 32,
         "rows": "launch", "near": 0.0, "host": False},
        # Sixty-four source candidates tuned side by side, one surrogate and one pool each.
        {"name": "score_many", "kind": "score", "batch": 64, "n": 512, "d": 32, "m": 65536, "k": 16,
         "rows": "launch", "near": 0.0, "host": False},
        # Pass ordering: one-hot position buckets of 32 passes, the widest rows.
        {"name": "score_passes", "kind": "score", "batch": 1, "n": 1024, "d": 128, "m": 1048576, "k": 256,
         "rows": "passes", "near": 0.0, "host": False},
        # A long history: the largest call.
        {"name": "score_history", "kind": "score", "batch": 1, "n": 4096, "d": 64, "m": 1048576, "k": 256,
         "rows": "mixed", "near": 0.0, "host": False},
        # A pool that the program holds in host memory, at sizes that divide nothing, an eighth of it neighbours of
        # replayed configurations (a local search around what has worked).
        {"name": "score_local_host", "kind": "score", "batch": 1, "n": 701, "d": 23, "m": 199999, "k": 50,
         "rows": "launch", "near": 0.125, "host": True},
        # One round of the smallest search: fit, update, next proposal -- latency and launches.
        {"name": "round_launch", "kind": "round", "batch": 1, "n": 64, "d": 6, "m": 4096, "q": 8, "rows": "launch"},
        # One round on the longest history.
        {"name": "round_history", "kind": "round", "batch": 1, "n": 3968, "d": 64, "m": 65536, "q": 128,
         "rows": "mixed"},
        # Hyper-parameters of one ordinary surrogate.
        {"name": "tune_flags", "kind": "tune", "batch": 1, "n": 300, "d": 16, "evals": 12, "rows": "launch"},
        # Hyper-parameters of sixty-four surrogates at once.
        {"name": "tune_many", "kind": "tune", "batch": 64, "n": 512, "d": 32, "evals": 8, "rows": "launch"},
        # The inner search as one call: ten rounds of eight replays.
        {"name": "search_flags", "kind": "search", "n": 100, "d": 16, "m": 32768, "q": 8, "rounds": 10,
         "rows": "launch"},
        # The Parzen estimator on a long history of 16-level parameters and switches.
        {"name": "tpe_history", "kind": "tpe", "n": 4096, "d": 64, "m": 1048576, "k": 256, "rows": "mixed",
         "grid": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "score", "score", "round", "round", "tune", "search", "tpe"])
    if kind == "score":
        rows = rng.choice(["launch", "mixed", "uniform", "passes"])
        batch = rng.choice([1, 1, 1, _log(rng, 2, 64)])
        near = rng.choice([0.0, 0.0, 0.125])
        n = _log(rng, 24, 1024 if near or batch > 1 else 4096)
        d = 128 if rows == "passes" else _log(rng, 3, 128)
        # no more arithmetic than the largest listed call, and a pool of at most 2^28 bytes; pools that lie close to
        # the history (few features, or neighbours of what was replayed) are smaller
        close = near or d < 32
        most = min(1 << 20, int((1 << 20) * (4096.0 / max(n, 1024 if close else 512)) ** 2 / batch / (16 if close else 1)),
                   (1 << 26) // (batch * d))
        m = _log(rng, 900, max(1800, most))
        return {"kind": kind, "batch": batch, "n": n, "d": d, "m": m, "k": _log(rng, 1, min(256, m)), "rows": rows,
                "near": near, "host": rng.random() < 0.25}
    if kind == "round":
        batch = rng.choice([1, 1, 1, _log(rng, 2, 16)])
        n = _log(rng, 20, 3900 if batch == 1 else 500)
        return {"kind": kind, "batch": batch, "n": n, "d": _log(rng, 3, 128), "m": _log(rng, 2000, 65536 // batch + 2000),
                "q": _log(rng, 1, 128 if batch == 1 else 32), "rows": rng.choice(["launch", "mixed", "uniform"])}
    if kind == "tune":
        batch = rng.choice([1, 1, _log(rng, 2, 64)])
        return {"kind": kind, "batch": batch, "n": _log(rng, 40, 1500 if batch == 1 else 400), "d": _log(rng, 3, 64),
                "evals": rng.randint(3, 12), "rows": rng.choice(["launch", "mixed", "uniform"])}
    if kind == "search":
        return {"kind": kind, "n": _log(rng, 20, 1000), "d": _log(rng, 6, 64), "m": _log(rng, 3000, 65536),
                "q": _log(rng, 2, 32), "rounds": rng.randint(3, 10), "rows": rng.choice(["mixed", "uniform"])}
    d = _log(rng, 4, 128)
    n = _log(rng, 40, 4096)
    rows = rng.choice(["launch", "mixed", "uniform"])
    # continuous values keep a component per observation: the pool is cut so that the largest call stays in range
    most = min(1 << 20, (1 << 26) // d)
    if rows == "uniform":
        most = min(most, int(4e10 / (n * d)))
    m = _log(rng, 2000, max(4000, most))
    return {"kind": kind, "n": n, "d": d, "m": m, "k": _log(rng, 1, 256), "rows": rows, "grid": rng.random() < 0.5}


# ------------------------------------------------------------------------------------------------ inputs
def _levels(rows, d):
    """Admissible values per feature; 0 for a continuous one."""
    if rows == "launch":
        return [_LAUNCH[j] if j < len(_LAUNCH) else 2 for j in range(d)]
    if rows == "mixed":
        return [16 if j < (d + 1) // 2 else 2 for j in range(d)]
    return [0] * d


def _draw_rows(gen, rows, count, d):
    if rows == "passes":   # pass p sits in one of four position buckets; rows have unit norm
        position = torch.rand((count, d // 4), generator=gen, device="cuda").argsort(dim=1)
        out = torch.zeros((count, d), device="cuda")
        return out.scatter_(1, 4 * torch.arange(d // 4, device="cuda") + position // max(1, d // 16),
                            1.0 / math.sqrt(d // 4))
    u = torch.rand((count, d), generator=gen, device="cuda")
    levels = torch.tensor(_levels(rows, d), device="cuda", dtype=torch.float32)
    if rows == "uniform":
        return u
    return torch.minimum((u * levels).floor(), levels - 1) / (levels - 1)


def _response(gen, x, noise):
    """Three waves and a bowl, the same surface for every row of x [count][d], standardised."""
    d = x.shape[1]
    wave = torch.randn((d, 3), generator=gen, device="cuda") * (2.0 / math.sqrt(d))
    phase = torch.rand(3, generator=gen, device="cuda") * (2 * math.pi)
    centre = torch.rand(d, generator=gen, device="cuda") * 0.6 + 0.2

    def surface(z):
        return (torch.sin(2 * math.pi * (z @ wave) + phase).sum(1) * 0.75 +
                ((z - centre) ** 2).sum(1) * min(1.0, 6.0 / d))

    clean = surface(x)
    mean, std = clean.mean(), clean.std() + 1e-6
    y = (clean - mean) / std + torch.randn(x.shape[0], generator=gen, device="cuda") * math.sqrt(noise)
    return y, lambda z: (surface(z) - mean) / std


def _neighbours(gen, history, rows, count):
    """Rows of the history with one feature moved by a step (two passes swapped into each other's buckets)."""
    out = history[torch.randint(0, history.shape[0], (count,), generator=gen, device="cuda")]
    d = out.shape[1]
    r = torch.arange(count, device="cuda")
    if rows == "passes":
        a = torch.randint(0, d // 4, (count,), generator=gen, device="cuda")
        b = (a + 1 + torch.randint(0, d // 4 - 1, (count,), generator=gen, device="cuda")) % (d // 4)
        four = torch.arange(4, device="cuda")
        ia, ib = 4 * a[:, None] + four, 4 * b[:, None] + four
        va, vb = out.gather(1, ia), out.gather(1, ib)
        return out.scatter(1, ia, vb).scatter(1, ib, va)
    j = torch.randint(0, d, (count,), generator=gen, device="cuda")
    levels = torch.tensor([max(2, v) if v else 33 for v in _levels(rows, d)], device="cuda", dtype=torch.float32)
    step = 1.0 / (levels[j] - 1)
    moved = out[r, j] + torch.where(out[r, j] + step <= 1.0 + 1e-6, step, -step)
    out[r, j] = moved.clamp(0.0, 1.0)
    return out


def _problem(case, gen, pool_rows, near=0.0, noise=1e-3):
    batch, n, d, rows = case.get("batch", 1), case["n"], case["d"], case["rows"]
    X = torch.stack([_draw_rows(gen, rows, n + case.get("q", 0), d) for _ in range(batch)])
    y, truth = zip(*[_response(gen, X[g], noise) for g in range(batch)])
    ell = torch.rand((batch, d), generator=gen, device="cuda") * 0.9 + 0.1
    pool = torch.empty((batch, pool_rows, d), device="cuda")
    for g in range(batch):
        pool[g] = _draw_rows(gen, rows, pool_rows, d)
        if near:
            count = int(near * pool_rows)
            at = torch.randperm(pool_rows, generator=gen, device="cuda")[:count]
            pool[g, at] = _neighbours(gen, X[g], rows, count)
    return X.contiguous(), torch.stack(y).contiguous(), ell, pool, truth


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    kind = case["kind"]
    # lengthscales that a fit would choose grow with the number of features; the literal ones keep rows apart
    wide = math.sqrt(max(1.0, case["d"] / 6.0))
    if kind == "score":
        X, y, ell, pool, _ = _problem(case, gen, case["m"], case["near"])
        ell = ell.cpu().numpy() * (wide if case["near"] else 1.0)
        state = {"case": case, "gp": r3.r3_gp_fit(X, y, ell, 1.0, 1e-3), "pool": pool}
        if case["host"]:
            b, m, k = case["batch"], case["m"], case["k"]
            state["pool"] = pool.cpu().pin_memory()
            state["out"] = [torch.empty((b, m), pin_memory=True) for _ in range(3)] + [
                torch.empty((b, k), dtype=torch.int32, pin_memory=True), torch.empty((b, k), pin_memory=True)]
        return state
    if kind == "round":
        X, y, ell, pool, _ = _problem(case, gen, case["m"])
        n = case["n"]
        return {"case": case, "X": X[:, :n].contiguous(), "y": y[:, :n].contiguous(), "Xnew": X[:, n:].contiguous(),
                "ynew": y[:, n:].contiguous(), "ell": ell.cpu().numpy() * wide, "pool": pool,
                "watch": torch.stack([_draw_rows(gen, case["rows"], 256, case["d"]) for _ in range(case["batch"])])}
    if kind == "tune":
        X, y, _, _, _ = _problem(case, gen, 1, noise=1e-2)
        return {"case": case, "X": X, "y": y, "ell": [[wide] * case["d"]] * case["batch"]}
    if kind == "search":
        X, y, ell, pool, truth = _problem(case, gen, case["m"])
        return {"case": case, "X": X[0, :case["n"]].contiguous(), "y": y[0, :case["n"]].contiguous(),
                "ell": ell[0].cpu().numpy() * wide, "pool": pool[0], "truth": truth[0]}
    X, y, _, pool, _ = _problem(case, gen, case["m"])
    levels = _levels(case["rows"], case["d"])
    # two admissible values: a categorical switch; more: ordinal, declared as a grid where the program knows it
    kinds = [2 if v == 2 else (-v if case["grid"] and 2 < v <= 64 else 0) for v in levels]
    return {"case": case, "X": X[0], "y": y[0], "pool": pool[0], "levels": kinds}


# ------------------------------------------------------------------------------------------------ the pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "score":
        if case["host"]:
            return r3.r3_gp_score_topk_host(state["gp"], state["pool"], case["k"], state["out"])
        return r3.r3_gp_score_topk(state["gp"], state["pool"], case["k"])
    if kind == "round":
        gp = r3.r3_gp_fit(state["X"], state["y"], state["ell"], 1.0, 1e-3)
        r3.r3_gp_append(gp, state["Xnew"], state["ynew"])
        idx, ei, _ = r3.r3_gp_propose(gp, state["pool"], case["q"])
        mu, sigma, _ = r3.r3_gp_score(gp, state["watch"])
        r3.r3_gp_check(gp)
        gp.close()
        return idx, ei, mu, sigma
    if kind == "tune":
        gp = r3.r3_gp_fit(state["X"], state["y"], state["ell"], 1.0, 0.05)
        ell, sf2, sn2, lml, _ = r3.r3_gp_optimize(gp, max_evals=case["evals"], gtol=1e-3)
        gp.close()
        return ell, sf2, sn2, lml
    if kind == "search":
        seen = []

        def replay(x):
            rows = torch.from_numpy(x).cuda()
            y = state["truth"](rows).cpu().numpy()
            seen.append((x, y))
            return y, [True] * len(y)

        found = r3.r3_bo_run(state["X"], state["y"], state["ell"], 1.0, 1e-3, state["pool"], replay, q=case["q"],
                             max_rounds=case["rounds"])
        return found["best_x"], found["best_y"], [x for x, _ in seen], [y for _, y in seen]
    tpe = r3.r3_tpe_fit(state["X"], state["y"], state["levels"])
    score = r3.r3_tpe_score(tpe, state["pool"])
    idx, val = r3.r3_topk(score, case["k"])
    r3.r3_tpe_check(tpe)
    tpe.close()
    return score, idx, val


# ------------------------------------------------------------------------------------------------ work and tolerance
def _fit_flops(n, d):
    return n ** 3 / 3.0 + n ** 3 / 3.0 + 3.0 * n * n * d / 2.0   # factor, inverse factor, Gram matrix (lower half)


def work(case):
    kind, n, d = case["kind"], case["n"], case["d"]
    b = case.get("batch", 1)
    if kind == "score":
        m = case["m"]
        return {"bytes": b * (4.0 * m * (d + 3) + 4.0 * n * (n + 1) / 2 + 4.0 * n * d + 8.0 * case["k"]),
                "flops": b * m * (2.0 * n * d + float(n) * n)}
    if kind == "round":
        m, q = case["m"], case["q"]
        t = n + q
        return {"bytes": b * 4.0 * (t * (d + 1) + m * d + 256 * d),
                "flops": b * (_fit_flops(n, d) + 2.0 * q * n * n + (m + 256) * (2.0 * t * d + float(t) * t))}
    if kind == "tune":   # an evaluation: factor, inverse, K^-1 and the pair sums of the gradient
        return {"bytes": b * 4.0 * n * (d + 1),
                "flops": b * case["evals"] * (_fit_flops(n, d) + n ** 3 / 3.0 + 3.0 * n * n * d / 2.0)}
    if kind == "search":
        total, q = 0.0, case["q"]
        for r in range(case["rounds"]):
            t = n + r * q
            total += (case["m"] - r * q) * (2.0 * t * d + float(t) * t) + 2.0 * q * t * t
        return {"bytes": 4.0 * (case["m"] * d * case["rounds"] + n * d), "flops": total + _fit_flops(n, d)}
    m = case["m"]
    # components that differ: at most one per admissible value, set and kind of bandwidth (inside or end of a run)
    terms = sum(0 if v == 2 or (case["grid"] and 2 < v <= 64) else (min(n + 2, 4 * v) if v else n + 2)
                for v in _levels(case["rows"], d))
    return {"bytes": 4.0 * (n * (d + 1) + m * (d + 1)), "flops": 5.0 * m * terms + 2.0 * m * d}


def tolerance(case):
    kind = case["kind"]
    if kind in ("score", "round"):
        # FP32-grade scoring.  Four times what the tensor-core and CUDA-core engines differ by on the listed and on
        # drawn cases (1.1e-5 and 9.5e-5, both in means that are sums of almost cancelling terms); near ties of the
        # selection may change places.
        return {"rel": 5e-5, "max": 4e-4, "differ": 0.01}
    if kind in ("tune", "search"):
        # FP64 throughout, results rounded to FP32 at the end: the order of the history changes at most a last bit
        return {"rel": 1e-6, "max": 1e-5}
    # FP32 sums of logarithms: an absolute error near 1e-5 in scores of some tens
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
