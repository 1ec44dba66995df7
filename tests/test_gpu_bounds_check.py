"""The bounds-checking build of the library (``build.py --check``, ``-DR3_BOUNDS_CHECK``): the scoring kernels, the guard, the
factorisation, the weights, the evidence and the proposal verify the indices of their operands and results (shared memory,
tensor memory and global) and report a violation through a status word instead of faulting.  It stands in for
compute-sanitizer, which is not available where the library is developed.  The small element-by-element cases (several
tiles, ragged tails in every dimension, both engines, multi-pass histories) run against that build in a child process: every
result must still match the oracle and no index check may fire (a fired check makes ``r3_gp_check``, or the fit or proposal
it happened in, fail with the line of the check).  The selection's own kernels and the Parzen estimator have no checks.
"""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_small_cases_pass_under_the_bounds_checking_build():
    from paper_2604_11109_b200 import build
    lib = build.build(check=True)
    assert os.path.exists(lib)
    env = dict(os.environ, R3_LIB_VARIANT="check")
    which = subprocess.run([sys.executable, "-c", "from paper_2604_11109_b200 import binding as b; b.load(); print(b.LIB_PATH)"],
                           cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert which.stdout.strip().endswith("libr3gp_check.so"), which.stdout + which.stderr
    run_checked(["test_gpu_parity.py", "test_gpu_failure_paths.py"],
                "small_cases or near_observations or random_shapes or paired or wait_that_runs_out or two_live")


def run_checked(files, sel):
    env = dict(os.environ, R3_LIB_VARIANT="check")
    r = subprocess.run([sys.executable, "-m", "pytest", *(os.path.join(ROOT, "tests", f) for f in files), "-m", "gpu", "-x",
                        "-q", "-k", sel, "-p", "no:cacheprovider"], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=1500)
    tail = (r.stdout + r.stderr)[-3000:]
    assert r.returncode == 0, tail
    assert " passed" in r.stdout and "failed" not in r.stdout, tail


@pytest.mark.parametrize("files,sel", [
    (["test_gpu_lml.py"], "random_problems or half_empty"),
    (["test_gpu_factor.py", "test_gpu_append.py"], "edges or weights or append"),
    (["test_gpu_propose.py", "test_gpu_rescue.py"], "propos or greedy or pick or recomputed"),
])
def test_fits_evidence_proposals_and_rescues_under_the_bounds_checking_build(files, sel):
    run_checked(files, sel)
