"""The autotuner does not choose between two timings of one program: a launch switch that changes
nothing for a batch (the cluster multigrid above three right-hand sides or with a larger coarsest
level, either switch in FP64 or 3-D) shares the default's timing."""
import os
import re

import workloads as W
from paper_2411_15897_gb300 import autotune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(monkeypatch, info, precision=1, problem=None):
    calls = []

    def noisy(problem, rb, env, opts, iters):
        calls.append((rb, tuple(sorted(env.items()))))
        return 1.0 / rb - 1e-6 * len(calls)            # every later timing a little better

    monkeypatch.setattr(autotune, "time_batch", noisy)
    monkeypatch.setattr(autotune, "_default_info", lambda p, o: info)
    p = problem or W.layered(64, 32, 4, seed=23, abc=6, nsrc=8, src_spacing=6)
    c = autotune.tune(p, nsrc=8, opts={"precision": precision}, measure=autotune.time_batch, device="test")
    return c, calls


def names(calls, rb):
    return [dict(e) for r, e in calls if r == rb]


def test_cluster_is_timed_only_where_it_runs(monkeypatch):
    c, calls = run(monkeypatch, {"levels": 6, "cluster_level": 2})
    for rb in (1, 2):
        assert len(names(calls, rb)) == 3
    for rb in (4, 8):
        assert names(calls, rb) == [{}, {"BAH_STAGED": "0"}]
        assert c.table[f"{rb}/no-cluster-mg"] == c.table[f"{rb}/default"]
    assert c.variant != "no-cluster-mg" and c.rhs_block == 8
    # every level below the first in the cluster: no Galerkin sweep outside it up to three right-hand sides
    _, calls = run(monkeypatch, {"levels": 4, "cluster_level": 1})
    assert names(calls, 1) == [{}, {"BAH_SMEM_MG": "0"}]
    # no cluster at all: a coarsest level above 256 points
    _, calls = run(monkeypatch, {"levels": 4, "cluster_level": 0})
    assert all({"BAH_SMEM_MG": "0"} not in names(calls, rb) for rb in (1, 2, 4, 8))


def test_one_program_in_fp64_and_3d(monkeypatch):
    c, calls = run(monkeypatch, {"levels": 4, "cluster_level": 0}, precision=0)
    assert len(calls) == len(autotune.candidates(8)) and c.variant == "default"
    p3 = W.random_medium((16, 8, 8), 3)
    c, calls = run(monkeypatch, {"levels": 3, "cluster_level": 0}, problem=p3)
    assert len(calls) == len(autotune.candidates(8)) and c.variant == "default"


def test_limit_is_the_library_s():
    src = open(os.path.join(ROOT, "paper_2411_15897_gb300", "csrc", "bah_internal.cuh")).read()
    assert int(re.search(r"kClusterRhs = (\d+);", src).group(1)) == autotune.CLUSTER_RHS
