"""The dense coarsest solve in block fixed point: a one-level hierarchy is that
solve alone, compared with the oracle's dense solve of the same block at point
counts around a warp's and a row block's multiples, and above 256 points, where
the right-hand side gives up bits for the longer sums."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, precond
from oracle import multigrid as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("n", [(4, 4), (11, 9), (16, 16), (21, 13), (40, 30)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_one_level_cycle_is_the_dense_solve(n, prec):
    p = W.random_medium(n, 5, abc=1)
    S = elastic.from_problem(p)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64 if prec == "fp64" else bah.BAH_MIXED, levels=1)
    pc = precond.multigrid(S, 1, precond.default_alpha(1), precision="fp64")
    # FP64: rounding times the blocks' condition numbers (below 1e4 here); mixed: the right-hand
    # side and the result are rounded to FP32 once each
    tol = 1e-11 if prec == "fp64" else 1e-3
    rng = np.random.default_rng(3)
    for b in range(3):
        v = rng.standard_normal(p.shape) + 1j * rng.standard_normal(p.shape)
        if b == 0:
            v[:, 0] = 0
        if b == 1:
            v[0, :] = 0
        x = s.block_cycle(b, torch.from_numpy(v).cuda()).cpu().numpy()
        cut = (lambda a: a[:, 1:] if b == 0 else (a[1:, :] if b == 1 else a))
        ref = mg.cycle(pc.hier[b], cut(v).ravel())
        got = cut(x).ravel()
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), b
    s.close()
