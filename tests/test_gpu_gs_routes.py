"""Gram-Schmidt at the sizes where its kernels change: partial sums added by the dot kernel's
last CTA or by a kernel of their own (61 and 65 CTAs), one tile per CTA with the deep and the
shallow ring (257 and 315 tiles), and one tile per warp (630 tiles in a batch of two).  FGMRES
iterates in FP64 mode against the oracle's FGMRES; the bound is the one the FP64 iterates are
held to in test_gpu_gram_schmidt.py."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, fgmres, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("n,nrhs", [((144, 144), 1), ((144, 152), 1), ((160, 168), 1), ((160, 168), 2)])
def test_iterates_match_oracle(n, nrhs):
    levels, steps = 4, 7
    p = W.random_medium(n, 12, abc=4)
    S = elastic.from_problem(p)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64, levels=levels, restart=5, maxit=steps, rhs_block=nrhs)
    b = np.stack([W.point_source(p)] + [W.random_vector(p.n, 70 + k) for k in range(nrhs - 1)])
    x, _, st = s.solve(torch.from_numpy(b).cuda(), rtol=1e-13)
    x = x.cpu().numpy()
    pc = precond.multigrid(S, levels, precond.default_alpha(levels))
    for k in range(nrhs):
        ref = fgmres.fgmres(lambda v: S.H @ v, W.padded_to_compact(b[k], p.n), pc.apply, restart=5, rtol=1e-13, maxit=steps)
        got = W.padded_to_compact(x[k], p.n)
        assert np.linalg.norm(got - ref.x) <= 1e-8 * np.linalg.norm(ref.x), (k, st[k])
    s.close()
