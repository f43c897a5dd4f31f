"""Grids with an odd number of points (one multigrid level): every array of a context starts on the
alignment of its entries whatever the point count, the exact-block setup's among them.  Iterates
against the oracle's, with multigrid and with exact blocks (block solves to 1e-12, iterates to 1e-9:
the block residuals enter three times and grow by the conditioning of small shifted blocks)."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, fgmres, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("n", [(5, 5), (9, 7), (33, 21)])
@pytest.mark.parametrize("exact", [False, True])
def test_iterates(n, exact):
    p = W.random_medium(n, 3, abc=2)
    S = elastic.from_problem(p)
    b = W.random_vector(n, 4)
    opts = dict(block_rtol=1e-12, block_maxit=400, block_alpha=0.5) if exact else {}
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64, levels=1, restart=10, maxit=4, **opts)
    x, _, _ = s.solve(torch.from_numpy(b).cuda(), rtol=1e-15)
    s.close()
    # one level: the cycle is the inverse of the shifted blocks
    pc = precond.multigrid(S, 1, 0.5 if exact else precond.default_alpha(1))
    ref = fgmres.fgmres(lambda v: S.H @ v, W.padded_to_compact(b, n), pc.apply, restart=10, rtol=1e-15, maxit=4)
    got = W.padded_to_compact(x.cpu().numpy(), n)
    assert np.linalg.norm(got - ref.x) <= (1e-9 if exact else 1e-11) * np.linalg.norm(ref.x)
