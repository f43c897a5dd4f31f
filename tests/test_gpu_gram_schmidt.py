"""The block fixed-point Gram-Schmidt at the sizes where it can go wrong:
vectors shorter than one 256-entry tile, partial last tiles, one row, row
groups of every size up to eight and several groups, more than 32 rows (the
coefficients keep one bit less), and batches.  FGMRES iterates in FP64 mode
against the oracle's FGMRES (modified Gram-Schmidt in FP64)."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, fgmres, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("n,levels,restart,steps", [
    ((8, 8), 2, 20, 1), ((8, 8), 2, 20, 6), ((12, 10), 2, 9, 9), ((24, 20), 2, 17, 21), ((64, 32), 3, 40, 39),
    ((64, 32), 3, 64, 60),
])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_iterates_match_oracle(n, levels, restart, steps, nrhs):
    p = W.random_medium(n, 11, abc=2) if n[0] < 64 else W.layered(64, 32, 3, 5, abc=4)
    S = elastic.from_problem(p)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64, levels=levels, restart=restart, maxit=steps, rhs_block=nrhs)
    b = np.stack([W.point_source(p)] + [W.random_vector(p.n, 60 + k) for k in range(nrhs - 1)])
    x, _, st = s.solve(torch.from_numpy(b).cuda(), rtol=1e-13)
    x = x.cpu().numpy()
    pc = precond.multigrid(S, levels, precond.default_alpha(levels))
    for k in range(nrhs):
        ref = fgmres.fgmres(lambda v: S.H @ v, W.padded_to_compact(b[k], p.n), pc.apply, restart=restart, rtol=1e-13,
                            maxit=steps)
        got = W.padded_to_compact(x[k], p.n)
        # the bound the FP64 iterates are held to elsewhere: rounding times the growth over one cycle
        assert np.linalg.norm(got - ref.x) <= 1e-8 * np.linalg.norm(ref.x), (k, st[k])
    s.close()
