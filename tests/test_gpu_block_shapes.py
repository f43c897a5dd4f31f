"""Block FGMRES where its kernels change: more than 8 columns (the 16-column kernels, a second column
group), grids whose point count is no multiple of a tile or below one, more than 64 rows (several
row chunks) and more than 256 (coefficients keep fewer bits).

FP64: iterates against the oracle's block FGMRES to 1e-11 (rounding, 2^-53, times some 300 rows and a
growth of two digits).  Mixed mode, whose cycles round to FP32: the least-squares residual of the
block Arnoldi relation equals the true residual of the iterate, which holds for any preconditioner as
long as the basis, its FP32 newest block and the coefficients belong together; the operator on FP32
vectors carries 48 bits, so 1e-9 of the right-hand side."""
import numpy as np
import pytest

import workloads as W
from oracle import block_fgmres as BF
from oracle import elastic, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("n,s,steps", [((20, 20), 8, 12), ((36, 20), 9, 8), ((64, 36), 16, 18), ((8, 8), 4, 5)])
def test_iterates(n, s, steps):
    p = W.random_medium(n, 7, abc=2)
    S = elastic.from_problem(p)
    b = np.stack([W.random_vector(n, 80 + q) for q in range(s)])
    d_b = torch.from_numpy(b).cuda()
    pc = precond.multigrid(S, 2, precond.default_alpha(2))
    Mb = lambda V: np.column_stack([pc.apply(V[:, c]) for c in range(V.shape[1])])
    ref = BF.block_fgmres(lambda V: S.H @ V, np.column_stack([W.padded_to_compact(v, n) for v in b]), Mb, restart=20,
                          rtol=1e-15, maxit=steps)
    for precision in (bah.BAH_FP64, bah.BAH_MIXED):
        sv = bah.Solver.from_problem(p, precision=precision, levels=2, restart=20, maxit=steps, rhs_block=s, block_krylov=1)
        x, _, stats = sv.solve(d_b, rtol=1e-15)
        x = x.cpu().numpy()
        sv.close()
        for q in range(s):
            assert stats[q]["iters"] == steps
            got = W.padded_to_compact(x[q], n)
            if precision == bah.BAH_FP64:
                assert np.linalg.norm(got - ref.X[:, q]) <= 1e-11 * np.linalg.norm(ref.X[:, q]), q
            bq = W.padded_to_compact(b[q], n)
            true = np.linalg.norm(bq - S.H @ got) / np.linalg.norm(bq)
            assert abs(true - stats[q]["relres_est"]) <= 1e-9, (precision, q, true, stats[q])
