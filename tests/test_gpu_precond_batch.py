"""The preconditioner on several vectors at once borrows its workspace from the flexible basis: one
right-hand side per context, every count of vectors (whole batches, ragged last ones, more than 32,
a workspace for fewer than two), both precisions, in place.  Each vector against the call on it alone
(1e-13 in FP64; in mixed mode the kernels and so the FP32 roundings differ: 2e-5) and one against the
oracle; and a solve before and after has the same bits, so the borrowed memory leaves no trace."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("precision", [bah.BAH_FP64, bah.BAH_MIXED])
@pytest.mark.parametrize("restart", [2, 5, 11, 20])
@pytest.mark.parametrize("n,levels", [((44, 28), 3), ((22, 10), 2)])
def test_vectors_together_and_alone(n, levels, restart, precision):
    p = W.random_medium(n, 17, abc=2)
    S = elastic.from_problem(p)
    mixed = precision == bah.BAH_MIXED
    pc = precond.multigrid(S, levels, precond.default_alpha(levels), precision="mixed" if mixed else "fp64")
    s = bah.Solver.from_problem(p, precision=precision, levels=levels, restart=restart, maxit=2 * restart + 1)
    b = torch.from_numpy(W.point_source(p)).cuda()
    before = s.solve(b, rtol=1e-14)[0].cpu().numpy()
    r = np.stack([W.random_vector(n, 300 + q) for q in range(33)])
    d_r = torch.from_numpy(r).cuda()
    alone = np.stack([s.apply_preconditioner(d_r[q]).cpu().numpy() for q in range(33)])
    ref = pc.apply(W.padded_to_compact(r[0], n))
    got = W.padded_to_compact(alone[0], n)
    assert np.linalg.norm(got - ref) <= (2e-4 if mixed else 1e-11) * np.linalg.norm(ref)
    for k in (2, 5, 33):
        inplace = d_r[:k].clone()
        bah.bah_apply_preconditioner(s.ctx, inplace, inplace, k)
        together = s.apply_preconditioner(d_r[:k])
        assert torch.equal(inplace, together)
        z = together.cpu().numpy()
        for q in range(k):
            assert np.linalg.norm(z[q] - alone[q]) <= (2e-5 if mixed else 1e-13) * np.linalg.norm(alone[q]), (k, q)
    after = s.solve(b, rtol=1e-14)[0].cpu().numpy()
    np.testing.assert_array_equal(after, before)
    s.close()
