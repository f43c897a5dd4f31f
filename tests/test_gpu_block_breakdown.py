"""Block FGMRES that breaks down: on a 4 x 4 grid (40 unknowns) a block of 16 columns has no 16
new directions left at its second step, so CholQR fails there while a third step is already
queued.  The call must return with its stream idle, so that the next call on the same context,
from another stream, has the workspace to itself."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("precision", [bah.BAH_FP64, bah.BAH_MIXED])
def test_failed_block_solve_leaves_the_stream_idle(precision):
    n, s = (4, 4), 16
    p = W.random_medium(n, 7, abc=1)
    opts = dict(precision=precision, levels=1, restart=8, rhs_block=s, block_krylov=1)
    b = torch.from_numpy(np.stack([W.random_vector(n, 80 + k) for k in range(s)])).cuda()

    def solve(solver, stream):
        with torch.cuda.stream(stream):
            x = torch.zeros_like(b)
            status, stats = bah.bah_solve(solver.ctx, b, x, s, 1e-14, stream)
        stream.synchronize()
        return x.cpu().numpy(), status, stats

    short = bah.Solver.from_problem(p, **opts, maxit=1)
    ref, _, _ = solve(short, torch.cuda.current_stream())
    sv = bah.Solver.from_problem(p, **opts, maxit=6)
    torch.cuda.synchronize()
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    status, _ = bah.bah_solve(sv.ctx, b, x, s, 1e-14, first)
    idle = first.query()
    torch.cuda.synchronize()
    assert status == bah.BAH_ERR_NONFINITE
    assert idle
    # the context still solves: one step to the tolerance that step reaches, from another stream
    with torch.cuda.stream(second):
        y = torch.zeros_like(b)
        st2, stats = bah.bah_solve(sv.ctx, b, y, s, 0.5, second)
    second.synchronize()
    assert st2 == bah.BAH_OK and all(q["iters"] == 1 for q in stats)
    np.testing.assert_array_equal(y.cpu().numpy(), ref)
