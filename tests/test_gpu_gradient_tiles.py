"""The gradient kernel at grid sizes around its 31 x 15-cell tiles (one tile,
one more column or row, partial tiles), against the oracle's gradient."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, gradient as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402
from paper_2411_15897_gb300 import misfit as M  # noqa: E402


@pytest.mark.parametrize("n", [(31, 15), (32, 16), (33, 17), (30, 31), (63, 14)])
@pytest.mark.parametrize("nsrc", [1, 3])
def test_gradient_tiles_match_oracle(n, nsrc):
    p = W.random_medium(n, 4, abc=2)
    S = elastic.from_problem(p)
    B = np.stack([W.point_source(p, (3 + 7 * k, 5)) for k in range(nsrc)])
    Bc = np.column_stack([W.padded_to_compact(b, p.n) for b in B])
    rows = G.receiver_rows(S, [(i, 2) for i in range(n[0])])
    rng = np.random.default_rng(8)
    D = rng.standard_normal((len(rows), nsrc)) + 1j * rng.standard_normal((len(rows), nsrc))
    _, g, X, Y = G.gradient(S, Bc, D, rows)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64)
    Xp, Yp = (np.stack([W.compact_to_padded(A[:, k], p.n) for k in range(nsrc)]) for A in (X, Y))
    gd = torch.zeros(3, S.ncells, dtype=torch.float64, device="cuda")
    bah.bah_gradient(s.ctx, torch.from_numpy(Xp).cuda(), torch.from_numpy(Yp).cuda(), nsrc, gd[0], gd[1], gd[2])
    gh = gd.cpu().numpy()
    for q, prm in enumerate(("lambda", "mu", "rho")):
        # sums of about 10 nsrc products per cell in FP64
        assert np.linalg.norm(gh[q] - g[prm].ravel()) <= 1e-12 * np.linalg.norm(g[prm]), prm
    # the adjoint sources: distinct receivers in parallel
    rec = M.receiver_indices(p.n, 2)
    x = torch.from_numpy(Xp).cuda()
    d = torch.from_numpy(np.ascontiguousarray(D.T)).cuda()
    adj = torch.full_like(x, 7.0)
    mis = torch.empty(nsrc, dtype=torch.float64, device="cuda")
    bah.bah_misfit(s.ctx, x, d, torch.from_numpy(rec).cuda(), rec.size, nsrc, adj, mis)
    ref = np.zeros_like(Xp).reshape(nsrc, -1)
    ref[:, rec] = Xp.reshape(nsrc, -1)[:, rec] - D.T
    assert np.array_equal(adj.cpu().numpy().reshape(nsrc, -1), ref)
    s.close()
