"""The fused level-0 visits at grid sizes around their tiles (30 x 14 coarse
points down; 62, 60 or 58 columns by 30, 28 or 26 rows up, for one, two or three
sweeps): one cycle per block on two levels against the oracle's cycle, the
points next to the grid's and the tiles' edges included."""
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


@pytest.mark.parametrize("n", [(8, 8), (58, 26), (60, 28), (62, 30), (64, 32), (122, 34)])
@pytest.mark.parametrize("nu", [(1, 1), (1, 2), (1, 3), (2, 2), (2, 3)])
@pytest.mark.parametrize("prec,intergrid", [("fp64", 0), ("mixed", 0), ("mixed", 1)])
def test_two_level_cycle_matches_oracle(n, nu, prec, intergrid):
    p = W.random_medium(n, 6, abc=2)
    S = elastic.from_problem(p)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64 if prec == "fp64" else bah.BAH_MIXED, levels=2, nu_pre=nu[0],
                                nu_post=nu[1], intergrid=intergrid)
    pc = precond.multigrid(S, 2, precond.default_alpha(2), precision=prec, nu_pre=nu[0], nu_post=nu[1],
                           intergrid="mixed" if intergrid else "bilinear")
    # as for the block cycles elsewhere: FP64 rounding, or FP32 on the oracle's bf16-rounded levels
    tol, tol_max = (1e-10, 1e-9) if prec == "fp64" else (2e-4, 2e-3)
    rng = np.random.default_rng(7)
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
        assert np.abs(got - ref).max() <= tol_max * np.abs(ref).max(), b
        if b < 2:
            assert np.all((x[:, 0] if b == 0 else x[0, :]) == 0)
    s.close()
