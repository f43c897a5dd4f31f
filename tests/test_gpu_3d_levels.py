"""Level kernels of the 3-D cycles at the sizes where their indexing can go wrong: columns that
do not fill a CTA (16- and 32-wide tiles), planes that are no multiple of four, two-point axes,
every parity of the sweeps' ping-pong, and a coarse level whose first sweep the restriction
writes.  One cycle of each block against the FP64 oracle (mixed mode: against the oracle's
bfloat16 stencils).

Tolerances: those of the cycles in test_gpu_3d.py, for the same reasons: 1e-10 in FP64 mode,
2e-4 in mixed mode.
"""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, multigrid as mg, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402

TOL = {"fp64": 1e-10, "mixed": 2e-4}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,levels,cyc,nu", [
    ((4, 4, 4), 2, "V", (1, 1)),
    ((36, 10, 6), 2, "V", (2, 1)),
    ((8, 34, 18), 2, "V", (3, 2)),
    ((68, 8, 12), 3, "W", (2, 2)),
    ((16, 24, 20), 3, "W", (1, 2)),
    ((12, 8, 20), 3, "V", (0, 3)),
])
def test_3d_cycle_at_ragged_sizes(prec, n, levels, cyc, nu):
    p = W.random_medium(n, 77, abc=1, h=(1 / 16, 1 / 14, 1 / 18))
    S = elastic.from_problem(p)
    alpha = precond.default_alpha(levels)
    weights = (0.8, 0.7, 0.4)
    s = bah.Solver.from_problem(p, precision=bah.BAH_FP64 if prec == "fp64" else bah.BAH_MIXED,
                                intergrid=bah.BAH_INTERGRID_MIXED, levels=levels, shift_alpha=alpha,
                                cycle=bah.BAH_CYCLE_V if cyc == "V" else bah.BAH_CYCLE_W, nu_pre=nu[0], nu_post=nu[1],
                                jacobi_w=weights)
    pc = precond.multigrid(S, levels, alpha, intergrid="mixed", precision=prec, cycle=cyc, nu_pre=nu[0], nu_post=nu[1],
                           weights=weights)
    rng = np.random.default_rng(9)
    shp = tuple(reversed(n))
    for q in range(4):
        v = rng.standard_normal(shp) + 1j * rng.standard_normal(shp)
        keep = [slice(None)] * 3
        if q < 3:
            keep[2 - q] = slice(1, None)
            edge = [slice(None)] * 3
            edge[2 - q] = 0
            v[tuple(edge)] = 0
        x = s.block_cycle(q, torch.from_numpy(v).to("cuda"))
        torch.cuda.synchronize()
        x = x.cpu().numpy()
        ref = mg.cycle(pc.hier[q], v[tuple(keep)].ravel())
        got = x[tuple(keep)].ravel()
        assert np.linalg.norm(got - ref) <= TOL[prec] * np.linalg.norm(ref), q
        if q < 3:
            assert np.all(x[tuple(edge)] == 0)
    s.close()
