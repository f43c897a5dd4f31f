"""H x and H^H x do not read the boundary-normal entries of x (they are no unknowns): a NaN or an
infinity there leaves the product as it is with zeros there, and a non-finite unknown at an end of
the grid reaches the rows of its column of H and no others."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


def solver(n, precision):
    kw = dict(intergrid=bah.BAH_INTERGRID_MIXED) if len(n) == 3 else {}
    p = W.random_medium(n, 21, abc=2)
    return p, bah.Solver.from_problem(p, precision=precision, levels=2, **kw)


@pytest.mark.parametrize("n", [(12, 10), (36, 20), (12, 10, 8), (34, 6, 10)])
@pytest.mark.parametrize("conj", [False, True])
def test_boundary_normal_entries_do_not_count(n, conj):
    p, s = solver(n, bah.BAH_FP64)
    v = W.random_vector(n, 31)
    ref = s.apply_operator(torch.from_numpy(v).cuda(), conj_transpose=conj).cpu().numpy()
    for bad in (np.nan, np.inf, 1e300):
        w = v.copy()
        for a in range(len(n)):
            at = [slice(None)] * len(n)
            at[len(n) - 1 - a] = 0
            w[a][tuple(at)] = bad
        got = s.apply_operator(torch.from_numpy(w).cuda(), conj_transpose=conj).cpu().numpy()
        np.testing.assert_array_equal(got, ref)
    s.close()


@pytest.mark.parametrize("n", [(12, 10), (12, 10, 8)])
def test_nonfinite_unknowns_reach_only_their_rows(n):
    p, s = solver(n, bah.BAH_MIXED)
    S = elastic.from_problem(p)
    d = len(n)
    for comp in range(d + 1):
        for corner in ((-1,) * d, (1,) * d):
            v = W.random_vector(n, 32)
            v[(comp,) + corner] = np.inf
            got = s.apply_operator(torch.from_numpy(v).cuda()).cpu().numpy()
            one = np.zeros_like(v)
            one[(comp,) + corner] = 1.0
            hit = S.H @ W.padded_to_compact(one, n) != 0
            np.testing.assert_array_equal(~np.isfinite(W.padded_to_compact(got, n)), hit)
    s.close()
