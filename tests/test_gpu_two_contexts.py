"""Contexts of different sizes alive at once: the cluster multigrid's shared memory (169 KB per CTA
for 512 x 512, 10 KB for 64 x 64) is asked for per context, and a context keeps solving, with the
same bits, after a smaller or a larger one was created."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


def iterate(s, p):
    x, _, st = s.solve(torch.from_numpy(W.point_source(p)).cuda(), rtol=1e-14)
    return x.cpu().numpy()


@pytest.mark.parametrize("first", ["large", "small"])
def test_a_context_outlives_the_creation_of_another(first):
    probs = {"large": W.layered(512, 512, 6, 2), "small": W.homogeneous(64, 64)}
    opts = dict(precision=bah.BAH_MIXED, maxit=3)
    ref = {}
    for k, p in probs.items():
        s = bah.Solver.from_problem(p, **opts)
        assert s.info["cluster_level"] > 0
        ref[k] = iterate(s, p)
        s.close()
    order = ["large", "small"] if first == "large" else ["small", "large"]
    held = {k: bah.Solver.from_problem(probs[k], **opts) for k in order}
    for k in order + order:
        np.testing.assert_array_equal(iterate(held[k], probs[k]), ref[k])
    for s in held.values():
        s.close()
