"""Where the small levels run: in one cluster's shared memory (mixed mode, up to three
right-hand sides, at most 256 points on the coarsest level) or as level kernels.  The batched
preconditioner on both sides of each line against the oracle, to the mixed-mode bound of
test_gpu_parity.py (2e-4)."""
import numpy as np
import pytest

import workloads as W
from oracle import elastic, precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402


@pytest.mark.parametrize("cycle", ["V", "W"])
@pytest.mark.parametrize("n,levels,cluster", [((64, 32), 4, True), ((64, 64), 3, True), ((68, 68), 3, False)])
def test_batched_preconditioner_matches_oracle(n, levels, cluster, cycle):
    p = W.random_medium(n, 23, abc=4)
    S = elastic.from_problem(p)
    pc = precond.multigrid(S, levels, precond.default_alpha(levels), precision="mixed", cycle=cycle)
    for k in (1, 3, 4):
        s = bah.Solver.from_problem(p, levels=levels, rhs_block=k,
                                    cycle=bah.BAH_CYCLE_W if cycle == "W" else bah.BAH_CYCLE_V)
        assert (s.info["cluster_level"] > 0) == cluster
        r = np.stack([W.random_vector(p.n, 80 + i) for i in range(k)])
        bah.bah_profile_control(s.ctx, 0, True)
        z = s.apply_preconditioner(torch.from_numpy(r).cuda())
        torch.cuda.synchronize()
        calls = bah.bah_profile_read(s.ctx)["classes"]["cluster"]["calls"]
        assert (calls > 0) == (cluster and k <= 3), (k, calls)
        z = z.cpu().numpy()
        for i in range(k):
            ref = pc.apply(W.padded_to_compact(r[i], p.n))
            assert np.linalg.norm(W.padded_to_compact(z[i], p.n) - ref) <= 2e-4 * np.linalg.norm(ref), (k, i)
        s.close()
