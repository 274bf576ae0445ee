"""The 3-DOF Mars sets of the FP32 path, computed without branches, against the
FP64 oracle with every choice of sets on and off, around whole warps of nodes.

Tolerance: the FP32 path's 1e-4 (normwise, floor 1) after equal iteration
counts, as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402

TOL = 1e-4


def rel(a, b):
    return float(np.abs(a - b).max() / max(1.0, np.abs(b).max()))


@pytest.mark.parametrize("lanes", [1, 2])
@pytest.mark.parametrize("N", [2, 31, 32, 95])
def test_mars_sets_on_and_off(N, lanes):
    # one instance for each choice of the lower thrust bound, the thrust ball and the glide-slope cone
    prob = W.mars_batch(8, seed=5, N=N, settings=dict(scp_iters=3, admm_iters=30, stop=0))
    prob.sets = prob.sets.copy()
    for b in range(8):
        for k in range(3):
            if b >> k & 1:
                prob.sets[b, k] = 0.0
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    ucn.ucn_problem_set_lanes(s.handle, lanes)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    xr, ur, _, _ = oracle.scp_solve(prob)
    assert rel(x.cpu().numpy(), xr) <= TOL and rel(u.cpu().numpy(), ur) <= TOL
    s.close()
