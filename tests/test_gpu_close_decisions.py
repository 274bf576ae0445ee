"""6-DOF landers of the Monte-Carlo batch whose FP32 solves meet an acceptance
test (Sec. III-A) that their last bits can turn: the solve must take the FP64
oracle's decisions on them.  One turned decision leaves the first four 1e-5 to
5e-3 off; the fifth's merits are not close.

Tolerance: the FP32 path's 1e-4 (normwise, floor 1), as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402

TOL = 1e-4


# (seed of the batch of 1000, instance)
@pytest.mark.parametrize("seed,b", [(7, 451), (28, 870), (13, 482), (8, 398), (7, 0)])
def test_six_dof_lander_takes_the_oracles_decisions(seed, b):
    st = dict(scp_iters=40, admm_iters=100, stop=0, rho_eq=1.0, rho_dyn=1.0, rho_geo=1.0, defect_tol=1e-2)
    prob = W.mars6_batch(1000, seed=seed, N=30, tf=5.0, settings=st).subset([b])
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    xr, ur, sr, _ = oracle.scp_solve(prob)
    assert int(s.stats_host()["accept_mask"][0]) == int(sr[0, 9])
    assert oracle.rel_err(x.cpu().numpy(), xr) <= TOL and oracle.rel_err(u.cpu().numpy(), ur) <= TOL
    s.close()
