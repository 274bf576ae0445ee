"""FP64 quadrotor batches on both sides of the rule that chooses between the fan and
the lane kernel (records of the latter in shared memory, 41 nodes, and in global
memory), against the FP64 oracle at 1e-9 as in test_gpu_fan.py."""
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402

TOL = 1e-9


@pytest.mark.parametrize("B,N,obs", [(69, 40, 10), (76, 40, 10), (140, 63, 3), (152, 63, 3), (104, 100, 4), (106, 100, 4),
                                     (130, (40, 120), 4), (152, (40, 120), 30)])
def test_both_sides_of_the_rule(B, N, obs):
    prob = W.quad_box(B, seed=17, N_range=N if isinstance(N, tuple) else (N, N), obs_range=(obs, obs),
                      settings=dict(scp_iters=2, admm_iters=15, stop=0, rho_eq=10.0, rho_dyn=10.0, rho_geo=10.0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    xr, ur, _, _ = oracle.scp_solve(prob)
    assert oracle.rel_err(x.cpu().numpy(), xr) <= TOL and oracle.rel_err(u.cpu().numpy(), ur) <= TOL
    s.close()
