"""FP32 scenario groups around the row kernel's 96 nodes: with at most one
obstacle the records of 97 to 99 nodes still fit a CTA's shared memory, and such
groups are solved as the shorter ones are.

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


def group(N, obs, K):
    return W.scenario_mpc(2, K, seed=3, N=N, n_obs=obs, settings=dict(scp_iters=3, admm_iters=30, stop=0))


@pytest.mark.parametrize("N,obs,K", [(95, 0, 2), (95, 1, 2), (96, 0, 2), (96, 1, 3), (98, 0, 2), (98, 1, 18)])
def test_groups_around_96_nodes(N, obs, K):
    prob = group(N, obs, K)
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    xr, ur, sr, _ = oracle.scp_solve(prob)
    np.testing.assert_array_equal(s.stats_host()["scp_iters"], sr[:, 7].astype(int))
    assert oracle.rel_err(x.cpu().numpy(), xr) <= TOL and oracle.rel_err(u.cpu().numpy(), ur) <= TOL
    s.close()


def test_longer_groups_stay_refused():
    with pytest.raises(ucn.UcnError, match="shared memory"):
        ucn.Solver(group(99, 1, 2), precision=ucn.UCN_PREC_FP32_REFINE)
