"""The consensus of a scenario group's first control (FP64 path): after one ADMM
iteration the scenarios' arguments are their exported u_0 (the duals start at
zero), and the accepted first control is their mean, clamped to the common box.

Bound: the mean of K doubles, one rounding per addition and one of the quotient, is
within (K + 1) 2^-53 of the exact one relative to the largest argument.  (The FP32
path re-bases the exported state in floats, which hides the arguments' last bits.)"""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402


@pytest.mark.parametrize("K,lanes", [(3, 4), (16, 4), (16, 1), (18, 4), (64, 4)])
def test_first_control_is_the_mean_of_the_arguments(K, lanes):
    P, N = 24, 12
    prob = W.scenario_mpc(P, K, seed=9, N=N, n_obs=2, settings=dict(scp_iters=1, admm_iters=1, stop=0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    ucn.ucn_problem_set_lanes(s.handle, lanes)
    x, u = s.scp_solve()
    state = s.state_export()
    torch.cuda.synchronize()
    took = s.stats_host()["accepted"].reshape(P, K)[:, 0] == 1
    assert took.any()
    u0 = u.cpu().numpy().reshape(P, K, N, 4)[:, :, 0]
    arg = state.cpu().numpy().reshape(P, K, -1)[:, :, (N + 1) * 12:(N + 1) * 12 + 4].astype(np.longdouble)
    s.close()
    lo = prob.ulo.reshape(P, K, 4).max(1)
    hi = prob.uhi.reshape(P, K, 4).min(1)
    r = prob.settings["tr_init"]
    ub = prob.uguess[prob.uoff].reshape(P, K, 4)
    mean = np.clip(arg.mean(1), np.maximum(lo, (ub - r).max(1)), np.minimum(hi, (ub + r).min(1)))
    big = np.abs(arg).max(1).astype(float)
    bound = (K + 1) * 2.0 ** -53 * big
    assert np.all(np.ptp(u0, axis=1)[took] == 0.0)
    assert np.all(np.abs(u0[:, 0] - mean)[took] <= bound[took])
