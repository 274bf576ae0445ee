"""The fan kernel (FP64 quadrotor, 8 to 32 lanes per node, an instance over a
cluster) against the FP64 oracle at 1e-9 (normwise, floor 1, as
test_gpu_parity.py): the batch sizes at which its lanes change, horizons around
the CTAs' shares of nodes, obstacle counts around the lanes, and the call beyond
its batches, which keeps the lane kernel."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402

TOL = 1e-9


def rel(a, b):
    return float(np.abs(a - b).max() / max(1.0, np.abs(b).max()))


def check(B, N, obs, **st):
    n, o = (N, N) if np.isscalar(N) else N, (obs, obs) if np.isscalar(obs) else obs
    prob = W.quad_box(B, seed=13, N_range=n, obs_range=o,
                      settings=dict(scp_iters=3, admm_iters=25, stop=0, rho_eq=10.0, rho_dyn=10.0, rho_geo=10.0, **st))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    x, u = s.scp_solve()
    state = s.state_export().cpu().numpy()
    torch.cuda.synchronize()
    st = s.stats_host()
    xr, ur, sr, _ = oracle.scp_solve(prob)
    np.testing.assert_array_equal(st["scp_iters"], sr[:, 7].astype(int))
    assert rel(x.cpu().numpy(), xr) <= TOL and rel(u.cpu().numpy(), ur) <= TOL
    assert np.isfinite(state).all()
    s.close()


# 32 lanes per node: 4 nodes per CTA, up to 16 CTAs, then more nodes each
@pytest.mark.parametrize("N", [1, 2, 3, 4, 7, 8, 31, 63, 64, 65, 126, 127])
def test_one_instance(N):
    check(1, N, 3)


# 16 lanes: 8 nodes per CTA, up to 8 CTAs
@pytest.mark.parametrize("N", [1, 7, 8, 15, 16, 63, 64, 127])
def test_a_few_instances(N):
    check(3, N, 5)


# 8 lanes: 16 nodes per CTA, up to 8 CTAs
@pytest.mark.parametrize("N", [1, 15, 16, 31, 32, 127])
def test_more_instances(N):
    check(20, N, 4)


@pytest.mark.parametrize("B,obs", [(1, 0), (1, 1), (1, 33), (3, 16), (3, 17), (20, 0), (20, 7), (20, 8), (20, 9), (20, 64)])
def test_obstacle_counts(B, obs):
    check(B, 12, obs)


@pytest.mark.parametrize("iters", [1, 2, 3])
@pytest.mark.parametrize("B", [1, 3, 20])
def test_short_admm_calls(B, iters):
    # the last iteration (residuals) is the first, the one after it, ...
    prob = W.quad_box(B, seed=14, N_range=(40, 40), obs_range=(6, 6),
                      settings=dict(scp_iters=4, admm_iters=iters, stop=0, rho_eq=10.0, rho_dyn=10.0, rho_geo=10.0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    xr, ur, sr, _ = oracle.scp_solve(prob)
    assert rel(x.cpu().numpy(), xr) <= TOL and rel(u.cpu().numpy(), ur) <= TOL
    st = s.stats_host()
    assert np.all(np.abs(st["primal_res"] - sr[:, 3]) <= TOL * np.maximum(1.0, sr[:, 3]))
    assert np.all(np.abs(st["dual_res"] - sr[:, 4]) <= TOL * np.maximum(1.0, sr[:, 4]))
    s.close()


def test_uneven_batch_and_the_batch_beyond():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check(sms, (3, 60), (0, 12))
    check(sms + 1, (3, 30), (0, 6))


# both sides of the rule that chooses between the fan and the lane kernel
@pytest.mark.parametrize("B,N", [(152, 31), (152, 32), (100, 40), (100, 60), (128, (20, 60)), (130, (60, 70))])
def test_batches_around_the_choice_of_kernel(B, N):
    check(B, N, 2)
