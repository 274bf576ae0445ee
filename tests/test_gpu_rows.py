"""The row kernel (FP32, four lanes per node, matrices in registers) against the
FP64 oracle at the sizes where its work splits: the register classes and the
CTAs of a cluster (64, 96, 128, ... nodes), warps with idle lanes, obstacle
counts around the four lanes, one-node-per-CTA remainders, scenario groups, and
the stand-alone ADMM call cold and continued.

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
SHORT = dict(scp_iters=3, admm_iters=30, stop=0)


def rel(a, b):
    return float(np.abs(a - b).max() / max(1.0, np.abs(b).max()))


def check(prob):
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    st = s.stats_host()
    xr, ur, sr, _ = oracle.scp_solve(prob)
    np.testing.assert_array_equal(st["scp_iters"], sr[:, 7].astype(int))
    assert rel(x.cpu().numpy(), xr) <= TOL and rel(u.cpu().numpy(), ur) <= TOL
    s.close()


def quad(N, obs, B=2, **st):
    n, o = (N, N) if np.isscalar(N) else N, (obs, obs) if np.isscalar(obs) else obs
    return W.quad_box(B, seed=11, N_range=n, obs_range=o, settings=dict(SHORT, rho_eq=10.0, rho_dyn=10.0, rho_geo=10.0, **st))


@pytest.mark.parametrize("N", [1, 2, 7, 62, 63, 64, 94, 95, 96, 97, 126, 127])
def test_quadrotor_horizons(N):
    check(quad(N, 3))


@pytest.mark.parametrize("obs", [0, 1, 3, 4, 5, 30, 64])
def test_quadrotor_obstacle_counts(obs):
    check(quad(33, obs))


def test_uneven_batch_over_a_cluster():
    # short instances leave whole CTAs of their cluster without a node
    check(quad((3, 120), (0, 30), B=7))


def test_uneven_batch_while_a_capture_holds_its_streams():
    # the parts' streams belong to the capture until it ends: a solve on another
    # stream meanwhile runs them on its own, with the same bits
    s = ucn.Solver(quad((20, 120), (0, 9), B=9), precision=ucn.UCN_PREC_FP32_REFINE)
    x0, u0 = s.tensor(s.prob.xguess), s.tensor(s.prob.uguess)
    s.scp_solve(x0, u0)
    torch.cuda.synchronize()
    ref = s.x_out.clone()
    s.x_out.zero_()
    other, held, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(held):
        graph.capture_begin(capture_error_mode="relaxed")
        s.scp_solve(x0, u0, stream=held)
        s.scp_solve(x0, u0, stream=other)
        graph.capture_end()
    torch.cuda.synchronize()
    assert torch.equal(s.x_out, ref)
    s.x_out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(s.x_out, ref)
    s.close()


@pytest.mark.parametrize("N", [1, 30, 63, 64, 127, 128, 200])
def test_quaternion_quadrotor_horizons(N):
    check(W.quat_study(2, seed=5, N=N, tf=0.12 * N, settings=dict(SHORT)))


@pytest.mark.parametrize("N", [1, 15, 63, 64, 129])
def test_six_dof_lander_horizons(N):
    check(W.mars6_batch(2, seed=7, N=N, tf=N / 6.0, settings=dict(SHORT)))


def test_six_dof_lander_without_some_sets():
    prob = W.mars6_batch(4, seed=8, N=12, tf=2.0, settings=dict(SHORT))
    prob.sets[0, 0] = 0.0            # no thrust lower bound
    prob.sets[1, 2] = prob.sets[1, 3] = 0.0   # no cones
    prob.sets[2, 4] = prob.sets[2, 5] = 0.0   # no tilt, no rate bound
    prob.sets[3, :] = 0.0
    check(prob)


@pytest.mark.parametrize("N,K", [(9, 3), (63, 2), (64, 2), (84, 2)])
def test_scenario_groups(N, K):
    check(W.scenario_mpc(2, K, seed=3, N=N, n_obs=5, settings=dict(SHORT)))


def test_a_group_beyond_the_record_limit_stays_refused():
    with pytest.raises(ucn.UcnError, match="shared memory"):
        ucn.Solver(W.scenario_mpc(2, 2, seed=3, N=95, n_obs=5, settings=dict(SHORT)), precision=ucn.UCN_PREC_FP32_REFINE)


@pytest.mark.parametrize("make", [lambda: quad(40, 6), lambda: quad(95, 6), lambda: quad((20, 110), (1, 9), B=3),
                                  lambda: W.quat_study(2, N=20, tf=2.4), lambda: W.quat_study(2, N=70, tf=8.4),
                                  lambda: W.mars6_batch(2, N=20, tf=3.4), lambda: W.mars6_batch(2, N=66, tf=11.0)])
def test_admm_call_cold_and_continued(make):
    prob = make()
    rng = np.random.default_rng(3)
    x = prob.xguess + 0.02 * rng.standard_normal(prob.xguess.shape)
    u = prob.uguess + 0.02 * rng.standard_normal(prob.uguess.shape)
    A = np.zeros((prob.total_u, prob.nx, prob.nx)); B = np.zeros((prob.total_u, prob.nx, prob.nu)); d = np.zeros((prob.total_u, prob.nx))
    for b in range(prob.batch):
        x[prob.xoff[b]] = prob.xinit[b]
        for i in range(int(prob.N[b])):
            g = prob.uoff[b] + i
            A[g], B[g], d[g], _ = oracle.linearize(prob.model, prob.params[b], prob.dt[b], x[prob.xoff[b] + i], u[g])
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    lin = [s.tensor(v) for v in (A, B, d)]
    args = (s.tensor(x), s.tensor(u), *lin, s.tensor(np.full(prob.batch, 0.7)))
    s.admm_solve(*args, 25, warm=False)
    xh, uh, res, status = s.admm_solve(*args, 20, warm=True)
    state = s.state_export().cpu().numpy()
    torch.cuda.synchronize()
    assert (status.cpu().numpy() == 0).all()
    mb, off = oracle.maxblk(prob), 0
    for b in range(prob.batch):
        N, xo, uo = int(prob.N[b]), prob.xoff[b], prob.uoff[b]
        q = (x[xo:xo + N + 1], u[uo:uo + N], A[uo:uo + N], B[uo:uo + N], d[uo:uo + N], 0.7)
        ref, _, _ = oracle.problem_admm(prob, b, *q, 25)
        ref, r, _ = oracle.problem_admm(prob, b, *q, 20, state=ref)
        size = oracle.state_size(N, prob.nx, prob.nu, mb)
        assert rel(state[off:off + size], ref) <= TOL
        un = oracle.unpack_state(ref, N, prob.nx, prob.nu, mb)
        assert rel(xh.cpu().numpy()[xo:xo + N + 1], un["xh"]) <= TOL and rel(uh.cpu().numpy()[uo:uo + N], un["uh"]) <= TOL
        assert rel(res.cpu().numpy()[b], np.array(r)) <= TOL
        off += size
    s.close()
