"""What the lanes and CTAs of the row and fan kernels pass to each other: the same
bits whatever the device is doing beside an instance, and on every repetition."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402


def linearised(prob, seed=3):
    """A nominal off the guess and its linearisation."""
    rng = np.random.default_rng(seed)
    x = prob.xguess + 0.02 * rng.standard_normal(prob.xguess.shape)
    u = prob.uguess + 0.02 * rng.standard_normal(prob.uguess.shape)
    x[prob.xoff] = prob.xinit
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    lin = s.linearize(s.tensor(x), s.tensor(u))
    torch.cuda.synchronize()
    s.close()
    return x, u, lin


def admm(prob, x, u, lin, iters):
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    xh, uh, res, status = s.admm_solve(s.tensor(x), s.tensor(u), *lin, s.tensor(np.full(prob.batch, 0.7)), iters)
    torch.cuda.synchronize()
    assert (status.cpu().numpy() == 0).all()
    out = xh.cpu().numpy(), uh.cpu().numpy(), res.cpu().numpy()
    s.close()
    return out


# instances over clusters of two (and four) CTAs, more than the device holds at a
# time: the CTAs of a cluster start while others still run
@pytest.mark.parametrize("make", [lambda: W.quad_box(400, seed=21, N_range=(110, 110), obs_range=(2, 6)),
                                  lambda: W.quat_study(400, seed=22, N=70, tf=8.4),
                                  lambda: W.quat_study(200, seed=23, N=200, tf=24.0)])
def test_admm_over_a_cluster_is_the_same_in_a_full_device_as_alone(make):
    prob = make()
    x, u, lin = linearised(prob)
    xh, uh, res = admm(prob, x, u, lin, 3)
    for b in (0, 1, 137, prob.batch - 1):
        xo, uo, N = prob.xoff[b], prob.uoff[b], int(prob.N[b])
        one = admm(prob.subset([b]), x[xo:xo + N + 1], u[uo:uo + N], [v[uo:uo + N].contiguous() for v in lin], 3)
        np.testing.assert_array_equal(one[0], xh[xo:xo + N + 1])
        np.testing.assert_array_equal(one[1], uh[uo:uo + N])
        np.testing.assert_array_equal(one[2][0], res[b])


def solve(s):
    x, u = s.scp_solve()
    torch.cuda.synchronize()
    return x.cpu().numpy().copy(), u.cpu().numpy().copy(), s.stats_host().copy()


def same(a, b):
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    for f in ("primal_res", "dual_res", "merit", "accept_mask"):
        np.testing.assert_array_equal(a[2][f], b[2][f])


# 32 lanes per node: two lanes share a row of every node, on one CTA boundary and on many
@pytest.mark.parametrize("N", [4, 50, 127])
@pytest.mark.parametrize("iters", [1, 40])
def test_fan_solves_repeat_their_bits(N, iters):
    prob = W.quad_box(2, seed=24, N_range=(N, N), obs_range=(3, 5), settings=dict(scp_iters=3, admm_iters=iters, stop=0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    first = solve(s)
    for _ in range(10):
        same(solve(s), first)
    s.close()


# the 17th row, carried by all four lanes of a node; one CTA and a cluster
@pytest.mark.parametrize("N", [1, 50, 70])
@pytest.mark.parametrize("iters", [1, 40])
def test_quaternion_solves_repeat_their_bits(N, iters):
    prob = W.quat_study(40, seed=25, N=N, tf=0.12 * N, settings=dict(scp_iters=3, admm_iters=iters, stop=0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    first = solve(s)
    for _ in range(10):
        same(solve(s), first)
    s.close()
