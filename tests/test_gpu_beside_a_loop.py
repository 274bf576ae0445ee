"""FP64 quadrotor solves beside a running request loop: the loop's CTAs stay on their
SMs until it has been idle for a while, and a solve does not wait for that.  Without
a loop the solve gives the bits it gave before one."""
import time

import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import serving, ucn  # noqa: E402

TOL = 1e-9
IDLE = 3.0


@pytest.mark.parametrize("ctas", [60, 100, 120])
@pytest.mark.parametrize("B", [1, 3, 24])
def test_an_fp64_solve_finds_its_place(ctas, B):
    prob = W.quad_box(B, seed=3, N_range=(50, 50), obs_range=(2, 4), settings=dict(scp_iters=2, admm_iters=30, stop=0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP64)
    x0, u0 = s.tensor(prob.xguess), s.tensor(prob.uguess)
    s.scp_solve(x0, u0)
    torch.cuda.synchronize()
    alone = s.x_out.clone()
    srv = serving.Server(1, ucn.UCN_PREC_FP32_REFINE, max_slots=64, max_horizon=120, max_obs=10, lanes=4,
                         settings=dict(W.quad_box(1).settings))
    stream, done = torch.cuda.Stream(), torch.cuda.Event()
    srv.loop_start(ctas=min(ctas, srv.loop_capacity()), idle_s=IDLE)
    time.sleep(0.1)
    t = time.perf_counter()
    x, u = s.scp_solve(x0, u0, stream=stream)
    done.record(stream)
    while not done.query():
        time.sleep(0.001)
    took = time.perf_counter() - t
    srv.loop_stop()
    srv.close()
    torch.cuda.synchronize()
    assert took < IDLE / 2, took
    xr, ur, _, _ = oracle.scp_solve(prob)
    assert oracle.rel_err(x.cpu().numpy(), xr) <= TOL and oracle.rel_err(u.cpu().numpy(), ur) <= TOL
    s.scp_solve(x0, u0)
    torch.cuda.synchronize()
    assert torch.equal(s.x_out, alone)
    s.close()
