"""An uneven FP32 batch in parts of one CTA shape each: the CTA order that a caller
sets and the threads per node change nothing in the results, nor do two threads
that solve one problem at the same time."""
import threading

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402


def solver():
    prob = W.quad_box(12, seed=31, N_range=(20, 127), obs_range=(0, 9), settings=dict(scp_iters=3, admm_iters=30, stop=0))
    s = ucn.Solver(prob, precision=ucn.UCN_PREC_FP32_REFINE)
    s.scp_solve()
    torch.cuda.synchronize()
    assert ucn.ucn_problem_last_launches(s.handle) == 3
    return s, s.x_out.clone(), s.u_out.clone()


def test_orders_and_lanes_leave_the_bits():
    s, x, u = solver()
    rng = np.random.default_rng(1)
    one = None
    for order in (None, np.arange(11, -1, -1, dtype=np.int32), rng.permutation(12).astype(np.int32)):
        ucn.ucn_problem_set_order(s.handle, order)
        s.x_out.zero_()
        s.scp_solve()
        torch.cuda.synchronize()
        assert torch.equal(s.x_out, x) and torch.equal(s.u_out, u)
        ucn.ucn_problem_set_lanes(s.handle, 1)   # one launch, in the order as it was set
        s.x_out.zero_()
        s.scp_solve()
        torch.cuda.synchronize()
        assert ucn.ucn_problem_last_launches(s.handle) == 1
        one = s.x_out.clone() if one is None else one
        assert torch.equal(s.x_out, one)
        ucn.ucn_problem_set_lanes(s.handle, 4)
    s.close()


def test_two_threads_on_one_problem():
    s, x, u = solver()
    x0, u0 = s.tensor(s.prob.xguess), s.tensor(s.prob.uguess)
    torch.cuda.synchronize()
    bad = []

    def work():
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            xo, uo = torch.zeros_like(x), torch.zeros_like(u)
            stats = torch.zeros_like(s.stats)
            status = torch.zeros_like(s.status)
            for _ in range(10):
                xo.zero_()
                ucn.ucn_scp_solve(s.handle, x0, u0, xo, uo, stats, status, stream)
                stream.synchronize()
                if not (torch.equal(xo, x) and torch.equal(uo, u)):
                    bad.append(1)
            stream.synchronize()

    ts = [threading.Thread(target=work) for _ in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
    s.close()
