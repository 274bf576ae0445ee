"""Device memory of a problem whose solves keep their records in shared memory:
no global records beside them."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402


def test_long_quaternion_problems_hold_no_global_records():
    # records of 121 nodes do not fit a CTA (the row kernel splits them over two); as
    # global records they would take 0.6 GB, the exported states take 0.19 GB
    B, N = 2000, 120
    prob = W.quat_study(B, seed=5, N=N, tf=0.12 * N, settings=dict(scp_iters=2, admm_iters=5, stop=0))
    ucn.Solver(prob.subset([0]), precision=ucn.UCN_PREC_FP32_REFINE).close()   # loads the library
    desc, keep = ucn.make_desc(prob, ucn.UCN_PREC_FP32_REFINE)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = ucn.ucn_problem_create(desc)
    used = before - torch.cuda.mem_get_info()[0]
    states = 8 * ucn.ucn_state_size(h)
    ucn.ucn_problem_destroy(h)
    assert used <= states + (64 << 20), (used, states)
