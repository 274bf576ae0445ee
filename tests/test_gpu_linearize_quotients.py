"""The linearisation (Eq. (2b)) divides by the model's constants with correctly
rounded quotients: of a quadrotor at rest and level, the rates answer to the
thrusts by h k, k = arm / J (km / Jz in yaw), through four equal RK4 stages -- the
entries of B are then those operations on the rounded quotient, bit for bit."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_10711_gb300 import ucn  # noqa: E402


@pytest.mark.parametrize("prec,t", [("UCN_PREC_FP64", np.float64), ("UCN_PREC_FP32_REFINE", np.float32)])
def test_rates_of_a_level_quadrotor(prec, t):
    n = 256
    prob = W.quad_box(n, seed=7, N_range=(3, 3), obs_range=(1, 1))
    rng = np.random.default_rng(7)
    prob.params = prob.params.copy()
    prob.params[:, 1:4] *= rng.uniform(0.5, 2.0, (n, 3))   # J
    prob.params[:, 4:6] *= rng.uniform(0.5, 2.0, (n, 2))   # arm, km
    x = np.zeros_like(prob.xguess)
    u = np.full_like(prob.uguess, 2.0)
    s = ucn.Solver(prob, precision=getattr(ucn, prec))
    B = s.linearize(s.tensor(x), s.tensor(u))[1].cpu().numpy()[::3]
    s.close()
    c = prob.params.astype(t)
    h6 = (prob.dt / 6.0).astype(t)
    k = np.stack([c[:, 4] / c[:, 1], c[:, 4] / c[:, 2], c[:, 5] / c[:, 3]], 1)   # rounded once each
    two = t(2)
    step = h6[:, None] * (((k + two * k) + two * k) + k)
    np.testing.assert_array_equal(B[:, 9, 1], step[:, 0].astype(np.float64))
    np.testing.assert_array_equal(B[:, 10, 2], step[:, 1].astype(np.float64))
    np.testing.assert_array_equal(B[:, 11, 0], step[:, 2].astype(np.float64))
