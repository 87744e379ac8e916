"""State mode's Taylor recursions at large theta_max: the Horner vectors grow with the norm of a slice (up to
e^theta times the state), and each is split on its own grid."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu


def one_norm(H):
    return float(np.max(np.sum(np.abs(H), axis=0)))


@pytest.mark.parametrize("theta", [0.9, 1.9, 3.8, 7.5])
@pytest.mark.parametrize("d,E,seed", [(5, 1, 1), (5, 1, 2), (5, 1, 3), (5, 1, 4), (24, 1, 1), (40, 2, 1), (154, 1, 1)])
def test_taylor_keeps_its_precision_at_large_norms(d, E, seed, theta):
    """A split product's cross terms are FP32 products of values 2^-12 below the vector: an error of 2^-36 of
    it.  A Horner step's error reaches the result multiplied by at most the sum of |X|^i / i!, e^|X|
    (2-norm), N slices' errors add up as sqrt(N), the fidelity's is twice the overlap's; and the states are
    FP32 values (2^-25).  On one grid for a whole application 2^-36 would be 2^-24 at theta = 7.5."""
    from paper_1612_04929_gb300 import build
    build.build()
    N = 30
    prob = sy.random_problem(d=d, M=1, N=N, S=1, seed=seed, E=E, dt=1.0, hk_scale=0.05, u_scale=0.1,
                             alpha=np.array([1.0, 0.0, 0.0, 0.0, 0.0]))
    if E > 1:
        prob.Hdet = 0.02 * prob.Hdet
    prob.dt = theta / (one_norm(prob.H0) + np.max(np.abs(prob.u)) * one_norm(prob.Hk[0])) / 1.05
    cost, grad, terms, info = run(prob, "fp32", propagation="state", theta_max=8.0)
    assert info["n"] == 0
    c_ref, g_ref, t_ref = orc.cost_and_grad(prob, prob.u)
    growth = np.exp(prob.dt * np.linalg.norm(prob.H0, 2))
    assert abs(terms[0] - t_ref[0]) <= 2.0 * np.sqrt(N) * 2.0 ** -36 * growth + 2.0 ** -25
    assert rel(grad, g_ref) <= 1e-5
