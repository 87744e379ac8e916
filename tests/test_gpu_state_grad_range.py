"""State mode's gradient for sparse controls contracts in FP64: controls scaled by 2^-k (their amplitudes by
2^k) and the cost's weight by 2^-60 scale the gradient and change no bit of it, also where the products of
its factors leave the range of FP32."""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_parity import run
from test_gpu_state_grad import sparse_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
@pytest.mark.parametrize("d,M", [(12, 1), (33, 2), (100, 2)])
@pytest.mark.parametrize("k", [40, 90])
def test_scaled_controls_scale_the_gradient(d, M, k, exponential):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sparse_problem(d=d, M=M, N=5, S=1, seed=1800 + d, dt=1.0 / d, alpha=np.array([1.0, 0, 0, 0, 0]))
    prob.Hk = prob.Hk.astype(np.complex64).astype(np.complex128)
    g0 = run(prob, "fp32", propagation="state", exponential=exponential)[1]
    prob.alpha = prob.alpha * 2.0 ** -60
    prob.Hk, prob.u = prob.Hk * 2.0 ** -k, prob.u * 2.0 ** k
    g1 = run(prob, "fp32", propagation="state", exponential=exponential)[1]
    assert np.array_equal(g1, g0 * 2.0 ** (-60 - k))
