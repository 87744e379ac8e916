"""Tensor-core products with fewer and with more output tiles than SMs (a persistent CTA takes several),
whole and ragged in rows, columns and the contraction, against the oracle."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(96, 3), (128, 5), (129, 120), (143, 64), (256, 48), (272, 30), (384, 13)])
def test_bf16_products_match_oracle(d, N):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sy.random_problem(d=d, M=1, N=N, S=3, seed=1300 + d, dt=1.0 / d, u_scale=0.8, alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    cost, grad, terms, info = run(prob, "bf16")
    c_ref, g_ref, t_ref = orc.cost_and_grad(prob, prob.u)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref)
    assert rel(grad, g_ref) <= 1e-5
