"""Tree products on the tensor cores: more products in a level than are sliced at once, several members,
and the ends of the size range, against the serial sweeps and the oracle."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N,E", [(128, 200, 8), (129, 21, 2), (191, 9, 3), (384, 14, 1), (385, 6, 1)])
def test_tree_products_match_serial_and_oracle(d, N, E):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sy.random_problem(d=d, M=1, N=N, E=E, S=d, seed=1400 + d, dt=1.0 / d, u_scale=0.8,
                             alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    cost, grad, terms, info = run(prob, "bf16")
    serial = run(prob, "bf16", sweep="serial")
    assert abs(cost - serial[0]) <= 1e-6 * abs(serial[0]) and rel(grad, serial[1]) <= 2e-6
    if N * E <= 50:
        c_ref, g_ref, _ = orc.cost_and_grad(prob, prob.u)
        assert abs(cost - c_ref) <= 1e-5 * abs(c_ref) and rel(grad, g_ref) <= 1e-5
