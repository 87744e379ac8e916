"""Gradient contraction over the controls' non-zero elements: every adjoint kernel that takes it, with
an all-zero control, a single-element one, ladder-like ones and more controls than warps, against the
oracle; and the dense contraction just above the density at which it takes over."""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_parity import check

pytestmark = pytest.mark.gpu

FORMS = [("fp64", 10, 10, {}), ("fp64", 24, 1, {}), ("fp64", 10, 3, dict(adjoint="recompute")), ("fp64", 50, 2, {}),
         ("fp64", 8, 1, dict(propagation="state")), ("fp32", 1, 1, {}), ("fp32", 11, 11, {}), ("fp32", 40, 1, {}),
         ("fp32", 11, 4, dict(taylor_scheme="horner")), ("fp32", 60, 1, {}), ("fp32", 60, 20, {}),
         ("fp32", 73, 20, {}), ("fp32", 74, 1, {}), ("fp32", 73, 3, dict(adjoint="recompute")),
         ("fp32", 40, 1, dict(propagation="state")), ("fp32", 33, 2, dict(propagation="state", exponential="chebyshev")),
         ("bf16", 73, 20, {})]


@pytest.mark.parametrize("keep", [0.02, 0.2, 0.3])
@pytest.mark.parametrize("precision,d,S,opt", FORMS)
def test_sparse_controls_match_oracle(precision, d, S, opt, keep):
    from paper_1612_04929_gb300 import build
    build.build()
    M = 18 if d < 20 else 3
    prob = sy.random_problem(d=d, M=M, N=6, S=S, seed=900 + d, nF=min(2, d - 1), dt=0.8 / np.sqrt(d) / M, u_scale=0.5)
    rng = np.random.default_rng(901)
    up = np.triu(rng.random((M, d, d)) < keep)
    mask = up | np.swapaxes(up, 1, 2)
    mask[0] = False                      # a control with no element
    mask[1 % M] = False
    mask[1 % M, d - 1, d - 1] = True     # a control with one
    prob.Hk = prob.Hk * mask
    check(prob, precision, **opt)
