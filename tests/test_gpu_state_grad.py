"""State mode's gradient kernel for sparse controls: both series at forced orders against the oracle's
derivative of the truncated series, and Chebyshev and Taylor at their default orders against the
oracle, at the edges of the 32-column chunks and rows a warp, one to several columns and members, one
term only, and sizes past the kernel's range (which keep the dense-block kernel)."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import check, rel, run

pytestmark = pytest.mark.gpu


def sparse_problem(**kw):
    prob = sy.random_problem(**kw)
    d, M = kw["d"], kw["M"]
    rng = np.random.default_rng(kw["seed"] + 1)
    up = np.triu(rng.random((M, d, d)) < 1.0 / d)
    prob.Hk = prob.Hk * (up | np.swapaxes(up, 1, 2) | np.eye(d, dtype=bool)[None])
    return prob


CASES = [dict(d=9, M=2, N=5, S=1), dict(d=32, M=17, N=4, S=3), dict(d=33, M=2, N=4, S=2, E=2), dict(d=64, M=2, N=3, S=1),
         dict(d=95, M=1, N=3, S=1), dict(d=128, M=2, N=3, S=1, E=2), dict(d=154, M=2, N=3, S=1), dict(d=160, M=1, N=2, S=2),
         dict(d=163, M=1, N=2, S=1)]


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"d{c['d']}S{c['S']}")
def test_default_orders_match_oracle(case, exponential):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sparse_problem(**case, seed=950 + case["d"], nF=1, dt=2.0 / case["d"], u_scale=0.8)
    check(prob, "fp32", propagation="state", exponential=exponential)


@pytest.mark.parametrize("pn", [(1, 0), (1, 3), (2, 1), (5, 2), (11, 0)])
def test_forced_orders_differentiate_the_series(pn):
    prob = sparse_problem(d=20, M=2, N=7, S=2, seed=980, nF=2, path=True, E=2, dt=0.1)
    cost, grad, terms, info = run(prob, "fp32", propagation="state", p_override=pn[0], n_override=pn[1])
    assert (info["p"], info["n"]) == pn
    c_t, g_t, _ = orc.taylor_cost_and_grad(prob, prob.u, *pn)
    assert abs(cost - c_t) <= 1e-5 * abs(c_t) and rel(grad, g_t) <= 1e-5


def test_one_chebyshev_term():
    """A degree-one expansion (loose tolerance, tiny theta): one rank-one term."""
    prob = sparse_problem(d=16, M=2, N=4, S=1, seed=981, nF=1, dt=1e-5)
    cost, grad, _, info = run(prob, "fp32", propagation="state", exponential="chebyshev", tol=1e-3)
    assert info["p"] == 1
    c_ref, g_ref, _ = orc.cost_and_grad(prob, prob.u)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref) and rel(grad, g_ref) <= 1e-3
