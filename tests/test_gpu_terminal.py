"""Costs that act on the final state alone: the costate starts from the terminal block and no
source or zero-carry pass runs.  Every layout (serial and segmented sweeps, one and several waves,
a ragged last segment, column panels with padding and zero-weight columns, ensembles) against the
oracle, and against the general path: a vanishing weight on C67 switches the sources back on."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5, "bf16": 1e-5}
CASES = [dict(d=3, M=2, N=7, S=1, seed=201), dict(d=9, M=2, N=53, S=9, seed=202, weights=True),
         dict(d=16, M=3, N=40, S=16, seed=203, E=3), dict(d=72, M=2, N=21, S=12, seed=204)]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("opt", [dict(), dict(sweep="serial"), dict(sweep="scan", ckpt_stride=5, wave_slices=10)],
                         ids=["auto", "serial", "waves"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"d{c['d']}S{c['S']}")
def test_terminal_cost_matches_oracle_and_general_path(case, opt, precision):
    from paper_1612_04929_gb300 import Context, build
    build.build()
    prob = sy.random_problem(**case, dt=0.2, u_scale=0.5, nF=2, alpha=np.array([1.0, 0.02, 0.01, 0.0, 0.0]))
    if case["S"] == 9:
        prob.col_weight[[2, 7]] = 0.0
    got = []
    for a67 in (0.0, 1e-300):
        prob.alpha = np.array([1.0, 0.02, 0.01, 0.0, a67])
        with Context(precision, **opt) as c:
            c.set_problem(prob)
            got.append(c.evaluate(prob.u))
    c_ref, g_ref, t_ref = orc.cost_and_grad(prob, prob.u)
    tol = TOL[precision]
    for cost, grad, terms in got:
        assert abs(cost - c_ref) <= tol * abs(c_ref)
        assert np.max(np.abs(terms - t_ref) / np.maximum(np.abs(t_ref), 1.0)) <= tol
        assert np.linalg.norm(grad - g_ref) <= tol * np.linalg.norm(g_ref)
