"""State mode's recursions across a cluster: every cluster size and row count a warp the dispatch
takes (few rows a CTA, ragged last CTA, one to six 32-column chunks, two and four rows a warp), both
series, several columns and members, waves, the empty series of a zero Hamiltonian, and sizes that
stay on the one-CTA form; all against the oracle."""
import pytest

import synthetic as sy
from test_gpu_parity import check

pytestmark = pytest.mark.gpu

# d: 2, 15 one CTA; 17 two; 33, 64 + 1 four / eight; 95, 97, 160, 165 chunk and row edges
CASES = [dict(d=2, M=1, N=5, S=1), dict(d=15, M=2, N=9, S=2), dict(d=17, M=2, N=9, S=1), dict(d=33, M=2, N=9, S=3),
         dict(d=65, M=2, N=7, S=1, E=2), dict(d=95, M=2, N=5, S=1), dict(d=97, M=1, N=4, S=2),
         dict(d=160, M=1, N=3, S=1), dict(d=165, M=1, N=3, S=1), dict(d=36, M=1, N=3, S=1, E=60),
         dict(d=40, M=1, N=3, S=1, E=150)]


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"d{c['d']}S{c['S']}E{c.get('E', 1)}")
def test_state_recursions_match_oracle(case, precision, exponential):
    from paper_1612_04929_gb300 import build
    build.build()
    if precision == "fp64" and case["d"] > 120:
        pytest.skip("the FP64 gradient kernel's d x d block exceeds shared memory")
    prob = sy.random_problem(**case, seed=800 + case["d"], nF=1, path=case["N"] > 5, dt=2.0 / case["d"], u_scale=0.8)
    tol = 1e-10 if precision == "fp64" else 1e-5
    check(prob, precision, tol=tol, propagation="state", exponential=exponential, wave_slices=4)


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
def test_zero_hamiltonian(exponential):
    prob = sy.random_problem(d=24, M=1, N=4, S=1, seed=830, nF=1, h0_scale=0.0, hk_scale=0.0)
    check(prob, "fp32", propagation="state", exponential=exponential)
