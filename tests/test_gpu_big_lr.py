"""The batched path's low-rank reverse mode (FP32 form, few columns): at forced (p, n) against the
oracle's derivative of the truncated series, over odd and even d (8- and 16-byte loads, 64- and
80-row contraction tiles), ranks from 1 to the largest that applies, orders without X^2 or X^3,
several controls (more than one contraction pass), members and padded column panels; and against
the block recursion at the same orders."""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_ps import against_truncated_series
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu

CASES = [
    (dict(d=69, M=1, N=4, S=1, seed=701, nF=1), (1, 0)),      # rank 1, one term, odd d
    (dict(d=80, M=2, N=5, S=1, seed=702, nF=2, E=2), (2, 1)),  # no X^3
    (dict(d=81, M=9, N=3, S=2, seed=703, nF=2), (3, 2)),       # rank 8, empty chain, nine controls
    (dict(d=96, M=2, N=3, S=3, seed=704, nF=2, path=True), (7, 2)),    # rank 12 = d / 8
    (dict(d=154, M=2, N=3, S=1, seed=705, nF=3), (14, 1)),     # two 80-row tiles
    (dict(d=161, M=2, N=2, S=1, seed=706, nF=3), (9, 3)),
    (dict(d=512, M=1, N=1, S=1, seed=707, nF=1), (6, 0)),      # the largest d: a column pair per thread
]


@pytest.mark.parametrize("case,pn", CASES, ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else f"d{c['d']}S{c['S']}")
def test_low_rank_batched_adjoint_differentiates_the_series(case, pn):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sy.random_problem(**case, dt=3.0 / case["d"], u_scale=0.8)
    info = against_truncated_series(prob, "fp32", *pn)
    assert info["kernel_path"] == 1 and info["adjoint_form"] == 0
    _, g, _, _ = run(prob, "fp32", p_override=pn[0], n_override=pn[1])
    _, g2, _, info2 = run(prob, "fp32", p_override=pn[0], n_override=pn[1], adjoint="recompute")
    assert info2["adjoint_form"] == 1 and rel(g, g2) <= 2e-6
