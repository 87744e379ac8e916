"""Full unitaries with a terminal cost: the recursions over the wave's binary tree, on the per-slice and
the batched path, for wave lengths around powers of two (whole and ragged last nodes, one slice in the
last wave), several waves (hand-over of the blocks, recomputation), members, targets and initial
blocks of other norms, each against the oracle and against the serial sweeps."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu

CASES = [(dict(d=48, M=2, N=17), {}), (dict(d=49, M=1, N=33), dict(wave_slices=16)), (dict(d=64, M=2, N=31, E=2), dict(wave_slices=8)),
         (dict(d=65, M=2, N=64), {}), (dict(d=70, M=2, N=40), dict(wave_slices=13, ckpt_stride=13)), (dict(d=81, M=1, N=18, E=3), {}),
         (dict(d=128, M=2, N=25), dict(wave_slices=12, ckpt_stride=4)), (dict(d=130, M=1, N=19), {}), (dict(d=256, M=1, N=17), {}),
         (dict(d=260, M=1, N=18), dict(wave_slices=1, sweep="scan", ckpt_stride=1))]


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("case,opt", CASES, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "auto")
def test_tree_matches_oracle_and_serial(case, opt, precision):
    from paper_1612_04929_gb300 import build
    build.build()
    d = case["d"]
    prob = sy.random_problem(**case, S=d, seed=1100 + d, dt=1.0 / d, u_scale=0.8, alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    if d in (49, 130):
        prob.psi0 = prob.psi0 * np.linspace(0.01, 3.0, d)[None, :]
        prob.psiT = prob.psiT * 40.0
        prob.col_weight = np.linspace(0.5, 1.5, d)
    cost, grad, terms, info = run(prob, precision, **opt)
    c_ref, g_ref, t_ref = orc.cost_and_grad(prob, prob.u)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref)
    assert np.max(np.abs(terms - t_ref) / np.maximum(np.abs(t_ref), 1.0)) <= 1e-5
    assert rel(grad, g_ref) <= 1e-5
    serial = run(prob, precision, sweep="serial")
    assert abs(cost - serial[0]) <= 1e-6 * abs(c_ref) and rel(grad, serial[1]) <= 2e-6
