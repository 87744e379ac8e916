"""Columns of very different norms.  A factor 2^-k on a column of the initial block and 2^k on the same
column of the target changes no term of the cost and no gradient in exact arithmetic, nor any FP32
rounding that is relative to the column, so a form that keeps its precision gives what it gives without
the factors.  The operands of the tensor-core product for Ubar are cut across columns, so it is left for
the FP32 product once the norms differ (2e-6 between the two forms, as between sweep forms elsewhere)."""
import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu


def scaled(prob, k):
    f = 2.0 ** np.where(np.arange(prob.psi0.shape[1]) % 3 == 0, k, 0.0)
    out = sy.Problem(**{**prob.__dict__})
    out.psi0, out.psiT = prob.psi0 / f, prob.psiT * f
    return out


# full unitaries (operands read in place; the tree) and a few columns (staged operands; the sweeps)
BF16 = [(dict(d=73, S=73, N=11), {}), (dict(d=130, S=130, N=11), {}), (dict(d=130, S=130, N=9), dict(sweep="serial")),
        (dict(d=74, S=20, N=9, E=2), {}), (dict(d=73, S=30, N=9), dict(taylor_scheme="horner"))]


@pytest.mark.parametrize("k", [3, 14, 30])
@pytest.mark.parametrize("case,opt", BF16, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "auto")
def test_bf16_keeps_columns_of_other_norms(case, opt, k):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sy.random_problem(**case, M=2, seed=1300 + case["d"], dt=1.0 / case["d"], u_scale=0.8,
                             alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    c_ref, g_ref, _ = orc.cost_and_grad(prob, prob.u)
    cost, grad, _, _ = run(scaled(prob, k), "bf16", **opt)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref) and rel(grad, g_ref) <= 1e-5
    assert rel(grad, run(prob, "bf16", **opt)[1]) <= 2e-6
