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
                             alpha=np.array([1.0, 0.0, 0.0, 0.0, 0.0]))
    c_ref, g_ref, _ = orc.cost_and_grad(prob, prob.u)
    cost, grad, _, _ = run(scaled(prob, k), "bf16", **opt)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref) and rel(grad, g_ref) <= 1e-5
    assert rel(grad, run(prob, "bf16", **opt)[1]) <= 2e-6


@pytest.mark.parametrize("k", [4, 14, 30])
@pytest.mark.parametrize("case,opt", [(dict(d=64, S=64, N=20), {}), (dict(d=65, S=65, N=9, E=2), dict(wave_slices=4, ckpt_stride=4)),
                                      (dict(d=130, S=130, N=11), {})],
                         ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()) or "auto")
def test_tree_splits_every_column_on_its_own_grid(case, opt, k):
    """The tree's blocks are split column by column: powers of two change nothing at all."""
    prob = sy.random_problem(**case, M=2, seed=1400 + case["d"], dt=1.0 / case["d"], u_scale=0.8,
                             alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    plain, other = run(prob, "fp32", **opt), run(scaled(prob, k), "fp32", **opt)
    assert plain[0] == other[0] and np.array_equal(plain[1], other[1])


def test_tensor_core_tree_splits_every_column_on_its_own_grid():
    prob = sy.random_problem(d=130, S=130, N=11, M=2, seed=1500, dt=1.0 / 130, u_scale=0.8,
                             alpha=np.array([1.0, 0.01, 0.02, 0.0, 0.0]))
    one, other = run(scaled(prob, 5), "bf16"), run(scaled(prob, 30), "bf16")   # both past the factor 8 of Ubar's slices
    assert one[0] == other[0] and np.array_equal(one[1], other[1])
