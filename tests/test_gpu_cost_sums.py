"""The per-slice cost sums of the FP32 forms: as accurate as FP64 sums of the same FP32 states, and over
the range of FP64 (unnormalised columns, whose products leave the range of FP32)."""
import math

import numpy as np
import pytest

import synthetic as sy
from oracle import qoc_oracle as orc
from test_gpu_parity import rel, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1612_04929_gb300 import build
    build.build()


@pytest.mark.parametrize("d,S,opt", [(256, 256, {}), (64, 64, {}), (300, 8, {}), (30, 8, {}), (120, 1, dict(propagation="state"))])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_sums_are_as_accurate_as_fp64(d, S, opt, seed):
    """A zero Hamiltonian leaves FP32-representable columns as they are, so the overlap and the forbidden
    population are known.  One column carries the weight.  An FP64 sum of d terms of random sign is off by
    about sqrt(d) 2^-53 of their root mean square (below 2e-16 here), the handful of FP64 operations
    after it by 2^-53 each: 1e-15."""
    prob = sy.random_problem(d=d, M=1, N=2, S=S, seed=seed, nF=d // 2, h0_scale=0.0, hk_scale=0.0,
                             alpha=np.array([1.0, 0.0, 0.0, 0.0, 0.0]))
    r32 = lambda a: a.astype(np.complex64).astype(np.complex128)
    prob.psi0 = r32(prob.psi0)
    prob.psiT = r32(prob.psi0 + 0.1 * prob.psiT)
    prob.col_weight = np.full(S, 1e-30)
    prob.col_weight[S // 2] = 1.0
    _, _, terms, _ = run(prob, "fp32", **opt)
    z, t = prob.psi0[:, S // 2], prob.psiT[:, S // 2]
    dot = lambda *ab: math.fsum(float(a) * float(b) for x, y in ab for a, b in zip(x, y))
    re, im = dot((t.real, z.real), (t.imag, z.imag)), dot((t.real, z.imag), (-t.imag, z.real))
    f = z[prob.forbidden]
    assert abs(terms[0] - (1.0 - (re * re + im * im))) <= 1e-15
    assert abs(terms[3] - 2 * dot((f.real, f.real), (f.imag, f.imag))) <= 1e-15


@pytest.mark.parametrize("precision,d,S", [("fp32", 16, 2), ("fp32", 40, 3), ("fp32", 70, 20), ("bf16", 70, 20), ("fp32", 50, 50)])
@pytest.mark.parametrize("m,path", [(1e-22, False), (1e20, False), (1e-15, True)])
def test_range(precision, d, S, m, path):
    """psi0 scaled by m and the targets by 1 / m: the overlaps stay, C5 scales by m^2."""
    prob = sy.random_problem(d=d, M=2, N=12, S=S, seed=7, nF=2, dt=1.0 / d, u_scale=0.8, path=path)
    prob.psi0, prob.psiT = prob.psi0 * m, prob.psiT / m
    if path:
        prob.psiT_path = prob.psiT_path / m
    prob.alpha = np.array([1.0, 0.01, 0.02, 0.5 / m ** 2, 0.3 if path else 0.0])
    cost, grad, terms, _ = run(prob, precision)
    c_ref, g_ref, t_ref = orc.cost_and_grad(prob, prob.u)
    assert abs(cost - c_ref) <= 1e-5 * abs(c_ref) and rel(grad, g_ref) <= 1e-5
    assert np.all(np.abs(terms - t_ref) <= 1e-5 * np.abs(t_ref))


@pytest.mark.parametrize("d,S", [(16, 2), (40, 3), (70, 20), (64, 64)])
def test_small_overlaps(d, S):
    """Overlaps far below the range of FP32 products, brought back by the weight of the fidelity."""
    prob = sy.random_problem(d=d, M=2, N=12, S=S, seed=8, dt=1.0 / d, u_scale=0.8, alpha=np.array([1e66, 0, 0, 0, 0]))
    prob.psi0, prob.psiT = prob.psi0 * 1e-22, prob.psiT * 1e-22
    _, grad, _, _ = run(prob, "fp32")
    assert rel(grad, orc.cost_and_grad(prob, prob.u)[1]) <= 1e-5
