"""Which kernels ran: the kernel classes that a profiled evaluation lists, at both sides of the rules that pick
the tree, its tensor-core products, the low-rank reverse mode, the cluster recursion and the rank-one gradient.
(The numerical tests of these forms would pass on the kernels they replace.)"""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_parity import check  # noqa: F401  (builds the library)
from test_gpu_ps import against_truncated_series
from test_gpu_state_grad import sparse_problem

pytestmark = pytest.mark.gpu


def classes(prob, precision, **opt):
    from paper_1612_04929_gb300 import Context, build
    build.build()
    with Context(precision, profile=True, **opt) as c:
        c.set_problem(prob)
        c.evaluate(prob.u)
        return set(c.profile())


GATE = np.array([1.0, 0.01, 0.02, 0.0, 0.0])
TREE = {"tree nodes", "tree states", "tree costates"}
TREE_TC = {t + " (tensor cores)" for t in TREE}


@pytest.mark.parametrize("precision,d,S,nF,opt,want", [
    ("fp32", 48, 48, 0, dict(N=200), TREE), ("fp32", 48, 48, 0, dict(N=199), set()), ("fp32", 63, 63, 0, dict(N=50, E=4), TREE),
    ("fp32", 63, 63, 0, {}, set()), ("fp32", 64, 64, 0, {}, TREE), ("fp32", 47, 47, 0, dict(N=200), set()),
    ("fp32", 64, 63, 0, {}, set()),
    ("fp32", 64, 64, 0, dict(sweep="serial"), set()), ("fp64", 64, 64, 0, {}, set()), ("fp32", 64, 64, 2, {}, set()),
    ("fp32", 130, 130, 0, {}, TREE), ("tf32", 70, 70, 0, {}, TREE), ("bf16", 127, 127, 0, {}, TREE),
    ("bf16", 128, 128, 0, {}, TREE_TC), ("bf16", 384, 384, 0, {}, TREE_TC), ("bf16", 385, 385, 0, {}, TREE)])
def test_tree(precision, d, S, nF, opt, want):
    alpha = GATE if nF == 0 else np.array([1.0, 0.01, 0.02, 0.5, 0.0])
    opt = dict(opt)
    prob = sy.random_problem(d=d, M=1, N=opt.pop("N", 17), E=opt.pop("E", 1), S=S, seed=11, nF=nF, dt=1.0 / d, alpha=alpha)
    got = classes(prob, precision, **opt)
    assert got & (TREE | TREE_TC) == want
    assert ("chain (replay)" in got or "chain" in got or "costate (final)" in got or "costate" in got) or want


@pytest.mark.parametrize("precision,d,S,opt,low", [
    ("fp32", 154, 1, {}, True), ("fp32", 96, 3, dict(p_override=5, n_override=2), True),      # rank d / 8
    ("fp32", 96, 3, dict(p_override=7, n_override=2), False),                                # its factors: too much shared memory
    ("fp32", 96, 4, dict(p_override=5, n_override=2), False), ("fp32", 80, 5, dict(p_override=7, n_override=1), True),
    ("fp32", 512, 1, dict(p_override=6, n_override=0), True), ("bf16", 154, 1, {}, False), ("fp64", 80, 1, {}, False),
    ("fp32", 154, 1, dict(adjoint="recompute"), False), ("fp32", 154, 1, dict(taylor_scheme="horner"), False)])
def test_low_rank_reverse_mode(precision, d, S, opt, low):
    prob = sy.random_problem(d=d, M=2, N=3, S=S, seed=12, nF=1, dt=0.5 / d)
    got = classes(prob, precision, **opt)
    assert ("expm_adj (low rank)" in got) == low and ("expm_adj" in got) != low


@pytest.mark.parametrize("d,S,pn", [(96, 3, (5, 2)), (73, 2, (14, 2)), (69, 2, (9, 2))])
def test_low_rank_at_its_largest_ranks(d, S, pn):
    prob = sy.random_problem(d=d, M=2, N=3, S=S, seed=15, nF=1, dt=3.0 / d, u_scale=0.8)
    assert "expm_adj (low rank)" in classes(prob, "fp32", p_override=pn[0], n_override=pn[1])
    against_truncated_series(prob, "fp32", *pn)


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
@pytest.mark.parametrize("precision,d,S,E,cluster", [("fp32", 2, 1, 1, True), ("fp32", 40, 3, 2, True), ("fp64", 33, 1, 1, True),
                                                     ("fp32", 165, 1, 1, True),   # the largest d of state mode
                                                     ("fp32", 24, 8, 60, False)])   # more than two chains an SM: wide panels
def test_state_recursion(precision, d, S, E, cluster, exponential):
    prob = sy.random_problem(d=d, M=1, N=3, S=S, seed=13, E=E, nF=1, dt=0.5 / d)
    got = classes(prob, precision, propagation="state", exponential=exponential, gradient="first_order")
    for way in ("forward", "costate"):
        assert ("state_chain (%s, cluster)" % way in got) == cluster and ("state_chain (%s)" % way in got) != cluster


@pytest.mark.parametrize("exponential", ["taylor", "chebyshev"])
@pytest.mark.parametrize("precision,d,dense,terms", [("fp32", 9, False, True), ("fp32", 24, False, True), ("fp32", 160, False, True), ("fp32", 161, False, False),
                                                     ("fp32", 40, True, False), ("fp64", 40, False, False)])
def test_state_gradient(precision, d, dense, terms, exponential):
    kw = dict(d=d, M=2, N=3, S=1, seed=14, nF=1, dt=0.5 / d)
    prob = sy.random_problem(**kw) if dense else sparse_problem(**kw)
    got = classes(prob, precision, propagation="state", exponential=exponential)
    assert ("expm_adj (rank-one terms)" in got) == terms and ("expm_adj" in got) != terms
