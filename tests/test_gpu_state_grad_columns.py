"""Which gradient kernel state mode takes for several columns of a small system (the faster one)."""
import pytest

from test_gpu_forms import classes
from test_gpu_parity import check
from test_gpu_state_grad import sparse_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,S,terms", [(23, 2, True), (23, 3, False), (24, 8, True), (16, 8, False)])
def test_state_gradient_of_several_columns(d, S, terms):
    prob = sparse_problem(d=d, M=2, N=3, S=S, seed=16, nF=1, dt=0.5 / d)
    assert ("expm_adj (rank-one terms)" in classes(prob, "fp32", propagation="state")) == terms
    check(prob, "fp32", propagation="state")
