"""The autotuner's cache: a choice made for one kind of cost is not applied to the other (a cost on the final
state alone runs other recursions than one with running terms)."""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [0.0, 0.5])
def test_terminal_and_running_costs_are_tuned_apart(first):
    from paper_1612_04929_gb300 import build
    build.build()
    N = 41 if first else 42                      # shapes that no other test tunes

    def candidates(a5):
        prob = sy.random_problem(d=50, M=1, N=N, S=50, seed=4, nF=1, dt=0.02, alpha=np.array([1.0, 0, 0, a5, 0]))
        return run(prob, "fp32", autotune=True)[3]["autotune_candidates"]

    other = 0.5 - first
    assert candidates(first) > 0 and candidates(other) > 0        # a search for each kind
    assert candidates(first) == 0 and candidates(other) == 0      # then the cached choices
