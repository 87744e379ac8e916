"""Device memory of a plan: no sources where the cost has none, and the tree's tensor-core planes within the
budget that sizes the wave."""
import numpy as np
import pytest

import synthetic as sy
from test_gpu_parity import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1612_04929_gb300 import build
    build.build()


@pytest.mark.parametrize("sweep", ["serial", "scan"])
def test_a_terminal_cost_holds_no_sources(sweep):
    d, S, N, E, W = 40, 4, 32, 2, 16
    held = {}
    for a5 in (0.0, 0.5):
        prob = sy.random_problem(d=d, M=1, N=N, S=S, E=E, seed=1, nF=2, dt=1.0 / d, alpha=np.array([1.0, 0, 0, a5, 0]))
        _, _, _, info = run(prob, "fp32", sweep=sweep, wave_slices=W, ckpt_stride=4)
        assert info["wave_slices"] == W
        held[a5] = info["device_bytes"]
    assert held[0.5] - held[0.0] == 2 * E * W * d * S * 8    # two wave sets of complex64 blocks


def test_the_tree_holds_no_sources():
    """Bytes per slice of the wave: propagators and their adjoints, states, costates (two sets), the operand
    scratch and stored products, which do not depend on the cost, tree nodes (two sets) and blocks."""
    d, N = 64, 64
    prob = sy.random_problem(d=d, M=1, N=N, S=d, seed=2, dt=1.0 / d, alpha=np.array([1.0, 0, 0, 0, 0]))
    held = {w: run(prob, "fp32", wave_slices=w, ckpt_stride=16)[3]["device_bytes"] for w in (16, 32)}
    flat = {}
    for w in (16, 32):   # a running cost: segmented sweeps, with sources
        p2 = sy.random_problem(d=d, M=1, N=N, S=d, seed=2, nF=1, dt=1.0 / d, alpha=np.array([1.0, 0, 0, 0.5, 0]))
        flat[w] = run(p2, "fp32", wave_slices=w, ckpt_stride=16)[3]["device_bytes"]
    dd = d * d
    tree = 16 * (2 * dd * 16 + dd * 16)                                       # nodes, blocks
    segments = 1 * (2 * 2 * dd * 16 + 2 * 8 * dd * 16 + dd * 8 + 3 * dd * 16)   # one more segment of 16: products, levels, blocks
    sources = 16 * 2 * dd * 8
    assert (held[32] - held[16]) - (flat[32] - flat[16]) == tree - segments - sources


def test_tensor_core_tree_planes_are_in_the_budget():
    """The wave is the largest that fits 32 GiB (an eighth of the free memory is more here)."""
    import torch
    if torch.cuda.mem_get_info()[0] < 8 * (33 << 30):
        pytest.skip("less free memory than the budget's upper limit asks for")
    d, N = 384, 1800
    prob = sy.random_problem(d=d, M=1, N=N, S=d, seed=3, dt=0.5 / d, alpha=np.array([1.0, 0, 0, 0, 0]))
    _, _, _, info = run(prob, "bf16")
    assert info["n_waves"] > 2                                                 # the memory decides
    top = info["p"] // 3 - (info["p"] % 3 == 0)
    stored = 2 * info["wave_slices"] * (top + info["n"] + 3) * d * d * 8       # operands kept for the adjoint: sized by
    blocks = (N // info["ckpt_stride"] + 1) * d * d * 16                       # the orders, at evaluation; checkpoints
    assert info["device_bytes"] - stored <= (32 << 30) + blocks + (64 << 20)
