"""The batched products' tiles: sizes that take each tile shape of the split and plain products, whole and
ragged (one row past a tile, one short of it), against the oracle's derivative of the truncated series."""
import pytest

import synthetic as sy
from test_gpu_ps import against_truncated_series

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [69, 79, 80, 81, 95, 96, 97, 127, 128, 129, 159, 160, 193])
def test_tile_shapes(d):
    from paper_1612_04929_gb300 import build
    build.build()
    prob = sy.random_problem(d=d, M=2, N=2, S=d // 4, seed=1000 + d, nF=2, dt=3.0 / d, u_scale=0.8)
    info = against_truncated_series(prob, "fp32", 8, 1)
    assert info["kernel_path"] == 1 and info["adjoint_form"] == 0
