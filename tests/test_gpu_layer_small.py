"""The kernels that take a small layer's pass at once (layer_small.cu) against the oracle: one state per CTA, groups of rows
that end short, one step, a sequence on the longest row groups, more threads than rows x columns and fewer, clusters of 8
and of 4 with the most sequences each takes, and one sequence more (which goes to the separate kernels)."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_layer_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,B,T,H,P", [("f32", 1, 1, 16, 8), ("f32", 1, 7, 8, 8), ("bf16", 1, 64, 32, 16), ("f32", 1, 500, 40, 24),
                                        ("f32", 1, 512, 16, 56), ("f32", 2, 33, 72, 40), ("bf16", 3, 4, 192, 120), ("f32", 14, 65, 24, 104),
                                        ("f32", 15, 18, 136, 48), ("bf16", 32, 50, 48, 32), ("f32", 32, 3, 200, 256), ("f32", 33, 50, 48, 32)])
@pytest.mark.parametrize("states", [False, True])
def test_small_layers(io, B, T, H, P, states):
    run(I.Workload("small", B=B, T=T, H=H, P=P, io_dtype=io, p_done=0.05 if states else 0.0, seed=B + T + H), with_x0=states, with_gxT=states)
