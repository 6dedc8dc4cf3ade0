"""The kernels at the two ends of a layer call, at the edges of their 32 x 32 tiles: discretisation with operand
packing, and the last sums of the backward pass (split-K partials, gAbar over sequences, dD over row groups)."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_layer_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,P", [(5, 600, 72, 40),     # six split-K partials (the 16-warp sums), ragged tiles both ways
                                     (600, 4, 40, 104),    # more than 512 rows of gAbar partials, brought down first
                                     (70, 3, 136, 8),      # one partial (the 8-warp sums), fewer states than a tile
                                     (1, 9, 8, 264)])      # fewer features than a tile
def test_tile_edges_fp32(B, T, H, P):
    run(I.Workload("params", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.05, seed=H + P), with_x0=True, with_gxT=True)


@pytest.mark.parametrize("B,T,H,P", [(3, 40, 128, 64), (2, 130, 384, 192), (130, 16, 128, 64)])
def test_operand_orders_bf16(B, T, H, P):
    # plain order, plain order with a half-filled last tile, and the interleaved order of the fused kernels
    run(I.Workload("params", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.05, seed=H + P), with_x0=True, with_gxT=True)
