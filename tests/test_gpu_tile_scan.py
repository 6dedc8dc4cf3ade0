"""Scans in the epilogue of the few-tile projections (csrc/gemm_tc_small.cu) against the oracle: sequences of 8 to 128 steps,
groups of rows that end short, tiles that hold one or several sequences and a last tile with fewer, clusters of 2 and of 4;
more sequences than rows of partial sums are kept; one step more than a tile (the streaming scans).  Stacks: a bf16 input of the first layer."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_layer_parity import run
from tests.test_gpu_stack_parity import run as run_stack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,P", [(1, 8, 256, 128), (17, 16, 256, 128), (5, 19, 256, 128), (3, 50, 256, 128), (16, 64, 256, 128), (9, 100, 512, 256),
                                     (7, 127, 256, 128), (8, 128, 512, 256), (5, 129, 256, 128), (520, 8, 128, 64), (13, 61, 384, 192),
                                     (40, 20, 128, 64)])
@pytest.mark.parametrize("states", [False, True])
def test_layers_fp32(B, T, H, P, states):
    from paper_2502_20168_b200 import binding as sb
    assert sb.ssm_layer_plan_string(sb.make_shape(B, T, H, P, "f32")).endswith("scans=in-epilogue" if T <= 128 else "scans=separate")
    run(I.Workload("tile", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.05 if states else 0.0, seed=B + T), with_x0=states, with_gxT=states)


@pytest.mark.parametrize("B,T,H,P", [(7, 50, 256, 128), (16, 64, 512, 256)])
def test_stacks_bf16(B, T, H, P):
    run_stack(I.Workload("tile_stack", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.02, n_layers=2, seed=B + T))
