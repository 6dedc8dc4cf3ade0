"""Stack kernels at the edges of their dispatch: widths on both sides of the warp-per-row LayerNorm's register tiles
(256, 512, 1024 features) and past them, more rows than its CTAs take at once, and more layers than one launch of the
parameter kernels takes (on the CUDA-core and on the plane path)."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_stack_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,B,T,H,P", [(2, 1, 5, 264, 16), (2, 3, 7, 520, 8), (1, 1, 11, 1024, 8), (2, 1, 9, 1032, 8),
                                       (1, 5, 1001, 64, 8)])
def test_layernorm_widths(L, B, T, H, P):
    run(I.Workload("stack_ln", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.05, n_layers=L, seed=H + T))


@pytest.mark.parametrize("L,H,P", [(18, 16, 8), (17, 256, 128)])
def test_more_layers_than_a_batch(L, H, P):
    run(I.Workload("stack_deep", B=2, T=12, H=H, P=P, io_dtype="bf16", p_done=0.05, n_layers=L, seed=L + H))
