"""The output projections on CTA pairs with tiles of 128 columns (csrc/gemm_tc.cu) against the oracle: a last wide tile that
would be half empty, one round of narrow tiles, rows that end inside a tile and inside a pair's first half, several
rounds, and the sizes on either side of the rule."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_layer_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,P", [(41, 100, 512, 256), (48, 200, 384, 192), (150, 130, 384, 64), (20, 100, 768, 256), (97, 99, 512, 128),
                                     (64, 100, 768, 128), (64, 100, 256, 128), (45, 213, 640, 128), (3, 3201, 384, 256)])
def test_output_projections_bf16(B, T, H, P):
    run(I.Workload("narrow", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.01, seed=B + H), with_x0=True, with_gxT=True)
