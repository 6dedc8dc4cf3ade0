"""Projections of few tiles (csrc/gemm_tc_small.cu) at the edges of their tiles: one row, one row more or less than a
128-row tile, output widths that leave the last 64-, 128- or 256-column tile partly empty, a contraction of one or
two k-blocks (clusters of at most as many CTAs), and the widest outputs."""
import numpy as np
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_half_glu import _run as run_gate
from tests.test_gpu_layer_parity import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,P", [(1, 1, 128, 64), (127, 1, 128, 64), (1, 129, 640, 64), (9, 57, 384, 320),
                                     (3, 43, 1152, 128), (60, 65, 384, 64), (31, 125, 768, 256),
                                     (31, 125, 512, 256)])   # CTA pairs, the last with one row tile
def test_bf16_edges(B, T, H, P):
    run(I.Workload("few", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.02, seed=B + H), with_x0=True, with_gxT=True)


@pytest.mark.parametrize("B,T,H,P", [(1, 1, 256, 128), (1, 127, 256, 128), (43, 3, 512, 128), (5, 205, 256, 384),
                                     (2, 64, 1024, 256), (37, 111, 256, 128),
                                     (1, 7, 128, 64), (2, 65, 128, 64), (5, 77, 384, 192), (9, 57, 640, 64)])
def test_fp32_edges(B, T, H, P):
    run(I.Workload("few32", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.02, seed=B + H), with_x0=True, with_gxT=True)


@pytest.mark.parametrize("rows,H", [(1, 128), (129, 256), (1000, 384), (3875, 512), (3875, 1024)])
def test_gate_edges_bf16(rows, H):
    run_gate(I.Workload("few_gate", B=1, T=rows, H=H, P=8, io_dtype="bf16", seed=rows + H))


@pytest.mark.parametrize("B,T,H,P", [(1, 65, 256, 128), (3, 4111, 256, 128), (2, 1025, 512, 384), (3, 1100, 384, 128), (3, 1100, 640, 64)])
def test_weight_gradients_from_planes_fp32(B, T, H, P):
    # one k-block and a row of the next; slices of several segments with a ragged end; one slice per tile; single CTAs on
    # long slices; pairs whose last tile is half empty
    run(I.Workload("nt32", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.01, seed=B + T), with_gxT=True)


@pytest.mark.parametrize("B,T,H,P", [(50, 131, 256, 128), (7, 301, 768, 384), (1, 12801, 256, 128), (37, 350, 384, 192)])
def test_many_tiles_fp32(B, T, H, P):
    """The persistent plane kernel: from 100 tiles on, a ragged last row of tiles, more tiles than CTAs.  Elementwise as
    everywhere but for dDelta, whose elements cancel to far below their scale in sums over thousands of rows (7 x 301 at
    (768, 384): scale 10^3, some elements below 1, where the worst is 2.5e-3 off, 2.7e-3 on the kernels that served these
    shapes before).  All parameter gradients also against their 2-norm.  Bound: operands are exact in their planes and
    dropped products are below 2^-24, so an element of a sum of n rows carries the rounding of its fp32 additions, sqrt(n)
    2^-24 of a term's size against sqrt(n) for the element: about 2^-24 per level of the chain rows -> states -> gradient;
    2^-24 x 64 = 4e-6 covers the three chained contractions (K up to 768 in steps of 16)."""
    from paper_2502_20168_b200 import harness
    from tests.util import TOL, assert_close, oracle_layer
    w = I.Workload("many32", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.01, seed=B + H)
    d = I.draw_layer(w, with_x0=True, with_gxT=True)
    res = harness.run_layer(d, "f32", with_x0=True, with_gxT=True)
    ref = oracle_layer(d, True, True)
    for k in ("y", "xT", "du", "dx0", "dLambda", "dB", "dC", "dD"):
        assert_close(k, res[k], ref[k], TOL["f32"])
    for k in ("dLambda", "dDelta", "dB", "dC", "dD"):
        off = np.linalg.norm(res[k] - ref[k]) / np.linalg.norm(ref[k])
        assert off <= 4e-6, (k, off)


def test_many_tiles_of_a_bf16_stack():
    # the first layer's bf16 input is one plane (three products), the last layer's output is bf16
    from tests.test_gpu_stack_parity import run as run_stack
    run_stack(I.Workload("many_stack", B=50, T=131, H=256, P=128, io_dtype="bf16", p_done=0.01, n_layers=2, seed=3))


@pytest.mark.parametrize("rows,H", [(5000, 512), (10300, 640)])
def test_gate_on_both_sides_of_the_pair_kernel_bf16(rows, H):
    run_gate(I.Workload("gate_pair", B=1, T=rows, H=H, P=8, io_dtype="bf16", seed=rows + H))
