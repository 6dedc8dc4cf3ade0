"""Sums and recurrences over many rows: how far the order of the fp32 operations lets their results drift from the oracle's."""
import numpy as np
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.util import oracle_layer

pytestmark = pytest.mark.gpu


def _off(got, ref):
    return float(np.linalg.norm(got - ref) / np.linalg.norm(ref))


def test_gate_weights_fp32_over_12800_rows():
    # 256 output tiles, which fill the GPU with a single slice: elementwise within the suite's bound, as with few rows
    from tests.test_gpu_half_glu import _run
    _run(I.Workload("glu_rows", B=1, T=12800, H=1024, P=8, io_dtype="f32", seed=3))


def test_layer_weights_fp32_off_the_tile_widths():
    """A chain of L additions of terms of random sign carries a relative rounding error of about sqrt(L / 6) 2^-24 (each
    addition rounds by 2^-24 / sqrt(3) of a partial sum that grows with the root of the terms).  Chains of at most 512 rows:
    5.5e-7; bound: twice that.  (One chain over all 8000 rows: 2.2e-6.)"""
    from paper_2502_20168_b200 import harness
    w = I.Workload("wide_odd", B=8, T=1000, H=1032, P=520, io_dtype="f32", p_done=0.002, seed=7)
    d = I.draw_layer(w)
    res = harness.run_layer(d, "f32")
    ref = oracle_layer(d)
    assert _off(res["dB"], ref["dB"]) <= 1.1e-6
    assert _off(res["dC"], ref["dC"]) <= 1.1e-6


def test_layer_weights_bf16_wide_outputs():
    """The tensor core truncates its fp32 accumulator at every addition: a chain of n additions whose partial sums grow with
    the root of their number is about n 2^-25 2/3 off its sum.  16384 rows in two slices of 128 blocks of 64 rows, four
    additions a block: 1.0e-5; bound: one and a half times that (the states' 16-bit mantissas add less).  One chain: 2.0e-5."""
    from paper_2502_20168_b200 import harness
    w = I.Workload("wide16", B=16, T=1024, H=1024, P=512, io_dtype="bf16", p_done=0.002, seed=7)
    d = I.draw_layer(w)
    res = harness.run_layer(d, "bf16")
    ref = oracle_layer(d)
    assert _off(res["dB"], ref["dB"]) <= 1.5e-5
    assert _off(res["dC"], ref["dC"]) <= 1.5e-5


@pytest.mark.parametrize("B,T,H,P", [(18, 1024, 256, 128), (18, 1088, 256, 128), (18, 2112, 256, 128), (17, 3203, 256, 128),   # CTA pairs
                                     (8, 1024, 384, 192), (8, 1088, 384, 192), (8, 2112, 384, 192), (7, 3203, 384, 192)])
def test_segments_of_a_slice_bf16(B, T, H, P):
    """Slices of 16 blocks of 64 rows (one segment), 17, 33 and about 50, the last one ragged.  The weights and the states
    carry 16 bits each (2^-17), and so does what the recurrence makes of them; bound: four such errors."""
    from paper_2502_20168_b200 import harness
    w = I.Workload("segs", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.01, seed=B + T)
    d = I.draw_layer(w)
    res = harness.run_layer(d, "bf16")
    ref = oracle_layer(d)
    for k in ("dB", "dC"):
        assert _off(res[k], ref[k]) <= 4 * 2.0 ** -17, k


@pytest.mark.parametrize("B,T,H,P", [(16, 1000, 512, 256), (6, 4096, 512, 256), (40, 1500, 256, 128), (150, 2048, 128, 64)])
def test_states_of_long_sequences_bf16(B, T, H, P):
    """The final state after T steps of slowly decaying states, on the kernels that scan in their epilogue (both CTAs of a
    pair on one sequence, or one each).  Bbar carries 16 bits: up to 2^-17 off, 2^-18 on average over a sum.  The
    multipliers over 16 and 128 steps are rounded once, by up to 2^-25 of their size, which a state that lives through T
    steps meets T / 16 times.  Bound: 2^-18 + T / 16 2^-25.  (A multiplier that carries the rounding of a single step 16
    times over is off by T / 2 2^-25 on average: 1.5e-5 after 1000 steps, 6e-5 after 4096.)"""
    from paper_2502_20168_b200 import harness
    w = I.Workload("long_x", B=B, T=T, H=H, P=P, io_dtype="bf16", p_done=0.0, seed=7)
    d = I.draw_layer(w)
    d["Delta"] = np.full_like(d["Delta"], 1e-3)
    res = harness.run_layer(d, "bf16")
    off = _off(res["xT"], oracle_layer(d)["xT"])
    print(f"T = {T}: xT {off:.2e} off")
    assert off <= 2.0 ** -18 + T / 16 * 2.0 ** -25


def test_layernorm_bias_gradient_over_a_million_rows():
    """dln_bias of the last layer is the plain sum of gout over the rows.  Chains of at most 16 rows a warp, 8 warps and groups
    of 64 such sums, the rest in double: about sqrt(L / 6) 2^-24 for each of these lengths, 1e-7, and the final rounding,
    3e-8; bound: twice their sum.  (443 rows a warp: 4.3e-7.)"""
    import torch
    from paper_2502_20168_b200 import binding as sb, harness
    w = I.Workload("ln_rows", B=1024, T=1024, H=128, P=8, io_dtype="f32", p_done=0.0, n_layers=2, seed=7)
    s = harness.StackBuffers(harness.device_drawn(w), "f32")
    s.forward()
    s.backward()
    sb.ssm_check(s.ws)
    ref = s.gout.double().sum((0, 1))
    off = torch.linalg.vector_norm(s.grads[-1]["dln_bias"] - ref) / torch.linalg.vector_norm(ref)
    assert float(off) <= 2.6e-7


@pytest.mark.parametrize("B,T,H,P", [(8, 1000, 384, 192), (8, 1000, 512, 256), (7, 1003, 640, 320), (8, 1000, 256, 192)])
def test_projections_fp32_in_segments(B, T, H, P):
    """fp32 layers of many tiles without the skip term: y and du are a projection, the recurrence and a projection.  The tensor
    core truncates at every addition, n 2^-25 2/3 for a chain of n (as above), and the two projections' losses add.  Chains
    of 16 additions of 16 products; bound: 2 x 16 x 2^-25 2/3 and 2^-24 for the rest.  (Chains of 24 and 32, over all of K: 7.7e-7
    and 1.0e-6.)  Inner lengths of one segment (256), of one and a half, two and two and a half."""
    from paper_2502_20168_b200 import harness
    w = I.Workload("planes_k", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.002, seed=7)
    d = I.draw_layer(w)
    d["D"] = np.zeros_like(d["D"])
    res = harness.run_layer(d, "f32")
    ref = oracle_layer(d)
    for k in ("y", "du"):
        off = _off(res[k], ref[k])
        print(f"({H}, {P}): {k} {off:.2e} off")
        assert off <= 2 * 16 * 2.0 ** -25 * 2 / 3 + 2.0 ** -24, k
