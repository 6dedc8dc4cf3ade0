"""The kernels that take a small layer's pass at once (layer_small.cu) against the oracle: one state per CTA, one step, the longest
sequence, more threads than rows x columns and fewer, clusters of 8 and of 4 with the most sequences each takes, groups of 4
to 17 rows per scanning thread that end full and short; weight gradients as slices and as products of their own; and the shapes
just past its limits, which go to the separate kernels."""
import numpy as np
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_layer_parity import run
from tests.util import oracle_layer

pytestmark = pytest.mark.gpu

ONE_KERNEL = [   # rows of a group in brackets where they are not 4
    ("f32", 1, 1, 16, 8), ("f32", 1, 7, 8, 8), ("bf16", 1, 64, 32, 16), ("f32", 1, 512, 16, 16), ("f32", 1, 512, 8, 8), ("f32", 2, 33, 72, 40),
    ("bf16", 3, 4, 192, 120), ("f32", 1, 13, 248, 120), ("f32", 14, 65, 24, 104), ("bf16", 32, 50, 48, 32), ("f32", 14, 1, 8, 8), ("f32", 2, 8, 248, 256),
    ("f32", 1, 64, 8, 136),      # [5], the last group 4
    ("f32", 4, 50, 24, 256),     # [7], the last group 1
    ("f32", 14, 100, 8, 120),    # [6]
    ("bf16", 20, 128, 32, 64),   # [8]
    ("f32", 15, 130, 8, 72),     # [10]
    ("f32", 32, 256, 8, 48),     # [13], the last group 9
    ("f32", 32, 64, 8, 208),     # [16]
    ("bf16", 15, 65, 8, 208),    # [17], the last group 14
]
SEPARATE = [
    ("f32", 33, 50, 48, 32),                                                  # sequences
    ("f32", 1, 500, 40, 24), ("f32", 1, 512, 16, 56), ("f32", 32, 3, 200, 256),   # shared memory
    ("f32", 1, 513, 8, 8), ("f32", 1, 8, 264, 8), ("f32", 1, 8, 8, 264),      # steps, features, states
]
PRODUCTS = [   # slices of the weight gradients would need more workspace than the separate kernels: their products take s
    ("f32", 15, 18, 136, 48), ("f32", 32, 10, 184, 128), ("f32", 14, 16, 192, 128), ("f32", 4, 2, 208, 256), ("f32", 5, 16, 88, 248),
    ("bf16", 32, 3, 104, 40), ("f32", 22, 20, 184, 8),
]


def _run(io, B, T, H, P, states, kernels, launches):
    from paper_2502_20168_b200 import binding as sb
    plan = sb.ssm_layer_plan_string(sb.make_shape(B, T, H, P, io))
    before = sb.ssm_launch_count()
    run(I.Workload("small", B=B, T=T, H=H, P=P, io_dtype=io, p_done=0.05 if states else 0.0, seed=B + T + H), with_x0=states, with_gxT=states)
    if B in (14, 32) and plan.endswith("separate"):
        return   # the most clusters a full B200 holds: one with its SMs grouped otherwise may hold fewer
    assert plan == f"projections=cuda-cores scans={kernels}"
    assert sb.ssm_launch_count() - before in launches


@pytest.mark.parametrize("io,B,T,H,P", ONE_KERNEL)
@pytest.mark.parametrize("states", [False, True])
def test_small_layers(io, B, T, H, P, states):
    _run(io, B, T, H, P, states, "one-kernel", [2 if B == 1 else 4])   # (several: and the last two kernels of the backward pass)


@pytest.mark.parametrize("io,B,T,H,P", PRODUCTS)
@pytest.mark.parametrize("states", [False, True])
def test_small_layers_with_separate_weight_gradients(io, B, T, H, P, states):
    _run(io, B, T, H, P, states, "one-kernel", [5])


@pytest.mark.parametrize("io,B,T,H,P", SEPARATE)
@pytest.mark.parametrize("states", [False, True])
def test_past_the_limits(io, B, T, H, P, states):
    _run(io, B, T, H, P, states, "separate", range(8, 12))


def _close_in_norm(res, ref, tol=1e-5):   # chains of a few dozen fp32 sums: 1e-6
    for k in ("y", "xT", "du", "dLambda", "dDelta", "dB", "dC", "dD"):
        assert np.isfinite(res[k]).all(), k
        assert np.linalg.norm((res[k] - ref[k]).ravel()) <= tol * np.linalg.norm(np.asarray(ref[k]).ravel()), k


@pytest.mark.parametrize("B,T,H,P", [(1, 16, 32, 16), (3, 9, 72, 40)])
def test_range_of_the_projected_inputs(B, T, H, P):
    """B u leaves the range of fp32, gamma B u and all that follows do not."""
    from paper_2502_20168_b200 import harness
    d = I.draw_layer(I.Workload("range", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.05, seed=3))
    d["Delta"] = np.full(P, 1e-3, np.float32)
    d["Bc"] = (d["Bc"] * np.float32(1e25)).astype(np.complex64)
    d["u"] = d["u"] * np.float32(5e14)
    d["Cc"] = (d["Cc"] * np.float32(1e-25)).astype(np.complex64)
    d["gy"] = d["gy"] * np.float32(1e-2)
    assert np.abs(np.einsum("bth,ph->btp", d["u"].astype(np.float64), d["Bc"].astype(np.complex128))).max() > 3.5e38
    _close_in_norm(harness.run_layer(d, "f32"), oracle_layer(d))


@pytest.mark.parametrize("B,T,H,P", [(1, 16, 32, 16), (3, 9, 72, 40)])
def test_range_of_the_states_gradients(B, T, H, P):
    """Steps longer than 1: conj(gamma) s leaves the range of fp32, s and conj(gamma B) s do not."""
    from paper_2502_20168_b200 import harness
    d = I.draw_layer(I.Workload("range", B=B, T=T, H=H, P=P, io_dtype="f32", seed=3))
    d["Delta"] = np.linspace(0.5, 9.0, P).astype(np.float32)
    d["Lambda"] = np.linspace(-0.2, -0.01, P).astype(np.complex64)
    d["Bc"] = (d["Bc"] * np.float32(1e-20)).astype(np.complex64)
    d["u"] = d["u"] * np.float32(1e-10)
    d["gy"] = d["gy"] * np.float32(3e37)
    d["D"] = d["D"] * np.float32(1e-20)
    ref = oracle_layer(d)
    Abar = np.exp(d["Lambda"].astype(np.complex128) * d["Delta"])
    first = np.abs(ref["dx0"] / Abar.conj())   # s of the first step
    assert first.max() < 3.4e38 < (first * np.abs((Abar - 1) / d["Lambda"])).max()
    _close_in_norm(harness.run_layer(d, "f32"), ref)
