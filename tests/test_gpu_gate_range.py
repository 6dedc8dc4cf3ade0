"""The half-GLU gate far out on the sigmoid, where v * sigmoid(z) is small but representable."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,rows,H", [("bf16", 300, 256), ("bf16", 33000, 512), ("bf16", 40, 24), ("f32", 40, 24)])
def test_gate_at_large_negative_arguments(io, rows, H):
    """v = 64 and W = -1.375 on the diagonal: GELU(v) = 64 and z = -88 exactly.  The few-tile kernel, the one on CTA pairs, and
    the elementwise kernels; bound: half a unit of the result's type (2^-9 for bf16) and 1e-5 for fp32's exponential."""
    import torch
    from paper_2502_20168_b200 import binding as sb
    dtype = torch.bfloat16 if io == "bf16" else torch.float32
    v = torch.full((1, rows, H), 64.0, device="cuda", dtype=dtype)
    gout = torch.ones_like(v) * 64
    W = torch.eye(H, device="cuda") * -1.375
    shape = sb.make_shape(1, rows, H, 8, io)
    ws = sb.alloc_workspace(sb.ssm_glu_workspace_bytes(shape))
    out, gv, dW = torch.empty_like(v), torch.empty_like(v), torch.empty_like(W)
    sb.ssm_glu_fwd(shape, W, v, out, ws)
    sb.ssm_glu_bwd(shape, W, v, gout, ws, gv, dW)
    sb.ssm_check(ws)
    s = 1.0 / (1.0 + math.exp(88.0))
    gz = 64.0 * 64.0 * s * (1.0 - s)
    tol = 2.0 ** -9 + 1e-5 if io == "bf16" else 1e-5
    for name, got, ref in (("out", out, 64.0 * s), ("gv", gv, 64.0 * s + gz * -1.375)):
        off = float((got.double() / ref - 1).abs().max())
        assert off <= tol, (name, off)
