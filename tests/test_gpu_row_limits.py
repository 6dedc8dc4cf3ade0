"""Row counts and widths past the limits of a grid's second and third dimension (65535 blocks)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io", ["f32", "bf16"])
def test_more_row_groups_than_a_grid_has_blocks_along_z(io):
    """8224 x 1024 rows are 65792 groups of 128: the sums for dD of a layer off the tile sizes.  The rows' gradients are
    compared with float64 sums; bound: fp32 sums of 128 rows, then of 64 partial sums at a time, stay below the suite's 1e-4."""
    import torch
    from paper_2502_20168_b200 import binding as sb, harness, inputs as I
    w = I.Workload("rows", B=8224, T=1024, H=8, P=8, io_dtype=io, p_done=0.0, seed=11)
    buf = harness.LayerBuffers(harness.device_drawn(w), io)
    buf.dD.fill_(float("nan"))
    buf.forward()
    buf.backward()
    sb.ssm_check(buf.ws)
    ref = torch.zeros(w.H, dtype=torch.float64, device="cuda")
    for u, gy in zip(buf.u.split(512), buf.gy.split(512)):
        ref += (u.double() * gy.double()).sum((0, 1))
    err = (buf.dD.double() - ref).abs() / (1 + ref.abs())
    assert float(err.max()) <= 1e-4
    # dB and dC, the products of the same launch: the sum of those of the two halves of the rows.  An element adds n rows in
    # fp32 in up to 64 slices; a chain of L additions of terms of random sign is off by about sqrt(L) 2^-24 of its sum, with
    # L = n / 64 = 131584 rows: 2.2e-5, relative to the 2-norm.
    whole = {k: getattr(buf, k).clone() for k in ("dB", "dC")}
    parts = {k: torch.zeros_like(v, dtype=torch.complex128) for k, v in whole.items()}
    for half in (slice(0, 4112), slice(4112, 8224)):
        d = {k: getattr(buf, k).cpu().numpy() for k in ("Lambda", "Delta", "Bc", "Cc", "D")}
        h = harness.LayerBuffers(dict(d, u=buf.u[half], gy=buf.gy[half], done=None), io)
        h.forward()
        h.backward()
        for k in parts:
            parts[k] += getattr(h, k)
        del h
    for k in parts:
        assert float(torch.linalg.vector_norm(whole[k] - parts[k]) / torch.linalg.vector_norm(parts[k])) <= 2.2e-5, k


def test_more_features_than_tiles_along_a_grid_dimension():
    """2097184 features are 65537 tiles of 32.  One step of a layer with 8 states: y and du elementwise against float64, dB and
    dC against the products they are (one row: no sums)."""
    import torch
    from paper_2502_20168_b200 import binding as sb, harness, inputs as I
    B, T, H, P = 1, 1, 2097184, 8
    d = I.draw_layer(I.Workload("wide", B=B, T=T, H=H, P=P, io_dtype="f32", p_done=0.0, seed=12))
    buf = harness.LayerBuffers(d, "f32")
    buf.forward()
    buf.backward()
    sb.ssm_check(buf.ws)
    c, r = torch.complex128, torch.float64
    Lam, dt, Bc, Cc = buf.Lambda.to(c), buf.Delta.to(r), buf.Bc.to(c), buf.Cc.to(c)
    u, gy, D = buf.u.to(r)[0, 0], buf.gy.to(r)[0, 0], buf.D.to(r)
    gamma = (torch.exp(Lam * dt) - 1) / Lam
    x = (gamma[:, None] * Bc) @ u.to(c)
    s = Cc.conj().T @ gy.to(c)
    assert float((buf.y[0, 0] - ((Cc @ x).real + D * u)).abs().max()) <= 1e-4
    assert float((buf.du[0, 0] - (((gamma[:, None] * Bc).conj().T @ s).real + D * gy)).abs().max()) <= 1e-4
    for got, ref in ((buf.dB, gamma.conj()[:, None] * s[:, None] * u), (buf.dC, gy[:, None] * x.conj()[None])):
        assert float(torch.linalg.vector_norm(got - ref) / torch.linalg.vector_norm(ref)) <= 1e-4
    assert torch.isfinite(buf.dLambda.real).all() and torch.isfinite(buf.dDelta).all()
