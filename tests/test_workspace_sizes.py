"""Workspace sizes (host only): a layer workspace sized for a batch serves every smaller batch of the same shape, as the last,
smaller batch of an epoch needs it.  Widths that the tensor cores do not take, over the range where one kernel takes a pass."""
import pytest


@pytest.fixture(scope="module")
def sb():
    from paper_2502_20168_b200 import build
    build.build()
    from paper_2502_20168_b200 import binding
    return binding


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("H,P", [(8, 8), (16, 56), (32, 16), (40, 24), (136, 48), (176, 72), (184, 128), (200, 256), (248, 8)])
def test_a_layer_workspace_serves_smaller_batches(sb, io, H, P):
    for T in (1, 2, 7, 10, 20, 50, 64, 128, 500, 512, 700):
        sizes = [sb.ssm_layer_workspace_bytes(sb.make_shape(B, T, H, P, io)) for B in (*range(1, 65), 100, 256)]
        assert sizes == sorted(sizes), (T, sizes)
