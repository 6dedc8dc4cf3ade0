"""The kernels of single-step mode at the edges of their dispatch: the CUDA-core pair (few trajectories, rows off its
groups of 8), the cluster kernel (one row more than a 128-row tile, widths that leave the last column tile of a cluster
empty or partly filled, more state columns than features and the other way round), and fp32 wider than it takes."""
import pytest

from paper_2502_20168_b200 import inputs as I
from tests.test_gpu_step_mode import _rollout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("io,B,H,P", [("f32", 1, 256, 128), ("f32", 13, 512, 128), ("bf16", 3, 128, 64), ("bf16", 29, 384, 448),
                                      ("bf16", 129, 512, 256), ("bf16", 300, 384, 64), ("bf16", 2100, 128, 192),
                                      ("bf16", 257, 640, 320), ("f32", 129, 256, 128), ("f32", 1100, 256, 128),
                                      ("f32", 130, 512, 128)])
def test_rollout(io, B, H, P, in_place):
    _rollout(I.Workload("step_k", B=B, T=1, H=H, P=P, io_dtype=io, p_done=0.1, seed=B + H), 3, in_place)


# One kernel in clusters of 4 to 16 CTAs: the most trajectories it takes and one group more (two kernels for the halves), widths that leave
# warps of a cluster without columns in one of the two halves, one trajectory; and a contraction of 640 (the halves).
FEW = [("f32", 112, 256, 128), ("f32", 113, 256, 128), ("f32", 32, 512, 64), ("f32", 33, 512, 256), ("f32", 9, 128, 256), ("f32", 1, 384, 192),
       ("f32", 17, 640, 64), ("f32", 1, 512, 256), ("f32", 224, 128, 64), ("bf16", 112, 256, 128), ("bf16", 5, 128, 128), ("bf16", 25, 256, 64),
       ("bf16", 224, 128, 64), ("bf16", 225, 128, 64), ("bf16", 250, 128, 64), ("bf16", 8, 384, 64)]


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("io,B,H,P", FEW)
def test_rollout_of_few_trajectories(io, B, H, P, in_place):
    _rollout(I.Workload("step_c", B=B, T=1, H=H, P=P, io_dtype=io, p_done=0.1, seed=B + H + P), 4, in_place)


@pytest.mark.parametrize("io,B,H,P", [("f32", 1, 512, 256), ("f32", 4, 384, 192), ("f32", 13, 512, 64), ("f32", 2, 256, 64), ("f32", 100, 128, 64),
                                      ("f32", 16, 256, 128), ("bf16", 1, 256, 64), ("bf16", 61, 128, 64), ("bf16", 2, 128, 128)])
def test_steps_in_a_graph_are_the_same_bits(io, B, H, P):
    """A step in a graph may take two kernels where the same step by itself takes one."""
    import torch
    from paper_2502_20168_b200 import binding as sb, harness
    w = I.Workload("step_g", B=B, T=1, H=H, P=P, io_dtype=io, p_done=0.1, seed=B + H)
    q = harness.LayerBuffers(harness.device_drawn(w), io)
    shape = sb.make_shape(B, 1, H, P, io)
    ws = sb.alloc_workspace(sb.ssm_step_workspace_bytes(shape))
    sb.ssm_step_prepare(shape, q.Lambda, q.Delta, q.Bc, q.Cc, ws)
    x = torch.view_as_complex(torch.randn((B, P, 2), device="cuda"))
    out = [(torch.empty_like(q.u), torch.empty_like(x)) for _ in range(2)]
    step = lambda y, xn: sb.ssm_step(shape, q.D, q.u, q.done, x, xn, y, ws)
    step(*out[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(*out[1])
    graph.replay()
    torch.cuda.synchronize()
    sb.ssm_check(ws)
    for a, b in zip(*out):
        assert torch.equal(a, b)
