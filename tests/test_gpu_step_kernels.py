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


# One kernel in clusters of 2 to 16 CTAs: the most trajectories it takes and one group more, widths that leave warps of a
# cluster without columns in one of the two halves, a contraction of 64 (half a warp's lanes) and of 640.
@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("io,B,H,P", [("f32", 112, 256, 128), ("f32", 113, 256, 128), ("f32", 32, 512, 64), ("f32", 33, 512, 256),
                                      ("f32", 9, 128, 256), ("f32", 1, 384, 192), ("f32", 17, 640, 64), ("bf16", 112, 256, 128),
                                      ("bf16", 5, 128, 128), ("bf16", 25, 256, 64), ("bf16", 250, 128, 64), ("bf16", 8, 384, 64)])
def test_rollout_of_few_trajectories(io, B, H, P, in_place):
    _rollout(I.Workload("step_c", B=B, T=1, H=H, P=P, io_dtype=io, p_done=0.1, seed=B + H + P), 4, in_place)
