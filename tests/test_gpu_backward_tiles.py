"""Tile edges of the tensor-core backward kernels against the CPU oracle (needs a B200): latents around the 32-column units, the
128-lane blocks, the head pairs and the ranges of one launch; lengths around the 128-token tiles; tokens whose decode weights reach
beyond the bound of the one-exponential form; enough tiles for every accumulator and ring to wrap."""
import pytest

from paper_2508_12594_b200 import workloads
from tests.test_gpu_backward import assert_grads_close, gpu_backward, oracle_backward

pytestmark = pytest.mark.gpu

CASES = [  # B, H, N, M, D, masked_fraction, k_std
    (1, 2, 128, 16, 16, 0.0, 0.8),
    (2, 2, 129, 48, 32, 0.2, 0.8),
    (1, 3, 127, 64, 16, 0.0, 0.8),
    (1, 2, 2700, 64, 32, 0.1, 0.8),
    (1, 2, 385, 80, 8, 0.0, 0.8),
    (1, 1, 257, 16, 64, 0.0, 0.8),
    (1, 2, 300, 128, 64, 0.3, 0.8),
    (1, 1, 260, 192, 64, 0.0, 0.8),
    (1, 1, 260, 208, 64, 0.1, 0.8),
    (1, 1, 300, 448, 32, 0.0, 0.8),
    (1, 1, 300, 464, 32, 0.2, 0.8),
    (1, 2, 200, 1024, 16, 0.0, 0.8),
    (1, 2, 200, 1040, 8, 0.1, 0.8),
    (1, 2, 300, 64, 32, 0.1, 6.0),
    (1, 2, 300, 144, 16, 0.0, 9.0),
    (1, 1, 300, 64, 64, 0.0, 4.0),
]


@pytest.mark.parametrize("B,H,N,M,D,masked,k_std", CASES)
def test_backward_tile_edges(oracle, B, H, N, M, D, masked, k_std):
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=masked, with_dy=True, k_std=k_std)
    assert_grads_close(gpu_backward(inp), oracle_backward(oracle, inp), "bf16", f"{B}x{H}x{N}x{M}x{D}")
