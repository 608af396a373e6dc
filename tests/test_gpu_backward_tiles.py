"""Tile edges of the tensor-core backward kernels against the CPU oracle (needs a B200): latents around the 32-column units, the
128-lane blocks, the head pairs and the ranges of one launch; lengths around the 128-token tiles; tokens whose decode weights reach
beyond the bound of the one-exponential form; enough tiles for every accumulator and ring to wrap."""
import numpy as np
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


@pytest.mark.parametrize("B,H,N,M,masked", [(1, 1, 64, 16, 0.0), (1, 2, 129, 48, 0.0), (2, 2, 700, 128, 0.2), (1, 2, 900, 144, 0.0),
                                            (4, 2, 2048, 64, 0.0), (1, 2, 20011, 32, 0.1), (1, 1, 40000, 256, 0.0),
                                            (1, 2, 1500, 160, 0.1), (1, 2, 1500, 176, 0.0)])
def test_wide_heads_keep_float32_accuracy_of_dq(oracle, B, H, N, M, masked):
    """dQ at D = 64: its kernel multiplies Z, dZ and dS in three parts, so that what is left is the forward's and the dZ pass' weights in
    two bf16 halves.  A factor in two halves is off by at most 2^-18 of itself, with random sign: less than 2^-18 of the norm in all.  (One
    more factor in halves, or sums truncated on the tensor core over a whole split, put dQ at 4.3e-6 to 5.6e-6.)"""
    inp = workloads.make_random(B, H, N, M, 64, dtype="bf16", seed=N + M, masked_fraction=masked, with_dy=True, k_std=0.125)
    got, want = gpu_backward(inp)["dQ"], oracle_backward(oracle, inp)["dQ"]
    assert np.linalg.norm(got - want) <= 2.0 ** -18 * np.linalg.norm(want)
