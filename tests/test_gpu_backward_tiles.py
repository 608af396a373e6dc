"""Tile edges of the tensor-core backward kernels against the CPU oracle (needs a B200): latents around the 32-column units, the
128-lane blocks, the head pairs and the ranges of one launch; lengths around the 128-token tiles; tokens whose decode weights reach
beyond the bound of the one-exponential form; enough tiles for every accumulator and ring to wrap."""
import numpy as np
import pytest
import torch

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
    (1, 1, 300, 512, 32, 0.1, 0.8),       # the most latents of one launch at D = 32, and ranges beyond
    (1, 1, 300, 528, 32, 0.1, 0.8),
    (1, 1, 260, 160, 64, 0.0, 0.8),       # third part of Z: the most latents
    (1, 2, 40000, 32, 32, 0.1, 0.8),      # two sets of warps, several tiles each
    (2, 1, 40000, 16, 8, 0.0, 0.8),
    (1, 2, 20001, 48, 16, 0.1, 0.8),
    (8, 4, 20001, 256, 8, 0.0, 0.8),      # several rounds of CTAs over the chip, token side
]


@pytest.mark.parametrize("B,H,N,M,D,masked,k_std", CASES)
def test_backward_tile_edges(oracle, B, H, N, M, D, masked, k_std):
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=masked, with_dy=True, k_std=k_std)
    assert_grads_close(gpu_backward(inp), oracle_backward(oracle, inp), "bf16", f"{B}x{H}x{N}x{M}x{D}")


@pytest.mark.parametrize("B,H,N,M,D,masked", [(1, 2, 300, 16, 32, 0.2), (1, 2, 2700, 96, 16, 0.0), (2, 1, 300, 144, 8, 0.1),
                                              (1, 1, 300, 48, 64, 0.1), (1, 1, 257, 640, 32, 0.0)])
def test_latents_of_very_different_norm(oracle, B, H, N, M, D, masked):
    """The latents' lse_enc spread over several hundred powers of two: no common factor can take W_enc from W_dec, and the token kernel
    exponentiates it by itself."""
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=masked, with_dy=True)
    inp.Q.mul_(torch.linspace(0.05, 30.0, M)[None, :, None].to(inp.Q.dtype))
    want = oracle_backward(oracle, inp)
    assert_grads_close(gpu_backward(inp), want, "bf16", f"spread {B}x{H}x{N}x{M}x{D}")


@pytest.mark.parametrize("B,H,N,M,D", [(1, 2, 20011, 96, 16), (1, 1, 40000, 32, 32), (1, 1, 9000, 128, 64), (1, 1, 9000, 640, 32)])
def test_features_with_a_mean(oracle, B, H, N, M, D):
    """Values around 1: the rows of Z are nearly equal, and dS is what is left of large numbers unless their mean is taken out first.  Then
    dK, before it is rounded to bfloat16, is off by the halves (2^-17 of itself) of the centred Z, of a weight and of dS, and by Z's own error, of
    the same kind: 2^-15 of the norm, allowed twice over.  (Without: 1.4e-4 to 1.8e-3, and up to 2.7 times that in the one-sweep form.)"""
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, with_dy=True, k_std=D ** -0.5)
    inp.V.mul_(D ** -0.5).add_(1.0)
    got, want = gpu_backward(inp)["dK"], oracle_backward(oracle, inp)["dK"]
    half_ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-300))) - 8)
    beyond = np.maximum(np.abs(got - want) - half_ulp, 0.0)
    assert np.linalg.norm(beyond) <= 2.0 ** -14 * np.linalg.norm(want)


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
