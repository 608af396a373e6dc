"""Tile edges of the tensor-core backward kernels against the CPU oracle (needs a B200): latents around the 32-column units, the
128-lane blocks, the head pairs and the ranges of one launch; lengths around the 128-token tiles; tokens whose decode weights reach
beyond the bound of the one-exponential form; enough tiles for every accumulator and ring to wrap."""
import numpy as np
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import dev, to_np64
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
    (1, 2, 300, 336, 32, 0.1, 6.0),       # the same in the kernels that D = 32 takes beyond 320 latents, in one launch and in two
    (1, 1, 300, 528, 32, 0.0, 6.0),
    (1, 1, 300, 512, 32, 0.1, 0.8),       # the most latents of one launch at D = 32, and ranges beyond
    (1, 1, 300, 528, 32, 0.1, 0.8),
    (1, 1, 260, 400, 64, 0.1, 0.8),       # three and four ranges: launches that neither begin nor end the sums, dd from either array
    (1, 1, 260, 592, 64, 0.1, 0.8),
    (1, 2, 200, 1040, 32, 0.1, 0.8),
    (1, 1, 260, 160, 64, 0.0, 0.8),       # third part of Z: the most latents
    (1, 2, 40000, 32, 32, 0.1, 0.8),      # two sets of warps, several tiles each
    (2, 1, 40000, 16, 8, 0.0, 0.8),
    (1, 2, 20001, 48, 16, 0.1, 0.8),
    (8, 4, 20001, 256, 8, 0.0, 0.8),      # 32 heads: once over the chip leaves 20 SMs idle
    (8, 4, 20001, 96, 64, 0.0, 0.8),      # several rounds of CTAs over the chip
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


def dk_error_bound(inp, u):
    """What dK of one batch item may be off by before it is stored, element by element (float64).  u: what an operand of the products loses, 2^-17 for two
    roundings of bf16 halves, 2^-24 for a float32.  Per (token, latent): W_dec (A - e) and W_enc (C - de) as they enter the last product, |A - e| <= |A - dd| + |dd - e|
    with e from Y as it is stored (a 2^-7 of |dY| |Y|; bfloat16), and W_dec against dd - e; the errors of A (Z and the weights it was
    formed with), as far as they do not move all of a token's alike; those of C (dZ likewise); the weights' own (a rounded score, its distance from a
    rounded log-sum-exp, the exponential)."""
    Q, K, V, dY = (t.double().numpy() for t in (inp.Q, inp.K, inp.V, inp.dY))
    out = np.zeros(K.shape)
    for h in range(Q.shape[0]):
        q, k, v, g = Q[h], K[0, :, h], V[0, :, h], dY[0, :, h]
        S = k @ q.T
        dec, enc = np.exp(S - S.max(1, keepdims=True)), np.exp(S - S.max(0))
        dec /= dec.sum(1, keepdims=True)
        enc /= enc.sum(0)
        Z, Z_abs, dZ, dZ_abs = enc.T @ v, enc.T @ np.abs(v), dec.T @ g, dec.T @ np.abs(g)
        centred = Z - Z.mean(0)
        A, C = g @ centred.T, v @ dZ.T
        dd, de = (dec * A).sum(1, keepdims=True), (enc * C).sum(0)
        guess = 2.0 ** -7 * (np.abs(g) * np.abs(dec @ Z)).sum(1, keepdims=True)
        weight = 2.0 ** -21 + 2.0 ** -22 * np.abs(S).max(1, keepdims=True)
        formed = u if inp.Q.dtype == torch.bfloat16 else u + weight.max()
        a = formed * np.abs(g) @ (np.abs(centred) + Z_abs).T
        others = (1.0 - dec) * a + (dec * a).sum(1, keepdims=True) - dec * a
        c = 4 * formed * (np.abs(v) @ dZ_abs.T + (dZ_abs * Z_abs).sum(1))
        out[0, :, h] = (dec * ((u + weight) * np.abs(A - dd) + 2 * u * guess + others) + enc * ((u + weight) * np.abs(C - de) + c)) @ np.abs(q)
    return out


@pytest.mark.parametrize("dtype,H,N,M,D,k_std", [
    ("bf16", 2, 1200, 64, 32, 2.0), ("bf16", 2, 1200, 64, 32, 5.0), ("bf16", 2, 1500, 48, 16, 4.0), ("bf16", 2, 1000, 96, 64, 2.0),
    ("bf16", 2, 900, 208, 64, 2.0), ("bf16", 4, 1100, 64, 8, 6.0), ("bf16", 4, 1000, 32, 4, 8.0), ("bf16", 2, 700, 640, 32, 3.0),
    ("bf16", 2, 2000, 64, 32, 0.2),
    ("f32", 2, 1200, 64, 32, 5.0), ("f32", 2, 1000, 64, 64, 5.0), ("f32", 2, 1000, 33, 16, 4.0), ("f16", 2, 1200, 64, 32, 5.0), ("f16", 2, 1000, 40, 8, 6.0)])
def test_rows_of_peaked_softmaxes(oracle, dtype, H, N, M, D, k_std):
    """A token that follows one latent has a small row of dK, left of large numbers: every element of it within what its own terms allow.  (bfloat16 without
    e 20 to 75 times that, with dd formed first, in a sweep of its own, 13 to 70 times; now at most 0.15 of it; float32 and
    float16 with dd summed in float32 and not over the sum of the weights 900 to 2000 times, now 0.05.)"""
    inp = workloads.make_random(1, H, N, M, D, dtype=dtype, seed=N + M, with_dy=True, k_std=k_std)
    got, want = gpu_backward(inp)["dK"], oracle_backward(oracle, inp)["dK"]
    bits, least = {"bf16": (8, -133), "f16": (11, -25), "f32": (24, -149)}[dtype]
    half_ulp = np.maximum(2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-300))) - bits), 2.0 ** least)
    assert (np.abs(got - want) <= half_ulp + dk_error_bound(inp, 2.0 ** (-17 if dtype == "bf16" else -24))).all()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 0.0, 1e30])
@pytest.mark.parametrize("M,D", [(64, 32), (144, 16), (336, 32), (528, 32), (208, 64)])
def test_any_stored_output(oracle, M, D, value):
    """The stored Y is a first guess only (D = 64, and D = 32 with more than 320 latents, in one launch and in two; the two sweeps do not read it): what a caller
    left there has no say in the gradients."""
    inp = workloads.make_random(2, 2, 300, M, D, dtype="bf16", seed=M, with_dy=True)
    Q, K, V, dY = (dev(t) for t in (inp.Q, inp.K, inp.V, inp.dY))
    desc = flare.make_desc(Q, K)
    Y, Z, le, ld = flare.forward(Q, K, V, want_stats=True)
    dQ, dK, dV = torch.empty(Q.shape, device="cuda"), torch.empty_like(K), torch.empty_like(V)
    flare.flare_backward(desc, Q, K, V, None, Y.fill_(value), dY, Z, le, ld, dQ, dK, dV, flare.alloc_workspace(desc, flare.OP_BACKWARD))
    assert_grads_close(dict(dQ=to_np64(dQ), dK=to_np64(dK), dV=to_np64(dV)), oracle_backward(oracle, inp), "bf16", f"Y = {value}, M = {M}, D = {D}")


def test_small_weights_of_a_range_of_latents(oracle):
    """Latents worked off in two ranges.  The first token's largest decode score is to the second range, 2^91 above its score to the first latent, whose decode
    weight is below 2^-126; its encode weight there, 2^-48, is 2^55 times any other: its row of dV is that weight times one row of dZ."""
    N, M, D = 1024, 208, 64
    inp = workloads.make_random(1, 1, N, M, D, dtype="bf16", seed=4, with_dy=True)
    inp.Q.zero_()
    inp.Q[0, 0, 0], inp.Q[0, 1:112, 1], inp.Q[0, 112:, 2] = 1.0, 1.0, 1.0
    inp.K.zero_()
    inp.K[0, 0, 0, :3] = torch.tensor([-26.25, -13.875, 59.0])
    inp.K[0, 200, 0, 1], inp.K[0, 300, 0, 2] = 57.5, 132.0      # (in other tiles) raise lse_enc of the first range's other latents, and of the second range's
    got, want = gpu_backward(inp)["dV"][0, 0, 0], oracle_backward(oracle, inp)["dV"][0, 0, 0]
    assert np.linalg.norm(want) > 2.0 ** -60
    assert np.linalg.norm(got - want) <= 2.0 ** -7 * np.linalg.norm(want)     # (one rounding of the stored value, and as much again)
