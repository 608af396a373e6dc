"""The two sweeps over the tokens of the bfloat16 backward (heads up to 32 wide) where they can go wrong, against the CPU oracle (needs a B200): latents
around the units of 64 and the most of one launch, ranges of unequal size side by side and one after the other, more tiles to a CTA than tensor memory adds up in a row (with one and with two
sets of warps), rows that leave by a tile's copy at the end of a batch item, narrow heads."""
import numpy as np
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import dev, to_np64
from tests.test_gpu_backward import assert_grads_close, gpu_backward, oracle_backward
from tests.test_gpu_backward_tiles import dk_error_bound
from tests.test_gpu_fullsize import _float64_z_and_dq

pytestmark = pytest.mark.gpu

CASES = [  # B, H, N, M, D, masked_fraction
    (1, 2, 60, 16, 32, 0.0),              # less than a tile
    (3, 2, 255, 32, 32, 0.2),             # rows past the end of an item are another item's
    (3, 3, 130, 48, 16, 0.1),
    (2, 2, 640, 112, 32, 0.0),
    (1, 2, 385, 176, 32, 0.1),
    (2, 4, 383, 80, 8, 0.1),
    (2, 4, 385, 64, 4, 0.1),
    (1, 1, 700, 320, 32, 0.1),            # the most latents at D = 32, few tiles and more than a hundred, and one more (other kernels)
    (4, 8, 700, 320, 32, 0.1),
    (1, 8, 250, 256, 32, 0.1),            # at 240 and 256 latents sixteen tiles, and more
    (1, 8, 300, 240, 32, 0.1),
    (1, 1, 700, 336, 32, 0.1),
    (1, 1, 300, 768, 16, 0.0),            # few tokens, ranges of latents side by side: the last of all sizes, one and several tiles to a CTA
    (1, 2, 300, 784, 16, 0.1),
    (1, 2, 260, 1552, 8, 0.0),
    (3, 3, 130, 544, 16, 0.1),
    (2, 2, 383, 400, 4, 0.1),
    (1, 4, 4000, 1040, 8, 0.0),
    (1, 9, 1100, 2048, 16, 0.1),
    (4, 8, 1024, 768, 16, 0.0),           # the most of one launch at D = 16
    (1, 64, 4800, 784, 16, 0.1),          # ranges one after the other: two, the second shorter; three
    (1, 64, 4800, 1552, 8, 0.0),
    (2, 32, 4800, 1040, 4, 0.1),
    (37, 4, 8400, 16, 8, 0.0),            # 66 tiles to a CTA, two sets of warps
    (37, 4, 8272, 16, 32, 0.0),           # 65 tiles, the last by itself; warps without columns run ahead of the others
    (37, 4, 8400, 48, 16, 0.1),           # one set
]


def some_heads(inp, heads):
    """The inputs of these heads alone (the oracle takes minutes for 64)."""
    cut = lambda x: None if x is None else x[:, :, heads].contiguous()
    return workloads.Inputs(Q=inp.Q[heads].contiguous(), K=cut(inp.K), V=cut(inp.V), key_mask=inp.key_mask, dY=cut(inp.dY))


def gradients_of(inp, heads):
    got = gpu_backward(inp)
    return dict(dQ=got["dQ"][heads], dK=got["dK"][:, :, heads], dV=got["dV"][:, :, heads])


@pytest.mark.parametrize("B,H,N,M,D,masked", CASES)
def test_backward_in_two_sweeps(oracle, B, H, N, M, D, masked):
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=masked, with_dy=True, k_std=0.8)
    heads = [0, H - 1] if H >= 32 else list(range(H))
    assert_grads_close(gradients_of(inp, heads), oracle_backward(oracle, some_heads(inp, heads)), "bf16", f"{B}x{H}x{N}x{M}x{D}")


# Ranges of latents side by side (few tokens) and one after the other (many).
RANGES = [(2, 700, 784, 16), (4, 500, 1552, 8), (4, 500, 1040, 4), (64, 4800, 784, 16), (64, 4800, 1552, 8)]


@pytest.mark.parametrize("H,N,M,D", RANGES)
def test_peaked_softmaxes_over_ranges_of_latents(oracle, H, N, M, D):
    """dd is what the ranges' shares of it add up to, each a float and what that lost: a token that follows one latent has a small row of dK, left of
    large numbers, within what its own terms allow element by element."""
    inp = workloads.make_random(1, H, N, M, D, dtype="bf16", seed=N + M, with_dy=True, k_std=80.0 / D if D > 4 else 12.0)
    heads = [0, H - 1]
    few = some_heads(inp, heads)
    got, want = gradients_of(inp, heads)["dK"], oracle_backward(oracle, few)["dK"]
    half_ulp = np.maximum(2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-300))) - 8), 2.0 ** -133)
    assert (np.abs(got - want) <= half_ulp + dk_error_bound(few, 2.0 ** -17)).all()


@pytest.mark.parametrize("H,N,M,D", RANGES)
def test_very_different_latents_over_ranges(oracle, H, N, M, D):
    """lse_enc spread over several hundred powers of two within a range and between ranges: a weight of the encode softmax has an exponential of its own."""
    inp = workloads.make_random(1, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=0.1, with_dy=True)
    inp.Q.mul_(torch.linspace(0.05, 30.0, M)[None, :, None].to(inp.Q.dtype))
    heads = [0, H - 1]
    assert_grads_close(gradients_of(inp, heads), oracle_backward(oracle, some_heads(inp, heads)), "bf16", f"spread {H}x{N}x{M}x{D}")


@pytest.mark.parametrize("H,N,M,D", RANGES)
def test_features_with_a_mean_over_ranges(oracle, H, N, M, D):
    """As in test_gpu_backward_tiles.py: dK within 2^-14 of its norm, beyond the rounding of what is stored, where the rows of Z are nearly equal."""
    inp = workloads.make_random(1, H, N, M, D, dtype="bf16", seed=N + M, with_dy=True, k_std=D ** -0.5)
    inp.V.mul_(D ** -0.5).add_(1.0)
    heads = [0, H - 1]
    got, want = gradients_of(inp, heads)["dK"], oracle_backward(oracle, some_heads(inp, heads))["dK"]
    half_ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-300))) - 8)
    assert np.linalg.norm(np.maximum(np.abs(got - want) - half_ulp, 0.0)) <= 2.0 ** -14 * np.linalg.norm(want)


@pytest.mark.parametrize("H,N,M,first", [(1, 1024, 784, 64), (64, 4800, 784, 448)])
def test_a_small_weight_of_one_range(oracle, H, N, M, first):
    """test_small_weights_of_a_range_of_latents of test_gpu_backward_tiles.py at D = 16, with the first range's `first` latents."""
    inp = workloads.make_random(1, H, N, M, 16, dtype="bf16", seed=4, with_dy=True)
    inp.Q.zero_()
    inp.Q[0, 0, 0], inp.Q[0, 1:first, 1], inp.Q[0, first:, 2] = 1.0, 1.0, 1.0
    inp.K.zero_()
    inp.K[0, 0, 0, :3] = torch.tensor([-26.25, -13.875, 59.0])
    inp.K[0, 200, 0, 1], inp.K[0, 300, 0, 2] = 57.5, 132.0
    got, want = gradients_of(inp, [0])["dV"][0, 0, 0], oracle_backward(oracle, some_heads(inp, [0]))["dV"][0, 0, 0]
    assert np.linalg.norm(want) > 2.0 ** -60
    assert np.linalg.norm(got - want) <= 2.0 ** -7 * np.linalg.norm(want)


@pytest.mark.parametrize("M,D", [(32, 32), (64, 32), (32, 16)])
def test_sums_over_tokens_are_made_of_few_parts(M, D):
    """The halves of the factors leave 2^-18 of dQ's norm.  The tensor core truncates its sums: a part added to one of uniform size loses 2^-24 / 3 of the whole on
    average.  A CTA has 14 tiles of eight parts, shared out to four sums (dQ at D = 32, M = 64: two): some 32 parts, in dZ and again in dQ.  (One sum of all: 5.5e-6 to 5.9e-6.)"""
    inp = workloads.make_random(1, 8, 65536, M, D, dtype="bf16", seed=65536 + M, with_dy=True, k_std=D ** -0.5)
    Q, K, V, dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.dY)
    _, dQ, _, _ = flare.forward_backward(Q, K, V, dY, check=True)
    want = torch.stack([_float64_z_and_dq(Q[h], K[0, :, h], V[0, :, h], dY[0, :, h])[1] for h in range(8)])
    assert (dQ - want).norm() <= (2.0 ** -18 + 2 * 32 * 2.0 ** -24 / 3) * want.norm()


def float64_gradients(Q, K, V, dY, Q_dec=None):
    """Of one head in float64 by plain torch, on the device, a slice of tokens at a time: dQ, dK and dV; with latent queries of its own for decode dQ of encode and
    of decode, the parts of dK from encode and from decode, and dV."""
    Qe, Qd, step = Q.double(), (Q if Q_dec is None else Q_dec).double(), 1 << 15
    at = range(0, K.shape[0], step)
    S = lambda a, q: K[a:a + step].double() @ q.T
    le = torch.logsumexp(torch.stack([torch.logsumexp(S(a, Qe), 0) for a in at]), 0)
    Z = sum(torch.exp(S(a, Qe) - le).T @ V[a:a + step].double() for a in at)
    dZ = sum(torch.softmax(S(a, Qd), 1).T @ dY[a:a + step].double() for a in at)
    de, dQe, dQd, dKe, dKd, dV = (dZ * Z).sum(1), torch.zeros_like(Qe), torch.zeros_like(Qd), [], [], []
    for a in at:
        k, v, g = (x[a:a + step].double() for x in (K, V, dY))
        Wd, We, A = torch.softmax(S(a, Qd), 1), torch.exp(S(a, Qe) - le), g @ Z.T
        dSd, dSe = Wd * (A - (Wd * A).sum(1, keepdim=True)), We * (v @ dZ.T - de)
        dQe += dSe.T @ k
        dQd += dSd.T @ k
        dKe.append(dSe @ Qe)
        dKd.append(dSd @ Qd)
        dV.append(We @ dZ)
    dKe, dKd, dV = torch.cat(dKe), torch.cat(dKd), torch.cat(dV)
    return (dQe + dQd, dKe + dKd, dV) if Q_dec is None else (dQe, dQd, dKe, dKd, dV)


@pytest.mark.parametrize("B,H,N,M,D", [(1, 8, 150001, 784, 16), (2, 8, 140000, 1040, 8), (1, 32, 40000, 784, 16)])
def test_chunks_of_tokens_between_ranges_of_latents(B, H, N, M, D):
    """More tokens than the rows that the ranges leave to one another have room for: several launches per range, each a chunk of the tokens.
    dQ: 2^-18 from the halves of its factors, and at most 512 parts in a row, in dZ and again in dQ (see above)."""
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, with_dy=True, k_std=D ** -0.5)
    Q, K, V, dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.dY)
    desc = flare.make_desc(Q, K)
    assert flare.flare_launch_count(desc, flare.OP_BACKWARD) > 3 + 2 * 2
    _, dQ, dK, dV = flare.forward_backward(Q, K, V, dY, check=True)
    for h in (0, H - 1):
        each = [float64_gradients(Q[h], K[b, :, h], V[b, :, h], dY[b, :, h]) for b in range(B)]
        got = dict(dQ=to_np64(dQ[h]), dK=to_np64(dK[:, :, h]), dV=to_np64(dV[:, :, h]))
        want = dict(dQ=to_np64(sum(x[0] for x in each)), dK=to_np64(torch.stack([x[1] for x in each])), dV=to_np64(torch.stack([x[2] for x in each])))
        assert_grads_close(got, want, "bf16", f"{B}x{H}x{N}x{M}x{D}")
        assert np.linalg.norm(got["dQ"] - want["dQ"]) <= (2.0 ** -18 + 2 * 512 * 2.0 ** -24 / 3) * np.linalg.norm(want["dQ"])


def test_separate_decode_queries_over_ranges_one_after_the_other():
    """The two runs of the sweeps each store their part of dK in bfloat16: it is off by a rounding of either part and one of their sum."""
    B, H, N, M, D = 1, 64, 4800, 784, 8
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=3, with_dy=True, k_std=0.8)
    Qe, K, V, dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.dY)
    Qd = dev(workloads.make_random(B, H, 1, M, D, dtype="bf16", seed=4).Q)
    desc = flare.make_desc(Qe, K)
    scratch = lambda op: torch.empty(flare.flare_variant_workspace_bytes(desc, op, False, True), dtype=torch.uint8, device="cuda")
    f32 = lambda *shape: torch.empty(*shape, dtype=torch.float32, device="cuda")
    Y, Z, le, ld, dQe, dQd, dK, dV = torch.empty_like(K), f32(B, H, M, D), f32(B, H, M), f32(B, N, H), f32(H, M, D), f32(H, M, D), torch.empty_like(K), torch.empty_like(V)
    flare.flare_forward_variant(desc, False, Qe, Qd, K, V, None, Y, Z, le, ld, scratch(flare.OP_FORWARD))
    ws = scratch(flare.OP_BACKWARD)
    flare.flare_backward_variant(desc, False, Qe, Qd, K, V, None, Y, dY, Z, le, ld, dQe, dQd, dK, dV, ws)
    flare.flare_check(ws)
    for h in (0, H - 1):
        we, wd, ke, kd, wv = (to_np64(x) for x in float64_gradients(Qe[h], K[0, :, h], V[0, :, h], dY[0, :, h], Qd[h]))
        got_k, rms = to_np64(dK[0, :, h]), np.sqrt(np.mean((ke + kd) ** 2))
        assert (np.abs(got_k - ke - kd) - 2.0 ** -8 * (np.abs(ke) + np.abs(kd) + np.abs(ke + kd))).max() <= 2e-2 * rms
        for got, want in ((dQe, we), (dQd, wd)):
            assert_grads_close(dict(dQ=to_np64(got[h]), dK=wv, dV=to_np64(dV[0, :, h])), dict(dQ=want, dK=wv, dV=wv), "bf16", f"head {h}")
