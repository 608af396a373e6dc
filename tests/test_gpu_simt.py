"""The float32 / float16 kernels at the edges of their tiles (needs a B200): rows in blocks of 8 per warp and up to 8 warps,
columns in tiles of 64 (32 at head width 64), against the oracle, forward and backward."""
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import assert_forward_close, gpu_forward, oracle_forward
from tests.test_gpu_backward import assert_grads_close, gpu_backward, oracle_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("B,H,N,M,D,masked", [
    (1, 2, 63, 8, 16, 0.0), (1, 2, 64, 9, 16, 0.2), (2, 1, 65, 16, 8, 0.0), (1, 2, 127, 17, 32, 0.3), (1, 1, 129, 33, 16, 0.0),
    (1, 2, 191, 64, 4, 0.0), (1, 1, 193, 65, 64, 0.2), (1, 1, 31, 257, 16, 0.0), (1, 1, 385, 129, 32, 0.0), (3, 8, 700, 20, 16, 0.1),
])
def test_tile_edges(oracle, B, H, N, M, D, masked, dtype):
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M, masked_fraction=masked, with_dy=True, k_std=0.8)
    what = f"{dtype} B{B}H{H}N{N}M{M}D{D}"
    assert_forward_close(gpu_forward(inp, scale=0.7, canary=True), oracle_forward(oracle, inp, 0.7), dtype, what)
    assert_grads_close(gpu_backward(inp, 0.7), oracle_backward(oracle, inp, 0.7), dtype, what)


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("B,H,N,M,D", [(1, 2, 700, 24, 4), (1, 1, 520, 40, 8), (1, 2, 1300, 16, 16), (1, 1, 600, 72, 32), (1, 1, 300, 33, 64)])
def test_scores_climb(oracle, B, H, N, M, D, dtype):
    """Scores that grow by tens along the tokens and along the latents: the softmax references move several times, in encode and decode.  A
    score of 64 is rounded by 2^-19, which the bounds of the other cases allow for."""
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M, k_std=0.8)
    inp.K.mul_(torch.linspace(0.05, 4.0, N)[None, :, None, None].to(inp.K.dtype))
    inp.Q.mul_(torch.linspace(0.5, 2.0, M)[None, :, None].to(inp.Q.dtype))
    scale = 2.0 * D ** -0.5
    assert_forward_close(gpu_forward(inp, scale), oracle_forward(oracle, inp, scale), dtype, f"climb {dtype} B{B}H{H}N{N}M{M}D{D}")


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("B,H,N,M,D,masked", [
    (1, 1, 1, 1, 4, 0.0), (1, 2, 7, 9, 16, 0.3), (1, 9, 1023, 64, 32, 0.1), (1, 9, 1024, 64, 32, 0.0), (1, 2, 2048, 32, 16, 0.0), (1, 3, 2041, 33, 8, 0.2),
    (2, 5, 512, 64, 32, 0.2), (2, 5, 1024, 31, 16, 0.0), (4, 9, 1017, 64, 8, 0.5), (1, 10, 130, 17, 4, 1.0),
])
def test_forward_in_one_launch(B, H, N, M, D, masked, dtype):
    """The form of small forwards against the general kernels (encode, then decode) on the same inputs: either side of the cluster sizes and of
    the most tokens, lengths that leave blocks a part of a tile or nothing, every token masked.  Both round the same float32 steps in another order:
    the bound of each against the oracle, twice; a stored float16 may land on the next value."""
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M, masked_fraction=masked, k_std=0.8)
    Q, K, V, mask = (None if t is None else t.cuda() for t in (inp.Q, inp.K, inp.V, inp.key_mask))
    desc = flare.make_desc(Q, K, 0.7)
    assert flare.flare_launch_count(desc, flare.OP_FORWARD) == 1
    Y, Z, le, ld = flare.forward(Q, K, V, mask, 0.7, want_stats=True)
    assert torch.equal(flare.forward(Q, K, V, mask, 0.7), Y)
    Z2, le2, Y2, ld2 = torch.empty_like(Z), torch.empty_like(le), torch.empty_like(Y), torch.empty_like(ld)
    flare.flare_encode(desc, Q, K, V, mask, Z2, le2, flare.alloc_workspace(desc, flare.OP_ENCODE))
    flare.flare_decode(desc, Q, K, Z2, Y2, ld2)
    for got, want, stored in ((Z, Z2, 0.0), (Y, Y2, 2.0 ** -10 if dtype == "f16" else 0.0), (le, le2, 0.0), (ld, ld2, 0.0)):
        got, want = got.double(), want.double()
        finite = want.isfinite()
        assert bool((finite | want.isneginf()).all()) and torch.equal(got.isfinite(), finite) and torch.equal(got.isneginf(), want.isneginf())
        if finite.any():
            got, want = got[finite], want[finite]
            rms = max(float(want.pow(2).mean().sqrt()), 1e-30)
            assert float(((got - want).abs() - stored * want.abs()).max()) <= 4e-5 * rms


@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("B,H,N,M,D,masked", [(1, 9, 1024, 64, 32, 0.1), (1, 2, 2048, 32, 16, 0.0), (2, 5, 512, 64, 32, 0.2), (2, 5, 1024, 64, 8, 0.1)])
def test_most_tokens_of_one_launch(oracle, B, H, N, M, D, masked, dtype):
    """The largest problems of that form, of sixteen and of eight blocks, against the oracle."""
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M, masked_fraction=masked, k_std=0.8)
    assert flare.flare_launch_count(flare.make_desc(inp.Q, inp.K, 0.7), flare.OP_FORWARD) == 1
    assert_forward_close(gpu_forward(inp, scale=0.7, canary=True), oracle_forward(oracle, inp, 0.7), dtype, f"{dtype} B{B}H{H}N{N}M{M}D{D}")


def test_weights_over_many_tokens():
    """One latent over 131072 tokens of nearly equal score: a row of dV is the token's weight times one vector, and the weight e^(score - lse) of a distance
    of 11.8.  That distance is rounded to multiples of 2^-20 (root mean square 2^-20 / sqrt(12) = 2.75e-7); the exponential, the score and the stored
    value add 2^-23 each at most.  (A product with log2(e) that is rounded once more: 4.7e-7.)"""
    inp = workloads.make_random(1, 1, 131072, 1, 8, dtype="f32", seed=9, with_dy=True, k_std=0.1)
    Q, K, V, dY = (t.cuda() for t in (inp.Q, inp.K, inp.V, inp.dY))
    dV = flare.forward_backward(Q, K, V, dY)[3].double()[0, :, 0]
    S = (K.double()[0, :, 0] * Q.double()[0, 0]).sum(1)
    ratio = (dV / (torch.softmax(S, 0)[:, None] * dY.double()[0, :, 0].sum(0))).mean(1)
    assert float((ratio / ratio.mean() - 1.0).pow(2).mean().sqrt()) <= 2.0 ** -20 / 12 ** 0.5 + 2.0 ** -23 * 0.5
