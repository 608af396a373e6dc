"""Edges of the forms of encode and decode that keep no running maximum (needs a B200): latents and tokens around their 64- and
32-column units, widths, masks, with and without log-sum-exp rows; sums of weights at either end of the range they accept."""
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import assert_forward_close, assert_stored_close, dev, gpu_forward, oracle_forward, to_np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stats", [True, False], ids=["train", "infer"])
@pytest.mark.parametrize("B,H,N,M,D,masked", [
    (1, 2, 63, 16, 16, 0.0), (1, 2, 65, 48, 32, 0.2), (2, 3, 129, 80, 8, 0.0), (1, 1, 300, 96, 32, 0.0), (1, 2, 1500, 112, 16, 0.3),
    (1, 2, 191, 144, 32, 0.0), (1, 1, 2700, 176, 16, 0.0), (1, 1, 200, 272, 8, 0.1), (1, 2, 321, 320, 32, 0.0), (1, 1, 130, 528, 16, 0.0),
    (1, 4, 700, 64, 4, 0.1), (1, 2, 200, 48, 8, 0.2), (2, 4, 129, 64, 8, 0.0), (1, 2, 2600, 16, 8, 0.0)])
def test_unit_edges(oracle, B, H, N, M, D, masked, stats):
    inp = workloads.make_random(B, H, N, M, D, dtype="bf16", seed=N + M, masked_fraction=masked, k_std=0.8)
    got = gpu_forward(inp, stats=stats, path=flare.PATH_FAST)
    assert_forward_close(got, oracle_forward(oracle, inp), "bf16", f"{B}x{H}x{N}x{M}x{D}")


@pytest.mark.parametrize("score,redo", [(72.0, True), (-72.0, True), (60.0, False), (-60.0, False)])
def test_sums_out_of_range_hand_over(oracle, score, redo):
    """All scores near one value: 2^(72 / ln 2) is past the largest sum the forms accept and 2^(-72 / ln 2) short of the smallest, though
    the norms alone pass; +-60 (2^+-87) is within the range."""
    inp = workloads.make_random(1, 2, 300, 96, 32, dtype="bf16", seed=5, k_std=0.02)
    a = (abs(score) / 32) ** 0.5
    inp.Q.mul_(0.02).add_(a if score > 0 else -a)
    inp.K.add_(a)
    Q, K, V = dev(inp.Q), dev(inp.K), dev(inp.V)
    desc = flare.make_desc(Q, K)
    ws = flare.alloc_workspace(desc, flare.OP_FORWARD)
    Y = torch.empty_like(K)
    flare.flare_set_path(flare.PATH_FAST)
    try:
        flare.flare_forward(desc, Q, K, V, None, Y, None, None, None, ws)
    finally:
        flare.flare_set_path(flare.PATH_AUTO)
    torch.cuda.synchronize()
    words = ws[:16].view(torch.int32).cpu()
    assert words[0] == 0 and bool(words[2]) == redo and bool(words[3]) == redo
    assert_stored_close(to_np64(Y), oracle_forward(oracle, inp)["Y"], "bf16", f"scores near {score}")


def test_masked_stretches_do_not_hand_over(oracle):
    """Whole tiles of masked tokens leave sums of exactly 0 behind, which are no reason for the exact form."""
    inp = workloads.make_random(1, 2, 3000, 48, 16, dtype="bf16", seed=9, masked_fraction=0.1, k_std=0.8)
    inp.key_mask[:, 300:2100] = 0
    Q, K, V, mask = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.key_mask)
    desc = flare.make_desc(Q, K)
    ws = flare.alloc_workspace(desc, flare.OP_FORWARD)
    Y, le = torch.empty_like(K), torch.empty(1, 2, 48, device="cuda")
    flare.flare_set_path(flare.PATH_FAST)
    try:
        flare.flare_forward(desc, Q, K, V, mask, Y, None, le, None, ws)
    finally:
        flare.flare_set_path(flare.PATH_AUTO)
    torch.cuda.synchronize()
    assert not ws[:16].view(torch.int32).cpu()[[0, 2, 3]].any()
    assert_stored_close(to_np64(Y), oracle_forward(oracle, inp)["Y"], "bf16", "masked stretches")
