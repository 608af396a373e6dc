"""flare_forward_host on batches that it works off in parts (needs a B200): whole and uneven parts, masks, float32; the rows of every part
against the CPU oracle, and the call's place in the order of its stream."""
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import assert_stored_close, oracle_forward, to_np64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,N,M,D,dtype,masked", [
    (3, 8, 8320, 32, 16, "bf16", 0.0),          # one item a part
    (5, 4, 8200, 16, 16, "bf16", 0.2),          # two items a part, one in the last
    (3, 4, 9001, 16, 16, "f32", 0.1),
    (2, 8, 8192, 64, 32, "bf16", 0.1)])
def test_parts(oracle, B, H, N, M, D, dtype, masked):
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=B + N, masked_fraction=masked, k_std=0.8)
    hQ, hK, hV = inp.Q.pin_memory(), inp.K.pin_memory(), inp.V.pin_memory()
    hmask = None if inp.key_mask is None else inp.key_mask.pin_memory()
    hY = torch.full_like(inp.K, 777.0).pin_memory()
    desc = flare.make_desc(inp.Q, inp.K)
    dQ, dK, dV, dY = (torch.full_like(t, 555.0, device="cuda") for t in (inp.Q, inp.K, inp.V, inp.K))
    dmask = None if hmask is None else torch.zeros_like(hmask, device="cuda")
    ws = flare.alloc_workspace(desc, flare.OP_FORWARD)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for _ in range(2):
            dY.fill_(555.0)
            flare.flare_forward_host(desc, hQ, hK, hV, hmask, hY, dQ, dK, dV, dmask, dY, ws, stream)
        after = dY.clone()                                       # queued behind the call: sees all of its rows
    stream.synchronize()
    flare.flare_check(ws)
    assert_stored_close(to_np64(hY), oracle_forward(oracle, inp)["Y"], dtype, f"{B}x{N} Y (host)")
    assert torch.equal(hY, after.cpu()) and torch.equal(dK.cpu(), inp.K)
