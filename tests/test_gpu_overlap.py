"""Calls queued behind one another on shared buffers, and the same calls in a captured graph (needs a B200).

The kernels of a call are launched so that each may be placed while the one before it runs out, and waits for it before it touches
memory.  What that could get wrong shows where one call's outputs or scratch are the next one's: different problems one after the
other in the same workspace, Z, log-sum-exp rows and gradients, without a pause, against the same calls with the device idle before
each.  Results are bitwise reproducible, so the comparison is exact.
"""
import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import dev

pytestmark = pytest.mark.gpu

SEQUENCES = [  # (B, H, N, M, D, dtype, masked, path, train) of each call
    # tensor cores: forms with and without a running maximum, head pairs, all widths, a training step between two forwards
    [(1, 2, 3000, 128, 16, "bf16", 0.0, flare.PATH_FAST, False), (2, 2, 700, 48, 32, "bf16", 0.2, flare.PATH_EXACT, True),
     (1, 2, 3000, 64, 16, "bf16", 0.1, flare.PATH_FAST, False), (1, 4, 900, 96, 64, "bf16", 0.0, flare.PATH_AUTO, True),
     (1, 2, 300, 272, 8, "bf16", 0.0, flare.PATH_FAST, True)],
    # latents worked off in ranges: decode's partial rows and the token kernel's sums go through memory from launch to launch
    [(1, 2, 500, 1040, 8, "bf16", 0.1, flare.PATH_FAST, True), (1, 1, 260, 208, 64, "bf16", 0.0, flare.PATH_AUTO, True),
     (1, 2, 500, 576, 16, "bf16", 0.0, flare.PATH_EXACT, False)],
    # double-precision MMA kernels, and the two families in turn (they clear the workspace's header in different places)
    [(1, 2, 1024, 16, 16, "f32", 0.0, flare.PATH_AUTO, False), (2, 4, 501, 64, 16, "f16", 0.1, flare.PATH_AUTO, True),
     (1, 2, 129, 128, 32, "bf16", 0.0, flare.PATH_FAST, True), (1, 2, 1024, 33, 8, "f32", 0.0, flare.PATH_AUTO, True)],
]


class _Call:
    """One forward, or forward and backward, whose outputs and scratch are views of buffers shared by the whole sequence."""

    def __init__(self, spec, shared):
        B, H, N, M, D, dtype, masked, self.path, self.train = spec
        inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M + D, masked_fraction=masked, with_dy=True, k_std=0.8)
        self.Q, self.K, self.V, self.mask, self.dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.key_mask), dev(inp.dY)
        self.desc = flare.make_desc(self.Q, self.K)
        f32 = torch.float32
        self.out = {"Y": shared.view("Y", self.K.shape, self.K.dtype), "Z": shared.view("Z", (B, H, M, D), f32)}
        if self.train:
            self.out.update(le=shared.view("le", (B, H, M), f32), ld=shared.view("ld", (B, N, H), f32),
                            dQ=shared.view("dQ", (H, M, D), f32), dK=shared.view("dK", self.K.shape, self.K.dtype),
                            dV=shared.view("dV", self.K.shape, self.K.dtype))
        self.ws = shared.view("ws", (shared.workspace,), torch.uint8)
        self.kept = {k: torch.empty_like(v) for k, v in self.out.items()}

    @staticmethod
    def workspace_bytes(spec):
        B, H, N, M, D, dtype = spec[:6]
        desc = flare.FlareDesc(B, H, N, M, D, {"f32": flare.DTYPE_F32, "bf16": flare.DTYPE_BF16, "f16": flare.DTYPE_F16}[dtype], 1.0)
        return max(flare.flare_workspace_bytes(desc, flare.OP_FORWARD), flare.flare_workspace_bytes(desc, flare.OP_BACKWARD))

    def __call__(self):
        o = self.out
        flare.flare_set_path(self.path)
        flare.flare_forward(self.desc, self.Q, self.K, self.V, self.mask, o["Y"], o["Z"], o.get("le"), o.get("ld"), self.ws)
        if self.train:
            flare.flare_backward(self.desc, self.Q, self.K, self.V, self.mask, o["Y"], self.dY, o["Z"], o["le"], o["ld"], o["dQ"], o["dK"],
                                 o["dV"], self.ws)
        flare.flare_set_path(flare.PATH_AUTO)
        for k, v in o.items():                                  # on the same stream: before the next call writes there
            self.kept[k].copy_(v)


class _Shared:
    def __init__(self, specs):
        self.workspace = max(_Call.workspace_bytes(s) for s in specs)
        self.buffers = {}

    def view(self, name, shape, dtype):
        n = torch.Size(shape).numel() * torch.empty(0, dtype=dtype).element_size()
        buf = self.buffers.setdefault(name, torch.zeros(max(8 << 20, self.workspace), dtype=torch.uint8, device="cuda"))
        assert n <= buf.numel()
        return buf[:n].view(dtype).view(shape)


@pytest.mark.parametrize("specs", SEQUENCES, ids=["tensor cores", "ranges", "double MMA"])
def test_calls_behind_one_another(specs):
    shared = _Shared(specs)
    calls = [_Call(s, shared) for s in specs]
    want = []
    for c in calls:                                             # one by one, the device idle before each
        torch.cuda.synchronize()
        c()
        torch.cuda.synchronize()
        flare.flare_check(c.ws)
        want.append({k: v.clone() for k, v in c.kept.items()})
        assert all(torch.isfinite(v.float()).all() for v in want[-1].values())

    def check(what):
        torch.cuda.synchronize()
        for c, w in zip(calls, want):
            for k in w:
                assert torch.equal(c.kept[k], w[k]), (what, c.desc.N, c.desc.M, c.desc.D, k)
                c.kept[k].zero_()

    for order in (calls, calls[::-1]):
        for c in order:
            c()
        check("queued")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for c in calls:
            c()
    for _ in range(3):
        graph.replay()
        check("captured")
    graph.replay()                                              # two replays without a pause between them
    graph.replay()
    check("replayed twice")


@pytest.mark.parametrize("train", [False, True])
def test_scratch_belongs_to_the_stream_of_the_call(train):
    """What a one-line call drops on return while its kernels are queued was allocated on their stream: the allocator may hand memory of the
    current stream on at once."""
    inp = workloads.make_random(1, 2, 3000, 64, 32, dtype="bf16", seed=3, with_dy=True)
    Q, K, V, dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.dY)

    def call(stream=None):
        return flare.forward_backward(Q, K, V, dY, stream=stream) if train else flare.forward(Q, K, V, want_stats=True, stream=stream)

    want = [t.clone() for t in call()]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    side = torch.cuda.Stream()
    got = call(side)
    torch.cuda.synchronize()
    assert all(torch.equal(g, w) for g, w in zip(got, want))
    held = sum(s["total_size"] for s in torch.cuda.memory_snapshot() if s["stream"] == side.cuda_stream)
    assert held >= flare.flare_workspace_bytes(flare.make_desc(Q, K), flare.OP_BACKWARD if train else flare.OP_FORWARD)
