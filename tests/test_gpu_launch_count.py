"""flare_launch_count against the kernel nodes of a captured call (needs a B200)."""
import ctypes

import pytest
import torch

from paper_2508_12594_b200 import flare, workloads
from tests._util import dev

pytestmark = pytest.mark.gpu


def kernels_in(call):
    """Kernels that `call` launches on the current stream: the kernel nodes of a graph captured around it."""
    call()                                                   # (attributes and modules are set up outside the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    rt = ctypes.CDLL("libcudart.so.12")
    raw, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert rt.cudaGraphGetNodes(raw, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(raw, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(0)                                    # cudaGraphNodeTypeKernel


@pytest.mark.parametrize("B,H,N,M,D,dtype", [
    (1, 2, 1000, 16, 16, "f32"), (1, 2, 5000, 64, 16, "f32"), (1, 1, 300, 256, 64, "f32"), (1, 1, 300, 528, 32, "f16"), (1, 1, 200, 2048, 64, "f32"),
    (1, 2, 1000, 64, 16, "bf16"), (1, 2, 40000, 128, 32, "bf16"), (1, 1, 300, 208, 64, "bf16"), (1, 1, 300, 400, 64, "bf16"),
    (1, 1, 300, 1040, 32, "bf16"), (2, 1, 300, 288, 8, "bf16"),
    (1, 2, 300, 784, 16, "bf16"), (1, 64, 4800, 784, 16, "bf16"), (1, 64, 25000, 784, 16, "bf16"), (4, 8, 700, 320, 32, "bf16"),
])
def test_counts_are_what_is_launched(B, H, N, M, D, dtype):
    inp = workloads.make_random(B, H, N, M, D, dtype=dtype, seed=N + M, with_dy=True)
    Q, K, V, dY = dev(inp.Q), dev(inp.K), dev(inp.V), dev(inp.dY)
    desc = flare.make_desc(Q, K)
    Y, Z, le, ld = flare.forward(Q, K, V, want_stats=True)
    dQ, dK, dV = torch.empty(H, M, D, device="cuda"), torch.empty_like(K), torch.empty_like(V)
    ws = {op: flare.alloc_workspace(desc, op) for op in (flare.OP_ENCODE, flare.OP_DECODE, flare.OP_FORWARD, flare.OP_BACKWARD)}
    calls = {flare.OP_ENCODE: lambda: flare.flare_encode(desc, Q, K, V, None, Z, le, ws[flare.OP_ENCODE]),
             flare.OP_DECODE: lambda: flare.flare_decode(desc, Q, K, Z, Y, ld, ws[flare.OP_DECODE]),
             flare.OP_FORWARD: lambda: flare.flare_forward(desc, Q, K, V, None, Y, Z, le, ld, ws[flare.OP_FORWARD]),
             flare.OP_BACKWARD: lambda: flare.flare_backward(desc, Q, K, V, None, Y, dY, Z, le, ld, dQ, dK, dV, ws[flare.OP_BACKWARD])}
    for op, call in calls.items():
        assert flare.flare_launch_count(desc, op) == kernels_in(call), op
