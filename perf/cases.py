"""Cases of work that users of the token mixer have it do, for timing it through its public entry points.

Every case is one shape and one way of calling: `forward` (inference with buffers and workspace kept between calls, as a
served model does), `call` (the one-line forward that allocates its outputs), `train` (forward and backward of one step),
`spectral` (Algorithm 1: statistics, Gram matrix, eigenvalues) and `host` (tensors in pinned host memory, as a data loader
leaves them).  Inputs follow the recipes of `paper_2508_12594_b200.workloads`, drawn on the GPU.
"""
import math

import torch

from paper_2508_12594_b200 import flare

_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(name, op, dtype, B, H, N, M, D, kind, masked=0.0):
    return {"name": name, "op": op, "dtype": dtype, "B": B, "H": H, "N": N, "M": M, "D": D, "kind": kind, "masked": masked}


def listed():
    return [
        # the smallest call: a thousand tokens in float32, what a test, a notebook or a small PDE mesh runs
        _case("call_f32_1k", "call", "f32", 1, 2, 1024, 16, 16, "iid"),
        # one training step on a small mesh with few latents
        _case("train_16k_m32", "train", "bf16", 1, 8, 16384, 32, 32, "scaled"),
        # inference over a batch of 2-D point clouds
        _case("forward_mesh2d", "forward", "bf16", 4, 8, 65536, 64, 16, "cloud"),
        # inference over a million points of a 3-D surface, the shape the benchmark is quoted on
        _case("forward_mesh3d_1m", "forward", "bf16", 1, 8, 1048576, 256, 16, "cloud"),
        # one training step on a batch of sequences padded to one length
        _case("train_padded", "train", "bf16", 32, 4, 4096, 128, 32, "scaled", 0.1),
        # one training step on a large mesh with many latents
        _case("train_131k_m512", "train", "bf16", 1, 8, 131072, 512, 32, "scaled"),
        # one training step of the million-point study: narrow heads, a thousand latents (the largest case)
        _case("train_field_1m", "train", "bf16", 1, 8, 1048576, 1024, 8, "cloud"),
        # wide heads and a length that is no multiple of anything
        _case("train_wide_heads", "train", "bf16", 2, 4, 20011, 128, 64, "scaled"),
        # training under float16 autocast, variable-length sequences
        _case("train_f16", "train", "f16", 4, 8, 10007, 64, 16, "scaled", 0.1),
        # training in float32, as gradient checks and small regressions are run
        _case("train_f32", "train", "f32", 2, 8, 9973, 64, 16, "iid"),
        # spectral analysis of the mixing matrices of one layer
        _case("spectral_131k", "spectral", "bf16", 1, 8, 131072, 128, 32, "scaled"),
        # inference from and to host memory
        _case("host_mesh2d", "host", "bf16", 4, 8, 65536, 64, 16, "cloud"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# per way of calling and type: (weight, tokens of the whole batch, most (latent, token) pairs over all heads, latents, head widths)
_RANGES = [
    ("call", "f32", 2, (512, 16384), 4e6, (8, 64), (8, 16, 32)),
    ("forward", "bf16", 5, (8192, 1048576), 2.2e9, (32, 512), (8, 16, 32)),
    ("train", "bf16", 6, (8192, 524288), 2.2e9, (32, 1024), (8, 16, 32)),
    ("train", "bf16", 2, (8192, 65536), 4e7, (32, 256), (64,)),
    ("train", "f16", 2, (4096, 65536), 4e7, (16, 128), (8, 16, 32)),
    ("train", "f32", 2, (4096, 65536), 4e7, (16, 128), (8, 16, 32)),
    ("spectral", "bf16", 2, (16384, 262144), 3e8, (32, 192), (16, 32)),
    ("host", "bf16", 2, (32768, 262144), 3e8, (32, 128), (16, 32)),
]


def draw(rng):
    op, dtype, _, tokens, most, latents, widths = rng.choices(_RANGES, weights=[r[2] for r in _RANGES])[0]
    D = rng.choice(widths)
    H = rng.choice((4, 8))
    M = _log_int(rng, *latents)
    if dtype == "bf16":
        M = max(16, (M + 8) // 16 * 16)
        if op == "spectral" and M > 128:
            M = M // 64 * 64
    T = min(_log_int(rng, *tokens), int(most / (H * M)))
    B = 1 if op == "spectral" else min(rng.choice((1, 1, 2, 4, 8)), max(1, T // 1024))
    N = max(1, T // B)
    if rng.random() < 0.5:                                   # half of the lengths as they fall, half whole tiles
        N = max(128, N // 128 * 128)
    kind = rng.choice(("cloud", "scaled"))
    masked = rng.choice((0.0, 0.1)) if op in ("forward", "train", "host") else 0.0
    return {"op": op, "dtype": dtype, "B": B, "H": H, "N": N, "M": M, "D": D, "kind": kind, "masked": masked}


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, H, N, M, D = (case[k] for k in "BHNMD")
    C, dt = H * D, _DTYPE[case["dtype"]]

    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    Q = randn(H, M, D).to(dt)
    if case["kind"] == "cloud":                              # projected features of points: coordinates and N(0, 1) channels
        Wk, Wv = randn(128, C) / 128 ** 0.5, randn(128, C) / 128 ** 0.5
        K, V = torch.empty(B, N, C, device="cuda", dtype=dt), torch.empty(B, N, C, device="cuda", dtype=dt)
        for b in range(B):
            X = randn(N, 128)
            X[:, :3] = torch.rand(N, 3, generator=g, device="cuda")
            K[b], V[b] = X @ Wk, X @ Wv
    else:
        s = 1.0 if case["kind"] == "iid" else D ** -0.5
        K, V = (randn(B, N, C) * s).to(dt), (randn(B, N, C) * s).to(dt)
    mask = None
    if case["masked"] > 0.0:                                 # padded tokens hold zeros
        mask = (torch.rand(B, N, generator=g, device="cuda") >= case["masked"]).to(torch.uint8)
        K, V = K * mask[:, :, None].to(dt), V * mask[:, :, None].to(dt)
    dY = randn(B, N, H, D).to(dt) if case["op"] == "train" else None
    return Q, K.view(B, N, H, D), V.view(B, N, H, D), mask, dY


def prepare(case, seed):
    B, H, N, M, D = (case[k] for k in "BHNMD")
    Q, K, V, mask, dY = _inputs(case, seed)
    s = {"op": case["op"], "Q": Q, "K": K, "V": V, "mask": mask, "dY": dY, "desc": flare.make_desc(Q, K)}

    def f32(*shape):
        return torch.empty(*shape, dtype=torch.float32, device="cuda")

    if case["op"] == "forward":
        s.update(Y=torch.empty_like(K), Z=f32(B, H, M, D), ws=flare.alloc_workspace(s["desc"], flare.OP_FORWARD))
    elif case["op"] == "spectral":
        s.update(Y=torch.empty_like(K), Z=f32(B, H, M, D), le=f32(B, H, M), ld=f32(B, N, H), G=f32(B, H, M, M), ev=f32(B, H, M),
                 ws=flare.alloc_workspace(s["desc"], flare.OP_FORWARD), wss=flare.alloc_workspace(s["desc"], flare.OP_SPECTRAL))
    elif case["op"] == "host":                               # the device tensors become the staging buffers
        s.update({"h" + k: s[k].cpu().pin_memory() for k in ("Q", "K", "V")})
        s.update(hmask=None if mask is None else mask.cpu().pin_memory(), hY=torch.empty_like(s["hK"]).pin_memory(),
                 Y=torch.empty_like(K), ws=flare.alloc_workspace(s["desc"], flare.OP_FORWARD))
    return s


def run(s):
    op = s["op"]
    if op == "call":
        return flare.forward(s["Q"], s["K"], s["V"])
    if op == "forward":
        flare.flare_forward(s["desc"], s["Q"], s["K"], s["V"], s["mask"], s["Y"], s["Z"], None, None, s["ws"])
        return s["Y"], s["Z"]
    if op == "train":
        return flare.forward_backward(s["Q"], s["K"], s["V"], s["dY"], s["mask"])
    if op == "spectral":
        flare.flare_forward(s["desc"], s["Q"], s["K"], s["V"], None, s["Y"], s["Z"], s["le"], s["ld"], s["ws"])
        flare.flare_spectral_gram(s["desc"], s["Q"], s["K"], s["le"], s["ld"], s["G"], s["wss"])
        flare.flare_spectral_eig(s["G"], s["ev"])
        return s["ev"], s["Z"], s["le"], s["ld"]
    flare.flare_forward_host(s["desc"], s["hQ"], s["hK"], s["hV"], s["hmask"], s["hY"], s["Q"], s["K"], s["V"], s["mask"], s["Y"],
                             s["ws"])
    return s["hY"]


def work(case):
    """Bytes: every tensor in or out once.  Operations: two per multiply-add of the contractions, each formed once."""
    B, H, N, M, D = (case[k] for k in "BHNMD")
    e = 4 if case["dtype"] == "f32" else 2
    tok, lat, mad = B * N * H * D * e, H * M * D * e, 2.0 * B * H * N * M * D
    mask = B * N if case["masked"] > 0.0 else 0
    if case["op"] == "train":                                # K, V, dY in, Y, dK, dV out; scores, their products and gradients
        return {"bytes": 6 * tok + lat + 4 * H * M * D + mask, "flops": 11 * mad}
    if case["op"] == "spectral":
        stats = 4 * (2 * B * H * M + B * N * H + B * H * M * D)
        return {"bytes": 2 * tok + lat + stats, "flops": 4 * mad + 2.0 * B * H * N * M * M + 4.0 / 3.0 * B * H * M ** 3}
    return {"bytes": 3 * tok + lat + mask + (4 * B * H * M * D if case["op"] == "forward" else 0), "flops": 4 * mad}


def tolerance(case):
    if case["op"] == "spectral":                             # eigenvalues of a float32 matrix of products of two bf16 halves
        return {"rel": 1e-3}
    # float32 sums; one rounding of stored float16 values; bfloat16 weights and stored values
    return {"rel": {"f32": 1e-5, "f16": 1e-3, "bf16": 1e-2}[case["dtype"]]}
