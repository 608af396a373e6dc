"""The C-ABI library loads and exports every symbol the header declares; host-side checks that need no GPU."""
import ctypes
import os
import re

import pytest

from paper_2508_12594_b200 import build, flare

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return flare.load()


def _declared():
    text = open(os.path.join(ROOT, "include", "flare.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(flare_[a-z_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared()
    assert {"flare_encode", "flare_decode", "flare_forward", "flare_backward"} <= set(names)
    raw = ctypes.CDLL(flare.LIB_PATH)
    for n in names:
        assert hasattr(raw, n), n
    assert sorted(flare.exported_symbols()) == names


def test_binding_argument_counts_match_the_header():
    """Every prototype in the header has as many parameters as the binding's ctypes signature."""
    text = open(os.path.join(ROOT, "include", "flare.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    protos = dict(re.findall(r"\b(flare_[a-z_]+)\s*\(([^)]*)\)\s*;", text))
    assert set(protos) == set(flare._SIGNATURES)
    for name, params in protos.items():
        n = 0 if params.strip() in ("", "void") else params.count(",") + 1
        assert n == len(flare._SIGNATURES[name][1]), name


def test_status_strings(lib):
    assert lib.flare_status_string(0) == b"ok"
    for s in range(1, 7):
        assert len(lib.flare_status_string(s)) > 0
    assert lib.flare_version() >= 100


def test_descriptor_validation_needs_no_device(lib):
    ok = flare.FlareDesc(1, 2, 1024, 16, 16, flare.DTYPE_F32, 1.0)
    assert flare.flare_workspace_bytes(ok, flare.OP_FORWARD) > 0
    assert flare.flare_encode_partials(ok) >= 1
    for bad in (flare.FlareDesc(0, 2, 8, 16, 16, 0, 1.0), flare.FlareDesc(1, 2, 8, 16, 12, 0, 1.0),
                flare.FlareDesc(1, 2, 8, 17, 16, flare.DTYPE_BF16, 1.0), flare.FlareDesc(1, 2, 8, 4096, 16, 1, 1.0),
                flare.FlareDesc(1, 2, 8, 16, 16, 7, 1.0), flare.FlareDesc(1, 2, 8, 16, 16, 0, float("nan"))):
        assert flare.flare_workspace_bytes(bad, flare.OP_FORWARD) == 0
    # null pointers are rejected before anything touches a device
    rc = lib.flare_encode(ctypes.byref(ok), None, None, None, None, None, None, None, 0, None)
    assert rc == flare.ERR_INVALID_ARG
    rc = lib.flare_decode(ctypes.byref(flare.FlareDesc(1, 2, 8, 16, 12, 0, 1.0)), None, None, None, None, None, None, 0, None)
    assert rc == flare.ERR_UNSUPPORTED


def test_every_head_width_of_the_paper_is_accepted(lib):
    """D = 4 and 8 (the paper's PDE models: C = 64 with 16 or 8 heads) up to 64, both dtypes, all operations."""
    for D in (4, 8, 16, 32, 64):
        for dtype in (flare.DTYPE_F32, flare.DTYPE_BF16):
            desc = flare.FlareDesc(2, 64 // D if D <= 16 else 2, 1000, 64, D, dtype, 1.0)
            for op in (flare.OP_ENCODE, flare.OP_FORWARD, flare.OP_BACKWARD):
                assert flare.flare_workspace_bytes(desc, op) > 0, (D, dtype, op)
    assert flare.flare_workspace_bytes(flare.FlareDesc(2, 4, 1000, 64, 2, flare.DTYPE_BF16, 1.0), flare.OP_FORWARD) == 0


def test_workspace_never_scales_with_n_times_m(lib):
    """Scratch is O(partials * B*H*M*(D+2)): growing N a thousandfold must not grow it by the same factor."""
    small = flare.FlareDesc(1, 8, 4096, 256, 16, flare.DTYPE_BF16, 1.0)
    big = flare.FlareDesc(1, 8, 1048576, 256, 16, flare.DTYPE_BF16, 1.0)
    ws, wb = flare.flare_workspace_bytes(small, 2), flare.flare_workspace_bytes(big, 2)
    assert wb < 1048576 * 256 * 2 / 8          # far below one N x M bf16 matrix of a single head
    rows = 8 * 256
    assert wb <= 256 + 4096 + flare.flare_encode_partials(big) * rows * (16 + 2) * 4 + rows * 16 * 4 + 4 * 256
    assert ws <= wb


def test_eigenvalues_of_empty_matrices_are_refused(lib):
    """The number of matrices is a quotient of sizes: no size may make it one by zero (the sixth: 2^32 squared is 0 in 64 bits)."""
    import torch
    for shape in ((0, 0), (3, 0, 0), (5, 0), (0,), (), (0, 1 << 32)):
        with pytest.raises((ValueError, flare.FlareError)):
            flare.flare_spectral_eig(torch.empty(shape), torch.empty(0))


# Shapes whose partial results in the exact form take 1.3 to 6.4 MB (splits x partial results a split x rows x (D + 2) floats).
STATIC_SCRATCH_SHAPES = [(2, 8, 16384, 2048, 16), (4, 16, 16384, 512, 16), (32, 4, 65536, 32, 64), (32, 4, 65536, 96, 32), (1, 8, 65536, 2048, 16),
                         (1, 8, 262144, 1024, 16), (1, 8, 1048576, 2048, 8), (4, 16, 1048576, 272, 8), (4, 4, 1048576, 1024, 4)]


@pytest.mark.parametrize("shape", STATIC_SCRATCH_SHAPES, ids=str)
def test_many_latents_fit_the_built_in_scratch(lib, shape):
    """flare_encode_static_scratch takes what fits its array in the exact form, also where another form runs."""
    desc = flare.FlareDesc(*shape, flare.DTYPE_BF16, 1.0)
    assert 0 < flare.flare_workspace_bytes(desc, flare.OP_ENCODE) <= flare.STATIC_SCRATCH_BYTES
    assert flare.flare_workspace_bytes(desc, flare.OP_FORWARD) >= flare.flare_workspace_bytes(desc, flare.OP_ENCODE)


def test_scratch_at_head_width_64_is_that_of_the_exact_form(lib):
    """D = 64 has no other form: one partial result per split and pair of latent blocks, up to 148 / (B H) splits."""
    desc = flare.FlareDesc(1, 4, 65536, 256, 64, flare.DTYPE_BF16, 1.0)
    assert flare.flare_encode_partials(desc) == 2 * (148 // 4)


@pytest.mark.parametrize("M,D,dtype,kernels", [
    (256, 64, flare.DTYPE_F32, 6), (528, 32, flare.DTYPE_F16, 6), (2048, 64, flare.DTYPE_F32, 6),     # one token kernel whatever M is
    (192, 64, flare.DTYPE_BF16, 6), (208, 64, flare.DTYPE_BF16, 7), (400, 64, flare.DTYPE_BF16, 8),   # up to 192 latents a launch at D = 64
    (512, 32, flare.DTYPE_BF16, 6), (528, 32, flare.DTYPE_BF16, 7),
    (256, 16, flare.DTYPE_BF16, 5), (512, 16, flare.DTYPE_BF16, 7), (784, 16, flare.DTYPE_BF16, 7), (2048, 8, flare.DTYPE_BF16, 7)])   # two sweeps
def test_launch_count_of_a_backward(lib, M, D, dtype, kernels):
    """Header, dZ and its reduction, the token kernel (bfloat16: one per range of latents), dQ and its reduction; two sweeps: header, the sweeps and their
    reductions, and with ranges of latents side by side, as few tokens want them, a kernel after each sweep that joins them."""
    assert flare.flare_launch_count(flare.FlareDesc(1, 2, 1000, M, D, dtype, 1.0), flare.OP_BACKWARD) == kernels


@pytest.mark.parametrize("B,H,N,D", [(1, 8, 1048576, 8), (1, 8, 1048576, 16), (4, 16, 262144, 16), (32, 4, 65536, 16)])
@pytest.mark.parametrize("M", [784, 1024, 2048])
def test_ranges_of_latents_take_bounded_scratch(lib, B, H, N, M, D):
    """Beyond the 768 latents of one launch a backward keeps float32 rows of dK and dV between its ranges of latents: at most 128 MB of them, whatever the number of
    tokens.  (All else grows as the latents do, or less.)"""
    need = lambda m: flare.flare_workspace_bytes(flare.FlareDesc(B, H, N, m, D, flare.DTYPE_BF16, 1.0), flare.OP_BACKWARD)
    assert 0 < need(M) <= need(768) * M / 768 + (128 << 20)


@pytest.mark.parametrize("B,H,N,M,kernels", [(1, 8, 65536, 768, 5), (1, 8, 65536, 784, 7), (1, 8, 65536, 1552, 9), (1, 8, 262144, 784, 15), (4, 8, 262144, 2048, 57)])
def test_launch_count_of_a_backward_over_ranges(lib, B, H, N, M, kernels):
    """Many tokens: each sweep is a launch per range of latents (up to 768), and per chunk of tokens where the rows between ranges would take more than 128 MB."""
    assert flare.flare_launch_count(flare.FlareDesc(B, H, N, M, 16, flare.DTYPE_BF16, 1.0), flare.OP_BACKWARD) == kernels
