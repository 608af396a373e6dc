"""Small float32 and float16 forwards where a cluster of blocks cannot be placed: the library's host code over a stand-in for the CUDA runtime (no GPU).

The stand-in answers as a B200 would, but for the one kernel that is launched in clusters: `fake_clusters` is what the occupancy query reports for it and
`fake_error` what its launch returns.  Launches are recorded by kernel, nothing runs."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_2508_12594_b200 import build, flare

FAKE = r"""
#include <cstring>
#include <map>
#include <string>
#include <cuda_runtime_api.h>
#include <crt/host_runtime.h>
static std::map<const void *, std::string> &names() { static std::map<const void *, std::string> m; return m; }
extern "C" {
int fake_clusters = 1, fake_error = 0, fake_launches = 0, fake_small = 0;
static cudaError_t launched(const void *f) {
    if (names()[f].find("forward_small") != std::string::npos) {
        if (fake_error) return (cudaError_t)fake_error;
        ++fake_small;
    }
    ++fake_launches;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 148;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { a->numRegs = 96; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *) {
    *n = names()[f].find("forward_small") != std::string::npos ? fake_clusters : 0;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **) { return launched(f); }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launched(f); }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { names()[host] = name; }
}
"""
# entry points of the runtime that no call here reaches
UNUSED = ["cudaEventCreateWithFlags", "cudaEventDestroy", "cudaEventRecord", "cudaGetDriverEntryPoint", "cudaGetSymbolAddress", "cudaMemcpyAsync",
          "cudaMemsetAsync", "cudaStreamCreateWithFlags", "cudaStreamDestroy", "cudaStreamIsCapturing", "cudaStreamSynchronize", "cudaStreamWaitEvent"]


@pytest.fixture()
def lib(tmp_path):
    """A library of its own for each test: what the device answered is kept per process."""
    build.build()
    (tmp_path / "fake.cpp").write_text(FAKE)
    (tmp_path / "unused.c").write_text("".join(f"int {name}(void) {{ return 801; }}\n" for name in UNUSED))
    include = os.path.join(os.path.dirname(os.path.dirname(build.NVCC)), "include")
    objects = sorted(glob.glob(os.path.join(build.OBJ, "*.o")))
    for cmd in (["gcc", "-fPIC", "-c", "-o", "unused.o", "unused.c"],
                ["g++", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", f"-I{include}", "-o", "libfake.so", "fake.cpp", "unused.o", *objects]):
        res = subprocess.run(cmd, cwd=tmp_path, capture_output=True, text=True)
        assert res.returncode == 0, res.stderr
    so = ctypes.CDLL(str(tmp_path / "libfake.so"))
    for name, (restype, argtypes) in flare._SIGNATURES.items():
        getattr(so, name).restype, getattr(so, name).argtypes = restype, argtypes
    return so


def forward(so, desc):
    """Status of a forward, and how many kernels it launched, the clusters' among them."""
    counts = [ctypes.c_int.in_dll(so, n) for n in ("fake_launches", "fake_small")]
    for c in counts:
        c.value = 0
    at = ctypes.c_void_p(1 << 20)                            # (never followed)
    rc = so.flare_forward(ctypes.byref(desc), at, at, at, None, at, None, None, None, at, so.flare_workspace_bytes(ctypes.byref(desc), flare.OP_FORWARD), None)
    return rc, counts[0].value, counts[1].value


# sixteen blocks per cluster, and eight
SMALL = [flare.FlareDesc(1, 2, 1024, 16, 16, flare.DTYPE_F32, 1.0), flare.FlareDesc(2, 9, 1017, 16, 8, flare.DTYPE_F16, 1.0)]


@pytest.mark.parametrize("desc", SMALL, ids=["sixteen", "eight"])
@pytest.mark.parametrize("clusters", [9, 0])
def test_device_without_room_for_a_cluster(lib, desc, clusters):
    """Encode, merge and decode where the device can place no cluster, and the count says so."""
    ctypes.c_int.in_dll(lib, "fake_clusters").value = clusters
    want = (0, 1, 1) if clusters else (0, 3, 0)
    assert forward(lib, desc) == want
    assert lib.flare_launch_count(ctypes.byref(desc), flare.OP_FORWARD) == want[1]


@pytest.mark.parametrize("desc", SMALL, ids=["sixteen", "eight"])
@pytest.mark.parametrize("error,fallen_back", [(912, True), (701, True), (719, False)])
def test_launch_of_a_cluster_refused(lib, desc, error, fallen_back):
    """A stream with fewer SMs than the device (invalid cluster size, out of resources): the general kernels.  Any other error is reported."""
    ctypes.c_int.in_dll(lib, "fake_error").value = error
    assert forward(lib, desc) == ((0, 3, 0) if fallen_back else (flare.ERR_CUDA, 0, 0))
