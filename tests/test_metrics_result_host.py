"""Where the four figures go, on the host: the library's objects linked against
a fake CUDA runtime that records launches and copies (no GPU).

The finalize kernel may store through the caller's pointer only where that is
memory of the launching device; memory of another GPU (a kernel's store there
needs peer access) and managed memory get a device-to-device copy.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1803_00737_gb300 import build as B

FAKE = r"""
#include <cuda_runtime_api.h>
#include <string.h>
int fake_device = 0, fake_type = cudaMemoryTypeDevice, fake_error = 0, copies = 0, launches = 0;
void *copy_dst;
size_t copy_bytes;
void **__cudaRegisterFatBinary(void *f) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterFunction(void **h, const char *f, char *d, const char *n, int t, void *a, void *b, void *c, void *e,
                            int *w) {}
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {}
int __cudaGetKernel(void *k, const void *f) { return 0; }
int __cudaLaunchKernel(void *k, dim3 g, dim3 b, void **a, size_t s, void *st) { return 0; }
int __cudaPopCallConfiguration(void *g, void *b, size_t *s, void *st) { return 0; }
int __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void *st) { return 0; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return 0; }
cudaError_t cudaGetLastError(void) { return 0; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) { *v = 152; return 0; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { return 0; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = 0; return 0; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s) { *n = 1; return 0; }
cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **a, size_t s, cudaStream_t st) { ++launches; return 0; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a) { ++launches; return 0; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t st) { return 0; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { return 0; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
    ++copies; copy_dst = d; copy_bytes = n; return 0;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof *a);
    if (fake_error) return cudaErrorInvalidValue;
    a->type = fake_type; a->device = fake_device;
    return 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc = "/usr/local/cuda/include"
    if shutil.which("gcc") is None or not os.path.isdir(inc):
        pytest.skip("no C compiler or CUDA headers")
    B.build()
    objs = sorted(os.path.join(B.OBJDIR, os.path.basename(s).replace(".cu", ".o")) for s in B.sources())
    if not all(os.path.exists(o) for o in objs):
        pytest.skip("the library was built elsewhere")
    d = tmp_path_factory.mktemp("fake")
    src, so = d / "fake.c", d / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-w", "-fPIC", f"-I{inc}", "-c", str(src), "-o", str(d / "fake.o")], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", str(so), str(d / "fake.o"), *objs], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("kind,device,error,copied", [
    (2, 0, 0, False),  # memory of the launching device
    (2, 1, 0, True),   # of another one
    (3, 0, 0, True),   # managed
    (0, 0, 0, True),   # not known to the runtime
    (2, 0, 1, True),   # the query fails
])
@pytest.mark.parametrize("call", ["metrics", "fuse_metrics", "score_finish"])
def test_figures_reach_other_memory_by_copy(lib, kind, device, error, copied, call):
    for name, v in (("fake_type", kind), ("fake_device", device), ("fake_error", error), ("copies", 0),
                    ("launches", 0)):
        ctypes.c_int.in_dll(lib, name).value = v
    vp, i64, sz = ctypes.c_void_p, ctypes.c_int64, ctypes.c_size_t
    lib.dwtfuse_metrics_workspace_size.restype = sz
    n = lib.dwtfuse_metrics_workspace_size()
    ms = (vp * 2)(0x3000000, 0x3100000)
    fused, pan, ws, out = vp(0x1000000), vp(0x2000000), vp(0x4000000), 0x5000000
    if call == "metrics":
        st = lib.dwtfuse_metrics(fused, 0, ms, pan, 0, 2, i64(64), i64(96), 32, ws, sz(n), vp(out), None)
    elif call == "fuse_metrics":
        st = lib.dwtfuse_fuse_metrics(pan, ms, 2, i64(64), i64(96), 1, 0, None, fused, ws, sz(n), vp(out), None)
    else:
        st = lib.dwtfuse_score_finish(ms, pan, 0, 2, i64(64), i64(96), fused, ws, sz(n), vp(out), None)
    assert st == 0
    assert ctypes.c_int.in_dll(lib, "launches").value == (2 if call == "score_finish" else 3)
    assert ctypes.c_int.in_dll(lib, "copies").value == copied
    if copied:
        assert vp.in_dll(lib, "copy_dst").value == out and sz.in_dll(lib, "copy_bytes").value == 32
