"""Parameters read back when the runtime refuses a copy: gwam_mlp_get_params_host compiled against stand-ins of the
copies and of the wait that return a chosen error (no GPU is touched), which it has to report as GWAM_ECUDA with the
wait having succeeded."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <cuda_runtime.h>
static cudaError_t rc_2d, rc_1d, rc_wait;
static int copies;
static cudaError_t fake_2d(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { ++copies; return rc_2d; }
static cudaError_t fake_1d(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { ++copies; return rc_1d; }
static cudaError_t fake_wait(cudaStream_t) { return rc_wait; }
static cudaError_t fake_last() { return cudaSuccess; }
#define cudaMemcpy2DAsync fake_2d
#define cudaMemcpyAsync fake_1d
#define cudaStreamSynchronize fake_wait
#define cudaGetLastError fake_last
#include "gwam_mlp.cu"
extern "C" int try_get(int e2d, int e1d, int ewait, int want_w, int want_b, int* n)
{
    gwam_mlp m;
    m.nl = 2;
    for (int l = 0; l <= 2; ++l) m.N[l] = m.D[l] = 64;
    rc_2d = (cudaError_t)e2d; rc_1d = (cudaError_t)e1d; rc_wait = (cudaError_t)ewait;
    copies = 0;
    float w[1], b[1];
    const int rc = gwam_mlp_get_params_host(&m, 1, 0, want_w ? w : nullptr, want_b ? b : nullptr);
    *n = copies;
    return rc;
}
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    from paper_2309_11257_gb300 import build
    d = tmp_path_factory.mktemp("shim")
    src, so = d / "shim.cu", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run([build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-diag-suppress", "177",
                                                  "-I", build.CSRC, "-shared", str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so), mode=os.RTLD_LAZY)


@pytest.mark.parametrize("e2d,e1d,ewait,w,b,ok", [(0, 0, 0, 1, 1, True), (0, 0, 0, 0, 0, True), (1, 0, 0, 1, 1, False),
                                                  (1, 0, 0, 1, 0, False), (0, 1, 0, 1, 1, False), (0, 1, 0, 0, 1, False),
                                                  (1, 0, 0, 0, 1, True), (0, 0, 1, 1, 1, False)])
def test_refused_copies_are_reported(shim, e2d, e1d, ewait, w, b, ok):
    n = C.c_int(-1)
    assert shim.try_get(e2d, e1d, ewait, w, b, C.byref(n)) == (0 if ok else -5)
    assert n.value == (w + b if not (w and e2d) else 1)
