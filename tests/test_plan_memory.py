"""Plan creation where device memory for the stored Gram matrices runs out
between the query of what is free and the allocation (another thread's or
process's): the matrices are an option of the plan's own choosing (c_supply 0),
so the plan keeps the factored loop; a caller that asked for them gets the
error.  The plan builder is compiled for the host against a CUDA runtime of
stubs whose cudaMalloc refuses large requests."""
import ctypes
import os
import subprocess

import pytest

from paper_2205_02646_gb300 import build, rljsde, synth

STUBS = r"""
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
#include "rljsde_internal.h"
extern "C" {
size_t stub_limit = ~(size_t)0;
long stub_live = 0;
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = (size_t)200 << 30; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (n > stub_limit) { *p = nullptr; return cudaErrorMemoryAllocation; }
    *p = std::malloc(64);
    ++stub_live;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { if (p) --stub_live; std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
namespace rljsde {
int build_stored_c(rljsde_plan *, const double *) { return RLJSDE_OK; }
int choose_launch(rljsde_plan *, int, int) { return RLJSDE_OK; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "stubs.cpp").write_text(STUBS)
    csrc, so = os.path.join(build.PKG, "csrc"), str(d / "plan.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    # (bound within the library: the process may hold the real runtime already)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-I", csrc, "-I",
                           os.path.join(build.ROOT, "include"), "-o", so, str(d / "stubs.cpp"), os.path.join(csrc, "plan.cpp")])
    out = ctypes.CDLL(so)
    out.rljsde_plan_destroy.restype = None
    return out


def params(lib, **kw):
    p = rljsde.Params()
    assert lib.rljsde_default_params(ctypes.byref(p)) == 0
    for k, v in kw.items():
        setattr(p, k, v)
    return p


def create(lib, p, limit):
    ctypes.c_size_t.in_dll(lib, "stub_limit").value = limit
    mask = synth.recurrent_mask(64, 64, 4, 1)
    h, info = ctypes.c_void_p(), rljsde.PlanInfo()
    st = lib.rljsde_plan_create(ctypes.byref(h), ctypes.c_void_p(mask.ctypes.data), 64, 64, ctypes.byref(p))
    if st == 0:
        assert lib.rljsde_plan_info(h, ctypes.byref(info)) == 0
        lib.rljsde_plan_destroy(h)
    assert ctypes.c_long.in_dll(lib, "stub_live").value == 0
    return st, info


@pytest.mark.parametrize("precision", [0, 1])
def test_no_memory_for_the_matrices(lib, precision):
    plenty, small = 1 << 40, 1 << 27                        # 100 table sets: 0.84 or 1.7 GB of matrices
    st, info = create(lib, params(lib, precision=precision), plenty)
    assert st == 0 and info.n_tables == 100 and info.n_stored_c_tables == 100 and info.device_c_bytes > small
    st, info = create(lib, params(lib, precision=precision), small)
    assert st == 0 and info.n_tables == 100
    assert (info.n_stored_c_tables, info.n_stored_c_blocks, info.device_c_bytes, info.n_launches) == (0, 0, 0, 1)
    if precision == 0:
        assert create(lib, params(lib, c_supply=1), small)[0] == 4                       # asked for: out of memory


def test_no_memory_at_all(lib):
    assert create(lib, params(lib), 1024)[0] == 4
