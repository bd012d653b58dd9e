"""Solves on two devices of one process, on the host alone: the CUDA calls that reach a device are replaced by fakes,
and a fake launch of more than eight blocks in a cluster fails unless its kernel has been allowed that on the device
in use, as the runtime documents it."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKES = r"""
#include <cuda_runtime_api.h>
#include <string.h>
enum { kMax = 4096 };
static int device = 0, nset = 0;
static struct { int device; const void *func; } set[kMax];
int fake_wide_launches = 0;
void fake_set_device(int d) { device = d; }

cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) { memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v && nset < kMax) {
        set[nset].device = device;
        set[nset++].func = f;
    }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
    for (unsigned i = 0; i < c->numAttrs; ++i) {
        if (c->attrs[i].id != cudaLaunchAttributeClusterDimension || c->attrs[i].val.clusterDim.x <= 8) continue;
        int allowed = 0;
        for (int k = 0; k < nset; ++k) allowed |= set[k].device == device && set[k].func == f;
        if (!allowed) return cudaErrorInvalidClusterSize;
        ++fake_wide_launches;
    }
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **a, size_t s, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *s, void **f, unsigned v, unsigned long long fl,
                                             enum cudaDriverEntryPointQueryResult *q) {
    *f = 0;
    return cudaErrorNotSupported;   // no tensor maps: plain loads
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) { return cudaSuccess; }
"""

PROGRAM = r"""
import ctypes as C, sys
from paper_1807_00467_gb300 import _lib

fake, L = C.CDLL(sys.argv[1]), _lib.load()
n, m, iters = (64, 64, 56), (33, 17, 15), 10          # 6311 quads: 13 blocks of a cluster
ig, gg = _lib.ImageGeom((C.c_int32 * 3)(*n), (C.c_double * 3)(1.0, 1.0, 1.5)), _lib.GridGeom((C.c_int32 * 3)(*m))
par, size, ptr = _lib.Params(10.0, 1.0, 0.001, 0.0, 0, 0.0, 0.25, 4.0), C.c_size_t(), C.c_void_p(1 << 30)
assert L.rg_workspace_size(C.byref(ig), C.byref(gg), 0, 0, iters, C.byref(size)) == 0
for device in (0, 1, 0):
    fake.fake_set_device(device)
    before = C.c_int.in_dll(fake, "fake_wide_launches").value
    ctx = C.c_void_p()
    assert L.rg_ctx_create(C.byref(ctx), C.byref(ig), C.byref(gg), 0, C.byref(par), 0, iters, ptr, size.value, None) == 0
    assert L.rg_set_images(ctx, ptr, ptr) == 0 and L.gn_linearize(ctx, ptr, ptr, ptr) == 0
    code = L.gn_pcg_solve(ctx, ptr, ptr, iters, None)
    assert code == 0, (device, code, L.rg_last_error(ctx))
    assert C.c_int.in_dll(fake, "fake_wide_launches").value == before + iters
    L.rg_ctx_destroy(ctx)
print("solved")
"""


def test_wide_clusters_on_both_devices(tmp_path):
    from paper_1807_00467_gb300 import build
    build.build()
    include = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("gcc") or not os.path.isdir(include):
        pytest.skip("needs gcc and the CUDA headers")
    src, lib = tmp_path / "fakes.c", tmp_path / "fakes.so"
    src.write_text(FAKES)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", include, str(src), "-o", str(lib)], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "LD_PRELOAD": str(lib)})
    assert r.returncode == 0 and "solved" in r.stdout, r.stdout + r.stderr
