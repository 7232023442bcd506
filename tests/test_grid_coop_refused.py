"""A grid solve in a context that refuses the cooperative launch (fewer SMs than the device has:
cudaErrorCooperativeLaunchTooLarge) goes on with the plain launches.  On the CPU: the library's objects
linked against a stand-in CUDA runtime whose memory is the host's, whose kernels do nothing and whose
residual norm, as the host reads it, is 1 until the third read."""
import os
import subprocess
import sys

import pytest

from paper_2210_14907_gb300 import build as B

FAKE = r"""
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>
int coop_asked, launched, reads;
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { ++launched; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative) {
      ++coop_asked;
      return cudaErrorCooperativeLaunchTooLarge;
    }
  ++launched;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  if (n == 16 * sizeof(double)) {  // the solver's scalars: ||r||^2 and ||b||^2
    ((double*)d)[4] = ((double*)d)[8] = ++reads < 3 ? 1.0 : 0.0;
    ((double*)d)[9] = 1.0;
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, enum cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = 0; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
}
"""

RUN = r"""
import ctypes as C, sys
sys.path.insert(0, sys.argv[2])
import paper_2210_14907_gb300 as nbm
lib = C.CDLL(sys.argv[1])
d = nbm.ProblemDesc(mu_plus=10.0)
p, buf, it, rel = C.c_void_p(), (C.c_double * 9261)(), C.c_int(), C.c_double()
assert lib.nbm_init_problem(C.byref(d.to_c()), C.byref(p)) == 0
f = getattr(lib, sys.argv[3])
f.argtypes = [C.c_void_p, C.c_int, C.c_double, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
rc = f(p, 20, 1e-9, 1000, buf, C.addressof(it), C.addressof(rel), None)
print(rc, it.value, C.c_int.in_dll(lib, "coop_asked").value, C.c_int.in_dll(lib, "launched").value)
"""


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("fake")
    src, out = d / "fake.cpp", d / "libnbm_fake.so"
    src.write_text(FAKE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    objs = [os.path.join(B.OUT, os.path.basename(s) + ".o") for s in B._sources()]
    subprocess.run(["g++", "-shared", "-fPIC", "-w", "-I", cuda, "-o", str(out), str(src), "-Wl,-Bsymbolic"] + objs,
                   check=True, capture_output=True, text=True)
    return str(out)


@pytest.mark.parametrize("call", ["nbm_grid_cg_solve", "nbm_grid_solve_refined"])
def test_solve_goes_on_without_the_cooperative_launch(fake_lib, call):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RUN, fake_lib, root, call], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-800:]
    rc, iters, asked, launched = map(int, r.stdout.split())
    assert rc == 0 and asked == 1 and launched >= 3 * iters > 0
