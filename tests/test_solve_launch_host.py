"""Which kernel a Poisson solve launches, on the CPU against a fake of the CUDA
runtime calls that the library makes (a shared object loaded ahead of the
runtime; kernels do nothing): small meshes run on one cluster of blocks where
the runtime says that it fits, and on the cooperative grid where it says that
none does (a process with a share of the SMs) or answers with an error."""
import json
import os
import subprocess
import sys


import __graft_entry__ as g

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <stdlib.h>
#include <string.h>
typedef void* P;
int fake_clusters, fake_error, n_cluster, n_coop;
int cudaOccupancyMaxActiveClusters(int* n, P f, P cfg) { *n = fake_clusters; return fake_error; }
int cudaLaunchKernelExC(P cfg, P f, P args) { ++n_cluster; return fake_clusters > 0 ? 0 : 912; }
int cudaLaunchCooperativeKernel(P f, ...) { ++n_coop; return 0; }
int cudaLaunchKernel(P f, ...) { return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { *v = a == 16 ? 152 : a == 97 ? 232448 : 1; return 0; }
int cudaFuncSetAttribute(P f, int a, int v) { return 0; }
int cudaGetLastError(void) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, P f, int b, size_t s) { *n = 2; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, P f, int b, size_t s, unsigned g) { *n = 2; return 0; }
int cudaMalloc(P* p, size_t n) { *p = calloc(1, n); return *p ? 0 : 2; }
int cudaFree(P p) { free(p); return 0; }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 30; return 0; }
int cudaMemcpy(P d, P s, size_t n, int k) { memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(P d, P s, size_t n, int k, P st) { memcpy(d, s, n); return 0; }
int cudaMemsetAsync(P d, int v, size_t n, P st) { memset(d, v, n); return 0; }
int cudaStreamSynchronize(P s) { return 0; }
int cudaGetSymbolAddress(P* p, P s) { *p = calloc(1, 8 << 20); return 0; }
/* device memory of device 0: type, device, device pointer, host pointer */
int cudaPointerGetAttributes(P at, P p) {
  memset(at, 0, 32);
  ((int*)at)[0] = 2;
  ((P*)at)[1] = p;
  return 0;
}
"""

CHILD = r"""
import ctypes, json, sys
fake = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
sys.path.insert(0, sys.argv[2])
from paper_2602_15130_gb300 import _lib, make_config, workloads
L = _lib.load()
I = lambda name: ctypes.c_int.in_dll(fake, name)
out = []
for clusters, error in ((1, 0), (0, 0), (0, 801), (1, 0)):
    I("fake_clusters").value, I("fake_error").value = clusters, error
    for what in ("fp64 8", "fp64 20", "fp64 21", "precision 8", "precision 12", "precision 40", "precision 41",
                 "noalloc 20", "noalloc 21"):
        form, n = what.split()
        n = int(n)
        I("n_cluster").value = I("n_coop").value = 0
        if form == "noalloc":
            buf = (ctypes.c_double * (3 * n ** 3))()
            at = ctypes.addressof(buf)
            st = L.pic_poisson_solve_noalloc(n, at, at, at, 1e-10, 10, None, None, None)
        else:
            p = workloads.base(n, 64, 0.01, 0, 1.0)
            c = make_config(workloads.mixed(p) if form == "precision" else p)
            ctx = ctypes.c_void_p()
            st = L.pic_create(ctypes.byref(c), None, None, ctypes.byref(ctx))
            if st == 0:
                st = L.pic_sample_mms(ctx, 0.0)
            L.pic_destroy(ctx)
        out.append([clusters > 0 and not error, what, st, I("n_cluster").value, I("n_coop").value])
print(json.dumps(out))
"""

ON_CLUSTER = {"fp64 8", "fp64 20", "precision 8", "precision 12", "precision 40", "noalloc 20"}


def test_small_solves_fall_back_to_the_grid(tmp_path):
    g.build()
    (tmp_path / "fake.c").write_text(FAKE)
    so = tmp_path / "fake.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(tmp_path / "fake.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(so), ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    for fits, what, status, n_cluster, n_coop in json.loads(r.stdout):
        want = (1, 0) if fits and what in ON_CLUSTER else (0, 1)
        assert (status, n_cluster, n_coop) == (0,) + want, (fits, what)
