"""A kernel's shared-memory limit is raised once on every device, tried again after a failure, and
kept per kernel: SmemLimit of common.cuh on the host, with the two runtime calls replaced."""
import ctypes
import glob
import os
import subprocess

import __graft_entry__ as G

SRC = r"""
#include <cuda_runtime.h>
static int device = 0, calls = 0, fail = 0;
static cudaError_t fake_device(int* d) { *d = device; return cudaSuccess; }
template <typename K>
static cudaError_t fake_attribute(K*, cudaFuncAttribute, int) {
  ++calls;
  return fail ? cudaErrorInvalidValue : cudaSuccess;
}
#define cudaGetDevice fake_device
#define cudaFuncSetAttribute fake_attribute
#include "%s/common.cuh"
__global__ void k_a() {}
__global__ void k_b() {}
// calls made so far after raising both kernels' limits on device d
extern "C" int raise_on(int d, int failing, int* status) {
  static mgk::SmemLimit a, b;
  device = d;
  fail = failing;
  status[0] = (int)a.raise(k_a, 65536);
  status[1] = (int)b.raise(k_b, 65536);
  return calls;
}
"""


def test_once_per_device(tmp_path):
    (tmp_path / "t.cu").write_text(SRC % G.CSRC)
    subprocess.run([G._nvcc(), *G.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", str(tmp_path / "t.so"),
                    str(tmp_path / "t.cu")], check=True, capture_output=True)
    L = ctypes.CDLL(str(tmp_path / "t.so"))
    st = (ctypes.c_int * 2)()
    seen = [(L.raise_on(d, f, st), tuple(st)) for d, f in ((0, 0), (0, 0), (1, 1), (1, 0), (1, 0), (0, 0), (70, 0), (70, 0))]
    assert [c for c, _ in seen] == [2, 2, 4, 6, 6, 6, 8, 10]   # beyond 64 devices: every time
    assert [s == (0, 0) for _, s in seen] == [True, True, False, True, True, True, True, True]


def test_no_launcher_keeps_it_for_one_device_only():
    for path in glob.glob(os.path.join(G.CSRC, "*.cu")):
        src = open(path).read()
        assert "static bool attr" not in src and "static const cudaError_t" not in src, path
