"""The row sums' launch on a device that cannot hold a cluster of 16 blocks (a partition of a GPU): the portable 8.
The CUDA runtime's answers come from a stand-in, so no GPU is needed."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#include <cuda_runtime_api.h>
#include <stdlib.h>
static int last, asked;
int last_cluster(void) { return last; }
int times_asked(void) { return asked; }
static int largest(void) { return atoi(getenv("LARGEST_CLUSTER")); }
static int cluster_of(const cudaLaunchConfig_t *c) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)c->attrs[i].val.clusterDim.x;
  return 1;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
  ++asked;
  *n = cluster_of(c) <= largest() ? 1 : 0;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  last = cluster_of(c);
  return last <= largest() ? cudaSuccess : cudaErrorInvalidClusterSize;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaPeekAtLastError(void) { return cudaSuccess; }
"""

CALLS = """
import ctypes as C, sys
L, R = C.CDLL(sys.argv[1]), C.CDLL(sys.argv[2])
p = C.c_void_p(256)
def call(rows, B, dtype):
    st = L.cr_reduce_rows(p, C.c_int64(rows), C.c_int64(B), p, C.c_int32(dtype), None)
    return [st, R.last_cluster()]
for dtype in (0, 1):
    print(*call(6, 262144, dtype), *call(6, 65536, dtype), *call(1, 20000, dtype), *call(6, 100, dtype), R.times_asked())
"""


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    from paper_2607_11340_gb300 import build_lib

    d = tmp_path_factory.mktemp("runtime")
    (d / "runtime.c").write_text(RUNTIME)
    so = str(d / "runtime.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build_lib.nvcc())), "include")
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", inc, str(d / "runtime.c"), "-o", so], check=True)
    return build_lib.build(), so


@pytest.mark.parametrize("largest", [16, 8])
def test_cluster_fits_the_device(runtime, largest):
    lib, so = runtime
    r = subprocess.run([sys.executable, "-c", CALLS, lib, so], capture_output=True, text=True, check=True,
                       env=dict(os.environ, LD_PRELOAD=so, LARGEST_CLUSTER=str(largest)))
    for i, line in enumerate(r.stdout.splitlines()):
        assert [int(x) for x in line.split()] == [0, largest, 0, largest, 0, 8, 0, 1, i + 1]  # asked once a type
    assert r.stdout.count("\n") == 2
