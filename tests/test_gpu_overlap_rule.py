"""Which grids take part in overlapped launches: a kernel of at most 1216
blocks, over all three extents of its grid, lets the next kernel be set up
while it runs (grid_begin() in csrc/common.cuh), a larger one does not.

Each case runs two kernels of its own: the first calls grid_begin() and then
keeps every block busy for a fixed time, the second is launched as dependent
and notes when it starts. It starts before the first one's end exactly when
the first one released it."""
import ctypes
import os
import subprocess

import pytest

from paper_2505_17287_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "common.cuh"
__device__ __forceinline__ unsigned long long now() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__global__ void k_first(unsigned long long *end, unsigned long long ns) {
    ibm::grid_begin();
    const unsigned long long t0 = now();
    while (now() - t0 < ns) {}
    atomicMax(end, now());
}
__global__ void k_second(unsigned long long *start) {
    *start = now();
    ibm::grid_wait();
}
// 1: the second kernel started before the first one's end; 0: after; -1: error
extern "C" int second_starts_early(int x, int y, int z) {
    unsigned long long *d = nullptr, h[2] = {0, 0};
    cudaStream_t s;
    if (cudaMalloc(&d, 16) != cudaSuccess || cudaStreamCreate(&s) != cudaSuccess) return -1;
    cudaMemsetAsync(d, 0, 16, s);
    k_first<<<dim3(x, y, z), 32, 0, s>>>(d, 200000ull);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, 1, 1);
    cfg.blockDim = dim3(1, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_second, d + 1);
    cudaMemcpyAsync(h, d, 16, cudaMemcpyDeviceToHost, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    cudaStreamDestroy(s);
    cudaFree(d);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? (h[1] < h[0] ? 1 : 0) : -1;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("overlap")
    src, lib = d / "probe.cu", d / "probe.so"
    src.write_text(SRC)
    subprocess.run([build.NVCC, *build.COMMON, "-I", build.CSRC, "-shared", "-cudart", "shared", "-o", str(lib),
                    str(src)], check=True, capture_output=True, text=True)
    f = ctypes.CDLL(os.fspath(lib)).second_starts_early
    f.argtypes, f.restype = [ctypes.c_int] * 3, ctypes.c_int
    f(1, 1, 1)   # (context and module set up)
    return f


@pytest.mark.parametrize("grid", [(1, 1, 1), (1216, 1, 1), (1217, 1, 1), (152, 8, 1), (152, 9, 1), (8, 8, 19),
                                  (8, 8, 20), (6, 32, 64), (12, 64, 3)])
def test_only_small_grids_release_the_next_kernel(probe, grid):
    n = grid[0] * grid[1] * grid[2]
    # (a host that is held up between the two launches starts the second late)
    got = [probe(*grid) for _ in range(5)]
    assert min(got) >= 0 and max(got) == (1 if n <= 1216 else 0), (grid, got)
