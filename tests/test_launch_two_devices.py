"""Launcher state on a process with two devices (CPU: the runtime is a fake).

The limit on a kernel's dynamic shared memory belongs to one device.  A program
compiled here launches the same large-shared-memory shape on device 0 and then
on device 1, twice each, against stand-ins for the runtime's queries; every
device's limit has to cover the launch before it is made.
"""
import os
import subprocess

from paper_1512_02818_gb300 import build

PROGRAM = r"""
#include <cuda_runtime.h>
#include <stdio.h>

static int device, limit[2] = {48 * 1024, 48 * 1024};
template <class K>
static cudaError_t fake_set(K, cudaFuncAttribute, int bytes) {
  limit[device] = bytes;
  return cudaSuccess;
}
template <class K>
static cudaError_t fake_get(cudaFuncAttributes* fa, K) {
  fa->numRegs = 64;
  return cudaSuccess;
}
static size_t asked;
template <class K>
static cudaError_t fake_occupancy(int* blocks, K, int, size_t smem) {
  asked = smem;  // the launch's own dynamic shared memory
  *blocks = 2;
  return cudaSuccess;
}
#define cudaFuncSetAttribute fake_set
#define cudaFuncGetAttributes fake_get
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_occupancy
#include "pdd_paths.cuh"

__global__ void nothing(pdd::PathArgsN<1>) {}

int main() {
  static std::atomic<int> state[pdd::kMaxBlockThreads / 32 + 1];
  for (int i = 0; i < 4; ++i) {
    device = i & 1;
    pdd::PathArgs a{};
    a.n_segs = 1;
    a.total = 512ull * 100000;
    a.seg[0].total = a.total;
    a.seg[0].n_nodes = 512;
    a.seg[0].n_paths = 100000;
    a.seg[0].h = 1e-3;
    pdd::LaunchInfo info{};
    // (there is no device here: the launch itself returns an error)
    (void)pdd::launch_persistent(nothing, a, 152, 0, &info, pdd::ExitRing<float, 2>::kBytes, 0, 0, 1,
                                 false, state);
    printf("%d %zu %d\n", device, asked, limit[device]);
  }
  return 0;
}
"""


def test_shared_memory_limit_is_set_on_every_device(tmp_path):
    src, exe = tmp_path / "two.cu", tmp_path / "two"
    src.write_text(PROGRAM)
    subprocess.check_call([build.nvcc_path(), "-O0", "-std=c++17", *build.ARCH, "-I", build.CSRC,
                           "-I", os.path.join(build.ROOT, "include"), str(src), "-o", str(exe)])
    lines = subprocess.check_output([str(exe)], text=True).split("\n")[:4]
    rows = [tuple(map(int, line.split())) for line in lines]
    assert [r[0] for r in rows] == [0, 1, 0, 1]
    for device, asked, limit in rows:
        assert asked > 48 * 1024 and limit >= asked, rows
