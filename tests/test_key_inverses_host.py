"""The fast key inverses of the assembly (csrc/lbm_internal.cuh, __host__
__device__), compiled as host code with nvcc and checked without a GPU.

Curves (curve_point / curve_local / curve_cell): in every aligned run of
8^levels keys the cell that the cube's frame gives each local key is the one
the general inverse gives the key, and as many cubes meet the box as it holds
aligned cubes.  Blocked order (blocked_cell, division by multiplication): the
same cell, or none, for every key of small boxes and for keys spread over key
spaces up to 2^31."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include <cstdlib>
#include "lbm_internal.cuh"
namespace lbm {
int fail(int status, const char*, ...) { return status; }
int cuda_fail(cudaError_t, const char*) { return LBM_ECUDA; }
void clear_error() {}
cudaError_t dev_alloc(void**, size_t, cudaStream_t, bool) { return cudaErrorMemoryAllocation; }
void dev_free(void*, cudaStream_t, bool) {}
}
#include "ASSEMBLY"
int main(int argc, char** argv) {
  int32_t dims[3] = {atoi(argv[1]), atoi(argv[2]), atoi(argv[3])};
  lbm_ordering ord{atoi(argv[4]), {1, 1, 1}, 0};
  for (int a = 0; a < 3 && argc > 7; ++a) ord.block[a] = atoi(argv[5 + a]);
  lbm::KeySpace ks;
  if (lbm::make_key_space(dims, ord, true, &ks)) return 2;
  if (ord.kind == LBM_ORDER_BLOCKED) {
    long bad = 0, inside = 0;
    const uint64_t end = ks.size + 5000, stride = end > 3000000 ? end / 1500000 | 1 : 1;
    for (uint64_t k = 0; k < end; k = k + stride < end || k == end - 1 ? k + stride : end - 1) {
      int64_t x, y, z;
      int32_t u, v, w;
      const bool in = lbm::cell_of(ks, k, x, y, z), fast = lbm::blocked_cell(ks, (uint32_t)k, u, v, w);
      bad += in != fast || (in && (x != u || y != v || z != w));
      inside += in;
    }
    printf("%ld %ld %llu\n", bad, inside, (unsigned long long)ks.size);
    return 0;
  }
  const uint64_t run = 1ull << (3 * ks.levels);
  long bad = 0, cubes = 0, inside = 0;
  for (uint64_t tile = 0; tile * run < ks.size; ++tile) {
    lbm::CurveFrame f;
    lbm::curve_point(ks, tile, 0, f.at);
    for (int a = 0; a < 3; ++a) {
      lbm::curve_point(ks, tile, a + 1, f.d[a]);
      for (int b = 0; b < 3; ++b) f.d[a][b] -= f.at[b];
    }
    int32_t low[3];
    for (int a = 0; a < 3; ++a) low[a] = f.at[a] & ~((1 << ks.levels) - 1);
    cubes += low[0] < dims[0] && low[1] < dims[1] && low[2] < dims[2];
    for (uint64_t l = 0; l < run; ++l) {
      uint32_t c[3];
      int32_t p[3];
      int64_t x, y, z;
      lbm::curve_local(ks, (uint32_t)l, c);
      lbm::curve_cell(f, c, p);
      inside += lbm::cell_of(ks, tile * run + l, x, y, z);
      bad += p[0] != x || p[1] != y || p[2] != z;
      for (int a = 0; a < 3; ++a) bad += (p[a] & ~((1 << ks.levels) - 1)) != low[a];
    }
  }
  printf("%ld %ld %ld\n", bad, cubes, inside);
  return 0;
}
'''


@pytest.fixture(scope="module")
def tool(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("curve")
    csrc = os.path.join(ROOT, "paper_1111_1129_gb300", "csrc")
    (d / "curve.cu").write_text(SRC.replace("ASSEMBLY", os.path.join(csrc, "assembly.cu")))
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                           "-I" + csrc, str(d / "curve.cu"), "-o", str(d / "curve")])
    return str(d / "curve")


@pytest.mark.parametrize("kind", [2, 3, 4])
@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 1), (3, 4, 5), (7, 8, 8), (16, 16, 16),
                                  (17, 5, 33), (64, 64, 64), (100, 20, 3), (1, 1, 130)])
def test_cubes_follow_the_curve(tool, kind, dims):
    out = subprocess.run([tool, *map(str, dims), str(kind)], capture_output=True, text=True,
                         check=True).stdout.split()
    bad, cubes, inside = map(int, out)
    assert bad == 0
    assert inside == dims[0] * dims[1] * dims[2]
    assert cubes == -(-dims[0] // 16) * -(-dims[1] // 16) * -(-dims[2] // 16)


@pytest.mark.parametrize("dims,block", [((7, 5, 9), (3, 2, 4)), ((16, 16, 16), (8, 8, 8)),
                                        ((100, 33, 20), (7, 33, 1)), ((1, 1, 50), (1, 1, 64)),
                                        ((1024, 256, 256), (8, 8, 8)), ((1023, 511, 999), (5, 9, 64)),
                                        ((1470000, 10, 100), (1000, 3, 7)), ((1280, 1280, 1280), (64, 64, 64))])
def test_blocked_cells(tool, dims, block):
    out = subprocess.run([tool, *map(str, dims), "1", *map(str, block)], capture_output=True,
                         text=True, check=True).stdout.split()
    bad, inside, size = map(int, out)
    assert size + 5000 < 2 ** 31
    assert bad == 0 and inside > 0
    if size < 2900000:
        assert inside == dims[0] * dims[1] * dims[2]
