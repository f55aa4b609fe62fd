"""Key spaces at the ends of their 64 bits (make_key_space in
csrc/assembly.cu), compiled as host code with nvcc and checked without a GPU.

Curve keys hold 21 bits per axis (Morton with 1 bit, Hilbert) or 20 (Morton
with 2 bits): an axis that needs more is refused with LBM_EOVERFLOW, for keys
and for the assembly alike, and the longest one that fits is not."""
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
// dims[3] kind block[3] walk: the status, and the key of the box's last cell
int main(int, char** argv) {
  int32_t dims[3] = {atoi(argv[1]), atoi(argv[2]), atoi(argv[3])};
  lbm_ordering ord{atoi(argv[4]), {atoi(argv[5]), atoi(argv[6]), atoi(argv[7])}, 0};
  lbm::KeySpace ks{};
  const int rc = lbm::make_key_space(dims, ord, atoi(argv[8]) != 0, &ks);
  unsigned long long k = 0;
  if (rc == LBM_OK) k = lbm::key_of(ks, dims[0] - 1, dims[1] - 1, dims[2] - 1);
  printf("%d %llu\n", rc, k);
  return 0;
}
'''
MORTON1, MORTON2, HILBERT = 2, 3, 4
OK, EOVERFLOW = 0, -2


@pytest.fixture(scope="module")
def tool(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("limits")
    csrc = os.path.join(ROOT, "paper_1111_1129_gb300", "csrc")
    (d / "limits.cu").write_text(SRC.replace("ASSEMBLY", os.path.join(csrc, "assembly.cu")))
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                           "-I" + csrc, str(d / "limits.cu"), "-o", str(d / "limits")])

    def run(dims, kind, block, walk):
        out = subprocess.run([str(d / "limits"), *map(str, dims), str(kind), *map(str, block),
                              str(int(walk))], capture_output=True, text=True, check=True)
        return tuple(map(int, out.stdout.split()))
    return run


@pytest.mark.parametrize("walk", [False, True])
@pytest.mark.parametrize("kind,bits", [(MORTON1, 21), (MORTON2, 20), (HILBERT, 21)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_curve_keys_are_not_cut(tool, kind, bits, axis, walk):
    dims = [1, 1, 1]
    dims[axis] = 2 ** bits
    rc, key = tool(dims, kind, (1, 1, 1), walk)
    assert rc == OK
    if kind != HILBERT:   # the last cell has every bit of its axis set
        group = 1 if kind == MORTON1 else 2
        assert key == sum(1 << (3 * group * (b // group) + group * axis + b % group)
                          for b in range(bits))
    dims[axis] += 1
    assert tool(dims, kind, (1, 1, 1), walk)[0] == EOVERFLOW


@pytest.mark.parametrize("dims,block", [((1, 1, 16), (2 ** 30, 2 ** 30, 4)),
                                        ((1, 4, 16), (2 ** 30, 2, 2 ** 31 - 1)),
                                        ((3, 1, 32), (2 ** 30, 2 ** 29, 8))])
def test_blocks_far_beyond_the_box_have_keys(tool, dims, block):
    """Keys keep the literal blocking factors, so their space may span more
    than 64 bits although every key of the box fits."""
    last = [d - 1 for d in dims]
    blocks = [-(-d // b) for d, b in zip(dims, block)]
    of = [c // b for c, b in zip(last, block)]
    at = [c % b for c, b in zip(last, block)]
    number = of[0] + blocks[0] * (of[1] + blocks[1] * of[2])
    key = (number * block[0] * block[1] * block[2] +
           at[0] + block[0] * (at[1] + block[1] * at[2]))
    assert key < 2 ** 64
    assert tool(dims, 1, block, False) == (OK, key)
