"""What a dictionary does without when device memory is refused (host logic,
CPU): the sizes of its tables and which of them the allocation leaves out, with
an allocator that takes up to a given number of bytes."""
import os
import shutil
import subprocess

import pytest

from paper_1806_04374_gb300 import build

SRC = r"""
#include <stdio.h>
#include <stdlib.h>
#include "dict_tables.h"
int main(int argc, char **argv) {
  const int M = atoi(argv[1]), H = atoi(argv[2]), R = atoi(argv[3]), L = atoi(argv[4]);
  const size_t room = strtoull(argv[5], nullptr, 10);
  const cudaError_t other = argc > 6 ? cudaErrorIllegalState : cudaSuccess;
  RefineTables t = plan_refine_tables(M, H, R, R % 2 ? R : R / 2, L);
  int calls = 0;
  void *base = nullptr;
  const cudaError_t e = alloc_refine_tables(t, [&](void **p, size_t n) {
    ++calls;
    if (other != cudaSuccess) return other;
    if (n > room) return cudaErrorMemoryAllocation;
    *p = &calls;
    return cudaSuccess;
  }, &base);
  printf("%d %d %d %zu %zu %zu %zu\n", (int)e, calls, base != nullptr, t.xgram, t.anorm, t.rows, t.gram);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("tables")
    src, exe = d / "t.cpp", str(d / "t")
    src.write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-I", build.CSRC, "-I", inc, str(src),
                    "-o", exe], check=True)

    def call(*a):
        out = subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout
        return [int(v) for v in out.split()]
    return call


@pytest.mark.parametrize("M, H, R, L", [(64, 9, 64, 112), (7, 9, 33, 112), (256, 13, 128, 256)])
def test_what_is_left_out(run, M, H, R, L):
    def up(v):
        return (v + 255) // 256 * 256
    x, a, r = up(M * M * H * 16), up(M * 8), up((R if R % 2 else R // 2) * M * L * 8)
    g = M * M * R * 8
    assert run(M, H, R, L, x + a + r + g) == [0, 1, 1, x, a, r, g]
    # one byte short of each amount: the next smaller set
    assert run(M, H, R, L, x + a + r + g - 1) == [0, 2, 1, x, a, r, 0]
    assert run(M, H, R, L, x + a + r) == [0, 2, 1, x, a, r, 0]
    assert run(M, H, R, L, x + a + r - 1) == [0, 3, 1, x, a, 0, 0]
    assert run(M, H, R, L, x + a) == [0, 3, 1, x, a, 0, 0]
    assert run(M, H, R, L, x + a - 1)[:3] == [2, 3, 0]  # cudaErrorMemoryAllocation
    # any other error is passed on at once
    assert run(M, H, R, L, 1 << 40, "other")[:3] == [401, 1, 0]


def test_large_gram_is_not_asked_for(run):
    v = run(1024, 9, 64, 112, 1 << 40)
    assert v[1] == 1 and v[6] == 0 and v[5] > 0
    v = run(1024, 9, 64, 112, v[3] + v[4])
    assert v[:3] == [0, 2, 1] and v[5] == 0
