"""The MMAs that one K block of a split contraction issues, replayed on the CPU (csrc/mma_schedule.h).

Every slice product (i, j) with i + j <= S + 1 belongs to the contraction once and no other does; a product
with j = 0 would read the shared memory in front of the B tiles. S = 8 has rows of A (i = 7, 8) whose
diagonals all lie past the last accumulator of its own.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1610_00823_gb300", "csrc")

PRINT = r"""
#include <cstdio>
#include <initializer_list>
#include "mma_schedule.h"
using namespace vfmm;
int main() {
    for (int S = kMinSlices; S <= kSlices; ++S)
        for (int N : {48, 64, 80})
            for (int i = 1; i <= S; ++i)
                for (int q = 0; q < mma_count(S, N, i); ++q) {
                    const MmaStep m = mma_step(S, N, i, q);
                    std::printf("%d %d %d %d %d %d\n", S, N, i, m.j, m.w, acc_of(i, m.j));
                }
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a host C++ compiler")
    d = tmp_path_factory.mktemp("mma_schedule")
    src, exe = d / "print.cpp", d / "print"
    src.write_text(PRINT)
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [tuple(int(x) for x in line.split()) for line in out.splitlines()]


@pytest.mark.parametrize("S", [6, 7, 8])
@pytest.mark.parametrize("N", [48, 64, 80])
def test_every_slice_product_is_issued_once(steps, S, N):
    done = {}
    for s, n, i, j, w, acc in steps:
        if (s, n) != (S, N):
            continue
        assert j >= 1 and w >= 1 and w * N <= 256
        for t in range(w):
            # columns of a wide MMA are consecutive accumulators: product (i, j + t) on its diagonal's,
            # diagonals 5 and up on the sixth
            assert acc + t == min(i + j + t - 2, 5)
            done[i, j + t] = done.get((i, j + t), 0) + 1
    want = {(i, j): 1 for i in range(1, S + 1) for j in range(1, S + 2 - i)}
    assert done == want and len(want) == S * (S + 1) // 2
