"""The twiddle rows of the line transforms, on the host: every supported size's
stages, the entries its rows take (counted here from the radices), and the fixed
array of the allocation-free solve, which has to hold the rows of every size it takes
(they do not grow with the size: 96 points need more than 128)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_12629_gb300", "csrc")
SIZES = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048]

PROGRAM = r"""
#include <cstdio>
#include "fft_plan.cuh"
using namespace cube2;
int main() {
    std::printf("%d %d\n", NOALLOC_MAX_N, NOALLOC_TWIDDLES);
    for (int n = 1; n <= 2048; ++n) {
        if (!stages_of(n, false)) continue;
        std::printf("%d %d", n, twiddle_entries(n));
        for (int xp = 0; xp < 2; ++xp) {
            std::printf(" :");
            for (int s = 0; s < stages_of(n, xp); ++s) std::printf(" %d", radix_at(n, s, xp));
        }
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("plan")
    src, exe = str(d / "plan.cpp"), str(d / "plan")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-D__host__=", "-D__device__=", "-I", CSRC, src, "-o", exe], check=True)
    head, *lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    sizes = {}
    for line in lines:
        first, tile, xpass = line.split(":")
        n, entries = map(int, first.split())
        sizes[n] = entries, [list(map(int, r.split())) for r in (tile, xpass)]
    return tuple(map(int, head.split())), sizes


@pytest.mark.parametrize("n", SIZES)
def test_rows_of_a_size(plan, n):
    entries, radices = plan[1][n]
    want = 0
    for r in radices:
        product = 1
        for k in r:
            product *= k
        assert product == n
        for order in (r, r[::-1]):     # forward and inverse, from the second stage on
            want += sum((k - 1) * (n // k) for k in order[1:])
    assert entries == want


def test_sizes(plan):
    assert sorted(plan[1]) == SIZES


def test_fixed_array_holds_every_size(plan):
    (max_n, capacity), sizes = plan
    for n in SIZES:
        if n <= max_n:
            assert sizes[n][0] <= capacity, n
