"""The choice of cutting few rods over several CTAs each (host code, no GPU): which cuts are taken, and what the
number of clusters that a device places side by side does to them."""
import os
import shutil
import subprocess

import pytest

from helpers import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "llg_internal.h"

static int g_limit, g_from_k;
// a device that runs at most g_limit clusters of g_from_k or more CTAs side by side, and any number of smaller ones
static int placed(const llg::KParams &, const llg::RodPlan &plan, int) { return plan.split >= g_from_k ? g_limit : 1000; }

int main(int argc, char **argv)
{
    if (argc != 8) return 2;
    llg::KParams p{};
    p.nx = std::atoi(argv[1]);
    p.ny = std::atoi(argv[2]);
    p.nz = std::atoi(argv[3]);
    p.ncells = p.nx * p.ny * p.nz;
    p.n_half = 1000;
    p.sample_every = 10;
    const int kind = std::atoi(argv[4]), n_real = std::atoi(argv[5]);
    g_limit = std::atoi(argv[6]);
    g_from_k = std::atoi(argv[7]);
    llg::RodPlan plan{};
    if (!llg::split_plan(p, n_real, 152, 232448, 0, llg::one_sm_us(p, kind), &plan, placed))
        std::printf("0 0 0 0 0\n");
    else
        std::printf("%d %d %d %d %d\n", plan.split, plan.pairs_per_thread, plan.physics_warps, plan.threads, plan.ctas);
    return 0;
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    """cut(dims, kind, n_real, limit, from_k) -> (CTAs per rod, pairs per thread, physics warps, threads, CTAs)."""
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    from paper_1912_00310_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("cut")
    src = d / "cut.cpp"
    src.write_text(PROGRAM)
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    exe = str(d / "cut")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1912_00310_gb300", "csrc"), "-I",
                    os.path.join(cuda, "include"), str(src), lib, "-Wl,-rpath," + os.path.dirname(lib), "-o", exe], check=True)

    def run(dims, kind, n_real, limit=1000, from_k=2):
        out = subprocess.run([exe, *map(str, (*dims, kind, n_real, limit, from_k))], check=True, capture_output=True, text=True)
        return tuple(map(int, out.stdout.split()))
    return run


# the GPU tests' ensembles (dims, kernel kind uncut, rods) -> CTAs per rod, pairs per thread
CASES = [((8, 24, 56), 2, 2, 8, 2), ((8, 24, 56), 2, 20, 6, 4), ((8, 24, 56), 2, 25, 5, 4), ((8, 24, 56), 2, 32, 4, 4),
         ((8, 24, 56), 2, 40, 6, 4), ((4, 12, 28), 3, 3, 7, 1), ((4, 12, 28), 3, 40, 3, 1), ((4, 12, 28), 3, 70, 2, 1),
         ((5, 11, 23), 1, 3, 8, 1), ((7, 9, 13), 1, 2, 7, 1), ((6, 16, 30), 1, 3, 8, 1), ((6, 16, 30), 1, 30, 4, 2),
         ((1, 15, 40), 1, 2, 8, 1), ((3, 30, 20), 1, 2, 7, 1), ((8, 5, 40), 2, 1, 8, 1), ((5, 24, 56), 2, 30, 8, 2),
         ((10, 20, 24), 2, 36, 4, 4), ((9, 20, 24), 2, 36, 4, 4), ((5, 11, 17), 1, 3, 6, 1)]


@pytest.mark.parametrize("dims,kind,n_real,k,pairs", CASES)
def test_cut_of_the_gpu_tests_ensembles(cut, dims, kind, n_real, k, pairs):
    """They cover 2 to 8 CTAs a rod, one, two and four pairs a thread, rows that fill their segments and rows
    that do not, odd widths, and more clusters than run at once; every thread has its place in a CTA."""
    got = cut(dims, kind, n_real)
    assert got[:2] == (k, pairs) and got[4] == n_real * k
    lines = max(dims[2] * (r + 1) // k - dims[2] * r // k for r in range(k))
    segments = -(-((dims[0] + 1) // 2) // pairs)
    assert got[2] * 32 >= segments * lines * dims[1] > (got[2] - 1) * 32 and got[3] == 32 * (got[2] + 1) <= 384


def test_cuts_covered():
    assert {c[3] for c in CASES} == {2, 3, 4, 5, 6, 7, 8}
    assert {(c[4], c[0][0] % (2 * c[4]) == 0) for c in CASES} == {(w, f) for w in (1, 2, 4) for f in (True, False)}


@pytest.mark.parametrize("dims,kind,n_real", [c[:3] for c in CASES])
def test_cut_follows_what_the_device_places(cut, dims, kind, n_real):
    """A device that cannot place clusters of 7 CTAs or more gets a smaller cut, one that places none, or too few
    at a time to pay, one rod per SM."""
    assert cut(dims, kind, n_real, 0, 7)[0] in (2, 3, 4, 5, 6)
    assert cut(dims, kind, n_real, 0, 2) == (0, 0, 0, 0, 0)
    assert cut(dims, kind, n_real, n_real, 2)[0] >= 2  # all at once
    assert cut(dims, kind, 120, 1, 2) == (0, 0, 0, 0, 0)


def test_small_rods_and_large_ensembles_are_not_cut(cut):
    assert cut((2, 6, 14), 3, 1)[0] == 0 and cut((1, 3, 7), 3, 1)[0] == 0
    assert cut((8, 24, 56), 2, 151)[0] == 0 and cut((4, 12, 28), 3, 151)[0] == 0
