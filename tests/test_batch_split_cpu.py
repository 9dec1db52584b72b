"""The choice of CTAs an instance of the batched step (csrc/batch_split.cuh,
host code) against the cluster sizes measured fastest."""
import os
import subprocess

import pytest

from paper_2412_16843_gb300 import build, inputs

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "batch_split.cuh"
int main(int argc, char** argv) {  // FP64, threads, sizes, slots of each, then the cell counts in decreasing order
    const bool fp64 = std::atoi(argv[1]) != 0;
    const int threads = std::atoi(argv[2]), sizes = std::atoi(argv[3]);
    int slots[8];
    for (int k = 0; k < sizes; ++k) slots[k] = std::atoi(argv[4 + k]);
    std::vector<long> cells;
    for (int i = 4 + sizes; i < argc; ++i) cells.push_back(std::atol(argv[i]));
    std::printf("%d\n", 1 << cdi::batch_split_choice(cells.data(), (int)cells.size(), slots, sizes, fp64, threads));
}
"""


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", build.CSRC, str(d / "h.cpp"), "-o", str(d / "h")], check=True)

    def run(cells, fp64=False, threads=1024, slots=(152, 76, 36, 15, 7)):
        args = [int(fp64), threads, len(slots)] + list(slots) + sorted(cells, reverse=True)
        return int(subprocess.run([str(d / "h")] + [str(a) for a in args], capture_output=True, text=True,
                                  check=True).stdout)

    return run


@pytest.mark.parametrize("fp64,threads,n,ctas", [
    (False, 1024, 32, 8), (False, 1024, 64, 8), (False, 1024, 128, 4), (False, 1024, 160, 4), (False, 1024, 256, 2),
    (False, 1024, 512, 2), (False, 256, 80, 8), (False, 512, 512, 2), (True, 512, 32, 16), (True, 1024, 48, 8),
    (True, 1024, 64, 8), (True, 1024, 256, 2), (True, 512, 512, 2)])
def test_sweep_takes_the_size_measured_fastest(choice, fp64, threads, n, ctas):
    """The fastest of the five sizes by 9 % or more where they were measured."""
    assert choice([w.cells for w in inputs.sweep_2d()[:n]], fp64, threads) == ctas


def test_3d_batches_take_the_size_measured_fastest(choice):
    for fp64 in (False, True):
        assert choice([(16, 24, 32, 48, 64)[i % 5] ** 3 for i in range(16)], fp64) == 16
        assert choice([(16, 24, 32, 48, 64)[i % 5] ** 3 for i in range(100)], fp64) == 4
    assert choice([(16, 24, 32)[i % 3] ** 3 for i in range(48)]) == 4


@pytest.mark.parametrize("fp64,cells,last", [(False, 64 * 32, 1), (True, 64 * 32, 1), (False, 16 ** 3, 1),
                                             (True, 16 ** 3, 2)])
def test_equal_grids_take_what_leaves_a_slot_for_each(choice, fp64, cells, last):
    """160 grids are two rounds of CTAs or three of pairs: the FP64 step of
    16^3 cells, 4.7 ms on one CTA and 2.9 on two, is through earlier in three."""
    assert [choice([cells] * n, fp64, 512) for n in (1, 10, 20, 60, 160)] == [16, 8, 4, 2, last]


def test_sizes_that_do_not_fit_are_not_taken(choice):
    assert choice([131072], slots=(152,)) == 1
    assert choice([131072], slots=(152, 76, 36)) == 4
    assert choice([2048] * 5, slots=(1,)) == 1
