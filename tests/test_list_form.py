"""Which traversal builds a system's lists: the rule, compiled by itself, against the times that were measured at its lines."""
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "list_form.cuh"
int main(int argc, char **argv) {
    const int64_t n = atoll(argv[1]);
    if (argc == 5) { printf("%d %d\n", mlip::lists_are_long(n, atoll(argv[2])), mlip::lists_expected_long(atof(argv[3]))); return 0; }
    if (argc == 3) { printf("%d\n", mlip::list_lane_row(n, atof(argv[2]), 148)); return 0; }
    const mlip::ListForm f = mlip::list_form(n, atoll(argv[2]), atoi(argv[3]) != 0);
    printf("%s %lld %lld\n", f == mlip::ListForm::WARP_1 ? "warp 1" : f == mlip::ListForm::WARP_8 ? "warp 8" : "lanes", (long long)((n + mlip::list_form_tile(f) - 1) / mlip::list_form_tile(f)), (long long)mlip::list_tile_words(n));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("list_form")
    (d / "rule.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", f"{ROOT}/paper_2608_16329_b200/csrc", "-o", str(d / "rule"), str(d / "rule.cpp")])
    return str(d / "rule")


@pytest.fixture(scope="module")
def rule(program):
    def ask(n, cells):
        rel, n_cells = all(c >= 3 for c in cells), cells[0] * cells[1] * cells[2]
        form, tiles, words = subprocess.check_output([program, str(n), str(n_cells), str(int(rel))], text=True).strip().rsplit(" ", 2)
        assert int(tiles) <= int(words)   # every tile has its look-back word
        return form
    return ask


@pytest.mark.parametrize("n,form", [(1, "warp 1"), (17999, "warp 1"), (18400, "warp 1"), (38416, "warp 1"), (49999, "warp 1"), (50000, "warp 8"), (1000000, "warp 8")])
def test_grids_of_two_cells_across(rule, n, form):
    assert rule(n, (2, 60, 60)) == form


@pytest.mark.parametrize("n,cells,form", [(17999, (9, 9, 9), "warp 1"), (19652, (8, 8, 8), "lanes"), (8001504, (64, 64, 64), "lanes")])
def test_condensed_systems(rule, n, cells, form):
    assert rule(n, cells) == form


# one atom per cell up to six, and a ball of 85,601 atoms in a wide box
@pytest.mark.parametrize("n,cells,form", [(20000, (27, 27, 27), "warp 1"), (18500, (18, 18, 18), "warp 1"), (18500, (16, 16, 16), "lanes"), (25000, (23, 23, 23), "warp 1"),
                                          (25000, (20, 20, 20), "lanes"), (70000, (41, 41, 41), "warp 8"), (70000, (32, 32, 32), "lanes"), (150000, (53, 53, 53), "warp 8"),
                                          (150000, (36, 36, 36), "lanes"), (300000, (66, 66, 66), "warp 8"), (1000000, (101, 101, 101), "warp 8"), (1000000, (87, 87, 87), "lanes"),
                                          (85601, (57, 57, 57), "warp 8")])
def test_sparse_systems(rule, n, cells, form):
    assert rule(n, cells) == form


@pytest.mark.parametrize("n,mean,least,most", [(18000, 61.6, 160, 640), (55296, 61.6, 160, 640), (80000, 61.6, 160, 640),   # half-empty boxes of 134-entry lists
                                               (432000, 80.0, 112, 124), (8001504, 123.2, 168, 180), (8001504, 0.5, 64, 64), (18000, 2000.0, 640, 640)])
def test_rows_of_the_lanes(program, n, mean, least, most):
    row = int(subprocess.check_output([program, str(n), str(mean)], text=True))
    assert least <= row <= most and row % 4 == 0
    per_sm = ((n + 63) // 64 + 147) // 148
    if row > max(1.3 * mean + 16, 64):   # longer than the mean asks for: every tile still runs at once
        assert per_sm * (64 * 2 * (row + 2) + 2 * 2 * 3 * 32 * 4 + 800 + 1024) <= 227 * 1024


# lists of more than 96 leading entries among all; the mean at the box's density: alloy of 134 entries (99 within 6.5 Angstrom), liquids of 0.08, 0.1 and 0.13 atoms per cubic Angstrom
@pytest.mark.parametrize("n_long,n,mean,by_count,by_density", [(0, 100000, 98.6, 0, 0), (10000, 100000, 92.0, 0, 0), (10001, 100000, 115.0, 1, 1), (100000, 100000, 150.0, 1, 1), (0, 0, 0.0, 0, 0)])
def test_atoms_one_after_the_other(program, n_long, n, mean, by_count, by_density):
    assert subprocess.check_output([program, str(n_long), str(n), str(mean), "-"], text=True).split() == [str(by_count), str(by_density)]
