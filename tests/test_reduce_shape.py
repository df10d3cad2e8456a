"""CPU checks of the rule that gives an item of the exact reduction its CTAs
(csrc/pp_reduce_shape.h, compiled by itself)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01655_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "pp_reduce_shape.h"
int main(int argc, char **argv)          // wide, items, cluster sizes: prints bins and the size chosen
{                                        // (or: "spend", n, weight, CTAs, tiles in sequence: the prices allowed)
    pp::ReduceShape r;
    if (argv[1][0] == 's') {
        r.ncl = 1;
        r.cl[0] = atoi(argv[4]);
        r.path[0] = atoi(argv[5]);
        pp::set_spending(r, atoi(argv[2]), atoi(argv[3]), 16);
        printf("%d %d\n", r.spending[0].evals[0], r.spending[0].evals[1]);
        return 0;
    }
    r.bins = 16;
    for (int i = 3; i < argc; ++i) {
        r.cl[r.ncl] = atoi(argv[i]);
        r.acc[r.ncl++] = 100 * atoi(argv[i]);
    }
    pp::set_wide(r, atoi(argv[1]));
    const int x = r.bins ? pp::cluster_index(r, atoi(argv[2])) : 0;
    printf("%d %d %d\n", r.bins, r.bins ? r.cl[x] : 0, r.bins ? r.acc[x] : 0);
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("shape")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I" + CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def run(wide, items, sizes):
        out = subprocess.run([str(d / "main"), str(wide), str(items), *map(str, sizes)], check=True,
                             capture_output=True, text=True).stdout
        return tuple(int(x) for x in out.split())
    return run


def test_sizes_that_the_device_does_not_run_are_not_chosen(choose):
    """Without a cluster of 16 on the device the item takes 8 CTAs, and a tree
    whose tiles fit only 16 is not reduced."""
    assert choose(0, 1, [16, 8, 4, 2, 1]) == (16, 8, 800)
    assert choose(0, 40, [16, 8, 4, 2, 1]) == (16, 2, 200)
    assert choose(0, 1, [16]) == (0, 0, 0)
    assert choose(7, 1, [16]) == (16, 16, 1600)


def test_ctas_by_items_in_flight(choose):
    """16 CTAs an item while the device runs seven of every eight at a time,
    then as many as 128 CTAs give."""
    assert [choose(7, i, [16, 8, 4, 2, 1])[1] for i in (1, 8, 9, 16, 17, 33, 65, 500)] == [16, 16, 8, 8, 4, 2, 1, 1]
    assert [choose(0, i, [6, 3, 2, 1])[1] for i in (1, 21, 22, 43, 65)] == [6, 6, 3, 2, 1]


def test_prices_allowed_by_what_the_sweep_takes(choose):
    """At least four (six prices' worth) or none: a chain of 800 rows is left to
    the sweep up to 128 columns, a star or a weighted chain of 800 is not, and
    from some thousand rows on all sixteen are allowed."""
    assert choose("spend", 800, (1, 1, 25)) == (0, 4)
    assert choose("spend", 800, (9, 1, 25)) == (15, 15)
    assert choose("spend", 800, (1, 1, 1)) == (16, 16)
    assert choose("spend", 128, (1, 1, 4)) == (5, 6)
    assert choose("spend", 400, (1, 1, 13)) == (0, 4)
    assert choose("spend", 12000, (1, 6, 8)) == (16, 16)
