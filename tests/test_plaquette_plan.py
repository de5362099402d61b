"""The cut of the plaquette kernel's work, compiled for the host: at every even
extent all time slices of all sites are covered, and the block with most to do
has little more than its share of the steps."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1010_1486_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "plaquette_plan.h"
int main()
{
    int ns, nt, sms;
    while (scanf("%d %d %d", &ns, &nt, &sms) == 3) {
        const su2::PlaquettePlan p = su2::plaquette_plan(ns * ns * ns, nt, sms);
        printf("%d %d %d %d\\n", p.pair_blocks, p.t_chunk, p.items, p.grid);
    }
}
"""
CUBES = [(n, n) for n in range(2, 130, 2)]
OTHERS = [(2, 60_000_000), (4, 64), (64, 4), (100, 6), (128, 8), (812, 2), (8, 256), (32, 4), (48, 96)]


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)
    shapes = [(ns, nt, sms) for ns, nt in CUBES + OTHERS for sms in (152, 148, 1)]
    out = subprocess.run([str(d / "plan")], input="\n".join(f"{a} {b} {c}" for a, b, c in shapes),
                         capture_output=True, text=True, check=True).stdout
    return dict(zip(shapes, ([int(v) for v in line.split()] for line in out.splitlines())))


def test_items_cover_the_lattice_once(plans):
    assert len(plans) == 3 * len(CUBES + OTHERS)
    for (ns, nt, sms), (pair_blocks, t_chunk, items, grid) in plans.items():
        chunks = -(-nt // t_chunk)
        assert (pair_blocks - 1) * 384 < ns ** 3 // 2 <= pair_blocks * 384
        assert 1 <= t_chunk <= nt and items == pair_blocks * chunks and grid == min(items, sms)


def test_no_extent_leaves_much_of_the_machine_idle(plans):
    for (ns, nt, sms), (pair_blocks, t_chunk, items, grid) in plans.items():
        longest = -(-items // sms) * t_chunk
        share = pair_blocks * nt / sms
        assert longest <= 1.25 * share + 1, (ns, nt, sms, longest, share)
