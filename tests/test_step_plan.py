"""The tiles that a step is cut into (plan_tiles, tile_span), on the CPU: the
host part of csrc/step_common.cuh compiled into a small program that prints, for
a number of rows and of CTAs resident at once, the grid and its tile sizes, for
the plain step and for the one with optional terms."""
import subprocess

import pytest

from paper_2601_16736_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "step_common.cuh"
int main(int argc, char **argv)
{
    for (int i = 1; i + 1 < argc; i += 2) {
        gs::StepArgs a = {};
        a.n_rows = atoi(argv[i]);
        unsigned grid = gs::plan_tiles<256, false>(a, atoi(argv[i + 1]));
        std::printf("%u %d %d %d\n", grid, a.n_big, a.big_rows, a.tail_rows);
        grid = gs::plan_tiles<256, true>(a, atoi(argv[i + 1]));
        std::printf("%u %d %d %d\n", grid, a.n_big, a.big_rows, a.tail_rows);
    }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-I", str(B.INCLUDE), "-I", str(B.CSRC), "-o", str(d / "plan"),
                    str(d / "plan.cu")], check=True, capture_output=True)

    def run(cases):
        out = subprocess.run([str(d / "plan"), *[str(x) for c in cases for x in c]], check=True, capture_output=True,
                             text=True).stdout
        got = [tuple(map(int, line.split())) for line in out.splitlines()]
        return [(n, terms, *got[2 * i + terms]) for i, (n, _) in enumerate(cases) for terms in (0, 1)]

    return run


def _sizes(wave):
    edges = [wave * t for t in (64, 128, 144, 160, 240, 256, 288, 512, 768, 1024, 2560)] + [wave * 1792 // 10]
    return sorted({max(1, e + d) for e in edges for d in (-257, -256, -1, 0, 1, 17, 255, 256)} |
                  {1, 15, 16, 100, 257, 5003, 100_000, 300_000, 1_000_003, 6_000_000, 2_000_000_011})


@pytest.mark.parametrize("wave", [0, 1, 3, 608, 760])
def test_tiles_cover_the_rows_once(plans, wave):
    for n, _, grid, n_big, big, tail in plans([(n, wave) for n in _sizes(wave)]):
        assert 0 < tail <= 256 and 0 < big <= 256 and tail % 16 == 0 and big % 16 == 0
        left = n - n_big * big                     # the rows of the tail_rows tiles
        assert n_big >= 0 and left >= 0
        assert n_big + (left + tail - 1) // tail == grid > 0


@pytest.mark.parametrize("wave", [608, 760])
def test_no_more_waves_than_whole_tiles(plans, wave):
    """A sparse tile takes much the same time whatever its rows: up to one wave
    of whole tiles, and beyond it with the optional terms, smaller tiles may fill
    the last wave but not begin another; the plain step adds at most an eighth
    of a wave."""
    for n, terms, grid, *_ in plans([(n, wave) for n in _sizes(wave)]):
        whole = -(-n // 256)
        if terms or whole <= wave:
            assert -(-grid // wave) == -(-whole // wave)
        else:
            assert grid <= whole + wave // 8 + 1
