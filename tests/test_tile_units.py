"""The cut of tile launches into units, built for the host.  Whatever a caller says of its tiles,
the units cover every tile and stay within what the kernels take; and the geometries that the
GPU tests name reach the paths that they are there for."""
import os
import shutil
import subprocess

import pytest

from test_philox_forms import ROOT, _cuda_include

NOISE, COPIES = 8, 4
RUN_MAX, TILE_MAX = 30, 1 << 20


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path_factory.mktemp("units") / "tile_units")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, os.path.join(ROOT, "tests", "tile_units_main.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)

    def run(cases):
        """Per case its plans as (ragged, units, log_parts, run), ragged None where there is one kernel."""
        out = subprocess.run([exe], input="".join("%d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                             check=True).stdout.splitlines()
        assert len(out) == len(cases)
        plans = []
        for line in out:
            v = [int(x) for x in line.split()]
            noise = [tuple(v[4 * i:4 * i + 4]) for i in range(NOISE)]
            rest = v[4 * NOISE:]
            plans.append(noise + [(None,) + tuple(rest[i:i + 3]) for i in range(0, len(rest), 3)])
        return plans

    return run


def test_units_cover_the_tiles_whatever_the_hint(plan):
    cases = [(n_tiles, n_alloc, elements, aligned)
             for n_tiles in (1, 2, 66, 499, 607, 609, 1217, 8_000, 245_645, (1 << 31) - 1)
             for n_alloc in (1_000, 1 << 20, 11_111_112, 1 << 33, 1 << 35)
             for elements in (0, 1, 77_777, 1 << 20, 11_111_112, 1 << 33, 1 << 35, 1 << 62)
             for aligned in (0, 1)]
    for case, plans in zip(cases, plan(cases)):
        for ragged, units, log, run in plans:
            assert 1 <= run <= RUN_MAX and (log == 0 or run == 1), case
            assert units == -(-case[0] // run) << log and units < 1 << 31, case
            assert 1024 << log <= 2 * TILE_MAX, case


def test_the_mean_length_and_place_choose_the_kernel(plan):
    geometry = [((1000, 1000 * 16384, 1000 * 16384, 1), 0), ((1000, 1000 * 16384, 1000 * 16384, 0), 1),
                ((1000, 1000 * 16384, 0, 0), 0), ((1000, 1 << 35, 1000 * 16384, 1), 1),
                ((1000, 1 << 30, 1000 * 4096, 1), 0), ((1000, 1 << 30, 1000 * 1000, 1), 1),
                ((1000, 1 << 30, 1000 * 6000, 1), 1), ((1000, 1 << 30, 1000 * 65_500, 1), 0),
                ((1000, 1 << 30, 1000 * 65_500, 0), 0)]
    for (_, ragged), plans in zip(geometry, plan([g for g, _ in geometry])):
        assert [p[0] for p in plans[:NOISE]] == [ragged] * NOISE


def test_short_tiles_in_a_large_arena_are_joined_as_in_a_small_one(plan):
    small, large = plan([(4000, 4_000_000, 4_000_000, 0), (4000, 64_000_000, 4_000_000, 0)])
    assert small == large


def test_geometries_of_the_gpu_tests(plan):
    """test_gpu_tile_units.py: runs of joined tiles with more than three waves of units, which are
    taken over early as well as late."""
    from test_gpu_tile_units import CASES, EARLY_RUNS
    late = 3 * 4 * 152
    for index, which in EARLY_RUNS.items():
        n, ranges, tile = CASES[index]
        n_tiles = sum(-(-(e - b) // tile) for b, e in ranges)
        aligned = all(b % 4 == 0 for b, e in ranges) and tile % 4 == 0
        plans = plan([(n_tiles, n, sum(e - b for b, e in ranges), aligned)])[0]
        taken = plans[0] if which == "perturb" else plans[NOISE + COPIES]  # by up to three noise vectors
        assert not taken[0] and taken[3] > 1 and taken[1] > late + 100, (index, taken)


@pytest.mark.parametrize("tile", [9_000, 12_000, 16_384, 20_000, 24_000, 50_000, 65_536])
def test_an_update_of_a_few_waves_gives_every_sm_its_blocks(plan, tile):
    for n in (2_200_000, 7_000_000, 11_111_112, 18_000_000):
        n_tiles = -(-n // tile)
        plans = plan([(n_tiles, n, n, 1)])[0]
        for _, units, log, run in plans[NOISE + COPIES + 1:NOISE + COPIES + 3]:  # by 4 and 32 noise vectors
            assert units >= 4 * 152 and run * tile >> log <= 2 * 16_384, (n, units, log, run)
