"""What the tile kernels take from a device tile table, built for the host: a tile outside the
arena, reversed ones whose length wraps round to a valid one among them, is taken by no
path."""
import itertools
import os
import shutil
import subprocess

import pytest

from test_philox_forms import ROOT, _cuda_include

TILE_MAX, PART = 1 << 20, 4096


def test_tiles_outside_the_arena_are_refused(tmp_path):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path / "tile_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, os.path.join(ROOT, "tests", "tile_check_main.cpp"), "-o", exe],
                   check=True, capture_output=True, text=True)
    n = 1_000_000
    points = [0, 1, 3, 4, PART - 4, PART, 4 * PART, n - 4 * PART, n - 1, n, n + 1, n + 4, 1 << 20, (1 << 20) + 1,
              (1 << 34) - 4 * PART, 1 << 34, (1 << 34) + 4, (1 << 64) - 4 * PART, (1 << 64) - PART, (1 << 64) - 4,
              (1 << 64) - 1]
    cases = [(b, e, a, PART, log) for b, e, a, log in itertools.product(points, points, (n, 1 << 35, (1 << 64) - 1),
                                                                        (0, 2))]
    out = subprocess.run([exe], input="".join("%d %d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.splitlines()
    assert len(out) == len(cases)
    taken = 0
    for (b, e, a, part, log), line in zip(cases, out):
        inside = b <= e <= a and e - b <= TILE_MAX
        whole = inside and e - b == part << log and b % 4 == 0 and e < 1 << 34
        assert [int(v) for v in line.split()] == [inside, whole], (b, e, a, log)
        taken += whole
    assert taken  # some are whole parts
