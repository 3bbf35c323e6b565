"""The folded Philox4x32-10 with keys folded for a counter's other words (the high word of
the noise counters past 2^32; the tensor id and high word of the partition's), built for the
host and checked word for word against the oracle's Philox."""
import itertools
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_philox_forms import ROOT, _cuda_include


def test_folded_keys_for_any_counter_match_the_oracle(tmp_path):
    import oracle
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path / "philox_counters")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, os.path.join(ROOT, "tests", "philox_counters_main.cpp"),
                    "-o", exe], check=True, capture_output=True, text=True)
    rng = np.random.default_rng(4)
    words = [0, 1, 2**31, 2**32 - 1] + [int(v) for v in rng.integers(0, 2**32, 3)]
    keys = [0, 33, 2**64 - 1, int(rng.integers(0, 2**63))]
    cases = [(k, c0, c1, c2, tag) for k, c0, c1, c2, tag in itertools.product(keys, words, words, words, (0, 2))]
    out = subprocess.run([exe], input="".join("%d %d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.splitlines()
    assert len(out) == len(cases)
    for (k, c0, c1, c2, tag), line in zip(cases, out):
        ref = oracle.philox4x32_10([c0, c1, c2, tag], [k & 0xFFFFFFFF, k >> 32])
        assert [int(v) for v in line.split()] == [int(v) for v in ref], (k, c0, c1, c2, tag)


def test_single_words_match_the_oracle(tmp_path):
    import oracle
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path / "philox_word")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, os.path.join(ROOT, "tests", "philox_word_main.cpp"),
                    "-o", exe], check=True, capture_output=True, text=True)
    rng = np.random.default_rng(5)
    cases = [(k, c) for k in [0, 33, 2**64 - 1] + [int(v) for v in rng.integers(0, 2**63, 20)]
             for c in [0, 1, 2**31, 2**32 - 1] + [int(v) for v in rng.integers(0, 2**32, 20)]]
    out = subprocess.run([exe], input="".join("%d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.splitlines()
    assert len(out) == len(cases)
    for (k, c), line in zip(cases, out):
        ref = oracle.philox4x32_10([c, 0, 0, 0], [k & 0xFFFFFFFF, k >> 32])
        assert [int(v) for v in line.split()] == [int(v) for v in ref], (k, c)


def test_high_keys_match_the_oracle(tmp_path):
    import oracle
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("g++ or the CUDA headers are not available")
    exe = str(tmp_path / "philox_high")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", inc, os.path.join(ROOT, "tests", "philox_high_main.cpp"),
                    "-o", exe], check=True, capture_output=True, text=True)
    rng = np.random.default_rng(6)
    words = [0, 1, 2, 2**31, 2**32 - 1] + [int(v) for v in rng.integers(0, 2**32, 3)]
    cases = [(k, c0, c1, tag) for k in (0, 33, 2**64 - 1, int(rng.integers(0, 2**63))) for c0 in words for c1 in words
             for tag in (0, 1)]
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.splitlines()
    assert len(out) == len(cases)
    for (k, c0, c1, tag), line in zip(cases, out):
        ref = oracle.philox4x32_10([c0, c1, 0, tag], [k & 0xFFFFFFFF, k >> 32])
        assert [int(v) for v in line.split()] == [int(v) for v in ref], (k, c0, c1, tag)
