"""Lazy evaluation compares what every seed newly covers with its gain: a wrong
gain is found also where a second one makes up for it in the sum."""

import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1212_4779_gb300", "csrc")


@pytest.fixture(scope="module")
def first_mismatch(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("celf") / "celf_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(HERE, "celf_check.cpp"), "-o", exe], check=True)

    def run(covered, gains):
        """covered: pairs newly covered by each seed."""
        at = np.concatenate([[0], np.cumsum(covered)])
        text = " ".join(str(int(v)) for v in [len(gains), *at, *gains])
        return int(subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout)

    return run


@pytest.mark.parametrize("k", [1, 2, 50])
def test_each_seed_is_compared(first_mismatch, k):
    gains = np.sort(np.random.default_rng(k).integers(1, 1 << 40, k))[::-1]
    assert first_mismatch(gains, gains) == -1
    for i in range(k):
        wrong = gains.copy()
        wrong[i] += 1
        assert first_mismatch(wrong, gains) == i
        if i + 1 < k:
            wrong[k - 1] -= 1  # the sums agree again
            assert first_mismatch(wrong, gains) == i
