"""The FP64 path's pair law at the edges of its integer arithmetic (no GPU).

Same probe and reference as test_pair64_cpu.py (60-digit arithmetic on the same FP64
differences) and, for the lengths of the three result vectors, its bound: 2^-50 of the
summed sizes of the terms.
"""
import os
import subprocess
from decimal import Decimal

import numpy as np
import pytest

from test_pair64_cpu import CUDA_INC, ROOT, _exact, probe   # noqa: F401  (probe: fixture)

ZERO = np.zeros(9)


def _within_sizes(got, eps, i, js):
    s, size, _ = _exact(eps, i, js)
    for f in range(3):
        err = sum((Decimal(float(got[3 * f + k])) - s[3 * f + k]) ** 2 for k in range(3)).sqrt()
        assert err <= size[f] * Decimal(2) ** -50, (f, float(err / size[f]), got, [float(x) for x in s])


def _lattice():
    """Largest component an exact power of two, a second one 2^-32 .. 2^-28 of it, either
    sign; the velocity along the separation, so that alpha carries the jerk."""
    for r0, eps in ((1.0, 0.0), (2.0 ** 18, 1e-4), (1024.0, 1e-6), (2.0 ** -7, 0.0)):
        for k in range(28, 33):
            for f in (1.0, 1.25, 1.5, -1.0, -1.25, -1.5):
                yield eps, [1.0, r0, f * r0 * 2.0 ** -k, 0, -r0, 0, 0, 0, 0, 0]
                yield eps, [1.0, 0, -f * r0 * 2.0 ** -k, -r0, 0, 0, 3 * r0, 0, 0, 1]


def test_separation_of_a_power_of_two(probe):   # noqa: F811
    for eps, j in _lattice():
        _within_sizes(probe(eps, ZERO, [j]), eps, ZERO, [j])


def test_shift_counts_in_range(tmp_path):
    """No shift by a negative count or by the width or more, over the same systems."""
    if not os.path.isdir(CUDA_INC):
        pytest.skip("needs the CUDA headers")
    exe = str(tmp_path / "pair64_probe_shifts")
    if subprocess.run(["g++", "-std=c++17", "-O1", "-fno-strict-aliasing", "-fsanitize=shift-exponent",
                       "-fno-sanitize-recover=shift-exponent", "-I", CUDA_INC, "-I", os.path.join(ROOT, "include"),
                       "-I", os.path.join(ROOT, "paper_1207_2367_gb300", "csrc"),
                       os.path.join(ROOT, "tests", "host", "pair64_probe.cpp"), "-o", exe]).returncode:
        pytest.skip("needs g++ with its undefined-behaviour sanitizer")
    words = []
    for eps, j in _lattice():
        words += [float(eps).hex(), "1"] + [float(x).hex() for x in (*ZERO, *j)]
    r = subprocess.run([exe], input=" ".join(words), capture_output=True, text=True)
    assert r.returncode == 0 and not r.stderr, r.stderr[:500]
