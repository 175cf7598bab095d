"""The FP64 path's fixed-point pair law against exact rational arithmetic (no GPU).

The header is compiled for the host with a small probe program
(tests/host/pair64_probe.cpp).  Reference: the pair law in decimal arithmetic of
60 digits on the same FP64 inputs (differences rounded to FP64, as the kernel
forms them).  Bounds: a term errs by a few 2^-55 of q |r|, q |v| and of
q (|a| + v^2 / R), the sizes its parts have before they cancel (the largest
coefficients, 12 of lambda w and 6 of kappa n, count as parts of the size);
rounding to FP64 adds 2^-53 of the sums.  2^-50 of the summed sizes holds all.
"""
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("pair64") / "pair64_probe")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fno-strict-aliasing", "-I", CUDA_INC, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1207_2367_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "pair64_probe.cpp"), "-o", exe], check=True)

    def run(eps, i, js):
        words = [float(eps).hex(), str(len(js))] + [float(x).hex() for x in i]
        for j in js:
            words += [float(x).hex() for x in j]
        out = subprocess.run([exe], input=" ".join(words), capture_output=True, text=True, check=True).stdout
        return np.array([float.fromhex(w) for w in out.split()])
    return run


def _exact(eps, i, js):
    """The nine sums, the summed sizes of A, J, S terms, and the potential."""
    getcontext().prec = 60
    s, size, phi = [Decimal(0)] * 9, [Decimal(0)] * 3, Decimal(0)
    e2 = Decimal(float(eps) * float(eps))
    for j in js:
        m = Decimal(float(j[0]))
        r, v, a = ([Decimal(float(np.float64(j[1 + 3 * f + k]) - np.float64(i[3 * f + k]))) for k in range(3)]
                   for f in range(3))
        r2 = sum(x * x for x in r) + e2
        if r2 == 0:
            continue
        R = r2.sqrt()
        q = m / (r2 * R)
        al = sum(x * y for x, y in zip(r, v)) / r2
        be = (sum(x * x for x in v) + sum(x * y for x, y in zip(r, a))) / r2 + al * al
        w = [y - 3 * al * x for x, y in zip(r, v)]
        u = [z - 6 * al * y - 3 * be * x for x, y, z in zip(r, w, a)]
        for f, vec in enumerate((r, w, u)):
            for k in range(3):
                s[3 * f + k] += q * vec[k]
        nr, nv, na = (sum(x * x for x in vec).sqrt() for vec in (r, v, a))
        size[0] += abs(q) * nr
        size[1] += abs(q) * nv
        size[2] += abs(q) * (na + nv * nv * min(nr / R, Decimal(1)) / R)
        if nr > 0:
            phi += m / R
    return s, size, phi


def _systems():
    g = np.random.default_rng(11)
    def js(n, rs=1.0, vs=1.0, as_=1.0, ms=1.0):
        return np.concatenate([ms * g.random((n, 1)) / n, rs * g.normal(size=(n, 3)), vs * g.normal(size=(n, 3)),
                               as_ * g.normal(size=(n, 3))], axis=1)
    i0 = 0.3 * g.normal(size=9)
    yield "ordinary", 1e-4, i0, js(300)
    for n in (1, 7, 8, 9, 31, 32, 33, 65):      # carries and folds of the integer sums
        yield f"{n} pairs", 1e-4, i0, js(n)
    yield "softening above the distances", 3.0, i0, js(100)
    for k in range(-12, 13, 4):                  # separations from far below to far above eps
        near = js(40, rs=2.0 ** k * 1e-3, vs=2.0 ** (k // 2))
        near[:, 1:4] += i0[:3]
        yield f"separations 2^{k} eps", 1e-3, i0, near
    wide = js(200)
    wide[:, 0] = 2.0 ** g.uniform(-300, 0, 200)
    wide[:, 1:4] *= 2.0 ** g.uniform(-20, 20, (200, 1))
    wide[:, 4:7] *= 2.0 ** g.uniform(-20, 20, (200, 1))
    wide[:, 7:10] *= 2.0 ** g.uniform(-40, 40, (200, 1))
    yield "exponents of every kind", 1e-8, np.zeros(9), wide
    yield "one axis", 1e-3, np.zeros(9), [[1.0, 1, 0, 0, -1, 0, 0, 2, 0, 0], [0.5, -3, 0, 0, 2, 0, 0, 0, 0, 0]]
    yield "powers of two", 0.0, np.zeros(9), [[2.0 ** -4, 1, 1, 1, 1, -1, 1, -1, 1, 1], [1.0, 2, 0, 0, 0, 4, 0, 0, 0, 8]]
    yield "at rest", 1e-3, np.zeros(9), [[1.0, 1, 2, 3, 0, 0, 0, 0, 0, 0]]
    yield "large values", 0.0, np.zeros(9), js(20, rs=1e140, vs=1e70, as_=1e20, ms=1e200)
    self_pair = js(33)
    self_pair[5] = np.concatenate([[0.1], i0])
    self_pair[9, 0] = 0.0                        # a massless (padding) record
    yield "own record", 1e-3, i0, self_pair
    yield "own record, no softening", 0.0, i0, self_pair


@pytest.mark.parametrize("name,eps,i,js", [pytest.param(*c, id=c[0].replace(" ", "_")) for c in _systems()])
def test_sums_against_exact_arithmetic(probe, name, eps, i, js):
    got = probe(eps, i, js)
    s, size, phi = _exact(eps, i, js)
    for f in range(3):
        err = sum((Decimal(float(got[3 * f + k])) - s[3 * f + k]) ** 2 for k in range(3)).sqrt()
        assert err <= size[f] * Decimal(2) ** -50, (name, f, float(err / size[f]))
    assert abs(Decimal(float(got[9])) - phi) <= phi * Decimal(2) ** -50


def test_nothing_to_add_is_exactly_zero(probe):
    i = np.arange(1.0, 10.0)
    own = np.concatenate([[1.0], i])
    pad = np.array([0.0, 1e18, 1e18, 1e18, 0, 0, 0, 0, 0, 0])
    for eps in (0.0, 1e-3):
        assert np.all(probe(eps, i, [own] + [pad] * 255) == 0.0)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("field", range(10))
def test_infinities_and_nan_show(probe, bad, field):
    j = np.array([[1.0, 1, 2, 3, .1, .2, .3, .4, .5, .6], [0.5, -1, 2, 1, .1, 0, .3, .4, 0, .6]])
    j[1, field] = bad
    assert np.all(np.isnan(probe(1e-3, np.zeros(9), j)[:9]))


def test_coincident_particles_without_softening(probe):
    """The forces leave the pair out (as the mixed path does); 1 / r in the potential is infinite."""
    j = [[1.0, 1, 2, 3, 1, 0, 0, 0, 0, 0], [1.0, 0, 0, 0, 1, 0, 0, 0, 0, 0]]
    ref = probe(0.0, np.zeros(9), j[:1])
    assert np.array_equal(probe(0.0, np.zeros(9), j)[:9], ref[:9])
