"""Every component of the FP64 path's sums on its own: thin discs, nearly aligned pairs,
small perturbations of a plane (no GPU; the probe of test_pair64_cpu.py).

Reference: 60-digit arithmetic on the FP64 differences.  Bound: the component's terms with
every product taken by its size, which is what FP64 instructions err in proportion to.
With u = 2^-53: the coefficients alpha, beta and q are rounded once (a little more than u
each, relative to the sizes of their terms), w = v - 3 alpha r adds a rounding, the two
steps of a - 6 alpha w - 3 beta r three more at most, q and the sum one each: 8 u of a
term, and u of the sums per addition, (8 + n) u for n pairs.
"""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from test_pair64_cpu import probe   # noqa: F401  (fixture)


def _sums_and_sizes(eps, i, js):
    getcontext().prec = 60
    s, size = [Decimal(0)] * 9, [Decimal(0)] * 9
    e2 = Decimal(float(eps) * float(eps))
    for j in js:
        m = Decimal(float(j[0]))
        r, v, a = ([Decimal(float(np.float64(j[1 + 3 * f + k]) - np.float64(i[3 * f + k]))) for k in range(3)]
                   for f in range(3))
        r2 = sum(x * x for x in r) + e2
        q = m / (r2 * r2.sqrt())
        for out, sign in ((s, lambda x: x), (size, abs)):
            rr, vv, aa = ([sign(x) for x in f] for f in (r, v, a))
            k3 = 3 if out is size else -3
            al = sum(x * y for x, y in zip(rr, vv)) / r2
            be = (sum(x * x for x in vv) + sum(x * y for x, y in zip(rr, aa))) / r2 + al * al
            w = [y + k3 * al * x for x, y in zip(rr, vv)]
            u = [z + 2 * k3 * al * y + k3 * be * x for x, y, z in zip(rr, w, aa)]
            for f, vec in enumerate((rr, w, u)):
                for k in range(3):
                    out[3 * f + k] += sign(q) * vec[k]
    return s, size


def _check(probe, eps, i, js):   # noqa: F811
    got = probe(eps, i, js)
    s, size = _sums_and_sizes(eps, i, js)
    for c in range(9):
        err = abs(Decimal(float(got[c])) - s[c])
        assert err <= (8 + len(js)) * size[c] * Decimal(2) ** -53, (c, float(got[c]), float(s[c]), float(err / size[c]))


@pytest.mark.parametrize("axis", range(3))
@pytest.mark.parametrize("flat", [2.0 ** -5, 1e-4, 1e-6, 1e-10, 1e-16, 1e-20, 1e-60])
def test_thin_disc(probe, flat, axis):   # noqa: F811
    g = np.random.default_rng(5)
    i, js = 0.3 * g.normal(size=9), g.normal(size=(60, 10))
    js[:, 0] = np.abs(js[:, 0]) / 60
    i[axis::3] *= flat
    js[:, 1 + axis::3] *= flat
    for eps in (1e-4, 0.0, 2.0):
        _check(probe, eps, i, js)
        _check(probe, eps, i, js[:1])


@pytest.mark.parametrize("t", [1e-6, 1e-10, 1e-18, 1e-19, 1e-40, 1e-150])
def test_nearly_aligned_pairs(probe, t):   # noqa: F811
    """Separation, velocity and acceleration along axes but for a small component each."""
    for eps in (0.0, 1e-3, 4.0):
        for r, v, a in (((1, t, 0), (-1, 0, 0), (2, 0, 0)), ((1, 0, 0), (t, 1, 0), (0, 0, 1)),
                        ((1, t, 0), (0, 1, 0), (0, 1, 0)), ((t, 1, t), (1, 0, t), (1, t * t, 0)),
                        ((0, 0, 1), (1, t, 0), (t, 0, 0)), ((3, 0, 0), (0, 0, 0), (t, 1, 0))):
            _check(probe, eps, np.zeros(9), [[0.7, *r, *v, *a]])
            _check(probe, eps, np.zeros(9), [[0.7, *r, *v, *a], [0.1, 5, 0, 0, 0, 3, 0, 0, 0, 2]])


def test_exponents_far_apart(probe):   # noqa: F811
    """Distant and close pairs in turn, separations around eps, sizes over many powers of two."""
    g = np.random.default_rng(3)
    for _ in range(150):
        eps = 2.0 ** g.integers(-12, 0)
        js = []
        for k in range(int(g.integers(1, 5))):
            d = 2.0 ** g.uniform(3, 9) if k % 2 == 0 else eps * 2.0 ** g.uniform(-16, 2)
            js.append([2.0 ** g.uniform(-20, 0), *(d * g.normal(size=3)), *(2.0 ** g.uniform(-8, 8, 3) * g.normal(size=3)),
                       *(2.0 ** g.uniform(-30, 8, 3) * g.normal(size=3))])
        _check(probe, eps, np.zeros(9), js)


def test_softened_pair_with_velocity_along_the_separation(probe):   # noqa: F811
    g = np.random.default_rng(8)
    for k in range(2, 17):
        for _ in range(6):
            d = g.normal(size=3)
            j = [1.0, *(2.0 ** -k * d), *(2.0 ** g.integers(-3, 3) * d), *(1e-9 * g.normal(size=3))]
            _check(probe, 1.0, np.zeros(9), [j])


def test_exponents_over_the_range(probe):   # noqa: F811
    """Components from 2^-400 to 2^200, zeros among them: a zero's product with a large number
    displaces nothing."""
    g = np.random.default_rng(21)
    for _ in range(200):
        j = np.zeros(10)
        for f, span in ((slice(0, 1), 100), (slice(1, 4), 100), (slice(4, 7), 100), (slice(7, 10), 200)):
            x = 2.0 ** g.uniform(-span, span) * g.normal(size=f.stop - f.start) * 2.0 ** g.uniform(-span, 0, f.stop - f.start)
            j[f] = np.where(g.random(x.size) < 0.2, 0.0, x)
        j[0] = abs(j[0])
        if not j[1:4].any():
            continue
        for eps in (0.0, 2.0 ** g.uniform(-40, 100)):
            _check(probe, eps, np.zeros(9), [j])


def test_denormal_differences_count(probe):   # noqa: F811
    """The integers hold normal numbers: a pair with a denormal one goes to FP64 instructions."""
    tiny = 2.0 ** -1060
    for j in ([1.0, tiny, 1, 0, 0, 0, 0, 2.0 ** 900, 0, 0], [1.0, 2, 0, 0, 0, tiny, 0, 0, 0, 0],
              [1.0, 2, 0, 0, 0, 0, 0, 0, 0, tiny], [2.0 ** -1070, 2.0 ** -200, 0, 0, 1, 0, 0, 0, 1, 0]):
        s, size = _sums_and_sizes(0.0, np.zeros(9), [j])
        got = probe(0.0, np.zeros(9), [j])
        for c in range(9):   # 16 2^-53: an FP64 step rounds each of some ten operations; denormal results to 2^-1074
            assert abs(Decimal(float(got[c])) - s[c]) <= size[c] * Decimal(2) ** -49 + Decimal(2) ** -1073, (j, c)


def test_softening_beyond_the_range_of_its_square(probe):   # noqa: F811
    """eps^2 = inf: no force, whatever the pair."""
    assert np.all(probe(1e200, np.zeros(9), [[1.0, 1, 2, 3, 4, 5, 6, 7, 8, 9]])[:9] == 0.0)
