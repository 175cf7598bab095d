"""FP64 energy at the edges of its tiles: every pair is taken once, by one of the
two tiles of 128 particles that hold it (own tile, tiles ahead of it modulo the
number of tiles, the opposite one by half of the tiles only).

Bound: the potential is a sum of N (N - 1) / 2 positive terms, each good to a few
2^-53, added in FP64 sums; 1e-13 relative holds the accumulated rounding at these N.
"""
import numpy as np
import pytest

from gpu_util import oracle_system, gpu_context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 127, 128, 129, 255, 256, 257, 384, 385, 511, 513, 640, 2048, 2177])
def test_every_pair_once(hg, n):
    sysm = oracle_system(n, 5, 1e-3, imf="salpeter")
    K, W = sysm.energy()
    ctx = gpu_context(hg, sysm, 0, 1e-3)
    try:
        k, w = hg.hg_energy(ctx)
    finally:
        hg.hg_free(ctx)
    assert k == pytest.approx(K, rel=1e-13) and w == pytest.approx(W, rel=1e-13)


def test_one_particle_has_no_potential(hg):
    ctx = hg.hg_init(np.array([1.0]), np.array([[1.0, 2.0, 3.0]]), np.array([[0.0, 1.0, 0.0]]), 0.0, 0.45,
                     hg.hg_default_opts(start_mode=1))
    try:
        assert hg.hg_energy(ctx) == (0.5, 0.0)
    finally:
        hg.hg_free(ctx)


def test_coincident_particles(hg):
    """Without softening 1 / r of two particles in one place is infinite; with it, 1 / eps."""
    x = np.zeros((300, 3))
    x[:, 0] = np.arange(300.0)
    x[290] = x[3]
    m = np.full(300, 1.0 / 300)
    for eps, check in ((0.0, np.isneginf), (1e-3, np.isfinite)):
        ctx = hg.hg_init(m, x, np.zeros((300, 3)), eps, 0.45, hg.hg_default_opts(start_mode=1))
        try:
            assert check(hg.hg_energy(ctx)[1])
        finally:
            hg.hg_free(ctx)
