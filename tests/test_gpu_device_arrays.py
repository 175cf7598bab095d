"""Explicit calls with the caller's device arrays: the list of hg_next_block and the
results of hg_evaluate are written by the kernels; host arrays get copies.  Same values
either way, at the edges of the one-CTA selection (8192 particles, rows of 1024)."""
import numpy as np
import pytest

from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _context(hg, n, precision, dt):
    p = inputs.plummer(n, 3)
    g = np.random.default_rng(n)
    st = {"mass": p.mass, "pos": p.pos, "vel": p.vel, "acc": g.normal(size=(n, 3)), "jerk": g.normal(size=(n, 3)),
          "snap": g.normal(size=(n, 3)), "crackle": np.zeros((n, 3)), "t": np.zeros(n), "dt": dt}
    ctx = hg.hg_init(p.mass, p.pos, p.vel, 1e-3, 0.45, hg.hg_default_opts(precision=precision, start_mode=1,
                                                                        dt_max=2.0 ** -4))
    hg.hg_set_state(ctx, st, 0.0)
    return ctx


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1023, 1024, 1025, 2500, 8191, 8192, 8193, 20000])
def test_next_block_lists(hg, n):
    import torch
    g = np.random.default_rng(7 + n)
    for share in (0.0, 0.02, 0.5, 1.0):          # besides one particle that is always due
        due = g.random(n) < share
        due[g.integers(n)] = True
        ctx = _context(hg, n, 0, np.where(due, 2.0 ** -9, 2.0 ** -6))
        try:
            want = np.flatnonzero(due)
            dev = torch.full((n + 3,), -7, dtype=torch.int32, device="cuda")
            t, m = hg.hg_next_block(ctx, dev)
            assert t == 2.0 ** -9 and m == want.size
            np.testing.assert_array_equal(dev[:m].cpu().numpy(), want)
            assert bool((dev[m:] == -7).all())
            host = np.full(n, -7, dtype=np.int32)
            assert hg.hg_next_block(ctx, host) == (t, m)
            np.testing.assert_array_equal(host[:m], want)
            short = torch.full((m,), -7, dtype=torch.int32, device="cuda")   # smaller than n: a copy
            assert hg.hg_next_block(ctx, short) == (t, m)
            np.testing.assert_array_equal(short.cpu().numpy(), want)
            assert hg.hg_next_block(ctx) == (t, m)
        finally:
            hg.hg_free(ctx)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,m", [(700, 1), (700, 700), (5000, 37), (20000, 20000)])
def test_results_in_device_arrays(hg, precision, n, m):
    import torch
    ctx = _context(hg, n, precision, np.full(n, 2.0 ** -6))
    try:
        idx = np.sort(np.random.default_rng(5).permutation(n)[:m]).astype(np.int32)
        hg.hg_predict(ctx, 2.0 ** -8)
        host = [np.empty((m, 3)) for _ in range(3)]
        hg.hg_evaluate(ctx, idx, m, *host)
        dev = [torch.full((m + 1, 3), -1.0, dtype=torch.float64, device="cuda") for _ in range(3)]
        hg.hg_evaluate(ctx, torch.tensor(idx, device="cuda"), m, *dev)
        for h, d in zip(host, dev):
            np.testing.assert_array_equal(d[:m].cpu().numpy(), h)
            assert bool((d[m:] == -1.0).all())
        one = torch.full((m, 3), -1.0, dtype=torch.float64, device="cuda")   # some wanted, some not
        hg.hg_evaluate(ctx, idx, m, None, one, None)
        np.testing.assert_array_equal(one.cpu().numpy(), host[1])
        hg.hg_evaluate(ctx, idx, m, one, one, one)                           # overlapping: the last one stays
        np.testing.assert_array_equal(one.cpu().numpy(), host[2])
        mix = np.empty((m, 3))
        hg.hg_evaluate(ctx, idx, m, one, mix, None)
        np.testing.assert_array_equal(one.cpu().numpy(), host[0])
        np.testing.assert_array_equal(mix, host[1])
    finally:
        hg.hg_free(ctx)
