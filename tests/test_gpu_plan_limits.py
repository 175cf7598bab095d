"""Graph steps whose plan does not come from the table of all block sizes, or that no
candidate of the planner fits, against the explicit calls, bit by bit."""
import numpy as np
import pytest

from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _contexts(hg, n, due_levels, **opts):
    p = inputs.plummer(n, 6)
    g = np.random.default_rng(1)
    dt = np.full(n, 2.0 ** -6)
    for level, share in due_levels:
        dt[g.permutation(n)[:max(1, int(share * n))]] = 2.0 ** -level
    st = {"mass": p.mass, "pos": p.pos, "vel": p.vel, "acc": -p.pos, "jerk": -p.vel, "snap": p.pos.copy(),
          "crackle": np.zeros((n, 3)), "t": np.zeros(n), "dt": dt}
    out = []
    for _ in range(2):
        c = hg.hg_init(p.mass, p.pos, p.vel, 1e-3, 0.45, hg.hg_default_opts(precision=1, start_mode=1, dt_max=2.0 ** -4,
                                                                           graph_steps=2, **opts))
        hg.hg_set_state(c, st, 0.0)
        out.append(c)
    return out


def _compare(hg, a, b, n, steps):
    """steps graph steps of a, the explicit calls of b."""
    hg.hg_step(a, steps)
    for _ in range(steps):
        t, m = hg.hg_next_block(b)
        hg.hg_predict(b, t)
        hg.hg_evaluate(b, None, m)
        hg.hg_correct(b, None, m)
    sa, sb = hg.new_state(n), hg.new_state(n)
    assert hg.hg_get_state(a, sa) == hg.hg_get_state(b, sb) > 0.0
    for f in hg.STATE_FIELDS:
        np.testing.assert_array_equal(sa[f], sb[f], err_msg=f)
    assert bool((sa["t"] > 0.0).any())
    return m


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 1])   # the last with a table, the first without
def test_plan_kernel_instead_of_the_table(hg, n):
    a, b = _contexts(hg, n, [(9, 3e-5), (10, 3e-6)])
    try:
        _compare(hg, a, b, n, 5)                          # both graphs, both entries; m of a few and a few dozen
    finally:
        hg.hg_free(a)
        hg.hg_free(b)


def test_block_that_no_split_fits(hg):
    n = 270000                                            # 8 chunks of m rows exceed the 4 n of the buffer
    a, b = _contexts(hg, n, [], jsplit=8)
    try:
        assert _compare(hg, a, b, n, 1) == n
        c, d = _contexts(hg, n, [], tpi=1, jsplit=1)
        try:
            hg.hg_step(c, 1)
            sa, sc = hg.new_state(n), hg.new_state(n)
            hg.hg_get_state(a, sa)
            hg.hg_get_state(c, sc)
            for f in ("acc", "jerk", "snap"):             # one thread over all j-records either way
                np.testing.assert_array_equal(sa[f], sc[f], err_msg=f)
        finally:
            hg.hg_free(c)
            hg.hg_free(d)
    finally:
        hg.hg_free(a)
        hg.hg_free(b)
