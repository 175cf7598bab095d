"""The plans of the graph steps' table, which one kernel forms for all block sizes, are the
planner's: graph steps of every block size from 1 to some dozens equal the explicit calls
bit by bit, with tuned entries and without."""
import numpy as np
import pytest

from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("n", [1, 5, 31, 300, 1027])
def test_table_plans_equal_the_planners(hg, n, tuned):
    p = inputs.plummer(max(n, 2), 8)
    mass, pos, vel = p.mass[:n], p.pos[:n], p.vel[:n]
    st = {"mass": mass, "pos": pos, "vel": vel, "acc": -pos, "jerk": -vel, "snap": pos.copy(), "crackle": np.zeros((n, 3)),
          "t": np.zeros(n)}
    ctx = []
    try:
        for _ in range(2):
            c = hg.hg_init(mass, pos, vel, 1e-2, 0.45, hg.hg_default_opts(precision=1, start_mode=1, dt_max=2.0 ** -4))
            ctx.append(c)
            if tuned:                       # 64 and 16 threads a particle, 2 tiles a chunk; an inadmissible one
                table = hg.hg_get_tuning(c)
                table[0], table[1], table[3] = 6 * 32 + 1, 4 * 32 + 1, 31
                hg.hg_set_tuning(c, table)
        for m in sorted({1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 33, n // 2, n - 1, n}):
            if not 1 <= m <= n:
                continue
            st["dt"] = np.where(np.arange(n) < m, 2.0 ** -10, 2.0 ** -6)
            for c in ctx:
                hg.hg_set_state(c, st, 0.0)
            hg.hg_step(ctx[0], 1)
            t, got = hg.hg_next_block(ctx[1])
            assert got == m
            hg.hg_predict(ctx[1], t)
            hg.hg_evaluate(ctx[1], None, m)
            hg.hg_correct(ctx[1], None, m)
            a, b = hg.new_state(n), hg.new_state(n)
            hg.hg_get_state(ctx[0], a)
            hg.hg_get_state(ctx[1], b)
            for f in hg.STATE_FIELDS:
                np.testing.assert_array_equal(a[f], b[f], err_msg=f"{f} m={m}")
    finally:
        for c in ctx:
            hg.hg_free(c)
