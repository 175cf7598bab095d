"""Graph steps alternate between two entries of the selection's scalars: any mix of
single steps, replays of graph_steps (odd or even), advances that stop, explicit block
calls and state changes gives the states of one replay after another."""
import numpy as np
import pytest

from gpu_util import DT_MAX, gpu_state
from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,clusters", [(0, 0), (1, 0), (1, 3)])
@pytest.mark.parametrize("graph_steps", [1, 3, 8])
def test_mixed_step_counts(hg, precision, clusters, graph_steps):
    n, eps = 1200, 1e-3
    p = inputs.plummer(n, 17)

    def context(k):
        o = hg.hg_default_opts(precision=precision, dt_max=DT_MAX, graph_steps=k)
        if clusters:
            return hg.hg_init_batch(np.linspace(0, n, clusters + 1).astype(np.int64), p.mass, p.pos, p.vel, eps, 0.45, o)
        return hg.hg_init(p.mass, p.pos, p.vel, eps, 0.45, o)

    def same(a, b):
        (sa, ta), (sb, tb) = gpu_state(hg, a, n), gpu_state(hg, b, n)
        assert ta == tb
        for f in hg.STATE_FIELDS:
            np.testing.assert_array_equal(sa[f], sb[f], err_msg=f)
        return sa, ta

    a, b = context(8), context(graph_steps)
    try:
        done = 0
        for k in (1, 2, 3, 5, 8, 1, 11):
            hg.hg_step(b, k)
            done += k
            hg.hg_step(a, k)
            s, t = same(a, b)
        t_end = t + 2.0 ** -9                       # stops between block times, the rest of a replay empty
        na, nb = hg.hg_advance(a, t_end), hg.hg_advance(b, t_end)
        assert na == nb
        done += na
        s, t = same(a, b)
        assert hg.hg_get_stats(b)["block_steps"] == done
        assert hg.hg_advance(b, t_end) == 0         # nothing due: the state stays
        same(a, b)
        hg.hg_step(b, 1)                            # now at the other entry
        t1, m = hg.hg_next_block(b)                 # explicit selection between graph steps
        assert m >= 1 and t1 > t
        hg.hg_step(b, 2)
        hg.hg_step(a, 3)
        s, t = same(a, b)
        hg.hg_step(b, 1)
        hg.hg_set_state(b, s, t)                    # back: the minimum is formed anew
        hg.hg_step(b, 4)
        hg.hg_step(a, 4)
        same(a, b)
    finally:
        hg.hg_free(a)
        hg.hg_free(b)
