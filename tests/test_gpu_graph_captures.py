"""Which graphs a call captures: both lengths (one step, graph_steps steps) at the first
call, the other entry's only when they are replayed.  Seen through fault injection: a
capture of 64 steps makes more than 150 checked CUDA calls, one of a single step and its
replay fewer than 40."""
import numpy as np
import pytest

from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clusters", [0, 3])
def test_single_steps_capture_no_long_graph(hg, clusters):
    n = 600
    p = inputs.plummer(n, 4)
    o = hg.hg_default_opts(precision=1, dt_max=2.0 ** -4, graph_steps=64)
    if clusters:
        ctx = hg.hg_init_batch(np.linspace(0, n, clusters + 1).astype(np.int64), p.mass, p.pos, p.vel, 1e-3, 0.45, o)
    else:
        ctx = hg.hg_init(p.mass, p.pos, p.vel, 1e-3, 0.45, o)
    try:
        hg.hg_step(ctx, 1)
        try:
            hg.hg_inject_fault(hg.HG_FAULT_CUDA, 100)
            for _ in range(2):                   # the other entry, then this one again
                hg.hg_step(ctx, 1)
        finally:
            hg.hg_inject_fault(hg.HG_FAULT_NONE)
        hg.hg_step(ctx, 130)                     # captures what it replays
        assert hg.hg_get_stats(ctx)["block_steps"] == 133
    finally:
        hg.hg_free(ctx)
