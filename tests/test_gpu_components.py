"""FP64 evaluations component by component: thin discs keep their small components, and an
infinite velocity spoils the jerk and the snap, not the acceleration.

Bound: the component's terms by their sizes (test_pair64_components_cpu.py).  numpy's FP64
sums err by up to 16 2^-53 of these (a dozen rounded operations a term) and 2^-53 per
addition, the kernel's by no more: (32 + 2 n) 2^-53.
"""
import numpy as np
import pytest

from paper_1207_2367_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sums_and_sizes(mass, x, v, a, eps, idx):
    out = []
    for sign in (lambda f: f, np.abs):
        r, w, d = (sign(f[None] - f[idx][:, None]) for f in (x, v, a))
        s3 = -3.0 if not out else 3.0
        r2 = ((x[None] - x[idx][:, None]) ** 2).sum(2) + eps * eps
        q = mass / (r2 * np.sqrt(r2))
        al = ((r * w).sum(2) / r2)[:, :, None]
        be = (((w * w).sum(2) + (r * d).sum(2)) / r2)[:, :, None] + al * al
        j = w + s3 * al * r
        s = d + 2 * s3 * al * j + s3 * be * r
        out.append([(q[:, :, None] * f).sum(1) for f in (r, j, s)])
    return out


@pytest.mark.parametrize("m", [1, 2, 9, 33, 200, 700])
@pytest.mark.parametrize("flat", [1e-3, 1e-8, 1e-16])
def test_thin_disc(hg, m, flat):
    n, eps = 700, 1e-3
    p = inputs.plummer(n, 9)
    g = np.random.default_rng(4)
    st = {"mass": p.mass, "pos": p.pos.copy(), "vel": p.vel.copy(), "acc": g.normal(size=(n, 3)),
          "jerk": np.zeros((n, 3)), "snap": np.zeros((n, 3)), "crackle": np.zeros((n, 3)), "t": np.zeros(n),
          "dt": np.full(n, 2.0 ** -6)}
    for f in ("pos", "vel", "acc"):
        st[f][:, 2] *= flat
    ctx = hg.hg_init(p.mass, st["pos"], st["vel"], eps, 0.45, hg.hg_default_opts(precision=0, start_mode=1, dt_max=2.0 ** -4))
    try:
        hg.hg_set_state(ctx, st, 0.0)
        hg.hg_predict(ctx, 0.0)
        idx = np.sort(g.permutation(n)[:m]).astype(np.int32)
        got = [np.empty((m, 3)) for _ in range(3)]
        hg.hg_evaluate(ctx, idx, m, *got)
    finally:
        hg.hg_free(ctx)
    want, size = _sums_and_sizes(p.mass, st["pos"], st["vel"], st["acc"], eps, idx)
    for a, b, s in zip(got, want, size):
        assert np.all(np.abs(a - b) <= (32 + 2 * n) * 2.0 ** -53 * s)


def test_infinite_velocity_leaves_the_acceleration(hg):
    import torch
    n = 300
    p = inputs.plummer(n, 2)
    mass, pos, vel = (torch.tensor(f, device="cuda") for f in (p.mass, p.pos, p.vel))
    zero = torch.zeros_like(pos)
    idx = torch.arange(n - 1, dtype=torch.int32, device="cuda")
    got = []
    for bad in (0.5, float("inf")):
        vel[n - 1, 0] = bad
        out = [torch.empty(n - 1, 3, dtype=torch.float64, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        hg.hg_evaluate_static(mass, pos, vel, zero, 1e-3, hg.HG_FP64, idx, n - 1, *out,
                              stream=torch.cuda.current_stream())
        torch.cuda.synchronize()
        got.append([f.cpu().numpy() for f in out])
    # q alone enters the acceleration: rounded once in integers, in some five FP64 steps otherwise
    r2 = ((p.pos[None] - p.pos[:-1][:, None]) ** 2).sum(2) + 1e-6
    size = (p.mass / r2 ** 1.5 * np.sqrt(r2)).sum(1)[:, None]
    assert np.all(np.abs(got[1][0] - got[0][0]) <= (16 + n) * 2.0 ** -53 * size)
    assert np.all(~np.isfinite(got[1][1]).all(axis=1)) and np.all(~np.isfinite(got[1][2]).all(axis=1))
