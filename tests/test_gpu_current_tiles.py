"""Grids with tile flags: the field kernels form J only where a step's deposits
can reach.  Elsewhere J must read zero, also where ions have left a tile with a
field behind and where the caller wrote J; E and B must not depend on what the
caller wrote into J."""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N, T = (512, 512), 16


def run(write_j, steps):
    from paper_2208_08038_gb300 import binding as B
    dx = synth.LAMBDA0 / 32
    rng = np.random.default_rng(3)
    x = (40.0 + 8.0 * rng.random((300, 2))) * dx
    u = np.tile([5.0, 0.0, 0.0], (300, 1))
    ctx = B.Context(2, N, (dx, dx), 0.6 * dx, (0, 0))
    sid = ctx.add_two_body(2.0, 0.0, synth.M_AU, 1e-3, 12.4e-9, [3.0])
    ctx.load_particles(sid, x, u)
    for k in range(6):
        f = 1e-2 * rng.standard_normal((1, N[1], N[0]))
        f[:, :, 300:] = 0.0
        ctx.write_field(k, f)
    ctx.step(2)
    if write_j:
        for k in (6, 7, 8):
            ctx.write_field(k, np.ones((1, N[1], N[0])))
    ctx.step(steps)
    ctx.sync()
    out = [ctx.read_field(k).reshape(N[1], N[0]).copy() for k in range(9)]
    pos = ctx.read_particles_by_id(sid, np.arange(300))[0][:, :2] / dx
    ctx.close()
    return out, pos


@pytest.mark.parametrize("steps", [1, 2, 90])
def test_current_only_where_ions_are(steps):
    a, pos = run(False, steps)
    b, _ = run(True, steps)
    for f, h in zip(a[:6], b[:6]):
        np.testing.assert_array_equal(f, h)
    near = np.zeros(N[::-1], bool)
    for i, j in np.unique((pos // T).astype(int), axis=0):
        near[(j - 2) * T:(j + 3) * T, (i - 2) * T:(i + 3) * T] = True
    assert near.any() and not near.all()
    fields = np.arange(N[0]) < 290  # columns whose tiles hold a field
    for f, h in zip(a[6:], b[6:]):
        assert np.abs(f[near]).max() > 0
        assert not f[~near].any()
        np.testing.assert_array_equal(f[:, fields], h[:, fields])
