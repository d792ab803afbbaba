"""2D tiles with few ions, sorted deposit: on a grid with few ions per tile on
average such tiles are pushed straight from and to the global arrays, on a grid
with more of them through shared-memory boxes.  Both must leave the same bits.

The second grid's extra ions rest in a region that no field reaches, where an
ion at rest with coinciding bodies deposits nothing: fields, currents and the
common ions must be equal exactly.  Counts of 32 and 33, 64 and 65 per tile stand at the
edges of the rule; ions sit at tile corners, on cell edges and by the periodic
and the open faces (whose boxes leave the grid), at rest, moving and with
torn bodies (a strong field)."""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N, T = (480, 400), 16


def ions(dx, rng, per_tile, open_x):
    tiles = [(i, j) for i in range(0, 8) for j in (0, 1, 5, 6, 24)]
    x = np.array([[(T * i + p[0]) * dx, (T * j + p[1]) * dx] for i, j in tiles
                  for p in np.vstack([[[0.0, 0.0], [15.999, 15.999], [0.4999, 8.5]], T * rng.random((per_tile, 2))])[:per_tile]])
    if open_x:
        x[:, 0] = np.maximum(x[:, 0], 3 * dx)  # nothing leaves the grid
    return x, 1e-2 * rng.standard_normal((len(x), 3)) * (rng.random((len(x), 1)) < 0.5) * synth.M_AU / 100


def run(extra, per_tile, open_x, a0):
    from paper_2208_08038_gb300 import binding as B
    dx = synth.LAMBDA0 / 32
    rng = np.random.default_rng(7 + per_tile)
    x, u = ions(dx, rng, per_tile, open_x)
    more = np.stack(np.meshgrid(np.arange(320, 400), np.arange(0, 400)), -1).reshape(-1, 2)[:extra] * dx + 0.3 * dx
    fields = [a0 * rng.standard_normal((1, N[1], N[0])) for _ in range(6)]
    for f in fields:
        f[:, :, 200:] = 0.0
    ctx = B.Context(2, N, (dx, dx), 0.6 * dx, (open_x, 0))
    sid = ctx.add_two_body(2.0, 0.0, synth.M_AU, 1e-3, 12.4e-9, [3.0])
    ctx.load_particles(sid, np.vstack([x, more]), np.vstack([u, np.zeros((len(more), 3))]))
    for k, f in enumerate(fields):
        ctx.write_field(k, f)
    ctx.step(4)
    ctx.sync()
    out = [ctx.read_field(k).copy() for k in range(9)] + list(ctx.read_particles_by_id(sid, np.arange(len(x))))
    ctx.close()
    return out


@pytest.mark.parametrize("per_tile,open_x,a0", [(1, 0, 1e-2), (3, 1, 0.5), (32, 0, 1e-2), (33, 1, 1e-2), (64, 1, 1e-2), (65, 0, 1e-2), (7, 0, 3.0)])
def test_few_ions_leave_the_same_bits(per_tile, open_x, a0):
    few = run(0, per_tile, open_x, a0)
    many = run(32000, per_tile, open_x, a0)
    for a, b in zip(few, many):
        np.testing.assert_array_equal(a, b)
    assert np.abs(few[6]).max() > 0
