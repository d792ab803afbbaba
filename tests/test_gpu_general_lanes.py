"""3D, sorted deposit: a particle whose nearest node changes in the step is
deposited by its whole warp.  What it adds must not depend on who shares the
warp with it: not on how many lanes have a particle, not on how many of the
others take the same path, not on the order of the load.  Equal bits, since
the current is a sum of integers.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N = (32, 16, 16)
DX = synth.LAMBDA0 / 16
DT = 0.95 * DX / np.sqrt(3.0)


def context():
    from paper_2208_08038_gb300 import binding as B
    return B.Context(3, N, (DX,) * 3, DT, (0, 0, 0))


def currents(ctx):
    ctx.sync()
    out = [ctx.read_field(c).copy() for c in (6, 7, 8)]
    ctx.close()
    return out


@pytest.mark.parametrize("count", [1, 2, 5, 31, 32, 33, 70])
@pytest.mark.parametrize("speed", [0.3, 3.0])
def test_current_does_not_depend_on_the_other_lanes(count, speed):
    """Free particles of one tile alone, and among particles at rest (which add
    zeros and fill the runs of 32)."""
    rng = np.random.default_rng(count)
    x = (8.0 + 8.0 * rng.random((count, 3))) * DX
    u = speed * rng.standard_normal((count, 3))
    rest = (8.0 + 8.0 * rng.random((517, 3))) * DX
    out = []
    for filler in (False, True):
        ctx = context()
        sid = ctx.add_free(-1.0, 1.0, 1e-3)
        if filler:
            order = rng.permutation(count + len(rest))
            ctx.load_particles(sid, np.vstack([x, rest])[order], np.vstack([u, np.zeros_like(rest)])[order])
        else:
            ctx.load_particles(sid, x, u)
        ctx.step(1)
        out.append(currents(ctx))
    assert all(np.abs(j).max() > 0 for j in out[0])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("sigma", [0.02, 0.5])
def test_current_does_not_depend_on_the_load_order(sigma):
    """Two-body ions and free particles, few or nearly all of them crossing, in
    fields that pull the ions' bodies apart."""
    rng = np.random.default_rng(8)
    cells = np.stack([m.ravel() for m in np.meshgrid(*[np.arange(n) for n in N], indexing="ij")], 1)
    x = (np.repeat(cells, 3, 0) + rng.random((3 * len(cells), 3))) * DX
    u = sigma * rng.standard_normal((len(x), 3))
    fields = [0.3 * rng.standard_normal(N[::-1]) for _ in range(6)]
    out = []
    for k in range(2):
        ctx = context()
        ion = ctx.add_two_body(2.0, 1.0, synth.M_AU, 1e-3, 12.4e-9, [3.0])
        free = ctx.add_free(-1.0, 1.0, 1e-3)
        order = np.arange(len(x) // 2) if k == 0 else rng.permutation(len(x) // 2)
        ctx.load_particles(ion, x[::2][order], synth.M_AU * u[::2][order])
        ctx.load_particles(free, x[1::2][order], u[1::2][order])
        for c in range(6):
            ctx.write_field(c, fields[c])
        ctx.step(3)
        out.append(currents(ctx))
    assert all(np.abs(j).max() > 0 for j in out[0])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
