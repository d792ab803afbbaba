"""The re-sort takes only the species of which a particle left its tile's
margin.  Two species of equal particles, one fast (it leaves its tiles in the
first steps and often), one slower (later), against the same particles in one
species, where every re-sort takes them all: the fields are sums of integers,
so they must have the same bits, and so must every particle.  A species left
unsorted when it needed it would give a domain error or another current.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N = {1: (256,), 2: (64, 48), 3: (32, 16, 24)}


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("fast_first", [0, 1])
def test_species_sorted_apart_leave_the_same_bits(D, fast_first):
    from paper_2208_08038_gb300 import binding as B
    n, dx, steps = N[D], synth.LAMBDA0 / 16, 40
    rng = np.random.default_rng(D)
    per = 1500
    xs = [rng.random((per, D)) * np.array(n) * dx for _ in range(2)]
    us = [s * rng.standard_normal((per, 3)) for s in (3.0, 0.4)]
    if not fast_first:
        xs, us = xs[::-1], us[::-1]
    out = []
    for apart in (True, False):
        ctx = B.Context(D, n, (dx,) * D, 0.95 * dx / np.sqrt(D), (0,) * D)
        if apart:
            sids = [ctx.add_free(-1.0, 1.0, 1e-3) for _ in range(2)]
            for sid, x, u in zip(sids, xs, us):
                ctx.load_particles(sid, x, u)
        else:
            sid = ctx.add_free(-1.0, 1.0, 1e-3)
            ctx.load_particles(sid, np.vstack(xs), np.vstack(us))
        for k in range(steps):
            ctx.step(1 if k % 2 else 3)
        ctx.sync()
        parts = ([np.concatenate([ctx.read_particles_by_id(s, np.arange(per))[q] for s in sids]) for q in (0, 2)] if apart
                 else [ctx.read_particles_by_id(sid, np.arange(2 * per))[q] for q in (0, 2)])
        out.append([ctx.read_field(c).copy() for c in range(9)] + parts)
        ctx.close()
    assert np.abs(out[0][0]).max() > 0
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
