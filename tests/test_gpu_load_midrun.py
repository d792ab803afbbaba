"""A species loaded in the middle of a run, while particles of another one have
left their tiles' margins and wait for the next step's sort: the load's own sort
must not make that one be forgotten.  The loaded particles' weight is below
the fixed-point unit of the current, so fields and the first species must have
the bits of a run without the load; so, too, with a refused load (a position
that is not finite) before the good one, which clears its error.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N = {1: (128,), 2: (48, 32), 3: (16, 16, 16)}
STEPS = 30
FIRST = {1: 8, 2: 2, 3: 1}  # the first step after which a particle can be out of its tile's margin


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("how", ["load", "medium", "lattice", "refused"])
def test_load_keeps_other_species_need_of_a_sort(D, how):
    from paper_2208_08038_gb300 import binding as B
    n, dx = N[D], synth.LAMBDA0 / 16
    rng = np.random.default_rng(D)
    x = rng.random((1200, D)) * np.array(n) * dx
    u = 2.0 * rng.standard_normal((1200, 3))
    centre = np.full((1, D), 8.5 * dx)
    out = []
    for load in (False, True):
        ctx = B.Context(D, n, (dx,) * D, 0.95 * dx / np.sqrt(D), (0,) * D)
        sid = ctx.add_free(-1.0, 1.0, 1e-3)
        more = [ctx.add_free(-1.0, 1.0, 1e-22) for _ in range(7)]  # (a context holds eight species)
        ctx.load_particles(sid, x, u)
        for k in range(STEPS):
            ctx.step(1)
            q = k - FIRST[D]
            if not load or q < 0 or q >= 7:
                continue
            if how == "refused":
                with pytest.raises(B.BPError) as e:
                    ctx.load_particles(more[q], np.full((3, D), np.nan))
                assert e.value.code == B.BP_ERR_NONFINITE
            if how == "medium":
                ctx.set_medium(more[q], (8,) * D, (9,) * D, 1, 3)
            elif how == "lattice":
                ctx.set_lattice(more[q], centre, 1, 0.0, 3)
            else:
                ctx.load_particles(more[q], centre)
        ctx.sync()
        got = ctx.read_particles_by_id(sid, np.arange(len(x)))
        out.append([ctx.read_field(c).copy() for c in range(9)] + [got[0], got[2], got[4]])
        ctx.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
