"""A sort whose grid barrier gives up: the error is reported and stays (steps,
graph steps and loads included) until bp_reset, after which the context
computes what a fresh one does.  The wait runs out because its poll limit is
set to zero: every block but the last to arrive gives up at the first barrier,
and that one at the second, where no other block arrives.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu


def workload():
    wl = synth.neutral_3d(seed=5, steps=24, n=(32, 16, 16), ppc=4, sigma_u=0.15, margin=2)
    wl.bc = (0, 0, 0)
    return wl


def fresh(wl):
    from paper_2208_08038_gb300 import binding as B
    ctx = B.Context(wl.D, wl.n, wl.dx, wl.dt, wl.bc)
    sp = wl.species[0]
    return ctx, ctx.add_two_body(sp.Zb, sp.qc, sp.mc, sp.w, sp.lambda0_m, sp.omega_b)


def run(ctx, sid, wl, steps):
    sp = wl.species[0]
    ctx.load_particles(sid, sp.x, sp.u)
    for c in range(3):
        ctx.write_field(c, np.random.default_rng(c).standard_normal(wl.n[::-1]) * 1e-2)
    ctx.step(steps)
    ctx.sync()
    return [ctx.read_field(c).copy() for c in range(9)] + list(ctx.read_particles_by_id(sid, np.arange(len(sp.x))))


@pytest.mark.parametrize("where", ["load", "medium", "step", "graph"])
def test_context_recovers_after_a_sort_that_gave_up(where):
    from paper_2208_08038_gb300 import binding as B
    wl = workload()
    ref, rid = fresh(wl)
    want = run(ref, rid, wl, 24)
    ref.close()

    ctx, sid = fresh(wl)
    sp = wl.species[0]

    def times_out(call):
        with pytest.raises(B.BPError) as e:
            call()
        assert e.value.code == B.BP_ERR_TIMEOUT

    if where in ("load", "medium"):
        ctx.set_sort_wait(0)
        if where == "load":
            ctx.load_particles(sid, sp.x, sp.u)
        else:
            ctx.set_medium(sid, (0, 0, 0), wl.n, 4, 1, 0.1)
    else:
        ctx.load_particles(sid, sp.x, sp.u)
        ctx.set_sort_wait(0)
        if where == "step":  # single steps until an ion has left its tile's margin
            for _ in range(24):
                ctx.step(1)
        else:
            ctx.step(24)
    times_out(ctx.sync)
    ctx.set_sort_wait(-1)
    # the error stays, and nothing runs on the half-sorted particles
    ctx.step(16)
    times_out(ctx.sync)
    other = ctx.add_free(-1.0, 1.0, 1e-3)
    times_out(lambda: ctx.load_particles(other, sp.x[:10], sp.u[:10]))
    times_out(ctx.sync)
    ctx.reset()
    ctx.sync()
    got = run(ctx, sid, wl, 24)
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
    ctx.close()
