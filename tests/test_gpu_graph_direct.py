"""Step graphs against direct launches: the same bits in fields, probe traces
and particles (sorted deposit).

A call of two or more steps replays graphs, and so does a single step from the
third such call in a row.  Two arms launch directly:
  timed   every step with the push timed: the number of timed push launches
          is the number of steps, so none went through a graph (this arm also
          takes the quiet-tile pass and its list on grids that otherwise go
          without);
  pairs   two single steps, then a call of no steps, which ends the row.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth
from _common import gpu_from_workload

pytestmark = pytest.mark.gpu


def hot_3d():
    """Fast thermal ions that cross tile margins: the re-sort runs."""
    wl = synth.neutral_3d(seed=2, steps=30, n=(48, 16, 16), ppc=4, sigma_u=0.15, margin=2)
    wl.bc = (0, 0, 0)
    wl.lasers[0].waist = 0.5 * synth.LAMBDA0
    wl.lasers[0].yc, wl.lasers[0].zc = 0.5 * 16 * wl.dx[1], 0.5 * 16 * wl.dx[2]
    wl.lasers[0].a0 = 0.05
    return wl


def few_2d():
    """1,024 tiles (per-tile field flags), few ions in most, open on both axes."""
    wl = synth.bragg_2d(n=512, sites=(10, 10), steps=60, waist_lambda=2.0, fwhm_lambda=2.0)
    wl.lasers[0].a0 = 0.05
    return wl


WORKLOADS = {"1d": lambda: synth.neutral_1d(steps=60), "2d": lambda: synth.refraction_2d(n=(64, 48), steps=40),
             "2d-flags-few-ions": few_2d, "3d-resorting": hot_3d}


def run(wl, arm, steps, cap):
    ctx, sids, pid = gpu_from_workload(wl, probe_cap=cap)
    if pid is None:  # a line of E_z nodes across the box
        pid = ctx.add_probe(2, np.array([20 + wl.n[0] * j for j in range(wl.n[1] if wl.D > 1 else 1)], dtype=np.int64), cap)
    if arm == "graph":
        ctx.step(steps)
    elif arm == "timed":
        ctx.time_push(True)
        ctx.step(steps // 2)
        for _ in range(steps - steps // 2):
            ctx.step(1)
    else:
        for k in range(steps):
            ctx.step(1)
            if k % 2:
                ctx.step(0)
    ctx.sync()
    if arm == "timed":
        assert ctx.push_time()[1] == steps
    out = [ctx.fields(), ctx.read_probe(pid)]
    for sid, sp in zip(sids, wl.species):
        out += list(ctx.read_particles_by_id(sid, np.arange(len(sp.x))))
    ctx.close()
    return out


@pytest.mark.parametrize("name", list(WORKLOADS))
@pytest.mark.parametrize("arm", ["timed", "pairs"])
def test_graph_steps_leave_the_bits_of_direct_steps(name, arm):
    wl = WORKLOADS[name]()
    steps = wl.steps
    cap = steps - 15 if name == "2d" else steps  # a probe that fills up
    got, want = run(wl, "graph", steps, cap), run(wl, arm, steps, cap)
    assert want[1].shape[0] == min(steps, cap)
    assert np.abs(want[0][:6]).max() > 0
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
