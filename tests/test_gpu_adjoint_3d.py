"""The discrete adjoint in 3D against the oracle's FP64 adjoint, on grids where
the transposed E update works in place (open faces on x alone, and none):
gradients with respect to omega_b at the tolerance of the 1D and 2D comparison
(test_gpu_adjoint.py).  (The gradients with respect to a group's position are
left out: in this homogeneous medium they cancel over the group's ions.)"""
import numpy as np
import pytest

import oracle as O
from paper_2208_08038_gb300 import synth
from paper_2208_08038_gb300.adjoint import SiteProblem
from _common import gpu_from_workload
from test_gpu_adjoint import GRAD_TOL
from test_oracle_adjoint import build_oracle, run_loss

pytestmark = pytest.mark.gpu

STEPS, GROUPS = 150, 6


def problem(open_x):
    wl = synth.neutral_3d(seed=4, steps=STEPS, n=(40, 8, 8), ppc=2, sigma_u=0.0, nb=0.05, margin=17)
    wl.bc = (open_x, 0, 0)
    L = wl.lasers[0]
    L.waist, L.fwhm, L.ia = 0.0, 1.5 * synth.T0, 4
    L.t0 = 1.5 * L.fwhm
    sp = wl.species[0]
    sp.pidx = (np.arange(len(sp.x)) * GROUPS // len(sp.x)).astype(np.int32)
    sp.omega_b = synth.uniform_params(3, GROUPS, 2.5, 3.5)
    wl.probe_comp = 1
    wl.probe_nodes = np.array([30 + 40 * (j + 8 * k) for j in range(0, 8, 3) for k in range(0, 8, 3)], dtype=np.int64)
    return wl


@pytest.mark.parametrize("open_x", [1, 0])
def test_gpu_adjoint_matches_oracle_in_3d(open_x):
    wl = problem(open_x)
    sp = wl.species[0]
    npts = len(wl.probe_nodes)
    _, target = run_loss(wl, STEPS, synth.uniform_params(33, GROUPS, 2.5, 3.5), np.zeros((STEPS, npts)))
    s, sid, pid = build_oracle(wl, sp.omega_b)
    a = O.Adjoint(s, sid)
    _, probe_o = a.forward(STEPS, pid, target)
    g_om, _ = a.backward(GROUPS, len(sp.x))
    a.close()
    s.close()
    ctx, sids, gpid = gpu_from_workload(wl, probe_cap=STEPS)
    prob = SiteProblem(ctx, sids[0], gpid, sp.pidx, sp.x, sp.pidx, STEPS, 16)
    probe = prob.run(sp.omega_b, np.zeros((GROUPS, 3)))
    assert np.abs(probe - probe_o).max() <= 1e-5 * np.abs(probe_o).max()
    go, _ = prob.gradients(2.0 * (probe_o - target), GROUPS)
    assert np.abs(go - g_om).max() <= GRAD_TOL * np.abs(g_om).max()
    ctx.close()
