"""Two-body ions whose bound electron is a cell or more from its nucleus, moved
by a warp each when few (up to 2,432 in a step) and by a thread each when many,
against the FP64 oracle: a uniform strong field tears every ion of a periodic
box in a few steps.

Tolerances: E, B and J relative L2 1e-4 and the bound electrons' momenta 1e-5,
the bounds of the other parity tests of a few steps (FP32 rounding of some 1e-7
a step; the electrons move at nearly the speed of light, so J has no small
differences of stored offsets).
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth
from _common import field_rel_l2, gpu_from_workload, oracle_from_workload, rel_l2

pytestmark = pytest.mark.gpu

N = {1: (64,), 2: (32, 48), 3: (16, 24, 16)}
STEPS = {1: 4, 2: 6, 3: 8}  # moves of 0.95 / sqrt(D) cells: two to four cells apart at the end


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("ions", [700, 2432, 2433, 6000])
def test_torn_ions_match_the_oracle(D, ions):
    n, dx = N[D], synth.LAMBDA0 / 16
    rng = np.random.default_rng(ions + D)
    x = rng.random((ions, D)) * np.array(n) * dx
    sp = synth.TwoBody(Zb=1.0, qc=0.0, mc=synth.M_AU, w=1e-4, lambda0_m=12.4e-9, omega_b=np.array([3.0]), x=x,
                       u=np.zeros((ions, 3)))
    wl = synth.Workload("torn", D, n, (dx,) * D, 0.95 * dx / np.sqrt(D), (0,) * D, STEPS[D], [sp], [], tile=None)
    ora, osid, _ = oracle_from_workload(wl)
    gpu, gsid, _ = gpu_from_workload(wl, tile=(0,) * D)
    ora.field(0)[...] = 20.0
    gpu.write_field(0, np.full(n[::-1], 20.0))
    ora.step(STEPS[D])
    gpu.step(STEPS[D])
    gpu.sync()
    x1, x2, _, u2 = ora.bodies(osid[0])
    assert np.linalg.norm(x1 - x2, axis=1).min() > 1.5 * dx  # every ion was far in the last steps
    assert field_rel_l2(gpu.fields(), ora.fields()) < 1e-4
    assert field_rel_l2(gpu.fields(), ora.fields(), comps=range(6, 9)) < 1e-4
    g = gpu.read_particles_by_id(gsid[0], np.arange(ions))
    assert rel_l2(g[3], u2) < 1e-5
    gpu.close()
    ora.close()
