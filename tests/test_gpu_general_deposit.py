"""Deposits whose nearest node changes in the step (four-node windows), in 1D,
2D and 3D: from a few such particles in a warp (3D: the warp shares out their
rows) to nearly every one (every lane its own), one body and two, against the
FP64 oracle after one step.

Tolerance: the one-step bound of the parity tests, 1e-5 relative L2 over E and
B (from zero fields, E is the step's current times dt).
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth
from _common import field_rel_l2, gpu_from_workload, oracle_from_workload

pytestmark = pytest.mark.gpu

N = {1: (64,), 2: (32, 48), 3: (16, 24, 16)}


def workload(D, speed, open_x, seed):
    n = N[D]
    dx = synth.LAMBDA0 / 16
    rng = np.random.default_rng(seed)
    lo = 4 if open_x else 0
    cells = np.stack([m.ravel() for m in np.meshgrid(*[np.arange(lo if a == 0 else 0, n[a] - (lo if a == 0 else 0))
                                                        for a in range(D)], indexing="ij")], 1)
    x = (np.repeat(cells, 3, 0) + rng.random((3 * len(cells), D))) * dx
    u = speed * rng.standard_normal((len(x), 3))
    sp = [synth.TwoBody(Zb=2.0, qc=1.0, mc=synth.M_AU, w=1e-3, lambda0_m=12.4e-9, omega_b=np.array([3.0]),
                        x=x[::2], u=1e-4 * u[::2] * synth.M_AU / 100),
          synth.Free(q=-1.0, m=1.0, w=1e-3, x=x[1::2], u=u[1::2])]
    dt = 0.95 * dx / np.sqrt(D)
    return synth.Workload("general", D, n, (dx,) * D, dt, (open_x,) + (0,) * (D - 1), 1, sp, [], tile=None)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("speed", [5e-3, 5e-2, 2.0])
def test_crossing_particles_match_the_oracle(D, speed, mode):
    wl = workload(D, speed, D % 2, seed=11 * D)
    ora, _, _ = oracle_from_workload(wl)
    gpu, sids, _ = gpu_from_workload(wl, deposit_mode=mode, tile=(0,) * D)
    ora.step(1)
    gpu.step(1)
    gpu.sync()
    assert field_rel_l2(gpu.fields(), ora.fields()) < 1e-5
    gpu.close()
