"""Dense streams of fast particles, sorted deposit: thousands of electrons per
cell that move the same way add to the same nodes, beyond what the two 32-bit
words of a node of the tile's box can hold (2^31 high-word units are some 2,100
of the largest contributions; low words, 2^16 adds of the largest).  The box
must be emptied before that, whichever path the particles take (crossing a
node or not), in one species or over several.

Tolerance: relative L2 against the FP64 oracle after one step, over E, B and
J, 1e-5 as in the other one-step tests: the particles move about a cell, so
the stored offset's quantum (2^-25 of a cell) and a handful of FP32 roundings
per contribution (6e-8 each) stay below 1e-6 of J, coherent sums included.
"""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth
from _common import field_rel_l2, gpu_from_workload, oracle_from_workload

pytestmark = pytest.mark.gpu

N = {1: (64,), 2: (32, 32), 3: (16, 16, 16)}
CELLS = {1: (14,), 2: (3, 3), 3: (2, 2, 2)}


def check(D, species, step):
    dx = synth.LAMBDA0 / 16
    wl = synth.Workload("stream", D, N[D], (dx,) * D, step * dx / np.sqrt(D), (0,) * D, 1, species, [], tile=None)
    ora, _, _ = oracle_from_workload(wl)
    gpu, _, _ = gpu_from_workload(wl, tile=(0,) * D)
    ora.step(1)
    gpu.step(1)
    gpu.sync()
    err = field_rel_l2(gpu.fields(), ora.fields(), comps=range(9))
    gpu.close()
    ora.close()
    assert err < 1e-5, err


def stream(D, per_cell, w, u, seed, at=2):
    dx = synth.LAMBDA0 / 16
    rng = np.random.default_rng(seed)
    cells = np.stack([m.ravel() for m in np.meshgrid(*[at + np.arange(n) for n in CELLS[D]], indexing="ij")], 1)
    x = (np.repeat(cells, per_cell, 0) + rng.random((per_cell * len(cells), D))) * dx
    return synth.Free(q=-1.0, m=1.0, w=w, x=x, u=np.tile(np.asarray(u, dtype=np.float64), (len(x), 1)))


@pytest.mark.parametrize("w", [1.0, 0.95, 0.7])
@pytest.mark.parametrize("D,u", [(1, (10.0, 0.0, 0.0)), (1, (0.0, -10.0, 0.0)), (2, (7.0, 7.0, 0.0)), (2, (0.0, 0.0, 10.0)),
                                 (3, (6.0, 6.0, -6.0))])
def test_dense_stream_matches_the_oracle(D, u, w):
    check(D, [stream(D, 4500 if D < 3 else 9000, w, u, 3)], 0.95)


def test_small_steps():
    """Moves of a third of a cell: most particles keep their nearest node."""
    check(1, [stream(1, 9000, 0.95, (10.0, 3.0, 0.0), 5)], 0.33)


def test_several_species():
    """The words fill over the species of a tile, ions among them."""
    ion = stream(2, 2000, 1.0, (0.0, 0.0, 0.0), 7)
    ions = synth.TwoBody(Zb=2.0, qc=1.0, mc=synth.M_AU, w=0.5, lambda0_m=12.4e-9, omega_b=np.array([3.0]), x=ion.x,
                         u=np.tile([10.0 * synth.M_AU, 0.0, 0.0], (len(ion.x), 1)))
    check(2, [stream(2, 1900, 0.95, (10.0, 0.0, 0.0), 8), ions, stream(2, 1900, 0.95, (10.0, 0.0, 0.0), 9)], 0.95)


@pytest.mark.parametrize("w", [1.0, 0.63, 0.81])
def test_many_equal_particles(w):
    """Equal particles at one place: equal remainders in the low words."""
    dx = synth.LAMBDA0 / 16
    n = 200000
    sp = synth.Free(q=-1.0, m=1.0, w=w, x=np.full((n, 1), 5.31 * dx), u=np.tile([0.013, 0.021, 0.0], (n, 1)))
    check(1, [sp], 0.95)
