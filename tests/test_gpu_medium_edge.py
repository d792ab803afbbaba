"""bp_set_medium where an in-cell offset rounds up to 1 in the grid's last cell.

Seed 1969 puts ion 64,094 of a 32-cell, 2048-per-cell medium at u = 1 - 2.8e-8
of cell 31: in FP32 the offset is 1, so the ion belongs to cell 0 of a periodic
axis and to the end of cell 31 of an open one; cell 32 is off the grid."""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

SEED, N, PPC, ION = 1969, 32, 2048, 64094


@pytest.mark.parametrize("open_x", [0, 1])
def test_offset_rounding_up_stays_on_the_grid(open_x):
    from paper_2208_08038_gb300 import binding as B
    dx = synth.LAMBDA0 / 64
    ctx = B.Context(1, (N,), (dx,), 0.95 * dx, (open_x,))
    sid = ctx.add_two_body(1.0, 0.0, synth.M_AU, 1e-3, 12.4e-9, [3.0])
    ctx.set_medium(sid, (0,), (N,), PPC, SEED)
    x1, _, _, _ = ctx.read_particles(sid, N * PPC)
    assert len(x1) == N * PPC
    want, _ = synth.medium(SEED, 1, (dx,), (0,), (N,), PPC)
    L = N * dx
    d = np.abs(x1[:, 0] - want[:, 0])
    # FP32 in-cell offsets: half an ulp below 1 is 2^-25 of a cell; the clamped ion one ulp
    assert np.minimum(d, L - d).max() <= 2.0 ** -24 * dx
    assert x1[:, 0].max() < L
    assert (x1[ION, 0] == 0.0) if not open_x else (x1[ION, 0] > L - 2.0 ** -23 * dx)
    ctx.step(3)
    ctx.sync()
    ctx.close()
