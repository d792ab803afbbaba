"""bp_set_lattice with odd numbers of ions and sites: the staging's arrays of
doubles must stay aligned (an odd number of ions put the site positions behind
an odd number of 4-byte indices).  Positions and momenta against the host
definition of the lattice, with and without parameter indices."""
import numpy as np
import pytest

from paper_2208_08038_gb300 import synth

pytestmark = pytest.mark.gpu

N = {1: (64,), 2: (32, 32), 3: (16, 16, 16)}


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("n_sites,per_site", [(1, 1), (3, 1), (7, 3), (5, 4), (4, 5)])
@pytest.mark.parametrize("params", [False, True])
def test_lattice_of_any_count(D, n_sites, per_site, params):
    from paper_2208_08038_gb300 import binding as B
    n, dx = N[D], synth.LAMBDA0 / 16
    rng = np.random.default_rng(n_sites)
    sites = (2.0 + rng.random((n_sites, D)) * (np.array(n) - 4.0)) * dx
    want, u = synth.lattice(9, sites, per_site, 0.05 * dx, 2e-3)
    ctx = B.Context(D, n, (dx,) * D, 0.95 * dx / np.sqrt(D), (0,) * D)
    omega = np.array([2.0, 3.0, 4.0])
    sid = ctx.add_two_body(1.0, 0.0, synth.M_AU, 1e-3, 12.4e-9, omega)
    sp = (np.arange(n_sites) % 3).astype(np.int32) if params else None
    ctx.set_lattice(sid, sites, per_site, 0.05 * dx, 9, 2e-3, sp)
    x1, _, u1, _, found = ctx.read_particles_by_id(sid, np.arange(n_sites * per_site))
    assert found.all()
    assert np.abs(x1[:, :D] - want).max() < 1e-6 * dx
    assert np.abs(u1 - u).max() <= 1e-6 * np.abs(u).max()
    ctx.step(2)
    ctx.sync()
    ctx.close()
