"""Lees-Edwards boundary with vertices more than a box height beyond the planes
(a run that blows up) and with a lattice lower than the stencil: every layer of
a stencil is a node of the lattice."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2305_02752_gb300 import hemo
from tests.helpers import assert_close, small_cell_shear

pytestmark = pytest.mark.gpu


def _config(n, nz):
    cfg = small_cell_shear(n=n, steps=3, seed=5, center=[n / 2.0, n / 2.0, nz / 2.0])
    rng = np.random.default_rng(5)
    return dataclasses.replace(cfg, nz=nz, mask=None, periodic=(1, 1, 1), wall_velocity=np.zeros((2, 3)),
                               init_velocity=0.003 * rng.normal(size=(nz, n, n, 3)))


@pytest.mark.parametrize('precision', ['f32', 'f64'])
@pytest.mark.parametrize('z', [95.0, -70.0, 1.0e4, -3.0e7])
def test_far_vertices(precision, z):
    """A cell put there through its saved state; its stencils wrap around the box
    any number of times.  Its forces and velocities stay finite."""
    cfg = _config(16, 16)
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.set_lees_edwards(0.02)
    sim.step(2)
    state = sim.save_state()
    sim.close()
    real = 8 if precision == 'f64' else 4
    at = 112 + 22 * real * 16 ** 3  # header, populations, velocity; then the centroids
    ctr = state[at:at + 24].view(np.float64)
    assert np.abs(ctr - cfg.centers[0]).max() < 0.5
    ctr[2] = z
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.set_lees_edwards(0.02)
    sim.load_state(state)
    sim.step(3)
    out = sim.get_fields()
    sim.close()
    for k in ('u', 'X', 'Fv'):
        assert np.isfinite(out[k]).all(), k
    assert np.abs(out['u']).max() < 0.3


@pytest.mark.parametrize('precision', ['f32', 'f64'])
@pytest.mark.parametrize('nz', [2, 3])
def test_low_lattice(precision, nz):
    """A cell several times as tall as the box runs (its images overlap it)."""
    cfg = _config(16, nz)
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.set_lees_edwards(0.0)
    sim.step(2)
    out = sim.get_fields()
    sim.close()
    assert np.isfinite(out['u']).all() and np.isfinite(out['X']).all()
    # without a displacement the images are those of a plain periodic box
    ref = O.from_config(cfg)
    ref.step(2)
    exp = ref.get()
    tol = 1e-10 if precision == 'f64' else 1e-4
    assert_close(out['u'], exp['u'], tol, 'u')
