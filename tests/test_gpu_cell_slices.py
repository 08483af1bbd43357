"""Membrane kernel with a cluster of CTAs per cell (few cells): every cluster
size, meshes smaller than the slices and mixed mesh types, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2305_02752_gb300 import inputs as I
from tests.helpers import assert_close, forces_close

pytestmark = pytest.mark.gpu


def _config(ncell, sub, platelets, seed=11):
    cfg = I.channel(nx=48, ny=43, nz=48, ncell=ncell, seed=seed, platelet_ratio=0.0, pack_iter=20, exact_iter=0)
    v, t = I.locality_order(*I.icosphere(sub))
    cfg.meshes[0].rest, cfg.meshes[0].tri = I.evans_fung(v, 7.0), t
    if platelets:
        cfg.meshes.append(I._platelet_type(cfg.meshes[0].kbt))
        cfg.cell_type = cfg.cell_type.copy()
        cfg.cell_type[ncell // 2:] = 1
    s = np.array([1.06, 0.97, 0.97255])
    cfg.rotations = cfg.rotations * s[None, None, :]  # stretched: forces far above rounding
    return cfg


@pytest.mark.parametrize('ncell,sub,platelets', [
    (1, 3, False),   # 16 slices of 642 vertices
    (2, 1, False),   # 42 vertices: some of the 16 slices empty
    (9, 2, True),    # 16 slices, 162-vertex meshes of two types
    (10, 2, False),  # 8
    (20, 1, True),   # 4
    (39, 1, False),  # 2
    (77, 1, False),  # one CTA per cell
])
@pytest.mark.parametrize('precision', ['f64', 'f32'])
def test_cell_slices(ncell, sub, platelets, precision):
    from paper_2305_02752_gb300 import hemo
    cfg = _config(ncell, sub, platelets)
    steps = 3
    ref = O.from_config(cfg)
    ref.step(steps)
    exp = ref.get()
    out = []
    for _ in range(2):
        sim = hemo.Simulation.from_config(cfg, precision)
        sim.step(steps)
        out.append(sim.get_fields())
        sim.close()
    for k in ('rho', 'u', 'X', 'Fv', 'cellstats'):
        assert np.array_equal(out[0][k], out[1][k]), k  # the same bits every run
    got = out[0]
    if precision == 'f64':
        assert_close(got['u'], exp['u'], 1e-12, 'u')
        assert_close(got['X'], exp['X'], 1e-12, 'X')
        forces_close(got['Fv'], exp['Fv'], cfg)
    else:
        assert_close(got['u'], exp['u'], 1e-5, 'u')
        assert np.abs(got['X'] - exp['X']).max() < steps * 1e-6 + 2e-6
    tol = 1e-12 if precision == 'f64' else 1e-5
    assert_close(got['cellstats'][:, 3:5], exp['cellstats'][:, 3:5], tol, 'area, volume')
    assert_close(got['cellstats'][:, 5], exp['cellstats'][:, 5], 1e-10 if precision == 'f64' else 1e-5, 'deformation')
