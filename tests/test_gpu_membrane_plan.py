"""Which cluster size the membrane kernel takes for a number of cells, and its
forces against the oracle at each."""
import numpy as np
import pytest

import oracle as O
from paper_2305_02752_gb300 import hemo, inputs as I
from tests.helpers import forces_close, rel_l2

pytestmark = pytest.mark.gpu


def _config(ncell):
    cfg = I.channel(nx=48, ny=43, nz=48, ncell=ncell, seed=11, platelet_ratio=0.0, pack_iter=20, exact_iter=0)
    v, t = I.locality_order(*I.icosphere(2))
    cfg.meshes[0].rest, cfg.meshes[0].tri = I.evans_fung(v, 7.0), t
    cfg.rotations = cfg.rotations * np.array([1.06, 0.97, 0.97255])[None, None, :]  # forces far above rounding
    return cfg


# as many CTAs per cell, a power of two up to 16, as leave every CTA an SM of
# its own on 152 of them (a cluster of 16 needs 16 free in one GPC, so that size
# is asked of one cell only)
@pytest.mark.parametrize('ncell,ctas', [(1, 16), (10, 8), (20, 4), (39, 2), (77, 1)])
@pytest.mark.parametrize('precision', ['f64', 'f32'])
def test_cluster_size(ncell, ctas, precision):
    cfg = _config(ncell)
    sim = hemo.Simulation.from_config(cfg, precision)
    assert sim.membrane_plan() == 0
    sim.step(1)
    assert sim.membrane_plan() == ctas
    got = sim.get_fields(hemo.HEMO_FORCES)['Fv']
    sim.close()
    ref = O.from_config(cfg)
    ref.step(1)
    exp = ref.get()['Fv']
    if precision == 'f64':
        assert forces_close(got, exp, cfg)
    else:
        # FP32 positions (2^-24 of a 3.5-unit radius) against strains of 3e-2 of
        # edges of 0.8 units: 2e-7 / 2.4e-2 per edge
        assert rel_l2(got, exp) < 1e-4
