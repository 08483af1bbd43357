"""FP32 spreading and interpolation at the edges of their bin sizes: bins of
a few vertices, around the sizes where the kernels switch paths or take
another chunk, and crowded ones, against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2305_02752_gb300 import inputs as I
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


def _crowd(ncell, subdiv, shape, seed=5, spread=0.6):
    """`ncell` cells about one point of a periodic box between walls, stretched
    so that the membrane forces are far above rounding."""
    nx, ny, nz = shape
    cfg = I.channel(nx=nx, ny=ny, nz=nz, ncell=1, seed=seed, pack_iter=1, exact_iter=0)
    rng = np.random.default_rng(seed)
    if subdiv is not None:
        v, t = I.locality_order(*I.icosphere(subdiv))
        cfg.meshes[0].rest, cfg.meshes[0].tri = I.evans_fung(v, 8.0), t
    c0 = np.array([nx / 2.0 + 0.3, ny / 2.0 - 0.4, nz / 2.0 + 0.1])
    cen = c0 + rng.normal(size=(ncell, 3)) * spread
    rot = np.stack([I.random_rotation(rng) @ np.diag([1.08, 0.96, 0.965]) for _ in range(ncell)])
    return dataclasses.replace(cfg, cell_type=np.zeros(ncell, np.int64), centers=cen, rotations=rot)


@pytest.mark.parametrize('ncell,subdiv,shape', [
    (1, 1, (24, 27, 24)),     # 42 vertices: every bin far below 64
    (1, None, (32, 29, 24)),  # one red cell: bins on both sides of 64
    (3, None, (24, 32, 24)),
    (9, None, (32, 33, 32)),  # bins of more than 256 and 512 vertices
    (16, 2, (16, 31, 24)),    # crowded small cells; two blocks along x
])
def test_spread_and_interpolate(ncell, subdiv, shape):
    from paper_2305_02752_gb300 import hemo
    cfg = _crowd(ncell, subdiv, shape)
    steps = 3
    ref = O.from_config(cfg)
    ref.step(steps)
    exp = ref.get()
    out = []
    for _ in range(2):
        sim = hemo.Simulation.from_config(cfg, 'f32')
        sim.step(steps)
        out.append(sim.get_fields())
        sim.close()
    for k in ('rho', 'u', 'X', 'Fv'):
        assert np.array_equal(out[0][k], out[1][k]), k  # the same bits every run
    assert_close(out[0]['u'], exp['u'], 1e-5, 'u')
    # positions move by about 0.02 a step: errors of FP32 offsets and velocity
    assert np.abs(out[0]['X'] - exp['X']).max() < steps * 1e-6 + 2e-6
