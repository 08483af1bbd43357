"""Field read-out into device memory where the last group of four is partly
filled: node and vertex-component counts of every remainder mod 4."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2305_02752_gb300 import hemo, inputs as I

pytestmark = pytest.mark.gpu

KEYS = ('rho', 'u', 'X', 'Fv', 'cellstats')
CASES = [((16, 13, 16), 4), ((17, 15, 19), 1), ((18, 15, 17), 2), ((17, 13, 15), 3)]


def _bipyramid():
    """Seven vertices, an odd number: five around, two tips."""
    a = 2 * np.pi * np.arange(5) / 5
    v = np.vstack([3.0 * np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 2.2], [0, 0, -2.2]]])
    t = [(k, (k + 1) % 5, 5) for k in range(5)] + [((k + 1) % 5, k, 6) for k in range(5)]
    return v, np.array(t, np.int32)


def test_cases_cover_every_remainder():
    assert {nx * ny * nz % 4 for (nx, ny, nz), _ in CASES} == {0, 1, 2, 3}
    assert {3 * 7 * ncell % 4 for _, ncell in CASES} == {0, 1, 2, 3}


@pytest.mark.parametrize('shape,ncell', CASES)
@pytest.mark.parametrize('precision', ['f32', 'f64', 'f16'])
def test_tails(shape, ncell, precision):
    cfg = I.channel(nx=shape[0], ny=shape[1], nz=shape[2], ncell=1, seed=3, pack_iter=1, exact_iter=0)
    v, t = _bipyramid()
    cen = np.array([[5.0, 6.0, 5.5], [11.0, 6.3, 9.0], [6.2, 6.6, 10.8], [11.5, 6.1, 4.0]])[:ncell]
    cfg = dataclasses.replace(cfg, meshes=[dataclasses.replace(cfg.meshes[0], rest=v, tri=t)],
                              cell_type=np.zeros(ncell, np.int64), centers=cen,
                              rotations=np.repeat(np.diag([1.03, 0.98, 0.99])[None], ncell, axis=0))
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.step(3)
    host = sim.get_fields()
    assert np.abs(host['Fv']).min(axis=0).max() > 0 and np.abs(host['u']).max() > 0
    real = torch.float64 if precision == 'f64' else torch.float32
    kinds = dict(rho=real, u=real, X=torch.float64, Fv=torch.float64, cellstats=torch.float64)
    # room behind every field, which stays as it is
    bufs = {k: torch.full((host[k].size + 8,), -7.0, dtype=kinds[k], device='cuda') for k in KEYS}
    sim.get_fields(out=bufs)
    for k in KEYS:
        got = bufs[k].cpu().numpy()
        assert np.array_equal(got[:-8].reshape(host[k].shape), host[k]), k
        assert (got[-8:] == -7.0).all(), k
    sim.close()
