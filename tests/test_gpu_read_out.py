"""Field read-out: into device memory (written there directly), into device
memory that is not aligned to 16 bytes, and into host memory give the same
values, for vertex and node counts of every remainder mod 4."""
import numpy as np
import pytest
import torch

from paper_2305_02752_gb300 import inputs as I

pytestmark = pytest.mark.gpu

KEYS = ('rho', 'u', 'X', 'Fv', 'cellstats')


@pytest.mark.parametrize('shape,ncell', [((16, 13, 16), 1), ((17, 15, 19), 2), ((24, 14, 25), 3), ((24, 16, 24), 5)])
@pytest.mark.parametrize('precision', ['f32', 'f64', 'bf16'])
def test_read_out_targets(shape, ncell, precision):
    from paper_2305_02752_gb300 import hemo
    nx, ny, nz = shape
    cfg = I.channel(nx=nx, ny=ny, nz=nz, ncell=ncell, seed=3, pack_iter=5, exact_iter=0)
    v, t = I.icosphere(1)
    cfg.meshes[0].rest, cfg.meshes[0].tri = I.evans_fung(v, 6.0), t  # 42 vertices a cell
    cfg.centers = np.clip(cfg.centers, 5.0, np.array([nx, ny, nz]) - 6.0)
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.step(3)
    host = sim.get_fields()
    real = torch.float64 if precision == 'f64' else torch.float32
    kinds = dict(rho=real, u=real, X=torch.float64, Fv=torch.float64, cellstats=torch.float64)
    for shift in (0, 1):  # 1: element-aligned only
        bufs = {k: torch.full((host[k].size + shift,), -7.0, dtype=kinds[k], device='cuda')[shift:] for k in KEYS}
        sim.get_fields(out=bufs)
        for k in KEYS:
            assert np.array_equal(bufs[k].cpu().numpy().reshape(host[k].shape), host[k]), (k, shift)
    # positions alone into host memory, forces alone into device memory
    F = torch.zeros(host['Fv'].shape, dtype=torch.float64, device='cuda')
    X = sim.get_fields(hemo.HEMO_VERTS)['X']
    sim.get_fields(hemo.HEMO_FORCES, out={'Fv': F})
    assert np.array_equal(X, host['X']) and np.array_equal(F.cpu().numpy(), host['Fv'])
    mixed = {'X': np.zeros_like(host['X']), 'Fv': torch.zeros_like(F)}
    sim.get_fields(hemo.HEMO_VERTS | hemo.HEMO_FORCES, out=mixed)
    assert np.array_equal(mixed['X'], host['X']) and np.array_equal(mixed['Fv'].cpu().numpy(), host['Fv'])
    sim.close()
