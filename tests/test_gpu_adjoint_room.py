"""FP64 membrane adjoint of many cells: its records take bounded room, and cells
beyond those that fit it at a time count like the others."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2305_02752_gb300 import hemo, inputs as I

pytestmark = pytest.mark.gpu

ROOM = 64 << 20


def _run(cfg, precision):
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.record(2)
    sim.step(2)
    _, dX = sim.deformation_loss()
    grad = sim.backward(dX)
    sim.close()
    return grad


def test_records_of_many_cells(monkeypatch):
    # 1000 cells (above 800 fill the room) on top of each other in a small box,
    # the last of a second type with a smaller mesh
    ncell, small = 1000, 100
    cfg = I.channel(nx=40, ny=41, nz=40, ncell=1, seed=3, pack_iter=1, exact_iter=0)
    rng = np.random.default_rng(4)
    meshes = []
    for sub, size in ((3, 7.0), (2, 5.0)):
        v, t = I.icosphere(sub)
        # soft, as the forces of all cells meet in the same nodes
        meshes.append(dataclasses.replace(cfg.meshes[0], rest=I.evans_fung(v, size), tri=t, kbt=cfg.meshes[0].kbt * 1e-3,
                                          k_area=5e-3, k_volume=2e-2))
    rot = np.stack([I.random_rotation(rng) @ np.diag([1.08, 0.96, 0.965]) for _ in range(ncell)])
    cfg = dataclasses.replace(cfg, meshes=meshes, cell_type=np.repeat([0, 1], [ncell - small, small]),
                              centers=20.0 + rng.uniform(-10, 10, size=(ncell, 3)), rotations=rot)
    asked = []
    alloc = torch.cuda.caching_allocator_alloc

    def count(nbytes, *args):
        asked.append(int(nbytes))
        return alloc(nbytes, *args)

    monkeypatch.setattr(torch.cuda, 'caching_allocator_alloc', count)
    got = _run(cfg, 'f64')
    assert max(asked) <= ROOM, max(asked)
    monkeypatch.undo()
    # the same cells with the second type first: other cells at a time, the same
    # sums up to the rounding of FP64 (1e-13, and 1e6 for terms that cancel; a
    # cell left out or counted twice changes its type's entries by 1e-3)
    order = np.argsort(-cfg.cell_type, kind='stable')
    other = _run(dataclasses.replace(cfg, cell_type=cfg.cell_type[order], centers=cfg.centers[order],
                                     rotations=cfg.rotations[order]), 'f64')
    exp = np.concatenate([other[4:8], other[:4]])  # (types are numbered as they are added)
    assert np.isfinite(got).all() and (got[:8] != 0).all()
    assert np.abs(got[:8] / exp - 1).max() < 1e-7, got[:8] / exp - 1
