"""Two simulations side by side whose membrane kernels take different amounts of
shared memory: the second does not take it from the first."""
import dataclasses

import numpy as np
import pytest

from paper_2305_02752_gb300 import hemo, inputs as I

pytestmark = pytest.mark.gpu


def _sphere(rings, around):
    """A closed mesh of rings * around + 2 vertices."""
    v = [[0, 0, 1.0]]
    for i in range(1, rings + 1):
        a = np.pi * i / (rings + 1)
        v += [[np.sin(a) * np.cos(b), np.sin(a) * np.sin(b), np.cos(a)] for b in 2 * np.pi * np.arange(around) / around]
    v.append([0, 0, -1.0])
    at = lambda i, k: 1 + i * around + k % around
    t = [(0, at(0, k), at(0, k + 1)) for k in range(around)]
    for i in range(rings - 1):
        for k in range(around):
            t += [(at(i, k), at(i + 1, k), at(i + 1, k + 1)), (at(i, k), at(i + 1, k + 1), at(i, k + 1))]
    t += [(len(v) - 1, at(rings - 1, k + 1), at(rings - 1, k)) for k in range(around)]
    return 3.5 * np.array(v), np.array(t, np.int32)


def _config(mesh, ncell=90):
    cfg = I.channel(nx=48, ny=43, nz=48, ncell=1, seed=3, pack_iter=1, exact_iter=0)
    rng = np.random.default_rng(5)
    v, t = mesh
    m = dataclasses.replace(cfg.meshes[0], rest=v, tri=t)
    return dataclasses.replace(cfg, meshes=[m], cell_type=np.zeros(ncell, np.int64),
                               centers=np.array([8.0, 8.0, 8.0]) + rng.random((ncell, 3)) * [30, 26, 30],
                               rotations=np.repeat(np.diag([1.01, 0.995, 0.995])[None], ncell, axis=0))


def test_smaller_mesh_beside_a_larger_one():
    big, small = _config(_sphere(20, 32)), _config(_sphere(16, 32))  # 642 and 514 vertices: 65 and 52 KB a cell
    a = hemo.Simulation.from_config(big, 'f32')
    a.step(1)
    assert a.membrane_plan() == 1  # one CTA per cell
    b = hemo.Simulation.from_config(small, 'f32')
    b.step(1)
    a.step(2)  # (a variant of the step that is captured only now)
    got = a.get_fields()
    a.close()
    b.close()
    ref = hemo.Simulation.from_config(big, 'f32')
    ref.step(3)
    exp = ref.get_fields()
    ref.close()
    for k in ('rho', 'u', 'X', 'Fv', 'cellstats'):
        assert np.array_equal(got[k], exp[k]), k
