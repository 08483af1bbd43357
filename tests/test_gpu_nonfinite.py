"""Values that are not finite in the coupling: forces raise the numeric status
in every precision."""
import dataclasses

import numpy as np
import pytest

from paper_2305_02752_gb300 import hemo, inputs as I

pytestmark = pytest.mark.gpu


def _config():
    cfg = I.channel(nx=24, ny=25, nz=24, ncell=1, seed=3, pack_iter=1, exact_iter=0)
    v, t = I.icosphere(2)
    # moduli so small that no finite force, however many are added, moves the
    # fluid by the 0.3 that the velocity's own check admits; links that may
    # shorten to nothing
    soft = dataclasses.replace(cfg.meshes[0], rest=I.evans_fung(v, 7.0), tri=t, k_area=1e-9, k_volume=1e-9, kbt=1e-12,
                               max_strain=2.0)
    return dataclasses.replace(cfg, meshes=[soft], centers=np.array([[12.0, 12.0, 12.0]]), body_force=np.zeros(3),
                               init_velocity=None)


@pytest.mark.parametrize('precision', ['f64', 'f32', 'f16'])
def test_collapsed_triangle_is_reported(precision):
    cfg = _config()
    sim = hemo.Simulation.from_config(cfg, precision)
    sim.step(2)
    X = sim.get_fields(hemo.HEMO_VERTS)['X']  # (raises on a status)
    sim.close()
    sim = hemo.Simulation.from_config(cfg, precision)
    a, b, _ = cfg.meshes[0].tri[0]
    X[a] = X[b]  # two triangles without area, an edge without length
    sim.set_vertices(X)
    with pytest.raises(hemo.HemoError) as e:
        sim.step(1)
        sim.sync()
    assert e.value.code == hemo.HEMO_ERR_NUMERIC
    sim.close()
