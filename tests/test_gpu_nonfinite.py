"""Values that are not finite in the coupling: forces raise the numeric status
in every precision; a vertex whose position is not a number spreads nothing."""
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


# rounding of the sums of about 1e3 operations per value, and of fixed-point
# scales that differ by a factor of two between the runs
@pytest.mark.parametrize('precision,tol', [('f32', 1e-5), ('f64', 1e-12)])
def test_position_not_a_number_spreads_nothing(precision, tol):
    cfg = I.channel(nx=24, ny=25, nz=24, ncell=1, seed=3, pack_iter=1, exact_iter=0)
    v, t = I.icosphere(3)
    mesh = dataclasses.replace(cfg.meshes[0], rest=I.evans_fung(v, 6.5), tri=t)
    # a stretched cell across x = 0 within one block of eight along y and z:
    # hundreds of vertices in the block that a NaN along x is binned into
    cfg = dataclasses.replace(cfg, meshes=[mesh], centers=np.array([[1.0, 12.0, 12.0]]), body_force=np.zeros(3),
                              rotations=np.diag([1.05, 0.97, 0.97])[None], init_velocity=None)
    nv, real = len(v), np.float64 if precision == 'f64' else np.float32

    def sim():
        s = hemo.Simulation.from_config(cfg, precision)
        s.set_time_scales(4)
        return s

    a = sim()
    a.step(1)
    state = a.save_state()
    first = a.get_fields()
    a.close()
    i = int(np.argmax(np.abs(first['Fv']).max(axis=1) < np.abs(first['Fv']).max()))  # not the vertex that sets the scale

    def poke(field, value):
        """The state with the entries of vertex i changed; the last sections are
        offsets, forces and previous velocities."""
        out = state.copy()
        n = 3 * nv * real().itemsize
        at = len(out) - {'off': 3, 'Fv': 2}[field] * n
        x = out[at:at + n].view(real)
        if field == 'Fv':  # (the section is the one meant)
            assert np.allclose(x.reshape(-1, 3), first['Fv'], rtol=1e-6, atol=0)
        x[3 * i:3 * i + len(value)] = value
        return out

    got = []
    for field, value in (('off', [np.nan]), ('Fv', [0.0, 0.0, 0.0])):
        s = sim()
        s.load_state(poke(field, value))
        s.step(1)  # forces held
        got.append(s.get_fields(hemo.HEMO_U)['u'])
        s.close()
    assert np.abs(got[0] - got[1]).max() <= tol * np.abs(got[1]).max()
