"""Internal viscosity's indicator with a vertex thrown far out: the triangles at
it are reported, not walked column by column."""
import numpy as np
import pytest

from paper_2305_02752_gb300 import hemo
from tests.helpers import small_cell_shear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('precision', ['f32', 'f64'])
@pytest.mark.parametrize('far', [60.0, 3.0e5, -4.0e12, np.nan])
def test_far_vertex_is_reported(precision, far):
    cfg = small_cell_shear(n=16, steps=2)
    sim = hemo.Simulation.from_config(cfg, precision)
    X = sim.get_fields(hemo.HEMO_VERTS)['X']
    before = sim.inside()
    assert before.any()
    X[5, :2] += far
    sim.set_vertices(X)
    with pytest.raises(hemo.HemoError) as e:
        sim.inside()
    assert e.value.code == hemo.HEMO_ERR_NUMERIC
    sim.close()


def test_wide_triangles_within_reach_are_not():
    """A cell larger than the box along x (the longest edges may be four times
    their rest length): accepted as before."""
    cfg = small_cell_shear(n=16, steps=2)
    sim = hemo.Simulation.from_config(cfg, 'f64')
    X = sim.get_fields(hemo.HEMO_VERTS)['X']
    c = X.mean(axis=0)
    X[:, 0] = c[0] + 2.5 * (X[:, 0] - c[0])
    sim.set_vertices(X)
    assert sim.inside().any()
    sim.close()
