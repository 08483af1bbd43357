"""16-bit storage: the default choice between the staged and the per-node
collision on both sides of its line, and the same bits from both."""
import numpy as np
import pytest

from paper_2305_02752_gb300 import hemo, inputs as I

pytestmark = pytest.mark.gpu


def _run(cfg, prec, options):
    sim = hemo.Simulation.from_config(cfg, prec, options=options)
    plan = sim.lattice_plan()
    sim.step(5)
    out = sim.get_fields(hemo.HEMO_RHO | hemo.HEMO_U)
    f = sim.populations()
    sim.close()
    return plan, f, out


@pytest.mark.parametrize('prec', ['f16', 'bf16'])
@pytest.mark.parametrize('shape,staged', [
    ((128, 138, 128), True),   # 2176 tiles: above 13 per multiprocessor of any device of up to 167
    ((64, 130, 256), True),    # the shortest rows staged by default
    ((56, 150, 256), False),   # shorter rows
    ((128, 66, 64), False),    # 512 tiles
    ((512, 20, 24), True),     # long rows, whatever the size
])
def test_default_staging(shape, staged, prec):
    nx, ny, nz = shape
    cfg = I.channel(nx=nx, ny=ny, nz=nz, ncell=0, pack_iter=1, exact_iter=0)
    rng = np.random.default_rng(8)
    cfg.init_velocity = cfg.init_velocity + 0.004 * rng.standard_normal(cfg.init_velocity.shape) * (cfg.mask == 0)[..., None]
    plan, f, out = _run(cfg, prec, 0)
    assert (plan[0] > 0) == staged, plan
    other = hemo.HEMO_OPT_UNSTAGED_COLLISION if staged else hemo.HEMO_OPT_STAGED_COLLISION
    plan1, f1, out1 = _run(cfg, prec, other)
    assert (plan1[0] > 0) != staged, plan1
    assert np.array_equal(f, f1)
    for k in ('rho', 'u'):
        assert np.array_equal(out[k], out1[k]), k
    if staged and nx < 512:  # a kernel that is asked for by name
        assert _run(cfg, prec, hemo.HEMO_OPT_PAIR_COLLISION)[0][0] == 0
