"""Bounds-checked build where the bins are listed by size and where cells are
split over a cluster of CTAs: no check fails and the bits are the default
build's."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = r'''
import sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_2305_02752_gb300 import hemo, inputs as I
cfg = I.channel(nx=48, ny=43, nz=48, ncell=16, seed=11, platelet_ratio=0.0, pack_iter=20, exact_iter=0)  # 10,272 vertices
sim = hemo.Simulation.from_config(cfg, sys.argv[1])
sim.step(4)
f = sim.get_fields()
assert sim.membrane_plan() > 1
sim.close()
np.savez(sys.argv[2], lib=np.array(hemo.LIB_PATH), **f)
'''


@pytest.mark.parametrize('precision', ['f32', 'f64'])
def test_same_bits(precision, tmp_path):
    out = []
    for checked in ('0', '1'):
        path = str(tmp_path / f'{checked}.npz')
        subprocess.run([sys.executable, '-c', RUN.format(root=ROOT), precision, path], check=True, cwd=ROOT,
                       env=dict(os.environ, HEMO_BOUNDS_CHECK=checked))  # (raises if a check failed)
        out.append(dict(np.load(path)))
    assert str(out[0].pop('lib')) != str(out[1].pop('lib'))
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
