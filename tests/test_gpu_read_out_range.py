"""Field read-out into a device allocation that ends before the field does: it
goes through the staging buffer and a copy, which the driver checks, not
through a kernel that would write past the end.  The staging buffer is refused
here, so nothing is copied either."""
import ctypes as C

import pytest
import torch

from paper_2305_02752_gb300 import hemo

pytestmark = pytest.mark.gpu


class _Raw:
    """`nbytes` of an allocation of their own."""

    def __init__(self, nbytes):
        self.p = C.c_void_p()
        assert hemo.lib().cudaMalloc(C.byref(self.p), C.c_size_t(nbytes)) == 0

    def data_ptr(self):
        return self.p.value

    def free(self):
        assert hemo.lib().cudaFree(self.p) == 0


def _refuse(*args):
    raise RuntimeError('out of memory')


@pytest.mark.parametrize('what,key,per_node', [(hemo.HEMO_RHO, 'rho', 1), (hemo.HEMO_U, 'u', 3)])
def test_short_destination_is_not_written(what, key, per_node, monkeypatch):
    sim = hemo.Simulation(96, 96, 96, precision='f32')  # 3.5 MB a component
    sim.step(2)
    need = 4 * per_node * sim.N
    whole, short = _Raw(need), _Raw(4096)
    monkeypatch.setattr(torch.cuda, 'caching_allocator_alloc', _refuse)
    sim.get_fields(what, out={key: whole})  # written directly: no staging buffer
    with pytest.raises(hemo.HemoError) as e:
        sim.get_fields(what, out={key: short})
    assert e.value.code == hemo.HEMO_ERR_OOM
    monkeypatch.undo()
    got = sim.get_fields(what)[key]  # the simulation goes on
    buf = torch.zeros(got.shape, dtype=torch.float32, device='cuda')
    sim.get_fields(what, out={key: buf})
    assert (buf.cpu().numpy() == got).all()
    sim.close()
    whole.free()
    short.free()
