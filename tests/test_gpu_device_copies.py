"""flood_read and flood_write_state on device memory: every alignment that the dense
side can have, against the host copies (exact).
"""
import ctypes as C

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 5), (31, 4), (32, 3), (255, 7), (256, 2), (2048, 3), (4099, 2), (3, 3000)])
@pytest.mark.parametrize("skip", [0, 1, 2])
def test_device_reads_and_writes_equal_the_host_ones(nx, ny, prec, skip):
    import torch
    Fm = F()
    p = inputs.lake_at_rest(nx, ny)
    sim, other = Fm.Sim(p, precision=prec), Fm.Sim(p, precision=prec)
    rng = np.random.default_rng(nx + ny)
    host = [rng.uniform(0.0, 1.0, s).astype(sim.dtype) for s in ((ny, nx), (ny, nx + 1), (ny + 1, nx))]
    sim.write_state(*host)
    dev = []
    for field, a in enumerate(host):
        buf = torch.full((a.size + skip + 4,), -1.0, dtype=torch.float64 if prec else torch.float32, device="cuda")
        t = buf[skip:skip + a.size]                  # starts `skip` elements past an aligned address
        Fm.flood_read(sim.h, field, C.c_void_p(t.data_ptr()), a.nbytes, 1)
        assert np.array_equal(t.cpu().numpy().reshape(a.shape), a)
        assert bool((buf[:skip] == -1).all()) and bool((buf[skip + a.size:] == -1).all())
        dev.append(t.view(*a.shape))
    other.write_state(*dev)
    for a, b in zip(host, other.state()):
        assert np.array_equal(a, b)
    sim.close()
    other.close()


def test_host_memory_passed_as_device_memory_is_not_handed_to_the_kernel():
    # the runtime's copy decides about it, as before: an error status or a copy, never a fault
    Fm = F()
    sim = Fm.Sim(inputs.lake_at_rest(40, 9))
    h = sim.read(Fm.FIELD_H)
    out = np.zeros_like(h)
    try:
        Fm.flood_read(sim.h, Fm.FIELD_H, C.c_void_p(out.ctypes.data), out.nbytes, 1)
        assert np.array_equal(out, h)
    except Fm.FloodError as e:
        assert e.status == Fm.ERR_CUDA
    sim.close()
