"""A device buffer that ends before the field does is an error, as it was from the runtime's copy, and
nothing is written past its end: the check is the host's, before any launch."""
import ctypes as C

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("field", [0, 1, 2])
def test_a_field_larger_than_the_buffers_allocation(field, prec):
    import torch
    import paper_2204_10323_gb300 as F
    p = inputs.lake_at_rest(4100, 4099)                # 67 MB a field and more: larger than any block that a few bytes share
    sim = F.Sim(p, precision=prec)
    before = sim.read(F.FIELD_H)
    small = torch.zeros(16, device="cuda")
    shape = ((4099, 4100), (4099, 4101), (4100, 4100))[field]
    n = int(np.prod(shape)) * (8 if prec else 4)
    with pytest.raises(F.FloodError) as e:
        F.flood_read(sim.h, field, C.c_void_p(small.data_ptr()), n, 1)
    assert e.value.status == F.ERR_CUDA
    assert not small.any()
    sim.close()
    sim = F.Sim(p, precision=prec)
    args = [C.c_void_p(small.data_ptr()) if k == field else None for k in range(3)]
    if args[0] is None:                                # a whole depth beside the short discharge
        h = torch.from_numpy(before).cuda()
        args[0] = C.c_void_p(h.data_ptr())
    with pytest.raises(F.FloodError) as e:
        F.flood_write_state(sim.h, *args, 1)
    assert e.value.status == F.ERR_CUDA
    sim.close()
