"""A state written to one strip of a decomposed grid through that strip's own handle swaps
the halves of its ping-pong buffers alone; the steps and exchanges after it take the half that
holds the new state.  Writing back the state that a strip has changes nothing, bit for bit.
"""
import ctypes as C

import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("part", [0, 1, 2])
@pytest.mark.parametrize("kernel", [1, 3, 4])
def test_state_written_to_one_part(part, kernel):
    import paper_2204_10323_gb300 as F
    p = inputs.random_small(130, 61, 12)
    out = []
    for rewrite in (False, True):
        d = F.Decomp(p, 3, 4, precision=F.F32, kernel=kernel)
        d.step(8)
        if rewrite:
            view = d.part_view(part)
            h, qx, qy = (np.ascontiguousarray(view.read(f)) for f in (F.FIELD_H, F.FIELD_QX, F.FIELD_QY))
            view.close()
            F.flood_write_state(d.part_handle(part), *(C.c_void_p(a.ctypes.data) for a in (h, qx, qy)), 0)
        d.step(13)
        d.sync()
        out.append(d.state())
        d.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
