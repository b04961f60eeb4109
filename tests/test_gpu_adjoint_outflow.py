"""The FP32 reverse step's derivative of an outflow face with respect to its cell's Manning n is rounded once per
operation: on a flat lake at rest every interior face is still, so one reverse step leaves dL/dn = (dt/dx) q / n at a
gauge in an outflow cell, with q the outflow that the step computed (exact: one division and one product)."""
import numpy as np
import pytest

from inputs import OUTFLOW, XMAX, Options, Problem, Section

pytestmark = pytest.mark.gpu


def test_outflow_derivative_is_correctly_rounded():
    import paper_2204_10323_gb300 as F
    nx, ny, dx, dt = 8, 2000, 4.0, 0.25
    rng = np.random.default_rng(4)
    n = rng.uniform(0.02, 0.09, (ny, nx)).astype(np.float32)
    p = Problem("outflow", nx, ny, dx, np.zeros((ny, nx)), n.astype(np.float64),
                [Section.cells(XMAX, 0, ny, OUTFLOW, 2e-3, nx, ny)],
                Options(dt_mode=1, dt_const=dt, dt_cap=dt, epoch_steps=4), h0=np.full((ny, nx), 0.75))
    gauges = np.stack([np.full(ny, nx - 1), np.arange(ny)], 1)
    s = F.Sim(p)
    g = s.adjoint(1, gauges, np.ones((1, ny)), n_checkpoints=1).astype(np.float32)
    s.step(1)
    q = s.read(F.FIELD_QX)[:, nx]
    s.close()
    assert (q > 0).all()
    want = np.float32(dt / dx) * (q / n[:, -1])        # the flux leaves: more n, less outflow, more depth
    assert np.array_equal(g[:, -1], want.astype(np.float32))
    assert not g[:, :-1].any()
