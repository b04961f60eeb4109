"""The FP64 kernels' division by dx, through one step: inflow through one-cell sections onto dry flat land, whose
faces are all zero but the inflow's, leaves the depth (dt q) / dx, which must be the division's own bits for divisors that
take the three operations and divisors that do not, ordinary, tiny (below 2^-700, subnormal) and huge (above
2^600) dividends and zero."""
import numpy as np
import pytest

from inputs import INFLOW, XMIN, Options, Problem, Section

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dx", [1.0, 2.0, 3.0, 5.0, 7.0, 0.3, 12.7, 33.3, 90.0, 1000.0, 49.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52,
                                1.0 / 3.0, 2.0 ** -20, 2.0 ** -21, 3e6])
def test_depth_after_inflow_is_the_quotient(dx):
    import paper_2204_10323_gb300 as F
    nx, ny = 3, 600
    rng = np.random.default_rng(int(dx * 1000) % 2 ** 31)
    Q = rng.uniform(1.0, 2.0, ny) * 2.0 ** rng.integers(-40, 40, ny)
    e = np.array([-1074, -1060, -1020, -760, -720, -705, -701, -700, -699, -690, 560, 590, 598, 599, 600, 601, 640])
    Q[:17 * 12] = rng.uniform(1.0, 2.0, 17 * 12) * 2.0 ** np.repeat(e, 12).astype(np.float64)
    Q[17 * 12] = 0.0
    secs = [Section.cells(XMIN, k, k + 1, INFLOW, 1e-3, nx, ny, [0.0], [Q[k]]) for k in range(ny)]
    dt = 1.0
    p = Problem("quotient", nx, ny, dx, np.zeros((ny, nx)), np.full((ny, nx), 0.05), secs,
                Options(dt_mode=1, dt_const=dt, dt_cap=dt, epoch_steps=1))
    s = F.Sim(p, precision=F.F64)
    s.step(1)
    q, h = s.read(F.FIELD_QX)[:, 0], s.read(F.FIELD_H)
    s.close()
    assert np.isfinite(q).all() and (q > 0).sum() > 500
    assert np.array_equal(h[:, 0], (dt * q) / dx)
    assert not h[:, 1:].any()
