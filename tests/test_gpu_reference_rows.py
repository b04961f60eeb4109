"""The IEEE-ordered kernel's strips of 31 columns and chunks of one to three rows at their edges, and its
integer maxima: ragged widths, dry and wet land, both precisions, the scheme options and gauges, against
the oracle (FP64 1e-10: cbrt and pow ulps and the ledger's order, as in the forward parity tests; FP32
1e-4 m after 24 steps), and infinities and NaN, which must stay where the plain comparisons leave them.
"""
import numpy as np
import pytest

import inputs
from inputs import Problem
import oracle

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


@pytest.mark.parametrize("prec,tol", [(1, 1e-10), (0, 1e-4)])
@pytest.mark.parametrize("theta,friction", [(1.0, 0), (0.9, 1)])
@pytest.mark.parametrize("nx,ny", [(1, 3), (30, 4), (31, 5), (32, 6), (33, 1), (61, 7), (62, 9), (63, 2), (800, 700), (1100, 1000)])
def test_strip_edges_match_the_oracle(nx, ny, theta, friction, prec, tol):
    Fm = F()
    p = inputs.random_small(nx, ny, nx + ny, wet=0.4)
    p.opts.theta, p.opts.friction = theta, friction
    if prec == 0:
        for a in ("z", "n", "h0", "qx0", "qy0"):
            setattr(p, a, getattr(p, a).astype(np.float32).astype(np.float64))
    steps = 24 if nx < 500 else 6
    s = Fm.Sim(p, precision=prec, kernel=Fm.KERNEL_REFERENCE)
    o = oracle.Oracle(p)
    gauges = np.array([[0, 0], [nx - 1, ny - 1], [min(30, nx - 1), 0], [min(31, nx - 1), ny // 2]])
    series = s.run_gauges(steps, gauges)
    o.run(steps)
    # (the FP32 bound is one of depths)
    for got, want in list(zip(s.state(), (o.h, o.qx, o.qy)))[:3 if prec else 1]:
        assert np.abs(got.astype(np.float64) - want).max() < tol
    assert np.array_equal(series[-1], s.read(Fm.FIELD_H)[gauges[:, 1], gauges[:, 0]].astype(np.float64))
    L, Lo = s.ledger(), o.ledger_dict()
    for k in ("V_in", "V_out", "V_clip"):
        assert L[k] == pytest.approx(Lo[k], rel=1e-10 if prec else 1e-4, abs=1e-9 if prec else 1e-4)
    s.close()


@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf])
def test_non_finite_depths_spread_like_the_plain_comparisons(bad):
    """One step from a state with a non-finite depth (device input is taken as it is): fmax passes over a NaN, so
    NumPy's fmax gives the faces."""
    import torch
    Fm = F()
    p = inputs.lake_at_rest(40, 6)
    s = Fm.Sim(p, precision=Fm.F64)
    h = p.h0.copy()
    h[3, 12] = bad
    s.write_state(torch.from_numpy(h).cuda())
    s.step(1)
    got = s.read(Fm.FIELD_QX)
    e = h + p.z
    with np.errstate(all="ignore"):
        hf = np.fmax(e[:, :-1], e[:, 1:]) - np.maximum(p.z[:, :-1], p.z[:, 1:])
        num = 0.0 - 9.81 * 0.05 * hf * (e[:, 1:] - e[:, :-1]) / p.dx
    want_nan = np.isnan(num) & (hf > 1e-3)
    assert np.array_equal(np.isnan(got[:, 1:-1]), want_nan)
    s.close()
