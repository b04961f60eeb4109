"""The Eq. 6 level search at its corners: one-cell sections, sections beyond one warp's cells,
very small and very large discharges, high ground (levels whose rounding is coarser than the
bracket), a zero discharge, both boundary forms, epochs of one step, against the oracle's
bisection on the same inputs.

Tolerance: every cell's share is rescaled to the section's discharge, so an error of the level
moves water between cells only, by (5/3) dW / h of a share.  FP64: dW <= 1e-12 m or a rounding of
W, 1e-9 relative for the 1 cm of the smallest case.  FP32 solves in single precision: dW is a rounding
of W (6e-8 W, W up to 3000 m over depths of 1 m: 3e-4), Eq. 5 1e-6: 1e-3.
"""
import numpy as np
import pytest

from inputs import INFLOW, OUTFLOW, XMAX, XMIN, Options, Problem, Section
import oracle

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ny,cells,Q,base,form,E", [
    (4, (1, 2), 5.0, 10.0, 0, 16), (64, (3, 40), 1e-3, 1.0, 0, 4), (64, (3, 40), 50.0, 3000.0, 0, 4),
    (64, (0, 64), 3e4, 10.0, 0, 4), (64, (3, 40), 5.0, -20.0, 0, 1), (64, (3, 40), 20.0, 0.0, 1, 4),
    (1500, (10, 1400), 900.0, 50.0, 0, 4), (40, (5, 38), 0.0, 10.0, 0, 4)])
def test_level_search_matches_the_bisection(prec, ny, cells, Q, base, form, E):
    Fm = F()
    rng = np.random.default_rng(ny + E)
    nx, dx = 6, 5.0
    f = lambda a: a.astype(np.float32).astype(np.float64)
    z = f(base + rng.uniform(0.0, 0.5, (ny, nx)))
    n = f(rng.uniform(0.02, 0.06, (ny, nx)))
    secs = [Section.cells(XMIN, cells[0], cells[1], INFLOW, 1e-3, nx, ny, [0.0, 100.0], [Q, 2.0 * Q]),
            Section.cells(XMAX, 0, ny, OUTFLOW, 1e-3, nx, ny)]
    p = Problem("level", nx, ny, dx, z, n, secs, Options(dt_mode=1, dt_const=0.01, dt_cap=0.01, epoch_steps=E, bc_form=form))
    s = Fm.Sim(p, precision=prec)
    o = oracle.Oracle(p)
    s.step(3)
    o.run(3)
    got, want = s.read(Fm.FIELD_QX)[:, 0].astype(np.float64), o.qx[:, 0]
    rtol = 1e-9 if prec else 1e-3
    assert np.abs(got - want).max() <= rtol * max(np.abs(want).max(), 1e-300)
    assert got.sum() == pytest.approx(want.sum(), rel=1e-12 if prec else 1e-6, abs=1e-30)
    s.close()
