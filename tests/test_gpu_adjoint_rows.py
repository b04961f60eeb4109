"""The FP32 reverse step's items at their edges: last strips one column wide, exactly
full and a column short, grids narrower than a lane, few rows, inflow and outflow on
every side, more gauges in one item than its list holds, repeated gauges, and more
steps than the log of the inflow pass, against the FP64 reverse sweep of the GPU
(itself pinned to the oracle).

Tolerance: every cell is wet and the water deep (0.6-0.8 m, steps of 0.1 s), so no
decision flips and the forward states differ by about 1e-6; a reverse step rounds some
twenty operations (6e-8 each) and the friction derivative amplifies a relative depth
error by 7/3: about 1e-5 a step at most, 1e-3 of the largest gradient over the 40 steps.
"""
import numpy as np
import pytest

from inputs import INFLOW, OUTFLOW, XMAX, XMIN, YMAX, YMIN, Options, Problem, Section

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


def case(nx, ny, seed):
    rng = np.random.default_rng(900 + seed)
    f = lambda a: a.astype(np.float32).astype(np.float64)
    z = f(1.0 - 1e-3 * np.arange(nx)[None, :] + rng.uniform(-0.02, 0.02, (ny, nx)))
    tab = ([0.0, 30.0], [0.3 * ny, 0.5 * ny])
    secs = [Section.cells(XMIN, 0, max(1, ny // 2), INFLOW, 2e-3, nx, ny, *tab),
            Section.cells(YMIN, nx // 3, nx // 3 + max(1, nx // 4), INFLOW, 1e-3, nx, ny, *tab),
            Section.cells(YMAX, 0, max(1, nx // 3), INFLOW, 1e-3, nx, ny, *tab),
            Section.cells(YMAX, max(1, nx // 3), nx, OUTFLOW, 1e-3, nx, ny),
            Section.cells(XMAX, ny // 4, ny, OUTFLOW, 2e-3, nx, ny)]
    if ny > 3:
        secs.append(Section.cells(XMAX, 0, ny // 4, INFLOW, 1e-3, nx, ny, *tab))
    return Problem("rows", nx, ny, 4.0, z, f(rng.uniform(0.03, 0.06, (ny, nx))), secs,
                   Options(dt_mode=1, dt_const=0.1, dt_cap=0.1, epoch_steps=8),
                   h0=f(0.6 + rng.uniform(0.0, 0.2, (ny, nx))))


def compare(p, gauges, steps, checkpoints):
    Fm = F()
    w = np.random.default_rng(steps).standard_normal((steps, len(gauges)))
    a, b = Fm.Sim(p, precision=Fm.F64), Fm.Sim(p)
    g64, h64 = a.adjoint(steps, gauges, w, n_checkpoints=checkpoints, want_dh0=True)
    g32, h32 = b.adjoint(steps, gauges, w, n_checkpoints=checkpoints, want_dh0=True)
    assert np.abs(g64).max() > 0
    assert np.abs(g32 - g64).max() <= 1e-3 * np.abs(g64).max()
    assert np.abs(h32 - h64).max() <= 1e-3 * np.abs(h64).max()
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(1, 7), (59, 5), (60, 7), (61, 6), (62, 9), (63, 4), (2, 9), (3, 5), (4, 4), (5, 33), (119, 6), (120, 7), (121, 8), (123, 9), (124, 30), (125, 3),
                                   (240, 17), (241, 2), (244, 1), (400, 61)])
def test_item_edges(nx, ny):
    gauges = np.array([[0, 0], [nx - 1, ny - 1], [nx // 2, ny // 2], [min(119, nx - 1), ny - 1], [min(120, nx - 1), 0]])
    compare(case(nx, ny, nx + ny), gauges, 40, 9)


def test_more_gauges_than_an_items_list():
    rng = np.random.default_rng(3)
    gauges = np.stack([rng.integers(0, 60, 90), rng.integers(0, 9, 90)], 1)      # with repeats
    compare(case(60, 9, 1), gauges, 24, 24)


def test_more_steps_than_the_inflow_log_holds():
    # 600 steps against a log of 512; the errors of 600 steps stay below the bound of 40 deep-water steps
    # because the perturbations leave through the outflow sections
    compare(case(40, 12, 2), np.array([[5, 5], [30, 2]]), 600, 40)


@pytest.mark.parametrize("theta,friction", [(1.0, 0), (0.9, 1)])
@pytest.mark.parametrize("precision", [0, 1])
def test_sections_that_share_a_corner_cell(precision, theta, friction):
    """Three inflow sections hold cell (0, 0), two the last one: their terms all reach dL/dn, in one order."""
    Fm = F()
    p = case(1, 7, 8)
    p.opts.theta, p.opts.friction = theta, friction
    w = np.random.default_rng(1).standard_normal((12, 2))
    out = []
    for _ in range(40):
        sim = Fm.Sim(p, precision=precision)
        out.append(sim.adjoint(12, np.array([[0, 0], [0, 6]]), w, n_checkpoints=12))
        sim.close()
    for g in out[1:]:
        assert np.array_equal(g, out[0])
