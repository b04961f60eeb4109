"""The temporal-blocking kernel's work items at their edges: grids whose last strip
is one column wide, exactly full or a column short, chunks shorter than the steps
per launch, borders in every lane position, and a cap that makes one warp walk many
items, against the single-step stream kernel.  Both evaluate the same explicitly
rounded operations, so the state is equal bit for bit; the boundary outflow and the
clipped volume are float sums over at most 32 rows folded in double (1e-6).
"""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


def pair(nx, ny, k, tile, theta, friction, steps, seed):
    Fm = F()
    p = inputs.random_small(nx, ny, seed)
    p.opts.theta, p.opts.friction, p.opts.epoch_steps = theta, friction, 24
    for a in ("z", "n", "h0", "qx0", "qy0"):
        setattr(p, a, getattr(p, a).astype(np.float32).astype(np.float64))
    ref = Fm.Sim(p, kernel=Fm.KERNEL_STREAM)
    sim = Fm.Sim(p, kernel=Fm.KERNEL_TILED, steps_per_launch=k, tile=tile)
    for s in (ref, sim):
        s.step(steps)
        s.sync()
    for name, a, b in zip(("h", "qx", "qy"), ref.state(), sim.state()):
        assert np.array_equal(a, b), (name, np.argwhere(a != b)[:4])
    A, B = ref.ledger(), sim.ledger()
    for key in ("t", "dt", "V_in", "h_max", "step"):
        assert A[key] == B[key], key
    for key in ("V_out", "V_clip"):
        assert B[key] == pytest.approx(A[key], rel=1e-6, abs=1e-9), key
    ref.close()
    sim.close()


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 116, 119, 120, 121, 123, 124, 125, 239, 240, 241, 244, 363])
@pytest.mark.parametrize("k,ny", [(4, 37), (3, 5), (2, 1), (1, 9), (8, 23)])
def test_strip_and_chunk_edges(nx, k, ny):
    pair(nx, ny, k, (0, 0), 1.0, 0, 27, 3 * nx + ny)


@pytest.mark.parametrize("theta,friction", [(1.0, 0), (0.9, 0), (1.0, 1), (0.9, 1)])
@pytest.mark.parametrize("nx,ny,rows", [(117, 9, 1), (236, 14, 2), (125, 40, 3), (241, 33, 5), (349, 66, 32), (120, 70, 0)])
def test_chunks_shorter_than_the_steps_of_a_launch(nx, ny, rows, theta, friction):
    pair(nx, ny, 4, (0, rows), theta, friction, 26, nx + rows)


@pytest.mark.parametrize("tile", [(1, 0), (3, 4), (2, 200)])
def test_few_warps_walk_many_items(tile):
    pair(300, 90, 4, tile, 1.0, 0, 50, 5)


@pytest.mark.parametrize("k,theta,friction", [(4, 1.0, 0), (3, 1.0, 0), (1, 1.0, 0), (4, 0.9, 1)])
@pytest.mark.parametrize("nx,ny,tile", [(7, 5, (0, 0)), (250, 61, (0, 9)), (130, 40, (2, 0))])
def test_gauges_inside_a_launch(nx, ny, tile, k, theta, friction):
    """Gauge depths after every step of a launch, in border and seam cells, more of them in one
    item than its list holds and repeated ones, against the stream kernel (bitwise)."""
    Fm = F()
    p = inputs.random_small(nx, ny, 3)
    p.opts.theta, p.opts.friction, p.opts.epoch_steps = theta, friction, 12
    for a in ("z", "n", "h0", "qx0", "qy0"):
        setattr(p, a, getattr(p, a).astype(np.float32).astype(np.float64))
    rng = np.random.default_rng(nx)
    some = np.stack([rng.integers(0, nx, 6), rng.integers(0, ny, 6)], 1)
    many = np.stack([rng.integers(0, min(nx, 40), 70), rng.integers(0, min(ny, 8), 70)], 1)
    edge = np.array([[0, 0], [nx - 1, ny - 1], [nx - 1, 0], [0, ny - 1], [min(119, nx - 1), ny // 2], [min(120, nx - 1), ny // 2]])
    for gauges in (some, edge, many):
        a = Fm.Sim(p, kernel=Fm.KERNEL_STREAM)
        b = Fm.Sim(p, kernel=Fm.KERNEL_TILED, steps_per_launch=k, tile=tile)
        assert np.array_equal(a.run_gauges(29, gauges), b.run_gauges(29, gauges))
        for x, y in zip(a.state(), b.state()):
            assert np.array_equal(x, y)
        a.close()
        b.close()
