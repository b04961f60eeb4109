"""Gauges in any number: spread over the grid or all in one patch, repeated, in random order, recorded through the
temporal-blocking kernel and its scheme options over whole launches and a short one, against the single-step
kernel's gather (bit for bit); their seeds in the FP32 reverse step against the FP64 one; and the time of a run
with thousands of them in one patch against the same run with one.
"""
import numpy as np
import pytest

import inputs
from inputs import OUTFLOW, XMAX, Options, Problem, Section

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


def gauges(kind, count, nx, ny, seed=0):
    rng = np.random.default_rng(seed)
    if kind == "spread":
        return np.stack([rng.integers(0, nx, count), rng.integers(0, ny, count)], 1)
    if kind == "row":                                  # all in one row, every column of it
        return np.stack([rng.permutation(count) % nx, np.full(count, ny // 2)], 1)
    side = int(np.ceil(np.sqrt(count)))                # a patch across a strip's end
    k = rng.permutation(count)
    return np.stack([min(100, nx - 1 - side) + k % side, min(20, ny - 1 - side) + k // side], 1)


@pytest.mark.parametrize("theta,friction", [(1.0, 0), (0.9, 0), (1.0, 1), (0.9, 1)])
@pytest.mark.parametrize("kind,count", [("spread", 1), ("spread", 32), ("spread", 33), ("spread", 700), ("patch", 40),
                                        ("patch", 900), ("row", 300), ("spread", 9000), ("spread", 110000)])
def test_series_equal_the_gathered_ones(kind, count, theta, friction):
    Fm = F()
    nx, ny, steps = 241, 67, 26
    p = inputs.random_small(nx, ny, 5)
    p.opts.theta, p.opts.friction, p.opts.epoch_steps = theta, friction, 16
    at = gauges(kind, count, nx, ny, count)
    out = []
    for kernel in (Fm.KERNEL_STREAM, Fm.KERNEL_TILED):
        s = Fm.Sim(p, kernel=kernel)
        out.append(s.run_gauges(steps, at))
        s.close()
    assert np.array_equal(out[0], out[1])


def test_series_without_memory_for_the_rows():
    """Single steps and gathers then, as for tall narrow grids over few steps."""
    Fm = F()
    p = inputs.random_small(241, 67, 5)
    at = gauges("spread", 40, 241, 67)
    out = []
    for fail in (-1, 0, 1, 2):                         # the cells, the series, the rows
        s = Fm.Sim(p, kernel=Fm.KERNEL_TILED)
        Fm.flood_debug_fail_alloc_after(fail)
        try:
            out.append(s.run_gauges(26, at))
        except Fm.FloodError as e:
            assert e.status == Fm.ERR_OOM and fail in (0, 1)
        finally:
            Fm.flood_debug_fail_alloc_after(-1)
        if fail in (0, 1):
            out.append(s.run_gauges(26, at))           # the handle is as before
        s.close()
    assert len(out) == 4 and all(np.array_equal(out[0], o) for o in out[1:])
    q = inputs.random_small(3, 20000, 5)
    at = gauges("spread", 40, 3, 20000)
    a, b = Fm.Sim(q, kernel=Fm.KERNEL_TILED), Fm.Sim(q, kernel=Fm.KERNEL_STREAM)
    for steps in (3, 9):
        assert np.array_equal(a.run_gauges(steps, at), b.run_gauges(steps, at))
    a.close()
    b.close()


@pytest.mark.parametrize("kind", ["spread", "patch"])
def test_series_of_many_gauges(kind):
    Fm = F()
    p = inputs.random_small(512, 400, 9)
    p.opts.epoch_steps = 16
    at = gauges(kind, 3000, 512, 400)
    out = []
    for kernel in (Fm.KERNEL_STREAM, Fm.KERNEL_TILED):
        s = Fm.Sim(p, kernel=kernel)
        out.append(s.run_gauges(64, at))
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("tile", [(1, 0), (0, 3), (2, 5)])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8])
def test_series_with_any_launch_shape(k, tile):
    Fm = F()
    p = inputs.random_small(250, 43, 6)
    p.opts.epoch_steps = 24
    at = gauges("spread", 500, 250, 43)
    out = []
    for opts in (dict(kernel=Fm.KERNEL_STREAM), dict(kernel=Fm.KERNEL_TILED, steps_per_launch=k, tile=tile)):
        s = Fm.Sim(p, **opts)
        out.append(s.run_gauges(31, at))
        s.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("kind,count", [("spread", 33), ("patch", 1600), ("row", 250), ("spread", 3000)])
def test_seeds_of_many_gauges(kind, count):
    """Wet land, 0.6-0.8 m, steps of 0.1 s: no decision flips, and a reverse step rounds some twenty operations (6e-8
    each) that the friction derivative amplifies by 7/3: 1e-5 a step, 1e-4 of the largest gradient over 8 steps."""
    Fm = F()
    nx, ny, steps = 190, 70, 8
    rng = np.random.default_rng(7)
    f = lambda a: a.astype(np.float32).astype(np.float64)
    z = f(1.0 - 1e-3 * np.arange(nx)[None, :] + rng.uniform(-0.02, 0.02, (ny, nx)))
    p = Problem("seeds", nx, ny, 4.0, z, f(rng.uniform(0.03, 0.06, (ny, nx))),
                [Section.cells(XMAX, 0, ny, OUTFLOW, 2e-3, nx, ny)],
                Options(dt_mode=1, dt_const=0.1, dt_cap=0.1, epoch_steps=8), h0=f(0.6 + rng.uniform(0.0, 0.2, (ny, nx))))
    at = gauges(kind, count, nx, ny, count)
    w = rng.standard_normal((steps, count))
    out = []
    for prec in (Fm.F64, Fm.F32):
        s = Fm.Sim(p, precision=prec)
        out.append(s.adjoint(steps, at, w, n_checkpoints=8, want_dh0=True))
        s.close()
    for a, b in zip(*out):
        assert np.abs(b - a).max() <= 1e-4 * np.abs(a).max()


def test_time_with_thousands_of_gauges_in_a_patch():
    """Single steps and a gather take about twice the launches of four steps on this grid, and each of them a few
    microseconds more for the gauges: five times one gauge's time is well above either way, a scan of all gauges by
    every item that holds some is a hundred times."""
    import torch
    Fm = F()
    nx = ny = 1024
    p = inputs.lake_at_rest(nx, ny)
    s = Fm.Sim(p)

    def best(at):
        out, times = torch.empty((64, len(at)), dtype=torch.float64, device="cuda"), []
        for _ in range(5):
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.run_gauges(64, at, out)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)
    patch = np.stack([400 + np.arange(4096) % 64, 400 + np.arange(4096) // 64], 1)
    assert best(patch) <= 5.0 * best(patch[:1])
    s.close()


def test_time_of_reverse_steps_with_thousands_of_gauges_in_a_patch():
    """A row of the patch takes 64 additions in turn, a few times what the row takes without; a scan of all gauges a row
    took 250 times as long as a step with one gauge."""
    Fm = F()
    s = Fm.Sim(inputs.lake_at_rest(1024, 1024))
    patch = np.stack([400 + np.arange(4096) % 64, 400 + np.arange(4096) // 64], 1)
    s.adjoint_profile(True)
    best = []
    for at in (patch, patch[:1]):
        times = []
        for _ in range(4):
            s.adjoint(16, at, np.ones((16, len(at))), n_checkpoints=16)
            times.append(s.adjoint_times()["reverse_ms"] / 16)
        best.append(min(times))
    assert best[0] <= 8.0 * best[1], best
    s.close()
