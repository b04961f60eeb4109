"""Launches that overlap the end of the one before: the order of everything they read and write, on one
stream with other work in between, on two streams at once, and captured by the caller (exact)."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu


def F():
    import paper_2204_10323_gb300 as F
    return F


def problem(seed, nx=300, ny=70):
    p = inputs.random_small(nx, ny, seed)
    for a in ("z", "n", "h0", "qx0", "qy0"):
        setattr(p, a, getattr(p, a).astype(np.float32).astype(np.float64))
    return p


def alone(p, prec, steps):
    Fm = F()
    s = Fm.Sim(p, precision=prec, kernel=Fm.KERNEL_REFERENCE if prec else Fm.KERNEL_STREAM)
    s.step(steps)
    out = s.state()
    s.close()
    return out


@pytest.mark.parametrize("prec", [0, 1])
def test_two_handles_interleaved_on_one_stream_and_on_two(prec):
    import torch
    Fm = F()
    probs = [problem(1), problem(2, 61, 44)]
    want = [alone(p, prec, 60) for p in probs]
    for streams in ([torch.cuda.current_stream()] * 2, [torch.cuda.Stream(), torch.cuda.Stream()]):
        sims = [Fm.Sim(p, precision=prec, stream=st) for p, st in zip(probs, streams)]
        noise = torch.zeros(1 << 20, device="cuda")
        for k in range(20):
            for s in sims:
                s.step(3)
            noise.add_(1.0)
        for s, w in zip(sims, want):
            for a, b in zip(s.state(), w):
                assert np.array_equal(a, b)
            s.close()


def test_an_epoch_captured_by_the_caller_replays():
    import torch
    Fm = F()
    p = problem(3)
    p.opts.epoch_steps = 8
    st = torch.cuda.Stream()
    s = Fm.Sim(p, stream=st)
    s.step(8)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        s.step(8)                              # two launches of four: the buffers end as they began
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(s.state(), alone(p, 0, 32)):
        assert np.array_equal(a, b)
    del graph
    s.close()
