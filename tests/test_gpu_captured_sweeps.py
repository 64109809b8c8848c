"""Sweeps that the caller captures into a graph of its own, replayed between calls of
either order of the launches: the chain is that of the same sweeps called one
after the other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns", [[4096], [1300] * 114, [300] * 320])
@pytest.mark.parametrize("captured", [(1, 1), (24,)])
def test_replays_between_calls(form, Ns, captured):
    import torch

    import paper_1211_1645_gb300 as hd
    R = len(Ns)
    eta = 0.69 if Ns[0] >= 700 else 0.60
    args = (Ns, [eta] * R, [0.15] * R, list(range(2, 2 + R)))
    stream = torch.cuda.Stream()
    g = hd.HardDisks(*args, precision=form)
    ref = hd.HardDisks(*args, precision=form, strips=1, replica_branches=1)
    g.set_stream(stream.cuda_stream)
    for x in (g, ref):
        x.sweep(1)
        x.sweep(24)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for n in captured:
            g.sweep(n)
    done = 25
    with torch.cuda.stream(stream):
        for n in (0, 2, 1, 1, 24, 0, 2):  # an even number of sweeps each time, as the graph was captured
            if n == 1:
                g.sweep(1)
                g.sweep(1)
            elif n:
                g.sweep(n)
            graph.replay()
            done += (2 if n == 1 else n) + sum(captured)
    ref.sweep(done - 25)
    assert np.array_equal(g.positions(), ref.positions())
    assert all(np.array_equal(a, b) for a, b in zip(g.stats(), ref.stats()))
    g.close()
    ref.close()
