"""Steps of one to three sweeps, whose few kernels follow one another closely: each
launch reads what the one before it wrote, never what was there before, with
every sweep kernel, as strips and branches, on the default and on a created
stream.  Exact against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OPTIONS = {
    "split": {"strips": 1, "replica_branches": 1},
    "strips": {"strips": 3},
    "branches": {},
    "wide cells": {"cell_min": 3.0},
    "two threads a cell": {"threads_per_cell": 2},
    "bulk copies": {"sweep_kernel": "tma"},
    "fused": {"sweep_kernel": "fused"},
    "persistent": {"sweep_kernel": "persistent"},
    "chosen by the library": {},
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns", [[700], [4096], [700, 1024], [20000]])
@pytest.mark.parametrize("name", list(OPTIONS))
def test_short_steps_match_the_oracle(oracle_mod, form, Ns, name):
    import torch

    import paper_1211_1645_gb300 as hd
    kw = OPTIONS[name]
    if (name == "strips" and len(Ns) > 1) or (name == "branches" and len(Ns) == 1):
        pytest.skip("one replica" if name == "strips" else "several replicas")
    R = len(Ns)
    chains = [oracle_mod.OracleChain(n, 0.69, 0.15, 2 + r, form=form, cell_min=kw.get("cell_min", 2.0)) for r, n in enumerate(Ns)]
    stream = torch.cuda.Stream()
    g = hd.HardDisks(Ns, [0.69] * R, [0.15] * R, list(range(2, 2 + R)), precision=form, **kw)
    for call in (lambda: g.run(1, 1, False), lambda: g.run(3, 1, False), lambda: g.run(2, 2, False),
                 lambda: g.set_stream(stream.cuda_stream), lambda: g.run(3, 1, False), lambda: g.run(2, 1, True),
                 lambda: g.sweep(1), lambda: [g.sweep(1) for _ in range(3)], lambda: g.run(2, 3, False)):
        before = g.geometry()["sweeps"]
        call()
        xy, (att, acc), off = g.positions(), g.stats(), 0
        for r, o in enumerate(chains):
            o.sweep(g.geometry()["sweeps"] - before)
            assert np.array_equal(xy[off:off + Ns[r]], o.positions())
            assert (int(att[r]), int(acc[r])) == o.stats()
            off += Ns[r]
    g.close()
