"""Whole-box sweeps beyond 400 disks and hard cells from registers against the
oracle, every position and count exact: the sizes on both sides of each rule
(one replica fixed and FP64, several replicas), several trials per cell, and
cells so wide that crowded ones exceed the shared pool and the hard lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import paper_1211_1645_gb300 as hd
    hd.load()
    return hd


# (N per replica, eta, delta, cell_min, trials per cell, sweeps)
CASES = {
    "22 cells a side": ([500], 0.70, 0.2, 2.0, 0, 30),
    "28 cells a side": ([700], 0.70, 0.2, 2.0, 0, 30),
    "30 cells a side": ([900], 0.70, 0.2, 2.0, 0, 30),
    "32 cells a side": ([1024], 0.70, 0.2, 2.0, 0, 30),
    "three trials": ([800], 0.66, 0.3, 2.0, 3, 15),
    "crowded, 20 cells": ([698], 0.70, 0.2, 2.78, 0, 12),
    "crowded, 28 cells": ([1369], 0.70, 0.2, 2.78, 0, 12),
    "crowded, 32 cells": ([1789], 0.70, 0.2, 2.78, 2, 12),
    "boxes of all sizes": ([1024, 40, 900, 256], 0.62, 0.3, 2.0, 0, 25),
    "crowded boxes": ([1572, 698], 0.70, 0.2, 2.78, 0, 9),
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("case", list(CASES))
def test_whole_boxes_match_the_oracle(hd, oracle_mod, form, case):
    Ns, eta, delta, cell_min, nt, sweeps = CASES[case]
    R = len(Ns)
    g = hd.HardDisks(Ns, [eta] * R, [delta] * R, list(range(7, 7 + R)), precision=form, cell_min=cell_min,
                     trials_per_cell=nt)
    g.sweep(1)
    g.run(1, sweeps, measure=False)
    xy, (att, acc) = g.positions(), g.stats()
    off = 0
    for r, n in enumerate(Ns):
        o = oracle_mod.OracleChain(n, eta, delta, 7 + r, form=form, cell_min=cell_min, nt=nt)
        o.sweep(sweeps + 1)
        assert (int(att[r]), int(acc[r])) == o.stats()
        assert np.array_equal(xy[off:off + n], o.positions())
        off += n
    g.close()
