"""The one-launch sweeps (whole small boxes, tiles of cells) against the
oracle, at the sizes where their geometry changes: the smallest box, the
largest box kept in one block and the first beyond it, tiles of one and of
several per axis, ragged counts, several trials per cell, crowded cells beyond
the shared pool, and batches that mix tile heights."""
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
    "smallest box": ([20], 0.30, 0.4, 2.0, 0, 40),
    "box of 20 cells": ([390], 0.70, 0.2, 2.0, 0, 30),
    "first on one tile": ([400], 0.66, 0.2, 2.0, 0, 30),
    "first on two tiles an axis": ([600], 0.70, 0.2, 2.0, 0, 30),
    "ragged": ([10007], 0.71, 0.15, 2.0, 0, 12),
    "trials": ([3001], 0.70, 0.2, 2.0, 3, 12),
    "boxes": ([256, 300, 121], 0.60, 0.3, 2.0, 0, 30),
    "mixed tile heights": ([256, 1024, 3000, 16384, 400], 0.66, 0.2, 2.0, 0, 12),
    "crowded beyond the pool": ([40000, 9000], 0.70, 0.2, 2.78, 0, 6),
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("case", list(CASES))
def test_one_launch_sweeps_match_the_oracle(hd, oracle_mod, form, case):
    Ns, eta, delta, cell_min, nt, sweeps = CASES[case]
    R = len(Ns)
    g = hd.HardDisks(Ns, [eta] * R, [delta] * R, list(range(41, 41 + R)), precision=form, cell_min=cell_min,
                     trials_per_cell=nt)
    launches = g.kernel_times()["sweep"][1]
    g.sweep(1)
    g.run(2, sweeps, measure=False)
    g.sweep(2)
    assert g.kernel_times()["sweep"][1] - launches == 4
    xy, (att, acc) = g.positions(), g.stats()
    off = 0
    for r, n in enumerate(Ns):
        o = oracle_mod.OracleChain(n, eta, delta, 41 + r, form=form, cell_min=cell_min, nt=nt)
        o.sweep(2 * sweeps + 3)
        assert (int(att[r]), int(acc[r])) == o.stats()
        assert np.array_equal(xy[off:off + n], o.positions())
        off += n
    # profiled steps run the split kernels on the same state and continue the chain
    g.profile(True)
    g.run(1, 3, measure=False)
    assert g.kernel_times()["pass"][1] == 12
    g.profile(False)
    g.sweep(2)
    ref = hd.HardDisks(Ns, [eta] * R, [delta] * R, list(range(41, 41 + R)), precision=form, cell_min=cell_min,
                       trials_per_cell=nt, strips=1, replica_branches=1)
    ref.sweep(2 * sweeps + 8)
    assert np.array_equal(g.positions(), ref.positions())
    assert all(np.array_equal(a, b) for a, b in zip(g.stats(), ref.stats()))
    g.close()
    ref.close()
