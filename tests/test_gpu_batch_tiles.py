"""Tiles of a batch that does not fill the GPU, split by each replica's share of
the idle SMs, against the oracle (exact): equal replicas, replicas of very
different sizes, more replicas than shares, and an odd share."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import paper_1211_1645_gb300 as hd
    hd.load()
    return hd


CASES = {
    "two": ([1500, 1500], 10),
    "very different": ([256, 1024, 20000], 8),
    "odd shares": ([3001, 5000, 1200, 9001, 2111], 8),
    "many": ([1300] * 37 + [2500], 5),
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("case", list(CASES))
def test_batches_on_shared_tiles_match_the_oracle(hd, oracle_mod, form, case):
    Ns, sweeps = CASES[case]
    R = len(Ns)
    g = hd.HardDisks(Ns, [0.69] * R, [0.2] * R, list(range(3, 3 + R)), precision=form)
    g.run(1, sweeps, measure=False)
    xy, (att, acc) = g.positions(), g.stats()
    off = 0
    for r, n in enumerate(Ns):
        o = oracle_mod.OracleChain(n, 0.69, 0.2, 3 + r, form=form)
        o.sweep(sweeps)
        assert (int(att[r]), int(acc[r])) == o.stats()
        assert np.array_equal(xy[off:off + n], o.positions())
        off += n
    g.close()
