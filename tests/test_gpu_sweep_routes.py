"""Which systems run their sweeps as one launch, on both sides of the rules on
disks per cell and on tiles per SM, and that either route makes the chain of
the serial split kernels (exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import paper_1211_1645_gb300 as hd
    hd.load()
    return hd


# (form, N per replica, cell_min, sweeps run as one launch)
CASES = [("fixed", [1000000], 2.2, False), ("fixed", [262144], 2.2, True), ("fixed", [1000000], 2.0, True),
         ("fp64", [524288], 2.6, False), ("fp64", [131072], 2.6, True), ("fixed", [100000] * 10, 2.0, False),
         ("fixed", [100000] * 3, 2.0, True), ("fixed", [20000] * 17, 2.0, True)]


@pytest.mark.parametrize("form,Ns,cell_min,one", CASES)
def test_route_and_chain(hd, form, Ns, cell_min, one):
    R = len(Ns)
    out = []
    for kw in ({}, {"strips": 1, "replica_branches": 1}):
        g = hd.HardDisks(Ns, [0.70] * R, [0.15] * R, list(range(2, 2 + R)), precision=form, cell_min=cell_min, **kw)
        g.run(1, 3, measure=False)
        assert (g.kernel_times()["sweep"][1] > 0) == (one and not kw)
        out.append((g.positions(), g.stats()))
        g.close()
    assert np.array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)
