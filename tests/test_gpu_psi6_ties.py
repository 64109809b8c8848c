"""psi_6 where the float search must hand over to the exact one: sixth and
seventh neighbours at equal or nearly equal distance, equal distances within
the six, three and four disks in a cell, neighbours beyond the stencil, and
boxes narrower and wider than a tile, against the oracle bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def compare(g, o):
    glob, loc = g.psi6()
    want, wglob = o.psi6()
    assert np.array_equal(loc, want)
    assert glob[0] == wglob


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("N, eta", [(256, 0.70), (1024, 0.5), (1089, 0.72), (65, 0.2)])
@pytest.mark.parametrize("noise", [0.0, 2.0 ** -24, 1e-6, 1e-5, 0.05])
def test_nearly_tied_neighbours(oracle_mod, form, N, eta, noise):
    import paper_1211_1645_gb300 as hd
    g = hd.HardDisks(N, eta, 0.1, 3, precision=form)
    o = oracle_mod.OracleChain(N, eta, 0.1, 3, form=form)
    if noise:
        xy = g.positions()
        xy += np.random.default_rng(N).choice([-noise, 0.0, noise], xy.shape)
        g.set_positions(xy)
        o.set_positions(xy)
    compare(g, o)
    g.close()


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("cell_min", [2.0, 2.8])
def test_crowded_and_repeated_after_an_error(oracle_mod, form, cell_min):
    import paper_1211_1645_gb300 as hd
    N = 3000
    g = hd.HardDisks(N, 0.70, 0.3, 3, precision=form, cell_min=cell_min)
    o = oracle_mod.OracleChain(N, 0.70, 0.3, 3, form=form, cell_min=cell_min)
    for _ in range(2):  # the sums start at zero each time
        g.sweep(15)
        o.sweep(15)
        compare(g, o)
    small = hd.HardDisks(5, 0.05, 0.1, 1, precision=form)
    for _ in range(2):
        with pytest.raises(hd.HDError):
            small.psi6()
    small.close()
    compare(g, o)
    g.close()
