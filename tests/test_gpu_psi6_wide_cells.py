"""psi_6 where cells hold up to nine disks, so that every disk takes the general
search: tied, nearly tied and relaxed neighbours against the oracle bit for
bit (the float pre-test may leave out only candidates beyond the sixth)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("N, eta, cell_min", [(256, 0.70, 2.9), (1024, 0.5, 3.3), (3000, 0.71, 3.9)])
@pytest.mark.parametrize("noise", [0.0, 2.0 ** -24, 1e-5, None])
def test_wide_cells_match_the_oracle(oracle_mod, form, N, eta, cell_min, noise):
    import paper_1211_1645_gb300 as hd
    g = hd.HardDisks(N, eta, 0.2, 3, precision=form, cell_min=cell_min)
    o = oracle_mod.OracleChain(N, eta, 0.2, 3, form=form, cell_min=cell_min)
    assert g.geometry()["capacity"] == 9
    if noise is None:  # a relaxed configuration
        g.sweep(30)
        o.sweep(30)
    elif noise:
        xy = g.positions()
        xy += np.random.default_rng(N).choice([-noise, 0.0, noise], xy.shape)
        g.set_positions(xy)
        o.set_positions(xy)
    glob, loc = g.psi6()
    want, wglob = o.psi6()
    assert np.array_equal(loc, want)
    assert glob[0] == wglob
    g.close()
