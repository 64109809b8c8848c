"""Binning of caller positions at the edges of the division-free path of the
FP64 form (coordinates on, and a few roundings around, cell boundaries), and
the contact histogram with pairs on its bin edges, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("N, eta", [(400, 0.30), (1000, 0.25)])
def test_coordinates_around_cell_boundaries(oracle_mod, form, N, eta):
    import paper_1211_1645_gb300 as hd
    g = hd.HardDisks(N, eta, 0.1, 3, precision=form)
    o = oracle_mod.OracleChain(N, eta, 0.1, 3, form=form)
    geo = g.geometry()
    L, w, m = geo["L"], geo["w"], geo["m"]
    rng = np.random.default_rng(N)
    xy = g.positions()
    pick = rng.random(N) < 0.7
    for c in range(2):  # the nearest boundary, shifted by nothing, a few ulps, or about 2^-30 of a cell
        edge = np.rint(xy[:, c] / w) * w
        step = rng.choice([0.0, 1.0, -1.0, 3.0, -2.0, 2.0 ** 21, -2.0 ** 21, 2.0 ** 24], N) * np.spacing(np.maximum(edge, w))
        xy[pick, c] = (edge + step)[pick]
    xy[0] = [0.0, -0.0]
    xy[1] = [L, np.nextafter(L, 0)]
    xy[2] = [-L * 2 + 1.0, L * 3 + 2.0]
    try:
        o.set_positions(xy)
    except Exception:
        pytest.skip("more disks in a cell than its capacity")
    g.set_positions(xy)
    assert np.array_equal(g.positions(), o.positions())
    assert np.array_equal(g.pressure()[2][0], o.histogram(50, 1e-3))
    g.sweep(3)
    o.sweep(3)
    assert np.array_equal(g.positions(), o.positions())
    g.close()


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("bins, dr, cell_min", [(5, 0.25, 2.0), (50, 0.0625, 2.0), (512, 2.0 ** -8, 2.0), (7, 0.5, 3.0), (40, 0.2, 2.0)])
def test_histogram_with_pairs_on_bin_edges(oracle_mod, form, bins, dr, cell_min):
    import paper_1211_1645_gb300 as hd
    N = 1600
    g = hd.HardDisks(N, 0.55, 0.2, 5, precision=form, hist_bins=bins, hist_dr=dr, cell_min=cell_min)
    o = oracle_mod.OracleChain(N, 0.55, 0.2, 5, form=form, cell_min=cell_min)
    L = g.geometry()["L"]
    side = np.arange(40)
    # spacings that are multiples of 2^-6: many distances exactly on an edge
    xy = np.stack(np.meshgrid(side * 2.25 + 0.125, side * 2.25 + 0.125), -1).reshape(-1, 2)
    xy[::3, 0] += 0.25 * np.random.default_rng(1).integers(0, 2, len(xy[::3]))
    assert xy.max() + 2.25 < L
    g.set_positions(xy)
    o.set_positions(xy)
    assert np.array_equal(g.pressure()[2][0], o.histogram(bins, dr))
    g.sweep(5)
    o.sweep(5)
    assert np.array_equal(g.pressure()[2][0], o.histogram(bins, dr))
    g.close()
