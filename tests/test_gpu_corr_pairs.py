"""The positional correlation from unordered pairs at the edges of its kernel's
range: one window, windows narrower than sigma, as many as fit 128, 64 and 32
threads' sums and the first count beyond (which takes the ordered-pair kernel),
a perfect lattice whose distances fall on window edges, capacity-9 cells,
overlapping disks and a batch, against the oracle's plain pair sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def check(oracle_mod, xy, hk0, L, nr, dr, C):
    want = oracle_mod.positional_corr(xy, hk0, L, (np.arange(nr) + 1) * dr)
    empty = np.isnan(want.real)
    assert np.array_equal(np.isnan(C.real), empty)
    # means of unit vectors: phases to (|h| + |k|) 2^-50 turns, sums of at most N^2 terms to N^2 eps
    tol = 2 * np.pi * np.abs(hk0).sum() * 2.0 ** -50 + 1e-11
    assert np.abs(C[~empty] - want[~empty]).max(initial=0.0) <= tol


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("nr, dr", [(1, 3.0), (7, 0.05), (36, 0.3), (37, 0.3), (74, 0.11), (75, 0.11), (148, 0.05),
                                    (149, 0.05), (150, 0.05), (1, 1e-42)])
def test_window_counts(oracle_mod, form, nr, dr):
    import paper_1211_1645_gb300 as hd
    g = hd.HardDisks(900, 0.6, 0.3, 5, precision=form)
    g.sweep(20)
    hk0 = np.array([11, -17])
    check(oracle_mod, g.positions(), hk0, g.geometry()["L"], nr, dr, g.positional_corr(hk0, nr, dr)[0])
    g.close()


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("cell_min", [2.0, 3.0])
def test_lattice_and_overlapping_input(oracle_mod, form, cell_min):
    import paper_1211_1645_gb300 as hd
    N = 1024
    g = hd.HardDisks(N, 0.5, 0.3, 5, precision=form, cell_min=cell_min)
    L = g.geometry()["L"]
    hk0 = np.array([32, 0])
    a = L / 32  # the lattice spacing: windows whose edges r +- sigma are lattice distances
    C = g.positional_corr(hk0, 8, (a - 1.0) / 2)[0]
    assert np.abs(C[~np.isnan(C.real)] - 1.0).max() <= 1e-10
    xy = np.random.default_rng(1).uniform(0, L, (N, 2))
    xy[:2] = xy[2:4]  # two pairs of coincident disks
    try:
        g.set_positions(xy)
    except Exception:  # more disks in a cell than its capacity: thin them out
        side = np.arange(32) * a
        xy = np.stack(np.meshgrid(side, side), -1).reshape(-1, 2) + np.random.default_rng(2).uniform(0, 0.9, (N, 2))
        xy[1] = xy[0]
        g.set_positions(xy)
    check(oracle_mod, g.positions(), np.array([3, 5]), L, 20, 0.4, g.positional_corr([3, 5], 20, 0.4)[0])
    g.close()


def test_batch_and_radius(oracle_mod):
    import paper_1211_1645_gb300 as hd
    Ns = [900, 1600, 1024]
    g = hd.HardDisks(Ns, [0.6] * 3, [0.2] * 3, [1, 2, 3], precision="fixed")
    g.sweep(10)
    hk0 = np.array([[5, 3], [-4, 9], [0, 7]])
    C = g.positional_corr(hk0, 15, 0.4)
    xy, off = g.positions(), 0
    for r, n in enumerate(Ns):
        check(oracle_mod, xy[off:off + n], hk0[r], g.geometry(r)["L"], 15, 0.4, C[r])
        off += n
    g.close()
    out = []
    for sigma in (1.0, 2.0, 0.5):  # the same chain in other units of length
        g = hd.HardDisks(1600, 0.6, 0.2 * sigma, 4, sigma=sigma, precision="fixed")
        g.sweep(10)
        out.append(g.positional_corr([6, 2], 10, 0.5 * sigma)[0])
        g.close()
    for C in out[1:]:
        assert np.abs(C[2:] - out[0][2:]).max() <= 1e-11
