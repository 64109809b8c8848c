"""The positional correlation with a length unit other than the disk radius:
the windows' reach follows from dr in units of sigma, so that no pair of the
outer windows is left out (sigma < 1) and no window that fits the box is
refused (sigma > 1), and a window far beyond the box is refused whatever its
size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("sigma, nr, dr", [(0.5, 20, 0.25), (0.5, 36, 0.25), (0.25, 150, 0.025), (2.0, 42, 1.0),
                                           (2.0, 20, 1.0), (16.0, 5, 6.0)])
def test_windows_in_other_units(oracle_mod, form, sigma, nr, dr):
    import paper_1211_1645_gb300 as hd
    g = hd.HardDisks(1600, 0.6, 0.2 * sigma, 4, sigma=sigma, precision=form)
    g.sweep(10)
    hk0 = np.array([6, 2])
    C = g.positional_corr(hk0, nr, dr)[0]
    want = oracle_mod.positional_corr(g.positions() / sigma, hk0, g.geometry()["L"], (np.arange(nr) + 1) * (dr / sigma))
    g.close()
    empty = np.isnan(want.real)
    assert np.array_equal(np.isnan(C.real), empty) and not empty.all()
    # means of unit vectors: phases to (|h| + |k|) 2^-50 turns, sums of at most N^2 terms to N^2 eps
    tol = 2 * np.pi * np.abs(hk0).sum() * 2.0 ** -50 + 1e-11
    assert np.abs(C[~empty] - want[~empty]).max(initial=0.0) <= tol


@pytest.mark.parametrize("sigma, dr", [(1.0, 50.0), (0.5, 25.0), (2.0, 100.0), (1.0, 1e12), (1.0, 1e300), (1e-3, 1e306),
                                       (1.0, float("inf"))])
def test_windows_beyond_the_box_are_refused(sigma, dr):
    import paper_1211_1645_gb300 as hd
    from paper_1211_1645_gb300.hd import HD_ERR_REACH
    g = hd.HardDisks(256, 0.6, 0.1 * sigma, 4, sigma=sigma)
    with pytest.raises(hd.HDError) as e:
        g.positional_corr([1, 0], 2, dr)
    assert e.value.status == HD_ERR_REACH
    g.close()
