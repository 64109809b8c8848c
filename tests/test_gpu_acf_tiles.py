"""The Psi_6 autocorrelation at the edges of its tiles of lags (128) and chunks
of times (128): one entry, one lag short of and beyond a tile, the longest lag,
and a series of several chunks, against the oracle's plain sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T, max_lag", [(1, 0), (127, 126), (128, 127), (129, 128), (300, 299), (1000, 257), (9000, 3)])
def test_acf_at_tile_edges(oracle_mod, T, max_lag):
    import paper_1211_1645_gb300 as hd
    R = 2
    g = hd.HardDisks([64] * R, [0.6] * R, [0.2] * R, [7, 8], precision="fixed")
    g.series_reserve(T)
    g.run(T, 1, True)
    s = g.series()
    psi = s[:, :, 2] + 1j * s[:, :, 3]
    C = g.psi6_acf(max_lag)
    for r in range(R):
        want = oracle_mod.psi6_acf(psi[:, r], max_lag)
        assert C[r, 0] == 1.0
        # sums of T products of magnitude <= 1 relative to <|psi|^2> T: T eps each side, and the division's few eps
        tol = 4 * T * np.finfo(float).eps / np.mean(np.abs(psi[:, r]) ** 2)
        assert np.abs(C[r] - want).max() <= tol
    g.close()
