"""Positions read out through a block's list of its disks, exact against the
oracle: block widths, a ragged last block, cells of up to nine disks, a sigma
other than one, and several replicas."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import paper_1211_1645_gb300 as hd
    hd.load()
    return hd


# (N per replica, sigma, cell_min, block_threads)
CASES = [([20], 1.0, 2.0, 128), ([500], 1.0, 2.0, 32), ([1000], 0.37, 2.0, 256), ([4000], 1.0, 2.75, 96),
         ([3001], 1.7, 3.1, 128), ([300, 20, 5000], 2.0, 2.0, 64)]


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns,sigma,cell_min,threads", CASES)
def test_positions_match_the_oracle(hd, oracle_mod, form, Ns, sigma, cell_min, threads):
    R = len(Ns)
    eta = 0.3 if min(Ns) <= 20 else 0.6
    g = hd.HardDisks(Ns, [eta] * R, [0.25 * sigma] * R, list(range(5, 5 + R)), sigma=sigma, precision=form,
                     cell_min=cell_min, block_threads=threads)
    g.sweep(3)
    xy = g.positions()
    off = 0
    for r, n in enumerate(Ns):
        o = oracle_mod.OracleChain(n, eta, 0.25, 5 + r, form=form, cell_min=cell_min)
        o.sweep(3)
        assert np.array_equal(xy[off:off + n], sigma * o.positions())
        off += n
    g.close()
