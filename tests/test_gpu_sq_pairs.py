"""The structure factor at wave vectors that share components, at the edges of
its tiles (32 disks, groups of threads, 256 and 512 wave vectors, 160 distinct
components) and with large, negative and repeated components, against the
oracle; a batch of replicas with different lists; and the list that shares too
little, which takes one plane wave per wave vector."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def window(side, h0, k0):
    return [[h0 + i // side, k0 + i % side] for i in range(side * side)]


LISTS = {
    "one": [[3, -7]],
    "origin and repeats": [[0, 0], [5, 2], [5, 2], [-5, -2]],
    "line of 32": [[0, k] for k in range(32)],
    "33": window(6, 10, -3)[:33],
    "128": window(12, -5, 20)[:128],
    "129": window(12, -5, 20)[:129],
    "257": window(17, 1, 1)[:257],
    "513": window(23, -11, 4)[:513],
    "80 + 80 components": [[i, j] for i in range(80) for j in (2 * i % 80, (2 * i + 1) % 80, (i + 40) % 80)],
    "81 + 80 components": [[i % 81, i % 80] for i in range(81 * 3)],
    "grid of 2 x 2": window(2, -1, -1),
    "grid of 3 x 3": window(3, 40, -1),
    "grid of 14 x 14": window(14, 5, -30),
    "grid of 29 x 29": window(29, -14, 3),
    "part of a grid": [[i, k] for i in range(9) for k in range(9) if i + k < 15],
    "grid at the ends": [[2147483646 + i, -2147483648 + k] for i in range(2) for k in range(2)],
    "large": [[100000, -99999], [-2000000000, 3], [7, 2000000000], [100000, 3], [7, -99999]],
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("name", list(LISTS))
def test_structure_factor_lists(oracle_mod, form, name):
    import paper_1211_1645_gb300 as hd
    hk = np.array(LISTS[name])
    for N in (31, 33, 1000):
        g = hd.HardDisks(N, 0.5, 0.3, 3, precision=form)
        g.sweep(10)
        xy, geo = g.positions(), g.geometry()
        S = g.structure_factor(hk)[0]
        # the phases in exact integers: positions and box as multiples of 2^-60 sigma
        X = [[int(c * 2.0 ** 30) * 2 ** 30 + int((c * 2.0 ** 30 % 1.0) * 2.0 ** 30) for c in row] for row in xy]
        L = int(geo["L"] * 2.0 ** 30) * 2 ** 30 + int((geo["L"] * 2.0 ** 30 % 1.0) * 2.0 ** 30)
        for q, (h, k) in enumerate(hk):
            t = np.array([((int(h) * x + int(k) * y) % L) / L for x, y in X])
            want = abs(np.exp(2j * np.pi * t).sum()) ** 2 / N
            # FP64 input bits below 2^-60 are dropped above; the direct form's double phase errs by (|h| + |k|) 2^-50 turns
            phase = (abs(int(h)) + abs(int(k))) * (2.0 ** -50 if form == "fp64" else 0.0) + 1e-14
            assert abs(S[q] - want) <= 2 * np.pi * phase * 2 * np.sqrt(N * max(want, 1.0)) + 1e-11
        g.close()


@pytest.mark.parametrize("form", ["fixed", "fp64"])
def test_structure_factor_of_a_batch(oracle_mod, form):
    import paper_1211_1645_gb300 as hd
    Ns = [400, 1000, 64]
    g = hd.HardDisks(Ns, [0.6] * 3, [0.2] * 3, [1, 2, 3], precision=form)
    g.sweep(8)
    rng = np.random.default_rng(2)
    hk = np.stack([rng.integers(-w, w + 1, (90, 2)) for w in (4, 9, 2)])
    S = g.structure_factor(hk)
    xy, off = g.positions(), 0
    for r, n in enumerate(Ns):
        want = oracle_mod.structure_factor(xy[off:off + n], hk[r], g.geometry(r)["L"])
        assert np.abs(S[r] - want).max() <= 1e-10 * max(1.0, want.max())
        off += n
    g.close()
