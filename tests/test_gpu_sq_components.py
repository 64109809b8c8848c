"""The structure factor's choice of way by the components of its wave vectors: on
both sides of its rules, in any order, with repeated wave vectors, and replicas
of different lists, each equal to the sum over the disks; and looking a list
over costs less than its sums."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import paper_1211_1645_gb300 as hd
    hd.load()
    return hd


def grid(h0, k0, nh, nk):
    return np.stack(np.meshgrid(np.arange(nh) + h0, np.arange(nk) + k0, indexing="ij"), -1).reshape(-1, 2)


RNG = np.random.default_rng(8)
LISTS = {
    "one": np.array([[3, -5]]),
    "grid": grid(-4, 7, 9, 11),
    "grid shuffled": RNG.permutation(grid(-4, 7, 9, 11)),
    "grid with repeats": np.concatenate([grid(2, 2, 6, 6), grid(2, 2, 6, 6)[::-3]]),
    "grid with gaps": 3 * grid(-5, 1, 9, 9),
    "line": np.stack([np.arange(80) - 40, np.zeros(80, int)], 1),
    "160 components": grid(0, -20, 80, 80)[::3],
    "161 components": grid(0, -20, 80, 81),
    "scattered": RNG.integers(-30, 31, (1500, 2)),
    "far apart": RNG.integers(-2000, 2001, (600, 2)),
    "steps of 512": np.stack([512 * 7 * np.arange(40), 1024 * np.arange(40) - 20000], 1),
}


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("N", [100, 127, 128, 400])
@pytest.mark.parametrize("name", list(LISTS))
def test_lists(hd, oracle_mod, form, N, name):
    hk = LISTS[name]
    g = hd.HardDisks(N, 0.6, 0.2, 3, precision=form)
    g.sweep(10)
    S = g.structure_factor(hk)[0]
    want = oracle_mod.structure_factor(g.positions(), hk, g.geometry()["L"])
    g.close()
    # amplitudes of N unit vectors whose phases err by (|h| + |k|) 2^-49 turns in the plain sum
    tol = 2 * N * (2 * np.pi * np.abs(hk).sum(1) * 2.0 ** -49 + 1e-13)
    assert np.all(np.abs(S - want) <= tol)


def test_replicas_of_different_lists(hd, oracle_mod):
    Ns = [400, 256, 900]
    g = hd.HardDisks(Ns, [0.6] * 3, [0.2] * 3, [1, 2, 3])
    g.sweep(5)
    xy, off = g.positions(), np.cumsum([0] + Ns)
    lists = [LISTS["grid"], LISTS["grid"] * [1, 2], np.repeat([[4, -4]], 99, 0)]
    for order in ((0, 1, 2), (2, 1, 0), (2, 2, 0), (0, 0, 0)):
        hk = np.stack([lists[i] for i in order])
        S = g.structure_factor(hk)
        for r in range(3):
            want = oracle_mod.structure_factor(xy[off[r]:off[r + 1]], hk[r], g.geometry(r)["L"])
            assert np.abs(S[r] - want).max() <= 1e-9 * max(1.0, want.max())
    g.close()


def test_a_list_beyond_the_limit_is_refused(hd):
    from paper_1211_1645_gb300.hd import HD_ERR_ARG
    R = 300  # 300 x 12 x 65536 partial sums
    g = hd.HardDisks([3000] * R, [0.6] * R, [0.2] * R, list(range(R)))
    with pytest.raises(hd.HDError) as e:
        g.structure_factor(np.zeros((65536, 2), np.int32))
    assert e.value.status == HD_ERR_ARG
    assert np.allclose(g.structure_factor(np.zeros((3, 2), np.int32)), 3000.0)
    g.close()


def timed(f):
    t = time.perf_counter()
    f()
    return time.perf_counter() - t


def test_long_scattered_list_of_a_small_system(hd):
    """30,000 wave vectors without shared components and 36 disks: about 0.5 ms of
    sums and copies, where sorting the list's components took another 2 ms."""
    hk = np.random.default_rng(1).integers(-30000, 30001, (30000, 2)).astype(np.int32)
    g = hd.HardDisks(36, 0.6, 0.2, 3)
    best = min(timed(lambda: g.structure_factor(hk)) for _ in range(30))
    g.close()
    assert best < 1.2e-3
