"""The tile sweep's float pre-test of the fixed-point form: a float estimate
outside [2^46 - M, 2^46 + M) (units of 2^-22 sigma, M the margin of
hd_bounds.h) is on the same side of contact as the exact integer test."""
import numpy as np
import pytest


def margin(W):
    u, R, E = 2.0 ** -24, 0.5 * W, 3.25
    return 2.0 * (4.0 * R * E + 2.0 * E * E + 4.0 * u * (R + E) ** 2)


@pytest.mark.parametrize("w", [2.0, 2.0009, 2.31, 2.78, 2.8284])
def test_estimates_outside_the_band_decide_exactly(w):
    rng = np.random.default_rng(5)
    W = int(round(w * 2 ** 24))
    M = margin(W)
    lo = np.nextafter(np.float32(2.0 ** 46 - M), np.float32(-np.inf))
    hi = np.nextafter(np.float32(2.0 ** 46 + M), np.float32(np.inf))
    n = 400000
    npos = rng.integers(0, W, (n, 2))
    off = rng.integers(-1, 2, (n, 2))
    # half of the pairs within a few units of contact at a random angle, the rest anywhere
    ang = rng.uniform(0, 2 * np.pi, n)
    near = np.rint(npos + 2.0 ** 25 * np.stack([np.cos(ang), np.sin(ang)], 1)).astype(np.int64) + rng.integers(-40, 41, (n, 2))
    q = near - off * W
    away = ((q < 0) | (q >= W)).any(axis=1)
    q[away] = rng.integers(0, W, (int(away.sum()), 2))
    exact = ((q + off * W - npos) ** 2).sum(axis=1) >= 1 << 50
    f = np.float32
    wf = f(0.25 * W)
    img, me = (q >> 2).astype(np.float32), (npos >> 2).astype(np.float32)
    base = np.where(off == 0, me, np.where(off < 0, me + wf, me - wf)).astype(np.float32)
    r = (img - base).astype(np.float32)
    y2 = (r[:, 1] * r[:, 1]).astype(np.float32)
    d2 = (r[:, 0].astype(np.float64) ** 2 + y2.astype(np.float64)).astype(np.float32)  # fused multiply-add: rounded once
    assert (~away).sum() > n // 20
    assert exact[d2 >= hi].all() and not exact[d2 < lo].any()
    band = (d2 >= lo) & (d2 < hi)
    assert 0 < band.sum() < n
