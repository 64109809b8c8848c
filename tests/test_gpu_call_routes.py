"""Which calls run their sweeps as one launch: both sides of the rules on the sweeps
of a call, the replicas and the rounds of boxes or tiles the SMs take, where
the launches per phase are the faster; and the chain of a context whose calls
change from one order to the other, with everything between them that touches
the cells, equal to the serial split kernels' (exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    import torch

    import paper_1211_1645_gb300 as hd
    hd.load()
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the rules count in SMs")
    return hd


# form, N, replicas, cell_min, call, sweeps, one launch
CASES = [
    ("fixed", 4096, 1, 2.0, "run", 1, False), ("fixed", 4096, 1, 2.0, "run", 2, True), ("fp64", 4096, 1, 2.0, "run", 1, True),
    ("fixed", 4096, 1, 2.0, "sweep", 1, True), ("fixed", 1000000, 1, 2.0, "run", 2, False),
    ("fixed", 800000, 1, 2.0, "sweep", 1, False), ("fixed", 800000, 1, 2.0, "sweep", 2, True),
    ("fixed", 1048576, 1, 2.0, "sweep", 1, True), ("fixed", 16384, 16, 2.5, "run", 2, False),
    ("fixed", 16384, 8, 2.5, "run", 2, True), ("fixed", 1000000, 1, 2.0, "run", 3, True), ("fp64", 524288, 1, 2.0, "sweep", 1, False),
    # more tiles than the SMs take in a few rounds
    ("fixed", 1300, 70, 2.0, "run", 24, True), ("fixed", 1300, 200, 2.0, "run", 24, False),
    ("fixed", 1300, 114, 2.0, "sweep", 24, True), ("fixed", 1300, 200, 2.0, "sweep", 24, False),
    ("fixed", 1300, 64, 2.0, "run", 24, True), ("fp64", 1300, 100, 2.0, "run", 12, True), ("fp64", 1300, 152, 2.0, "run", 12, False),
    ("fixed", 16384, 64, 2.0, "run", 1, True), ("fixed", 40000, 31, 2.0, "run", 12, False),
    ("fixed", 40000, 31, 2.0, "sweep", 12, True), ("fp64", 65536, 8, 2.0, "run", 12, False),
    ("fp64", 65536, 8, 2.0, "sweep", 12, True), ("fixed", 16384, 31, 2.5, "run", 12, False),
    ("fixed", 4096, 31, 2.5, "run", 12, True),
    # boxes
    ("fixed", 36, 600, 2.0, "run", 24, True), ("fixed", 36, 800, 2.0, "run", 24, False),
    ("fixed", 36, 800, 2.0, "sweep", 24, True), ("fixed", 36, 800, 2.0, "sweep", 1, False),
    ("fp64", 36, 760, 2.0, "run", 24, True), ("fp64", 36, 1000, 2.0, "run", 24, False), ("fp64", 1000, 1000, 2.0, "run", 3, True),
    ("fixed", 400, 608, 2.5, "run", 12, False),
]


@pytest.mark.parametrize("form,N,R,cell_min,call,n,one", CASES)
def test_route(hd, form, N, R, cell_min, call, n, one):
    eta = 0.70 if N >= 1000 else 0.60
    g = hd.HardDisks([N] * R, [eta] * R, [0.1] * R, list(range(R)), precision=form, cell_min=cell_min)
    if call == "run":
        g.run(1, n, measure=False)
    else:
        g.sweep(n)
    assert (g.kernel_times()["sweep"][1] > 0) == one
    g.stats()  # and no error on the device
    g.close()


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns", [[4096], [700], [262144], [1300] * 100, [300] * 320, [20000, 3000, 900]])
def test_chain_over_changing_routes(hd, form, Ns):
    R = len(Ns)
    eta = 0.69 if min(Ns) >= 700 else 0.60
    args = (Ns, [eta] * R, [0.15] * R, list(range(2, 2 + R)))
    g = hd.HardDisks(*args, precision=form)
    ref = hd.HardDisks(*args, precision=form, strips=1, replica_branches=1)
    both = (g, ref)

    def same():
        assert np.array_equal(g.positions(), ref.positions())
        assert all(np.array_equal(a, b) for a, b in zip(g.stats(), ref.stats()))

    for k, (call, n) in enumerate([("run", 1), ("sweep", 3), ("run", 1), ("run", 6), ("sweep", 1), ("run", 2), ("sweep", 2),
                                   ("run", 1), ("profile", 2), ("sweep", 5), ("profile", 1), ("run", 25)]):
        for x in both:
            if call == "sweep":
                x.sweep(n)
            else:
                x.profile(call == "profile")
                x.run(2, n, measure=False)
                x.profile(False)
        if k % 3 == 2:
            same()
        if k == 3:
            blob = g.checkpoint()
        if k == 5:  # back to an earlier state, from the route in use to the other
            for x in both:
                x.restore(blob)
        if k == 7:
            xy = ref.positions()
            for x in both:
                x.set_positions(xy)
        if k == 8:
            for x in both:
                with pytest.raises(hd.HDError):
                    x.set_positions(np.full_like(xy, np.nan))
    same()
    psi = [x.psi6(False)[0] for x in both]
    assert np.array_equal(*psi)
    g.close()
    ref.close()
