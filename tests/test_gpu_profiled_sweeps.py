"""hd_sweep while profiling: the launches it times are the ones it makes without
profiling (the sweeps of a draw table in one launch where the library chooses
the order), and the chain is the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns", [[256], [1000], [4096], [400, 576], [4096, 6400]])  # boxes, tiles, batches of both
@pytest.mark.parametrize("n", [1, 7, 260])
def test_profiled_sweeps_are_those_that_run(form, Ns, n):
    import paper_1211_1645_gb300 as hd
    R = len(Ns)
    a, b = (hd.HardDisks(Ns, [0.70] * R, [0.1] * R, list(range(5, 5 + R)), precision=form) for _ in range(2))
    before = {k: v[1] for k, v in b.kernel_times().items()}
    b.sweep(n)
    made = {k: v[1] - before[k] for k, v in b.kernel_times().items()}
    a.profile(True)
    a.sweep(n)
    kt = a.kernel_times()
    a.profile(False)
    assert {k: v[1] for k, v in kt.items()} == made and made["sweep"] == -(-n // 256)
    assert all((ms > 0.0) == (count > 0) for ms, count in kt.values())
    a.sweep(3)  # and the chain goes on
    b.sweep(3)
    assert np.array_equal(a.positions(), b.positions())
    assert all(np.array_equal(x, y) for x, y in zip(a.stats(), b.stats()))
    a.close()
    b.close()
