"""The tile sweep's bounded waits.  With HD_TEST_TILE_STALL=1 at creation the first
work item of every launch is never taken, so the tiles around it wait for a
sweep that does not come; the waits give up after 4096 polls, every block
leaves, the call reports HD_ERR_TIMEOUT and the context stays in its error
state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fixed", "fp64"])
@pytest.mark.parametrize("Ns, sweeps", [([4096], 3), ([65536], 20), ([4096, 6400, 2500], 256)])
def test_wait_gives_up_and_sticks(oracle_mod, monkeypatch, form, Ns, sweeps):
    import paper_1211_1645_gb300 as hd
    from paper_1211_1645_gb300.hd import HD_ERR_STATE, HD_ERR_TIMEOUT
    R = len(Ns)

    def make():
        return hd.HardDisks(Ns, [0.70] * R, [0.1] * R, list(range(3, 3 + R)), precision=form)

    monkeypatch.setenv("HD_TEST_TILE_STALL", "1")
    g = make()
    monkeypatch.delenv("HD_TEST_TILE_STALL")
    g.sweep(sweeps)
    with pytest.raises(hd.HDError) as e:
        g.stats()
    assert e.value.status == HD_ERR_TIMEOUT
    for call in (lambda: g.sweep(1), g.positions, g.stats):
        with pytest.raises(hd.HDError) as e:
            call()
        assert e.value.status == HD_ERR_STATE
    g.close()
    ok = make()  # a new context without the hook runs the chain
    ok.sweep(3)
    o = oracle_mod.OracleChain(Ns[0], 0.70, 0.1, 3, form=form)
    o.sweep(3)
    assert np.array_equal(ok.positions()[:Ns[0]], o.positions())
    ok.close()
