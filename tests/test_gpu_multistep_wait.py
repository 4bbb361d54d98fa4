"""The bounded wait of a multi-step launch for its own blocks: with a limit of 0 polls every block
leaves at the first barrier, and every call that waits for the stream reports it; with the default
limit restored a handle of its own steps as ever."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattice(streaming, precision, q=19):
    from paper_2305_09910_gb300 import lbm

    lat = lbm.Lattice(64, 24, 20, stencil=q, tau=0.6, closure="smag", streaming=streaming, precision=precision,
                      faces=("periodic", "periodic", "wall", "wall", "periodic", "periodic"))
    lat.set_force(1e-5)
    lat.init_equilibrium()
    lat.step(2)  # steady: the next steps go into one launch
    lat.sync()
    return lat


def _calls(lat):
    from paper_2305_09910_gb300 import lbm

    n = lat.nx * lat.ny * lat.nz
    return {"sync": lat.sync, "reduce": lambda: lbm.lbm_reduce(lat.h), "populations": lat.get_populations,
            "moments": lambda: lbm.lbm_moments(lat.h, np.zeros(n, np.float32), np.zeros(3 * n, np.float32)),
            "stats": lambda: lbm.lbm_stats_get(lat.h, lat.ny)}


@pytest.mark.parametrize("first", ["sync", "reduce", "populations", "moments", "stats"])
@pytest.mark.parametrize("streaming,precision,q", [("aa", "f32", 19), ("pull", "f16", 19), ("pull", "f32", 27)])
def test_a_wait_that_gives_up_is_reported(first, streaming, precision, q):
    from paper_2305_09910_gb300 import lbm

    lat = _lattice(streaming, precision, q)
    calls = _calls(lat)
    for call in calls.values():
        call()  # no error before
    lbm.lbm_debug_set_wait_polls(lat.h, 0)
    lat.step(6)
    for name in (first, "sync", "reduce"):
        with pytest.raises(lbm.LbmError) as e:
            calls[name]()
        assert e.value.status == lbm.LBM_ECUDA and "unusable" in str(e.value), (name, e.value)
    for step in (lambda: lat.step(1), lambda: lat.step(4)):
        with pytest.raises(lbm.LbmError) as e:
            step()
        assert e.value.status == lbm.LBM_ECUDA
    lat.close()


@pytest.mark.parametrize("polls", [-1, 1 << 20])
def test_a_wait_that_does_not_give_up(polls):
    from paper_2305_09910_gb300 import lbm

    a, b = _lattice("aa", "f32"), _lattice("aa", "f32")
    lbm.lbm_debug_set_wait_polls(a.h, 0)
    lbm.lbm_debug_set_wait_polls(a.h, polls)
    a.step(9)
    for _ in range(9):
        b.step(1)
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.sync()
    a.close()
    b.close()
