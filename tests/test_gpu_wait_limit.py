"""Barrier waits that give up (GPU required).

Several steps in one launch wait at a barrier over the grid between steps, for
a bounded number of polls; LBM_BARRIER_POLLS, read when a context or a server
is created, sets that number.  At 0 every wait gives up at once, the kernels
return, and no call may hand out the torn state: not the first read after the
steps, not a later one, and not the server.
"""
import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FLAGS = I.nozzle_flags(24, 8, 80)
FLOW = dict(nu=0.02, u_in=0.02, d_in=24.0, profile="parabolic", noise_amp=0.02, noise_seed=3)


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def lattice(lbm, precision):
    G = lbm.Lattice(FLAGS, precision)
    G.set_params(**FLOW)
    G.init_equilibrium(1.0, (0.0, 0.0, 0.0))
    return G


READS = {
    "sync": lambda G: G.sync(),
    "moments": lambda G: G.moments(),
    "moments_box": lambda G: G.moments(1),
    "populations": lambda G: G.get_populations(),
    "populations_box": lambda G: G.get_populations(1),
    "totals": lambda G: G.totals(),
    "averages": lambda G: G.stats_get(),
    "full_averages": lambda G: G.stats_get_full(),
    "checkpoint": lambda G: G.checkpoint(),
}


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
@pytest.mark.parametrize("first", sorted(READS))
def test_torn_state_is_not_read(lbm, monkeypatch, first, precision):
    monkeypatch.setenv("LBM_BARRIER_POLLS", "0")
    with lattice(lbm, precision) as G:
        G.stats_begin(1, full=True)
        G.step(16)
        for call in (READS[first], READS["sync"], READS["moments"], READS["averages"], lambda g: g.step(1)):
            with pytest.raises(lbm.LbmError) as e:
                call(G)
            assert e.value.status == lbm.LBM_ERR_TIMEOUT
        # a new state is a new start (fewer steps than go in one launch)
        G.init_equilibrium(1.0, (0.0, 0.0, 0.0))
        G.step(5).sync()
        monkeypatch.delenv("LBM_BARRIER_POLLS")
        with lattice(lbm, precision) as H:
            H.step(5).sync()
            assert np.array_equal(G.get_populations(), H.get_populations())


def test_server_fails_the_requests_of_a_torn_tick(lbm, monkeypatch):
    monkeypatch.setenv("LBM_BARRIER_POLLS", "0")
    S = lbm.Server(8 << 30, max_slots=4, steps_per_tick=16)
    ids = [S.submit(FLAGS, 40, p, **FLOW) for p in ("fp32", "fp16s")]
    with pytest.raises(lbm.LbmError) as e:
        for _ in range(10000):
            S.tick()
    assert e.value.status == lbm.LBM_ERR_TIMEOUT
    for _ in range(10000):  # the second request, if it was not admitted with the first
        if all(S.poll(i)[0] == lbm.LBM_REQ_FAILED for i in ids):
            break
        try:
            S.tick()
        except lbm.LbmError as again:
            assert again.status == lbm.LBM_ERR_TIMEOUT
    for i in ids:
        assert S.poll(i)[0] == lbm.LBM_REQ_FAILED
        with pytest.raises(lbm.LbmError) as e:
            S.result(i)
        assert e.value.status == lbm.LBM_ERR_TIMEOUT
    # one step has no barrier: the server goes on
    one = S.submit(FLAGS, 1, "fp32", **FLOW)
    for _ in range(10000):
        S.tick()
        if S.poll(one)[0] == lbm.LBM_REQ_DONE:
            break
    rho, u = S.result(one)
    with lattice(lbm, "fp32") as G:
        G.step(1).sync()
        r, v = G.moments()
    assert np.array_equal(rho, r) and np.array_equal(u, v)
    S.close()
