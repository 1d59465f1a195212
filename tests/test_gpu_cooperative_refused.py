"""Where the device refuses a cooperative launch, steps run one by one (GPU required).

LBM_COOPERATIVE_BLOCKS, read when the launch is sized, asks for a number of
blocks that the device cannot hold at once: the runtime refuses the launch
with an error, nothing runs, and lbm_step and the server's tick take the same
steps in ordinary launches, to the same bits.
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


def stepped(lbm, precision):
    with lbm.Lattice(FLAGS, precision) as G:
        G.set_params(**FLOW)
        G.init_equilibrium(1.0, (0.0, 0.0, 0.0))
        G.stats_begin(3)
        G.set_check_every(20)
        G.step(33).step(9).sync()
        mean, square, samples = G.stats_get()
        return G.kernel_launches(), samples, [G.get_populations(), mean, square]


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_steps_run_one_by_one(lbm, monkeypatch, precision):
    monkeypatch.delenv("LBM_COOPERATIVE_BLOCKS", raising=False)
    a = stepped(lbm, precision)
    monkeypatch.setenv("LBM_COOPERATIVE_BLOCKS", "1000000")
    b = stepped(lbm, precision)
    assert a[0] < b[0] and a[1] == b[1] == 14
    for x, y in zip(a[2], b[2]):
        assert np.isfinite(x).all() and np.array_equal(x, y)


def served(lbm):
    S = lbm.Server(8 << 30, max_slots=4, steps_per_tick=16)
    ids = [S.submit(FLAGS, n, p, **FLOW) for n, p in ((37, "fp32"), (50, "fp16s"), (3, "fp16s"))]
    done = (lbm.LBM_REQ_DONE, lbm.LBM_REQ_FAILED)
    while not all(S.poll(i)[0] in done for i in ids):
        S.tick()
    out = [S.result(i) for i in ids]
    S.close()
    return out


def test_server_ticks_run_step_by_step(lbm, monkeypatch):
    monkeypatch.delenv("LBM_COOPERATIVE_BLOCKS", raising=False)
    a = served(lbm)
    monkeypatch.setenv("LBM_COOPERATIVE_BLOCKS", "1000000")
    b = served(lbm)
    for (r, u), (q, v) in zip(a, b):
        assert np.isfinite(r).all() and np.array_equal(r, q) and np.array_equal(u, v)


@pytest.mark.parametrize("updates", [1, 200000, 700000])
def test_long_ticks_go_in_several_launches(lbm, monkeypatch, updates):
    """Past a number of cell updates (LBM_LAUNCH_UPDATES) a tick's steps go in
    several launches of one, a few, or, once a lattice has finished, all steps:
    the same results."""
    monkeypatch.delenv("LBM_LAUNCH_UPDATES", raising=False)
    a = served(lbm)
    monkeypatch.setenv("LBM_LAUNCH_UPDATES", str(updates))
    b = served(lbm)
    for (r, u), (q, v) in zip(a, b):
        assert np.isfinite(r).all() and np.array_equal(r, q) and np.array_equal(u, v)
