"""Several small lattices on streams of their own (GPU required).

Their several-step launches run side by side or one after the other; results
must equal, bit for bit, those of each lattice alone, from one host thread and
from a thread per lattice, with lattices on half the grid, on the whole grid,
and on per-step launches together.
"""
import threading

import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELDS = [(I.nozzle_flags(12, 4, 60), "fp32"), (I.nozzle_flags(24, 8, 80), "fp16s"),
          (np.ones((40, 60, 72), dtype=np.uint8), "fp32"), (I.nozzle_flags(18, 6, 90), "fp64"),
          (np.ones((48, 48, 48), dtype=np.uint8), "fp16s"), (I.nozzle_flags(24, 8, 120), "fp32")]


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def lattice(lbm, k, stream=None):
    flags, precision = FIELDS[k]
    G = lbm.Lattice(flags, precision, periodic=7 if (flags == 1).all() else 0, stream=stream)
    G.set_params(nu=0.02, u_in=0.02, d_in=float(flags.shape[2]), noise_amp=0.02, noise_seed=3)
    n = G.n_active
    G.init_fields(I.random_density_field(n, 0.01, 5 + k), I.random_velocity_field(n, 0.03, 60 + k))
    return G


@pytest.mark.parametrize("threads", [False, True])
def test_lattices_on_their_own_streams(lbm, threads):
    alone = []
    for k in range(len(FIELDS)):
        with lattice(lbm, k) as G:
            G.step(40).step(21).sync()
            alone.append(G.get_populations())
    streams = [torch.cuda.Stream() for _ in FIELDS]
    lats = [lattice(lbm, k, s) for k, s in enumerate(streams)]
    if threads:
        work = [threading.Thread(target=lambda G=G: G.step(40).step(21).sync()) for G in lats]
        for t in work:
            t.start()
        for t in work:
            t.join()
    else:
        for n in (40, 21):
            for G in lats:
                G.step(n)
    for G, a in zip(lats, alone):
        assert np.array_equal(G.sync().get_populations(), a)
        G.close()
