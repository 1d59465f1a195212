"""Lattices of many rounds of work (GPU required).

The staged FP16S kernel in its steady state (each warp refills its stages and
draws runs of units many times over) against the chunk kernel, bit for bit;
transfers in parts on two streams, above 2^20 cells that do not divide by the
number of parts, against the box layout and the host's own arithmetic; and
FP16S statistics of the several-step kernel at other ghost rates.
"""
import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NOZZLE = (84, 28, 700)  # 2.9 million cells
FIELDS = {
    "box": (np.ones((136, 136, 136), dtype=np.uint8), 7, False),
    "box_uneven": (np.ones((121, 150, 147), dtype=np.uint8), 6, False),
    "nozzle": (I.nozzle_flags(*NOZZLE), 0, False),
    "nozzle_smooth": (I.nozzle_flags(*NOZZLE), 0, True),
}


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def populations(lbm, monkeypatch, name, kernel):
    flags, periodic, smooth = FIELDS[name]
    if kernel:
        monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
    else:
        monkeypatch.delenv("LBM_FLUID_KERNEL", raising=False)
    with lbm.Lattice(flags, "fp16s", periodic=periodic) as G:
        G.set_params(nu=0.01, u_in=0.02, d_in=float(flags.shape[2]), noise_amp=0.02, noise_seed=3)
        if smooth:
            G.set_wall_q(*I.nozzle_wall_q(*NOZZLE, flags=flags))
        n = G.n_active
        G.init_fields(I.random_density_field(n, 0.02, 5), I.random_velocity_field(n, 0.05, 6))
        G.stats_begin(2)
        G.step(9).sync()
        return [G.get_populations()] + list(G.stats_get()[:2])


@pytest.mark.parametrize("name", sorted(FIELDS))
def test_staged_kernel_in_its_steady_state(lbm, monkeypatch, name):
    a = populations(lbm, monkeypatch, name, None)
    b = populations(lbm, monkeypatch, name, "chunk")
    for x, y in zip(a, b):
        assert np.isfinite(x).all() and np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16s"])
def test_transfers_in_parts(lbm, precision):
    f = np.ones((101, 104, 105), dtype=np.uint8)
    f[40:43, 50, 3:9] = 0
    with lbm.Lattice(f, precision, periodic=7) as G:
        n = G.n_active
        assert n > 2 ** 20 and n % 4 != 0
        rho, u = I.random_density_field(n, 0.01, 5), I.random_velocity_field(n, 0.03, 6)
        G.set_params(nu=0.01)
        G.init_fields(rho, u)
        r, v = G.moments()
        tol = {"fp64": 1e-14, "fp32": 1e-6, "fp16s": 1e-3}[precision]  # storage roundings of 27 populations
        assert np.abs(r - rho).max() < tol and np.abs(v - u).max() < tol
        active = f.reshape(-1) != 0
        box = [np.zeros(f.size), np.zeros((f.size, 3))]
        box[0][active], box[1][active] = rho, u
        p = G.get_populations()
        rb, vb = G.moments(1)
        assert np.array_equal(rb[active], r) and np.array_equal(vb[active], v)
        assert not rb[~active].any() and not vb[~active].any()
        G.init_fields(box[0], box[1], layout=1)
        assert np.array_equal(G.get_populations(), p)
        only = G.moments()[1]
        assert np.array_equal(only, v)


@pytest.mark.parametrize("ghost", [(1.0 / (3.0 * 0.02 + 0.5),) * 4, (1.2, 1.1, 0.9, 1.3)])
def test_statistics_of_several_steps_at_other_rates(lbm, monkeypatch, ghost):
    out = []
    for kernel in (None, "chunk"):
        if kernel:
            monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
        else:
            monkeypatch.delenv("LBM_FLUID_KERNEL", raising=False)
        with lbm.Lattice(I.nozzle_flags(12, 4, 45), "fp16s") as G:
            G.set_params(nu=0.02, ghost=ghost, u_in=0.02, d_in=12.0, noise_amp=0.02, noise_seed=3)
            n = G.n_active
            G.init_fields(I.random_density_field(n, 0.01, 5), I.random_velocity_field(n, 0.03, 6))
            G.stats_begin(3, full=True)
            G.step(20).sync()
            s = G.stats_get_full()
            out.append([s["samples"], G.get_populations()] + [s[k] for k in ("u", "uu", "sigma", "rho")])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
