"""Several steps in one launch against the per-step kernels (GPU required).

Small lattices take eight or more steps in one cooperative launch.  Every
cell runs the same code as in the per-step kernels, which a fluid kernel
asked for by name still runs, so populations and sampled statistics must
agree bit for bit (tolerance zero): both row axes, periodic rows, walls in
every direction, interpolated walls, inlet/outlet nodes with noise and ramp,
odd and even step counts, sampling strides, health checks in between, fewer
items than warps, and the three collision forms.
"""
import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

from gpu_util import gpu_lattice, max_rel, oracle_lattice, random_state, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOX = 1


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def ragged():
    f = np.ones((9, 8, 70), dtype=np.uint8)
    f[np.random.default_rng(4).random(f.shape) < 0.03] = 0
    return f


FIELDS = {
    "one_cell": (np.ones((1, 1, 1), dtype=np.uint8), 7, "x"),
    "box": (np.ones((20, 18, 33), dtype=np.uint8), 7, "x"),
    "ragged": (ragged(), 5, "x"),
    "nozzle": (I.nozzle_flags(12, 4, 45), 0, "z"),
    "nozzle_x_rows": (I.nozzle_flags(12, 4, 45), 0, "x"),
    "several_rounds": (np.ones((40, 60, 72), dtype=np.uint8), 7, "x"),
}


def run(lbm, monkeypatch, kernel, precision, name, steps, ghost=(1.0,) * 4, check=0, walls=False):
    flags, periodic, rows = FIELDS[name]
    if kernel:
        monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
    else:
        monkeypatch.delenv("LBM_FLUID_KERNEL", raising=False)
    with lbm.Lattice(flags, precision, periodic=periodic, row_axis=rows) as G:
        G.set_params(nu=0.02, ghost=ghost, u_in=0.02, d_in=12.0, profile="parabolic", noise_amp=0.02, noise_seed=3,
                     inlet_ramp=9)
        if walls:
            G.set_wall_q(*I.nozzle_wall_q(12, 4, 45))
        n = G.n_active
        G.init_fields(I.random_density_field(n, 0.01, 5), I.random_velocity_field(n, 0.03, 6))
        G.set_check_every(check)
        n0 = G.kernel_launches()
        G.step(steps)
        launches = G.kernel_launches() - n0
        if precision == "fp16s":  # with statistics on, FP16S steps go one by one
            G.step(steps + 1).sync()
            return launches, 0, [G.get_populations()]
        G.stats_begin(3, full=True)
        G.step(steps + 1).sync()
        s = G.stats_get_full()
        return launches, s["samples"], [G.get_populations()] + [s[k] for k in ("u", "uu", "sigma", "rho")]


def same(lbm, monkeypatch, precision, name, steps, **kw):
    a = run(lbm, monkeypatch, None, precision, name, steps, **kw)
    b = run(lbm, monkeypatch, "tile", precision, name, steps, **kw)
    assert a[1] == b[1] and a[0] < b[0]
    for x, y in zip(a[2], b[2]):
        assert np.isfinite(x).all() and np.array_equal(x, y)


@pytest.mark.parametrize("name", sorted(FIELDS))
@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_one_launch_equals_one_by_one(lbm, monkeypatch, precision, name):
    same(lbm, monkeypatch, precision, name, 9)


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_interpolated_walls_and_health_checks(lbm, monkeypatch, precision):
    same(lbm, monkeypatch, precision, "nozzle", 28, check=11, walls=True)


OMEGA = 1.0 / (3.0 * 0.02 + 0.5)


@pytest.mark.parametrize("ghost", [(OMEGA,) * 4, (1.2, 1.1, 0.9, 1.3)])
@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_other_collision_forms(lbm, monkeypatch, precision, ghost):
    same(lbm, monkeypatch, precision, "nozzle", 8, ghost=ghost)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5), ("fp16s", 1e-3)])
@pytest.mark.parametrize("nu", [0.02, 0.3])
def test_lattice_bgk_against_the_oracle(orc, lbm, precision, tol, nu):
    """Every ghost rate at omega: the lattice BGK form against the oracle's
    general collision, populations (FP64) or velocity."""
    ghost = (1.0 / (3.0 * nu + 0.5),) * 4
    flags = I.nozzle_flags(12, 4, 45)
    bc = dict(profile="parabolic", u_in=0.02, d_in=12.0, noise_amp=0.02, seed=5)
    O = oracle_lattice(orc, flags, nu, ghost=ghost, **bc)
    f0 = random_state(orc, flags, 21)
    O.set_populations(f0)
    G = gpu_lattice(lbm, flags, precision, nu, ghost=ghost, **bc)
    G.set_populations(f0, layout=BOX)
    O.step(9)
    G.step(9).sync()
    act = flags.reshape(-1) != 0
    if precision == "fp64":
        assert max_rel(G.get_populations(BOX)[act], O.f[act]) < tol
    else:
        assert rel_l2(G.moments(BOX)[1][act], O.moments()[act, 1:]) < tol
