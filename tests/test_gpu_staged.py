"""The staged FP16S fluid kernel against the chunk kernel (GPU required).

Both round every operation of the rate-1 collision explicitly and in the same
order, so the populations must agree bit for bit (tolerance zero) whatever
way the cells are grouped: units that start mid-sector, units cut by row
ends, obstacles and absent chunks, plain units with wrap-around copies at
even row ends, split ones at odd ends, single-unit lattices, walls in every
direction, interpolated walls, inlet/outlet nodes, and the fused statistics.
"""
import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOX = 1


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def ragged(shape, seed):
    f = np.ones(shape, dtype=np.uint8)
    f[np.random.default_rng(seed).random(shape) < 0.03] = 0
    return f


def duct():
    f = np.ones((150, 7, 9), dtype=np.uint8)
    f[60:90, 2:5, 3:7] = 0
    f[0], f[-1] = 2, 3
    return f


FIELDS = {
    "one_unit": (np.ones((1, 1, 64), dtype=np.uint8), 7, "x"),
    "row_64": (np.ones((3, 4, 64), dtype=np.uint8), 7, "x"),
    "row_65": (np.ones((3, 4, 65), dtype=np.uint8), 7, "x"),
    "row_128": (np.ones((4, 3, 128), dtype=np.uint8), 7, "x"),
    "row_200_walls": (np.ones((5, 4, 200), dtype=np.uint8), 0, "x"),
    "row_9": (np.ones((5, 4, 9), dtype=np.uint8), 1, "x"),
    "ragged_x": (ragged((6, 7, 150), 1), 5, "x"),
    "ragged_z": (ragged((150, 7, 6), 2), 2, "z"),
    "duct_z": (duct(), 0, "z"),
    "duct_x": (duct(), 0, "x"),
    "nozzle": (I.nozzle_flags(12, 4, 140), 0, "z"),
}


def run(lbm, monkeypatch, kernel, name, walls=False):
    flags, periodic, rows = FIELDS[name]
    monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
    with lbm.Lattice(flags, "fp16s", periodic=periodic, row_axis=rows) as G:
        nx = flags.shape[2]
        G.set_params(nu=0.02, u_in=0.02, d_in=float(nx), profile="parabolic", noise_amp=0.02, noise_seed=3)
        if walls:
            G.set_wall_q(*I.nozzle_wall_q(12, 4, 140))
        n = G.n_active
        G.init_fields(I.random_density_field(n, 0.01, 5), I.random_velocity_field(n, 0.03, 6))
        G.step(3)
        G.stats_begin(1, full=True)
        G.step(4).sync()
        s = G.stats_get_full()
        return [G.get_populations()] + [s[k] for k in ("u", "uu", "sigma", "rho")]


@pytest.mark.parametrize("name", sorted(FIELDS))
def test_staged_kernel_equals_chunk_kernel(lbm, monkeypatch, name):
    for a, b in zip(run(lbm, monkeypatch, "staged", name), run(lbm, monkeypatch, "chunk", name)):
        assert np.isfinite(a).all() and np.array_equal(a, b)


def test_staged_kernel_with_interpolated_walls(lbm, monkeypatch):
    for a, b in zip(run(lbm, monkeypatch, "staged", "nozzle", True), run(lbm, monkeypatch, "chunk", "nozzle", True)):
        assert np.isfinite(a).all() and np.array_equal(a, b)


@pytest.mark.parametrize("name,walls", [("duct_x", False), ("duct_z", False), ("ragged_z", False), ("nozzle", False),
                                        ("nozzle", True)])
def test_steps_with_statistics_differ_by_roundings_alone(lbm, monkeypatch, name, walls):
    """With statistics on, FP16S keeps other roundings of the same update (in
    the chunk kernel): after one step each population is within one FP16 step
    of the other form's, 2^-10 of its deviation, and the FP32 arithmetic's
    error, 1e-8 (27 roundings of deviations below 0.01)."""
    flags, periodic, rows = FIELDS[name]
    w = np.array([(1 / 6, 2 / 3, 1 / 6)[i % 3] * (1 / 6, 2 / 3, 1 / 6)[i // 3 % 3] * (1 / 6, 2 / 3, 1 / 6)[i // 9]
                  for i in range(27)])
    out = []
    for kernel in (None, "chunk"):
        if kernel:
            monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
        else:
            monkeypatch.delenv("LBM_FLUID_KERNEL", raising=False)
        with lbm.Lattice(flags, "fp16s", periodic=periodic, row_axis=rows) as G:
            G.set_params(nu=0.02, u_in=0.02, d_in=float(flags.shape[2]), profile="parabolic", noise_amp=0.02,
                         noise_seed=3)
            if walls:
                G.set_wall_q(*I.nozzle_wall_q(12, 4, 140))
            n = G.n_active
            G.init_fields(I.random_density_field(n, 0.01, 5), I.random_velocity_field(n, 0.03, 6))
            G.stats_begin(1, full=True)
            G.step(1).sync()
            assert G.stats_get_full()["samples"] == 1
            out.append(G.get_populations())
    a, b = out
    assert np.isfinite(a).all()
    assert (np.abs(a - b) <= 2.0 ** -10 * np.maximum(np.abs(a - w), np.abs(b - w)) + 1e-8).all()
