"""One set of roundings for FP16S steps at the default ghost rates (GPU required).

FP16 storage carries a last-bit difference of the FP32 arithmetic on to the
size of its own noise, so a run is only repeatable if a cell rounds alike
whatever kernel updates it.  Sampling statistics must leave the populations
alone (tolerance zero), and the states reached must be the stored ones, by
their SHA-256: both row axes, periodic rows, walls in every direction,
interpolated walls, inlet/outlet nodes with noise and ramp, steps one by one
and several in a launch, the staged kernel, and the request server.
"""
import hashlib

import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


def ragged():
    f = np.ones((30, 31, 70), dtype=np.uint8)
    f[np.random.default_rng(4).random(f.shape) < 0.02] = 0
    return f


NOZZLE = (24, 8, 80)
FIELDS = {  # flags, periodic axes, row axis, interpolated walls
    "box": (np.ones((30, 32, 70), dtype=np.uint8), 7, "x", False),
    "ragged_x": (ragged(), 5, "x", False),
    "ragged_z": (ragged(), 4, "z", False),
    "nozzle_x": (I.nozzle_flags(*NOZZLE), 0, "x", False),
    "nozzle_z": (I.nozzle_flags(*NOZZLE), 0, "z", False),
    "smooth_x": (I.nozzle_flags(*NOZZLE), 0, "x", True),
    "smooth_z": (I.nozzle_flags(*NOZZLE), 0, "z", True),
}


def state(lbm, name, parts, stats=False):
    """Populations after the given runs of steps, and the averages."""
    flags, periodic, rows, smooth = FIELDS[name]
    with lbm.Lattice(flags, "fp16s", periodic=periodic, row_axis=rows) as G:
        G.set_params(nu=0.02, u_in=0.05, d_in=24.0, profile="parabolic", noise_amp=0.02, noise_seed=3, inlet_ramp=9)
        if smooth:
            G.set_wall_q(*I.nozzle_wall_q(*NOZZLE))
        n = G.n_active
        G.init_fields(I.random_density_field(n, 0.05, 5), I.random_velocity_field(n, 0.15, 6))
        if stats:
            G.stats_begin(1, full=True)
        for k in parts:
            G.step(k)
        G.sync()
        s = G.stats_get_full() if stats else None
        return [G.get_populations()] + ([s[k] for k in ("u", "uu", "sigma", "rho")] if stats else [])


def served(lbm, smooth_start):
    S = lbm.Server(8 << 30, max_slots=4, steps_per_tick=16)
    p = dict(nu=0.02, u_in=0.08, d_in=24.0, profile="parabolic", noise_amp=0.4, noise_seed=3,
             inlet_ramp=30 if smooth_start else 0)
    rid = S.submit(I.nozzle_flags(24, 8, 40), 60, "fp16s", **p)
    while S.poll(rid)[0] not in (lbm.LBM_REQ_DONE, lbm.LBM_REQ_FAILED):
        S.tick()
    out = S.result(rid)
    S.close()
    return [np.float32(a) for a in out]


def digest(arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update(np.ascontiguousarray(a).tobytes())
    return h.hexdigest()[:16]


# states reached by the release before the staged kernel
STORED = {"box": "20c632bab537616f", "nozzle_x": "a349f7129e3d1341", "nozzle_z": "b6f7e5d0fd0dcec2",
          "ragged_x": "a5d110a033a66116", "ragged_z": "5f992b9ebf51eb18", "smooth_x": "e1f9b2daba667b18",
          "smooth_z": "45e278260e655e51"}
AVERAGED = {"box": "2701ab302aa3217d", "nozzle_x": "197c346e119810fe", "nozzle_z": "e18f97cad312b7a7",
            "ragged_x": "62b20e9948b765fe", "ragged_z": "358cca1ce20b5ebb", "smooth_x": "6a7915800da8d5ee",
            "smooth_z": "69f53b94fd685f02"}
SERVED = {False: "efabbea6e3389201", True: "dcd49e39443f219e"}


@pytest.mark.parametrize("kernel", [None, "chunk", "staged", "tile", "pairs"])
@pytest.mark.parametrize("name", sorted(FIELDS))
def test_states_are_the_stored_ones(lbm, monkeypatch, name, kernel):
    if kernel:
        monkeypatch.setenv("LBM_FLUID_KERNEL", kernel)
    else:
        monkeypatch.delenv("LBM_FLUID_KERNEL", raising=False)
    assert digest(state(lbm, name, (3, 12))) == STORED[name]
    assert digest(state(lbm, name, (3, 12), stats=True)) == AVERAGED[name]


@pytest.mark.parametrize("smooth_start", [False, True])
def test_served_states_are_the_stored_ones(lbm, smooth_start):
    assert digest(served(lbm, smooth_start)) == SERVED[smooth_start]


@pytest.mark.parametrize("parts", [(1, 4), (15,)])
@pytest.mark.parametrize("name", sorted(FIELDS))
def test_sampling_leaves_the_populations_alone(lbm, name, parts):
    a, b = state(lbm, name, parts), state(lbm, name, parts, stats=True)
    assert np.isfinite(a[0]).all() and np.array_equal(a[0], b[0])


@pytest.mark.parametrize("full", [False, True])
def test_sampling_leaves_a_large_lattice_alone(lbm, full):
    """The same above the staged kernel's threshold."""
    out = []
    for stats in (False, True):
        with lbm.Lattice(np.ones((136, 136, 136), dtype=np.uint8), "fp16s", periodic=7) as G:
            G.set_params(nu=0.005)
            n = G.n_active
            G.init_fields(I.random_density_field(n, 0.02, 5), I.random_velocity_field(n, 0.1, 6))
            if stats:
                G.stats_begin(2, full=full)
            G.step(20).sync()
            out.append(G.get_populations())
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
