"""Admission to the request server's memory budget (CPU only).

A request that fits a budget today has to fit it tomorrow: the device
footprint of a served lattice is no larger than that of the first releases,
stored here in bytes (FP32, FP16S).
"""
import numpy as np
import pytest

from paper_2204_10566_gb300 import inputs as I

FIELDS = {
    "pipe_18x150": (lambda: I.pipe_flags(18, 150), 0, 12700448, 7231008),
    "nozzle_24x160": (lambda: I.nozzle_flags(24, 8, 160), 0, 21368240, 11876016),
    "pipe_33x275": (lambda: I.pipe_flags(33, 275), 0, 70957028, 40769252),
    "nozzle_48x400": (lambda: I.nozzle_flags(48, 16, 400), 0, 197628752, 111176272),
    "box_64": (lambda: np.ones((64, 64, 64), dtype=np.uint8), 7, 82815488, 47411200),
    "box_33": (lambda: np.ones((33, 33, 33), dtype=np.uint8), 7, 13086340, 7431300),
}


@pytest.fixture(scope="module")
def lbm():
    from paper_2204_10566_gb300 import build

    build.build()
    from paper_2204_10566_gb300 import lbm as m

    return m


@pytest.mark.parametrize("name", sorted(FIELDS))
def test_what_fitted_still_fits(lbm, name):
    make, periodic, fp32, fp16s = FIELDS[name]
    for precision, budget in (("fp32", fp32), ("fp16s", fp16s)):
        info = lbm.check_request(make(), 10, precision, periodic=periodic, budget_bytes=budget, nu=0.01)
        assert info["footprint"] <= budget
