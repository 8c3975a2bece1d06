"""Wide lattices of a few rows on moments, with Eq. Gravity_2: the walk's grid has at most as many
CTAs as the handle has partial sums, so <rho> and the status word stay what they are. Against the FP64
oracle; tolerances as in test_gpu_walk.py.
"""
import numpy as np
import pytest

from oracle import lbm as olbm
from oracle import thermal as oth
from paper_2301_12869_gb300 import lbm
from test_gpu_walk import T_C, cuda_lib, read, setup, tolerance  # noqa: F401 (the fixture is used)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny, precision, zh", [
    (4096, 8, "fp32", True), (2048, 4, "fp32", True), (8192, 3, "fp32", True), (1924, 3, "fp32", True),
    (2048, 1, "fp32", False), (2048, 2, "fp32", False), (4096, 2, "fp32", False), (8192, 9, "fp64", True),
])
def test_steps_match_oracle(nx, ny, precision, zh):
    p, op, rho0, f = setup(nx, ny, precision, 2, zh)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        for n in (6, 3):
            lbm.lbm_step(h, n)
            f = olbm.run(f, op, n)
            assert np.max(np.abs(read(h, p) - f)) <= tolerance(precision, 9)
        assert lbm.lbm_status(h) == lbm.LBM_OK
    finally:
        lbm.lbm_destroy(h)


def test_thermal_steps_match_oracle():
    nx, ny = 4096, 8
    p, op, rho0, f = setup(nx, ny, "fp32", 2, False, thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C)
    th = oth.Thermal(c_v=p.c_v, kappa=p.kappa, T_bot=p.T_bot, T_top=p.T_top)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        T, Tg = np.empty((ny, nx)), np.empty((ny, nx))
        lbm.lbm_get_temperature(h, T)
        lbm.lbm_step(h, 6)
        for _ in range(6):
            f, T = oth.thermal_step(f, T, op, th)
        lbm.lbm_get_temperature(h, Tg)
        tol = tolerance("fp32", 6)
        assert np.max(np.abs(read(h, p) - f)) <= tol and np.max(np.abs(Tg - T)) <= tol
        assert lbm.lbm_status(h) == lbm.LBM_OK
    finally:
        lbm.lbm_destroy(h)
