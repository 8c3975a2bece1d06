"""Which step an FP64 lattice takes, on moments or on populations (lbm_walk.cu: walk_pays): the faster
one by the times measured on a GB300, without a GPU, and that a handle takes it."""
import ctypes

import numpy as np
import pytest

from paper_2301_12869_gb300 import lbm
from test_gpu_walk import read, setup
from test_walk_plan import FP32, FP64, NSM, plan  # noqa: F401 (the fixture is used)

# nx, ny, form, the population step's band and strip, and us a step: on moments, on populations, and
# of the population step before it collided from three moments
MEASURED = [
    (4, 17000, 1, 4, 23, 84.9, 163.2, 216.5), (8, 9000, 2, 8, 12, 47.7, 94.5, 123.5),
    (16, 5000, 1, 16, 7, 54.3, 56.7, 74.2), (24, 3000, 2, 24, 4, 47.5, 42.2, 52.8),
    (28, 2500, 1, 28, 4, 50.0, 37.4, 47.9), (32, 2100, 1, 32, 3, 49.2, 30.9, 39.1),
    (32, 2100, 2, 32, 3, 48.4, 34.6, 43.0), (48, 2000, 2, 48, 3, 47.7, 50.3, 64.2),
    (56, 1300, 1, 56, 2, 48.8, 35.1, 45.1), (60, 1200, 2, 60, 2, 34.1, 38.7, 48.4),
    (64, 1100, 2, 64, 2, 48.6, 38.1, 47.9), (64, 3000, 1, 64, 4, 81.8, 58.2, 76.2),
    (100, 3000, 1, 100, 4, 101.1, 102.9, 136.9), (120, 600, 2, 120, 1, 33.1, 41.6, 53.6),
    (180, 400, 1, 128, 2, 34.3, 53.8, 70.6), (260, 300, 2, 128, 2, 47.3, 61.7, 81.1),
    (512, 512, 1, 128, 3, 83.6, 81.0, 107.6), (1024, 70, 1, 128, 1, 49.1, 37.5, 49.4),
    (1024, 1024, 2, 128, 11, 230.2, 259.7, 344.1), (1024, 4096, 1, 128, 44, 805.4, 967.1, 1288.9),
    (16384, 16, 1, 128, 4, 73.1, 99.6, 132.7), (65536, 4, 2, 128, 4, 98.3, 86.8, 114.9),
]


@pytest.fixture(scope="module")
def pays(plan):  # noqa: F811
    fn = ctypes.CDLL(lbm.LIB_PATH)["_ZN3lbm9walk_paysEiRKNS_10WalkTilingEiiii"]
    fn.restype = ctypes.c_bool

    def call(precision, nx, ny, form, band, strip):
        ok, t = plan(precision, nx, ny, False, 1 << 20)
        assert ok
        return fn(precision, ctypes.byref(t), NSM, band, strip, form)

    return call


@pytest.mark.parametrize("row", MEASURED, ids=lambda r: "%dx%d-%d" % r[:3])
def test_the_faster_step(pays, row):
    nx, ny, form, band, strip, walk, step, before = row
    took, other = (walk, step) if pays(FP64, nx, ny, form, band, strip) else (step, walk)
    assert took < before and took <= 1.08 * other


def test_fp32_always_walks(pays):
    assert all(pays(FP32, nx, ny, 1, min(nx, 512), 1) for nx, ny in ((4, 100), (32, 2100), (1024, 70), (65536, 4)))


@pytest.mark.gpu
@pytest.mark.parametrize("nx, ny, form, populations", [(32, 2100, 1, True), (64, 1100, 2, True), (260, 300, 2, False)])
def test_a_handle_takes_it(plan, nx, ny, form, populations):  # noqa: F811
    """The two steps round differently: a block of steps has the bits of single steps between reads,
    which are population steps, exactly where populations are faster."""
    p, _, rho0, f = setup(nx, ny, "fp64", form, False)
    out = []
    for block in (8, 1):
        h = lbm.lbm_init(p, rho0)
        try:
            lbm.lbm_set_state(h, f)
            for _ in range(0, 8, block):
                lbm.lbm_step(h, block)
                state = read(h, p)
            out.append(state)
        finally:
            lbm.lbm_destroy(h)
    assert np.array_equal(*out) == populations
    assert np.max(np.abs(out[0] - out[1])) <= 1e-14
