"""When a handle changes between its two forms, populations and moments: what a call takes shows in the
last bits of its result (the two steps round differently), so the routes are compared bit by bit.
"""
import numpy as np
import pytest

from paper_2301_12869_gb300 import lbm
from test_gpu_walk import cuda_lib, read, setup  # noqa: F401 (the fixture is used)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny, precision, zh", [(256, 200, "fp32", False), (256, 200, "fp32", True),
                                                   (256, 257, "fp64", False)])
def test_single_steps_between_reads_are_population_steps(nx, ny, precision, zh):
    """After a block of steps on moments, a loop of one step and a read of the populations takes one
    population step a turn, not a walk and a collision that forms the populations again."""
    p, _, rho0, f = setup(nx, ny, precision, 2, zh)
    out = []
    for populations in (False, True):
        h = lbm.lbm_init(p, rho0)
        try:
            lbm.lbm_set_state(h, f)
            lbm.lbm_step(h, 9)
            states = [read(h, p)]
            if populations:
                lbm.lbm_set_tiling(h, 0)  # the state as populations, as lbm_set_tiling leaves it
            for _ in range(3):
                lbm.lbm_step(h, 1)
                states.append(read(h, p))
            out.append(states)
        finally:
            lbm.lbm_destroy(h)
    for k, (a, b) in enumerate(zip(*out)):
        assert np.array_equal(a, b), k


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("zh", [False, True])
def test_mass_of_a_state_on_moments(form, zh):
    """The collision keeps a node's mass, so the mass of the populations after n steps is the sum of the
    densities they collided from: taken from there without forming the populations, it is that sum to
    1e-13 (sums of the rounded FP32 populations differ from it by 1e-11)."""
    nx, ny = 256, 200
    p, _, rho0, f = setup(nx, ny, "fp32", form, zh)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        lbm.lbm_step(h, 8)
        rho = np.empty((ny, nx))
        for _ in range(2):
            lbm.lbm_moments(h, rho)
            lbm.lbm_step(h, 1)
            assert lbm.lbm_reduce(h, lbm.LBM_REDUCE_MASS)[0] == pytest.approx(float(np.sum(rho)), rel=1e-13)
            assert lbm.lbm_reduce(h, lbm.LBM_REDUCE_MEAN_RHO)[0] == pytest.approx(float(np.mean(rho)), rel=1e-13)
        mass = lbm.lbm_reduce(h, lbm.LBM_REDUCE_MASS)[0]
        got = read(h, p)
        assert mass == pytest.approx(float(np.sum(got)), rel=1e-9)
        assert lbm.lbm_reduce(h, lbm.LBM_REDUCE_MASS)[0] == pytest.approx(float(np.sum(got)), rel=1e-13)
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("nx, ny, precision, steps, chip", [
    (100, 160, "fp32", 8, False), (20, 800, "fp32", 8, False), (64, 256, "fp32", 8, True), (100, 128, "fp32", 8, True),
    (20, 100, "fp64", 4, False), (24, 80, "fp64", 4, True)])
def test_padded_rows_count_for_the_steps_on_chip(nx, ny, precision, steps, chip):
    """A row on chip takes a power of two of lanes. Lattices that fill less than their share are
    stepped as in calls too short for the chip: the same bits as such calls."""
    p, _, rho0, f = setup(nx, ny, precision, 2, True)
    out = []
    for block in (steps, steps // 2):
        h = lbm.lbm_init(p, rho0)
        try:
            lbm.lbm_set_state(h, f)
            for _ in range(0, steps, block):
                lbm.lbm_step(h, block)
            out.append(read(h, p))
        finally:
            lbm.lbm_destroy(h)
    assert np.array_equal(*out) != chip


@pytest.mark.parametrize("nx, ny, precision", [(256, 200, "fp32"), (64, 64, "fp32"), (260, 300, "fp64")])
def test_single_steps_without_reads_walk(nx, ny, precision):
    """From the fourth step on, steps in calls of one are steps on moments like a block's."""
    p, _, rho0, f = setup(nx, ny, precision, 2, False)
    out = []
    for calls in ([1] * 10, [1, 1, 1, 7], [10]):
        h = lbm.lbm_init(p, rho0)
        try:
            lbm.lbm_set_state(h, f)
            for n in calls:
                lbm.lbm_step(h, n)
            out.append(read(h, p))
        finally:
            lbm.lbm_destroy(h)
    assert np.array_equal(out[0], out[1]) and not np.array_equal(out[0], out[2])


@pytest.mark.parametrize("nx, ny, precision, steps, walk", [
    (4, 3000, "fp32", 1, True), (512, 512, "fp32", 1, False), (256, 200, "fp32", 8, True), (12, 6000, "fp64", 1, False),
    (12, 6000, "fp64", 4, True), (100, 3000, "fp64", 4, False), (1024, 256, "fp64", 1, False)])
def test_steps_and_reads_in_turn_take_the_cheaper_route(nx, ny, precision, steps, walk):
    """After a read of the populations: a population step's bits, or a walk's. us a turn on a GB300, on
    populations and walking: 4 x 3000 FP32 37 and 23, 100 x 3000 FP64 with 4 steps 432 and 635."""
    p, _, rho0, f = setup(nx, ny, precision, 1, False)
    out = []
    for route in ("turns", "walk", "populations"):
        h = lbm.lbm_init(p, rho0)
        try:
            lbm.lbm_set_state(h, f)
            lbm.lbm_step(h, 7)
            if route == "populations":  # single steps from a state that was set
                for _ in range(steps):
                    lbm.lbm_set_state(h, read(h, p))
                    lbm.lbm_step(h, 1)
            else:
                if route == "turns":
                    read(h, p)
                lbm.lbm_step(h, steps)
            out.append(read(h, p))
        finally:
            lbm.lbm_destroy(h)
    assert np.array_equal(out[0], out[1 if walk else 2]) and not np.array_equal(out[1], out[2])
