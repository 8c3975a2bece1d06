"""Steps and reads of a handle captured in a CUDA graph, mixed with direct calls: a replay changes the
state without the handle's knowledge, so after a captured call every read and step has to find what the
replays left. Against the FP64 oracle; tolerances as in test_gpu_walk.py, with 1e-13 in FP64 for up to
45 steps (a state a step old differs by 1e-4 and more).
"""
import numpy as np
import pytest

from oracle import lbm as olbm
from oracle import thermal as oth
from paper_2301_12869_gb300 import lbm
from test_gpu_walk import T_C, cuda_lib, read, setup, tolerance  # noqa: F401 (the fixture is used)

pytestmark = pytest.mark.gpu

# on the walk (FP32, FP64) and, in calls of 8 steps or more, on chip
WALKED = [(256, 200, "fp32", False), (256, 200, "fp32", True), (256, 257, "fp64", True)]
SMALL = [(64, 40, "fp32", True), (4, 60, "fp64", True)]


class Replayed:
    """A handle on its own stream; graphs of calls captured on it."""

    def __init__(self, nx, ny, precision, form, zh, gy=None, **kw):
        import torch

        self.torch = torch
        self.p, self.op, rho0, f = setup(nx, ny, precision, form, zh, **kw)
        if gy is not None:
            self.p.gy, self.op.g = gy, (self.p.gx, gy)
        self.s = torch.cuda.Stream()
        self.h = lbm.lbm_init(self.p, rho0, stream=self.s.cuda_stream)
        lbm.lbm_set_state(self.h, f)
        self.f = read(self.h, self.p)
        self.tol = 1e-13 if precision == "fp64" else tolerance(precision, 45)

    def capture(self, calls):
        g = self.torch.cuda.CUDAGraph()
        self.torch.cuda.synchronize()
        with self.torch.cuda.graph(g, stream=self.s):
            calls()
        return g

    def replay(self, g, steps=0):
        with self.torch.cuda.stream(self.s):
            g.replay()
        self.f = olbm.run(self.f, self.op, steps)

    def step(self, n):
        lbm.lbm_step(self.h, n)
        self.f = olbm.run(self.f, self.op, n)

    def check(self, got=None):
        got = read(self.h, self.p) if got is None else got
        assert np.max(np.abs(got - self.f)) <= self.tol
        mass = lbm.lbm_reduce(self.h, lbm.LBM_REDUCE_MASS)[0]
        assert mass == pytest.approx(float(np.sum(got)), rel=1e-9)
        rho = np.empty((self.p.ny, self.p.nx))
        lbm.lbm_moments(self.h, rho)
        assert np.max(np.abs(rho - olbm.macroscopic(self.f, self.op).rho)) <= self.tol


@pytest.fixture
def make():
    made = []

    def one(*args, **kw):
        made.append(Replayed(*args, **kw))
        return made[-1]

    yield one
    for r in made:
        r.torch.cuda.synchronize()
        lbm.lbm_destroy(r.h)


@pytest.mark.parametrize("read_before", [False, True])
@pytest.mark.parametrize("case", WALKED + SMALL)
@pytest.mark.parametrize("block", [2, 10])
def test_reads_between_replays(make, case, block, read_before):
    nx, ny, precision, zh = case
    r = make(nx, ny, precision, 2, zh)
    r.step(9)
    if read_before:
        r.check()
    g = r.capture(lambda: lbm.lbm_step(r.h, block))
    for _ in range(2):
        r.replay(g, block)
        r.check()
    r.step(1)
    r.check()


@pytest.mark.parametrize("case", WALKED + SMALL)
@pytest.mark.parametrize("block", [2, 10])
def test_direct_steps_between_replays(make, case, block):
    nx, ny, precision, zh = case
    r = make(nx, ny, precision, 2, zh)
    g = r.capture(lambda: lbm.lbm_step(r.h, block))  # captured from populations
    r.replay(g, block)
    r.step(10)
    r.replay(g, block)
    r.check()
    r.step(1)
    r.replay(r.capture(lambda: lbm.lbm_step(r.h, 1)), 1)  # an odd step back to the graph's buffers
    r.step(2)
    r.replay(g, block)
    r.check()


def test_sums_between_replays_on_chip(make):
    """lbm_moments forms the sums of <rho>; the next replay makes them old. Mass is not kept by Zou-He
    walls: with the sums of the replay before, the last step is off by g_y times its change (1e-8)."""
    nx, ny = 4, 60
    r = make(nx, ny, "fp64", 2, True, gy=-5e-3)
    g = r.capture(lambda: lbm.lbm_step(r.h, 10))
    rho = np.empty((ny, nx))
    for _ in range(2):
        r.replay(g, 10)
        lbm.lbm_moments(r.h, rho)
    r.replay(g, 10)
    r.step(1)
    r.check()


@pytest.mark.parametrize("case", WALKED + SMALL)
def test_captured_reads(make, case):
    """A captured read of the state is of the state at each replay, also after lbm_set_state."""
    nx, ny, precision, zh = case
    r = make(nx, ny, precision, 2, zh)
    r.step(9)  # held as moments
    out = r.torch.zeros((9, ny, nx), dtype=r.torch.float64, device="cuda")
    rho = r.torch.zeros((ny, nx), dtype=r.torch.float64, device="cuda")

    def calls():
        lbm.lbm_moments(r.h, rho)
        lbm.lbm_get_state(r.h, out)

    g = r.capture(calls)
    for advance in (lambda: None, lambda: r.step(2), lambda: r.step(12)):
        advance()
        r.replay(g)
        r.torch.cuda.synchronize()
        assert np.max(np.abs(rho.cpu().numpy() - olbm.macroscopic(r.f, r.op).rho)) <= r.tol
        r.check(out.cpu().numpy())
    lbm.lbm_set_state(r.h, r.f[:, ::-1].copy())
    r.f = read(r.h, r.p)
    r.replay(g)
    r.torch.cuda.synchronize()
    r.check(out.cpu().numpy())


@pytest.mark.parametrize("case", WALKED + SMALL)
def test_a_graph_that_is_never_replayed(make, case):
    nx, ny, precision, zh = case
    r = make(nx, ny, precision, 2, zh)
    r.step(9)
    r.capture(lambda: lbm.lbm_step(r.h, 2))
    r.check()
    r.step(6)
    r.check()


def test_set_state_between_replays(make):
    r = make(256, 200, "fp32", 2, False)
    r.step(9)
    g = r.capture(lambda: lbm.lbm_step(r.h, 2))
    lbm.lbm_set_state(r.h, r.f[:, :, ::-1].copy())
    r.f = read(r.h, r.p)
    r.replay(g, 2)
    r.check()


@pytest.mark.parametrize("read_first", [False, True])
def test_parameters_set_in_a_capture(make, read_first):
    """The populations belong to the parameters of the step that made them."""
    r = make(256, 200, "fp32", 1, True)
    r.step(9)
    r.p.gy, r.p.gravity_form = 2e-4, 2
    g = r.capture(lambda: (lbm.lbm_set_params(r.h, r.p), lbm.lbm_step(r.h, 2)))
    if read_first:
        assert np.max(np.abs(read(r.h, r.p) - r.f)) <= r.tol
    r.op.g, r.op.form = (r.p.gx, r.p.gy), 2
    for _ in range(2):
        r.replay(g, 2)
        r.check()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_thermal_replays(make, precision):
    nx, ny = 256, 260
    r = make(nx, ny, precision, 2, False, thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C)
    th = oth.Thermal(c_v=r.p.c_v, kappa=r.p.kappa, T_bot=r.p.T_bot, T_top=r.p.T_top)
    T, Tg = np.empty((ny, nx)), np.empty((ny, nx))
    lbm.lbm_get_temperature(r.h, T)
    f = r.f

    def advance(n):
        nonlocal f, T
        for _ in range(n):
            f, T = oth.thermal_step(f, T, r.op, th)

    lbm.lbm_step(r.h, 6)
    advance(6)
    g = r.capture(lambda: lbm.lbm_step(r.h, 2))
    for _ in range(2):
        r.replay(g)
        advance(2)
        lbm.lbm_get_temperature(r.h, Tg)
        assert np.max(np.abs(read(r.h, r.p) - f)) <= r.tol and np.max(np.abs(Tg - T)) <= r.tol
