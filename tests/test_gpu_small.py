"""Small lattices of a handle, stepped on chip a block at a time, against the FP64 oracle: at both
sides of the sizes that choose them (FP32 2^14 nodes and 128 columns, FP64 2^11 and 32), with
single steps, reads and parameter changes between the blocks, and in a replayed CUDA graph.

Tolerances as in test_gpu_parity.py: FP64 1e-14 a few steps on; FP32 1e-6 sqrt(n) + 1e-6.
"""
import ctypes
import os

import numpy as np
import pytest

from oracle import lbm as olbm
from paper_2301_12869_gb300 import _build, lbm
from test_gpu_walk import T_C, read, setup, tolerance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    if not os.path.exists(lbm.LIB_PATH):
        _build.build()
    lbm.load()


@pytest.mark.parametrize("nx, ny, precision, form, zh", [
    (4, 4096, "fp32", 2, False), (4, 4097, "fp32", 1, False), (128, 128, "fp32", 2, True), (128, 129, "fp32", 2, False),
    (132, 40, "fp32", 1, False), (68, 240, "fp32", 2, False), (16, 3, "fp32", 2, True), (4, 1, "fp32", 1, False),
    (32, 64, "fp64", 2, False), (32, 65, "fp64", 1, False), (34, 60, "fp64", 2, False), (2, 1024, "fp64", 2, True),
    (22, 93, "fp64", 1, True), (4, 1, "fp64", 2, False),
])
def test_blocks_and_single_steps(nx, ny, precision, form, zh):
    p, op, rho0, f = setup(nx, ny, precision, form, zh)
    tol = tolerance(precision, 31)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        for block in ((9,), (1,), (2, 1, 1, 1), (1, 8), (7,)):  # the state is read after each
            for n in block:
                lbm.lbm_step(h, n)
            f = olbm.run(f, op, sum(block))
            got = read(h, p)
            assert np.max(np.abs(got - f)) <= tol, block
            assert lbm.lbm_reduce(h, lbm.LBM_REDUCE_MASS)[0] == pytest.approx(float(np.sum(got)), rel=1e-12)
        rho = np.empty((ny, nx))
        lbm.lbm_moments(h, rho)
        assert np.max(np.abs(rho - olbm.macroscopic(f, op).rho)) <= tol
        assert lbm.lbm_status(h) == lbm.LBM_OK
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_parameters_change_between_blocks(precision):
    """To a general relaxation time (the population step), another gravity form, and back."""
    p, op, rho0, f = setup(8, 100, precision, 2, False)
    tol = tolerance(precision, 27)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        for tau, form in ((1.0, 2), (0.9, 1), (1.0, 2)):
            p.tau_nu, p.gravity_form = tau, form
            op.tau_nu, op.form = tau, form
            lbm.lbm_set_params(h, p)
            lbm.lbm_step(h, 9)
            f = olbm.run(f, op, 9)
        assert np.max(np.abs(read(h, p) - f)) <= tol
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("nx, ny, precision", [(4, 60, "fp64"), (64, 40, "fp32"), (256, 200, "fp32")])
@pytest.mark.parametrize("before", [0, 9])
@pytest.mark.parametrize("block", [2, 10])
def test_captured_steps_replay(nx, ny, precision, before, block):
    """Steps captured in a CUDA graph (an even number: two buffers take turns) and replayed, from
    a state just set or already stepped, on the walk and on chip; then steps without the graph."""
    import torch

    p, op, rho0, f = setup(nx, ny, precision, 2, False)
    tol = tolerance(precision, before + 3 * block + 2)
    s = torch.cuda.Stream()
    h = lbm.lbm_init(p, rho0, stream=s.cuda_stream)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        lbm.lbm_step(h, before)
        if before:
            read(h, p)  # the sums of an on-chip block are not formed until something needs them
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            lbm.lbm_step(h, block)
        with torch.cuda.stream(s):
            for _ in range(3):
                g.replay()
        lbm.lbm_step(h, 2)
        f = olbm.run(f, op, before + 3 * block + 2)
        assert np.max(np.abs(read(h, p) - f)) <= tol
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("offset", [0, 1])
def test_state_in_and_out_keep_every_value(precision, offset):
    """Device states on 16- and 8-byte boundaries: each value minus its share of the reference,
    rounded once to the storage type - ties, denormals, infinities and NaN among them - and back."""
    import torch

    nx, ny = 64, 37
    n = nx * ny
    rho_ref = 0.0 if offset else 0.173
    rng = np.random.default_rng(5)
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        v = rng.normal(size=9 * n) * np.exp2(rng.integers(-160, 132, 9 * n))
        half = np.float32(rng.normal(size=n)).astype(np.float64)  # halfway between two FP32 values
        v[:n] = half + np.float64(np.spacing(np.float32(half))) / 2
        v[n:n + 12] = [0.0, -0.0, np.inf, -np.inf, np.nan, 2.0**-126, -2.0**-126 * (1 - 2.0**-25), 2.0**-149, 2.0**-150,
                       3.4028235677973366e38, 2.0**127, 1 - 2.0**-26]
        raw = torch.zeros(9 * n + 1, dtype=torch.float64, device="cuda")
        src = raw[offset:offset + 9 * n]
        src.copy_(torch.from_numpy(v))
        assert src.data_ptr() % 16 == 8 * offset
        w = np.repeat(np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4), n) * rho_ref
        want = v - w
        if precision == "fp32":
            want = want.astype(np.float32).astype(np.float64)
        want = want + w
    h = lbm.lbm_init(lbm.make_params(nx, ny, 0.85 * T_C, precision, a=0.25, rho_ref=rho_ref), np.full((ny, nx), 0.1))
    out = torch.zeros(9 * n + 1, dtype=torch.float64, device="cuda")[offset:offset + 9 * n]
    try:
        lib = lbm.load()
        assert lib.lbm_set_state(h, ctypes.c_void_p(src.data_ptr()), lbm.LBM_DEVICE, 0) == lbm.LBM_OK
        assert lib.lbm_get_state(h, ctypes.c_void_p(out.data_ptr()), lbm.LBM_DEVICE, None) == lbm.LBM_OK
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        lbm.lbm_destroy(h)
    assert np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("thermal", [0, 1])
def test_density_alone_is_the_density_with_the_velocity(thermal):
    """rho of a state held as moments, without the stencil and with it."""
    nx, ny = 256, 257
    kw = dict(thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C) if thermal else {}
    p, _, rho0, f = setup(nx, ny, "fp64", 1, False, **kw)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        lbm.lbm_step(h, 6)
        rho, rho2, ux = np.empty((ny, nx)), np.empty((ny, nx)), np.empty((ny, nx))
        lbm.lbm_moments(h, rho)
        lbm.lbm_moments(h, rho2, ux)
        assert np.array_equal(rho, rho2)
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("factor, code", [(1.0, lbm.LBM_OK), (40.0, lbm.LBM_ENONPHYS)])
def test_density_alone_reports_what_psi_would(precision, factor, code):
    """A temperature at which p_EOS > rho/3 is set under a state held as moments: psi^2 < 0 is
    reported by rho alone, before any step."""
    nx, ny = 256, 257
    p, _, rho0, f = setup(nx, ny, precision, 1, False, thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        lbm.lbm_step(h, 6)
        lbm.lbm_set_temperature(h, np.full((ny, nx), 0.85 * T_C * factor))
        rho = np.empty((ny, nx))
        rc = lbm.load().lbm_moments(h, rho.ctypes.data_as(ctypes.c_void_p), None, None, lbm.LBM_HOST)
        assert rc == code and np.all(rho > 0)
    finally:
        lbm.lbm_destroy(h)
