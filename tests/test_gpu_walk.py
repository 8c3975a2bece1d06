"""The step on moments (all relaxation times 1) against the FP64 oracle at the edges of its
layout: segments of 8, 16 and 32 lanes (12, 28 and 60 owned columns), strips cut by the walls,
one to a few rows, both precisions, both gravity forms, both wall types, the thermal variant.

Tolerances as in test_gpu_parity.py: FP64 1e-14 a few steps on; FP32 1e-6 sqrt(n) + 1e-6.
"""
import ctypes
import math
import os

import numpy as np
import pytest

from oracle import eos
from oracle import lbm as olbm
from oracle import thermal as oth
from paper_2301_12869_gb300 import _build, inputs, lbm

pytestmark = pytest.mark.gpu

A, B, R = 0.25, 4.0, 1.0
_, T_C, _ = eos.critical_point(A, B, R)


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    if not os.path.exists(lbm.LIB_PATH):
        _build.build()
    lbm.load()


def setup(nx, ny, precision, form, zh, **kw):
    p = lbm.make_params(nx, ny, 0.85 * T_C, precision, a=A, form=form, g=(2e-5, -5e-5),
                        wall=lbm.LBM_WALL_ZOU_HE if zh else lbm.LBM_WALL_BOUNCE_BACK, **kw)
    op = olbm.Params(nx=nx, ny=ny, a=p.a, b=p.b, R=p.R, T=p.T, G=p.G, sigma=p.sigma, g=(p.gx, p.gy), form=form,
                     wall="zou-he" if zh else "bounce-back")
    rv, rl, _ = eos.maxwell(0.85 * T_C, A, B, R)
    rho0 = inputs.column_rho0(nx, ny, rl, rv, ny // 2, noise_amp=1e-3)
    return p, op, rho0, inputs.perturbed_populations(rho0, 1e-2, seed=nx + ny)


def read(h, p):
    f = np.empty((9, p.ny, p.nx))
    lbm.lbm_get_state(h, f)
    return f


def tolerance(precision, steps):
    return 1e-14 if precision == "fp64" else 1e-6 * math.sqrt(steps) + 1e-6


@pytest.mark.parametrize("nx, ny, precision, form, zh", [
    (4, 1, "fp32", 1, False), (4, 2, "fp32", 2, False), (12, 3, "fp32", 2, True), (16, 4, "fp32", 1, True),
    (24, 5, "fp32", 2, False), (28, 7, "fp32", 1, False), (32, 6, "fp32", 2, True), (60, 33, "fp32", 2, False),
    (64, 9, "fp32", 2, True), (120, 31, "fp32", 1, False), (124, 130, "fp32", 2, False), (1028, 64, "fp32", 2, True),
    (4, 900, "fp32", 2, False), (256, 260, "fp64", 2, False), (1040, 65, "fp64", 2, True), (62, 1100, "fp64", 1, False),
    (2, 200, "fp64", 2, False), (4, 200, "fp64", 1, True), (10, 37, "fp64", 2, True), (130, 41, "fp64", 2, False),
])
def test_step_on_moments_matches_oracle(nx, ny, precision, form, zh):
    p, op, rho0, f = setup(nx, ny, precision, form, zh)
    tol = tolerance(precision, 9)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        lbm.lbm_step(h, 6)  # populations -> moments, and on
        rho = np.empty((ny, nx))
        lbm.lbm_moments(h, rho)
        f = olbm.run(f, op, 6)
        assert np.max(np.abs(rho - olbm.macroscopic(f, op).rho)) <= tol
        lbm.lbm_step(h, 1)  # goes on from the moments
        f = olbm.step(f, op)
        got = read(h, p)
        assert np.max(np.abs(got - f)) <= tol
        mass = lbm.lbm_reduce(h, lbm.LBM_REDUCE_MASS)[0]
        assert mass == pytest.approx(float(np.sum(got)), rel=1e-12)  # of the populations read
        lbm.lbm_step(h, 2)  # the populations were read: the moments are still there
        f = olbm.run(f, op, 2)
        assert np.max(np.abs(read(h, p) - f)) <= tol
        ux, uy = np.empty((ny, nx)), np.empty((ny, nx))
        lbm.lbm_moments(h, None, ux, uy)
        mac = olbm.macroscopic(f, op)
        utol = (10 if precision == "fp64" else 30) * tol / mac.rho.min()
        assert np.max(np.abs(ux - mac.u[0])) <= utol and np.max(np.abs(uy - mac.u[1])) <= utol
        assert lbm.lbm_status(h) == lbm.LBM_OK
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("precision, zh", [("fp32", False), ("fp32", True), ("fp64", True)])
def test_parameters_change_between_steps(precision, zh):
    """lbm_set_params on a state held as moments: the populations belong to the old parameters,
    what the walls send back to the new ones; then another tile (populations again) and back."""
    nx, ny = (64, 40) if precision == "fp32" else (256, 257)
    p, op, rho0, f = setup(nx, ny, precision, 1, zh)
    tol = tolerance(precision, 12)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        lbm.lbm_step(h, 4)
        f = olbm.run(f, op, 4)
        p.gravity_form, p.gy, p.T = 2, 1e-4, 0.83 * T_C
        lbm.lbm_set_params(h, p)
        op.form, op.g, op.T = 2, (p.gx, p.gy), p.T
        assert np.max(np.abs(read(h, p) - f)) <= tol
        lbm.lbm_step(h, 4)
        f = olbm.run(f, op, 4)
        if not zh:
            lbm.lbm_set_tiling(h, 1)
        lbm.lbm_step(h, 1)
        lbm.lbm_set_tiling(h, 0)
        lbm.lbm_step(h, 5)
        f = olbm.run(f, op, 6)
        assert np.max(np.abs(read(h, p) - f)) <= tol
    finally:
        lbm.lbm_destroy(h)


@pytest.mark.parametrize("nx, ny, precision, zh", [(60, 21, "fp32", False), (124, 8, "fp32", True),
                                                   (256, 260, "fp64", False), (20, 30, "fp64", True)])
def test_thermal_step_on_moments(nx, ny, precision, zh):
    p, op, rho0, f = setup(nx, ny, precision, 2, zh, thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C)
    th = oth.Thermal(c_v=p.c_v, kappa=p.kappa, T_bot=p.T_bot, T_top=p.T_top)
    tol = tolerance(precision, 6)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_set_state(h, f)
        f = read(h, p)
        T = np.empty((ny, nx))
        lbm.lbm_get_temperature(h, T)
        for n in (5, 1):
            lbm.lbm_step(h, n)
            for _ in range(n):
                f, T = oth.thermal_step(f, T, op, th)
            Tg = np.empty((ny, nx))
            lbm.lbm_get_temperature(h, Tg)
            assert np.max(np.abs(read(h, p) - f)) <= tol
            assert np.max(np.abs(Tg - T)) <= tol
    finally:
        lbm.lbm_destroy(h)


def test_moments_into_arrays_off_a_16_byte_boundary():
    """Outputs are doubles on any 8-byte boundary, from a state held as moments too."""
    import torch

    p, op, rho0, f = setup(64, 20, "fp32", 2, False)
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_step(h, 8)
        want = torch.empty((3, 20, 64), dtype=torch.float64, device="cuda")
        lbm.lbm_moments(h, want[0], want[1], want[2])
        n = 20 * 64
        raw = torch.zeros(3 * (n + 1), dtype=torch.float64, device="cuda")
        ptrs = [raw.data_ptr() + 8 * (1 + k * (n + (n % 2))) for k in range(3)]
        assert all(q % 16 == 8 for q in ptrs)
        rc = lbm.load().lbm_moments(h, *[ctypes.c_void_p(q) for q in ptrs], lbm.LBM_DEVICE)
        assert rc == lbm.LBM_OK
        torch.cuda.synchronize()
        for k in range(3):
            off = (ptrs[k] - raw.data_ptr()) // 8
            assert torch.equal(raw[off:off + n].view(20, 64), want[k])
    finally:
        lbm.lbm_destroy(h)


def test_nonphysical_density_is_flagged_on_moments():
    p = lbm.make_params(8, 12, 0.8 * T_C, "fp32", a=A)
    rho0 = np.full((12, 8), 0.1)
    rho0[4:7, :] = 0.7  # p_EOS > rho / 3
    h = lbm.lbm_init(p, rho0)
    try:
        lbm.lbm_step(h, 4)
        assert lbm.lbm_status(h) == lbm.LBM_ENONPHYS
    finally:
        lbm.lbm_destroy(h)
