"""Columns iterated on chip (every relaxation time 1) against the FP64 oracle at the edges of
their layout: rows that fill a warp, a CTA or a cluster's share and one more, padded row widths,
single tall columns split over a cluster, both gravity forms and wall types; and the residual.

Tolerances: a few steps add a few ulp each - FP64 1e-14, double-float 1e-12, FP32
1e-6 sqrt(n) + 1e-6, as in the batch tests.
"""
import math
import os

import numpy as np
import pytest

from oracle import eos
from oracle import lbm as olbm
from paper_2301_12869_gb300 import _build, inputs, lbm

pytestmark = pytest.mark.gpu

A = 0.25
_, T_C, _ = eos.critical_point(A, 4.0, 1.0)
TOL = {"fp64": 1e-14, "dd": 1e-12}


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    if not os.path.exists(lbm.LIB_PATH):
        _build.build()
    lbm.load()


def columns(nx, heights):
    """Own T, g and form per column; densities with an x dependence, so that the shifts count."""
    cols, rhos = [], []
    for k, ny in enumerate(heights):
        T = (0.80 + 0.02 * (k % 6)) * T_C
        rv, rl, _ = eos.maxwell(T, A, 4.0, 1.0)
        cols.append(dict(ny=ny, T=T, gx=1e-5, gy=-2e-5, form=1 + k % 2))
        rhos.append(inputs.column_rho0(nx, ny, rl, rv, ny // 2, width=4.0, noise_amp=1e-3, noise_band=ny, seed=k))
    return cols, rhos


def split(flat, nx, heights):
    out, off = [], 0
    for ny in heights:
        out.append(flat[off:off + 9 * nx * ny].reshape(9, ny, nx))
        off += 9 * nx * ny
    return out


def run(nx, heights, precision, zh, steps, check_every=1000):
    cols, rhos = columns(nx, heights)
    p = lbm.make_params(nx, 8, 0.8 * T_C, precision, a=A,
                        wall=lbm.LBM_WALL_ZOU_HE if zh else lbm.LBM_WALL_BOUNCE_BACK)
    b = lbm.lbm_batch_init(p, cols, np.concatenate([r.ravel() for r in rhos]))
    try:
        n = 9 * nx * sum(heights)
        f0, f1 = np.empty(n), np.empty(n)
        lbm.lbm_batch_get_state(b, f0)
        lbm.lbm_batch_run(b, 0.0, steps, check_every)
        lbm.lbm_batch_get_state(b, f1)
        st, res, status = lbm.lbm_batch_results(b, len(cols))
    finally:
        lbm.lbm_batch_destroy(b)
    assert np.all(st == steps) and np.all(status == 0)
    ops = [olbm.Params(nx=nx, ny=c["ny"], a=A, T=c["T"], g=(c["gx"], c["gy"]), form=c["form"],
                       wall="zou-he" if zh else "bounce-back") for c in cols]
    return split(f0, nx, heights), split(f1, nx, heights), ops, res


@pytest.mark.parametrize("precision", ["fp32", "dd", "fp64"])
@pytest.mark.parametrize("nx, heights, zh", [
    (4, (3, 4, 5, 31, 32, 33, 63, 64, 65, 127, 128, 129), False),
    (4, (255, 256, 257, 511, 513, 1024), False),
    (4, (1024,), False),              # one column over a cluster
    (4, (1023, 700), True),
    (4, (3, 9, 64, 100, 130), True),
    (8, (5, 40, 77), False),          # wider rows: powers of two,
    (12, (3, 33), True),              # and rows padded to one
    (20, (7, 50, 210), False),
    (64, (9, 30), False),             # FP64 rows beyond a warp keep the general kernel
])
def test_columns_match_oracle(precision, nx, heights, zh):
    steps = 6
    f0, f1, ops, _ = run(nx, heights, precision, zh, steps)
    tol = TOL.get(precision, 1e-6 * math.sqrt(steps) + 1e-6)
    for g0, g1, op in zip(f0, f1, ops):
        err = float(np.max(np.abs(g1 - olbm.run(g0, op, steps))))
        assert err <= tol, (op.ny, op.form, err)


def test_two_wide_fp64_columns():
    f0, f1, ops, _ = run(2, (4, 61, 300), "fp64", False, 6)
    for g0, g1, op in zip(f0, f1, ops):
        assert np.max(np.abs(g1 - olbm.run(g0, op, 6))) <= 1e-14


@pytest.mark.parametrize("zh", [False, True])
@pytest.mark.parametrize("precision, check_every", [("fp32", 2), ("fp32", 5), ("dd", 5), ("fp64", 2)])
def test_residual_of_the_last_check(precision, check_every, zh):
    """max |rho_t - rho_(t-1)| of the streamed densities at the last check: FP32 densities are
    compared beyond FP32, so it follows the oracle's from the same state to a few FP32 ulp of
    the populations (5e-9 here), not of the density (3e-8)."""
    heights, steps = (20, 64, 300), 2 * check_every
    f0, _, ops, res = run(4, heights, precision, zh, steps, check_every)
    for g0, op, r in zip(f0, ops, res):
        f = olbm.run(g0, op, steps - 2)
        before = olbm.macroscopic(f, op).rho
        want = olbm.residual(olbm.macroscopic(olbm.step(f, op), op).rho, before)
        assert abs(r - want) <= (2e-7 if precision == "fp32" else 1e-12 + 1e-6 * want), (op.ny, r, want)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_extrapolated_run_reaches_the_same_steady_state(precision):
    """The extrapolation works on the moments here: same state as without it (1e-5, as the batch
    tests hold it), in no more steps in all."""
    heights = (40, 64, 300)
    cols, rhos = columns(4, heights)
    rhos = [np.repeat(r.mean(axis=1, keepdims=True), 4, axis=1) for r in rhos]
    for c in cols:
        c["gx"] = 0.0
    tol = 3e-8 if precision == "fp32" else 1e-10
    out = []
    for checks in (0, 5):
        b = lbm.lbm_batch_init(lbm.make_params(4, 8, 0.8 * T_C, precision, a=A), cols, np.concatenate([r.ravel() for r in rhos]))
        try:
            lbm.lbm_batch_set_acceleration(b, checks)
            lbm.lbm_batch_run(b, tol, 400000, 100)
            st, res, status = lbm.lbm_batch_results(b, len(cols))
            rho = np.empty(4 * sum(heights))
            lbm.lbm_batch_moments(b, rho)
            out.append((st, res, status, rho))
        finally:
            lbm.lbm_batch_destroy(b)
    for st, res, status, _ in out:
        assert np.all(status == 0) and np.all(res <= tol), (st, res)
    assert np.sum(out[1][0]) <= np.sum(out[0][0])
    if precision == "fp64":
        assert np.max(np.abs(out[0][3] - out[1][3])) <= 1e-5
