"""What columns on chip do at a residual check: the residual itself, formed in FP64 from the library's
own states, and one extrapolation cycle, formed in FP64 from the library's own snapshots."""
import numpy as np
import pytest

from oracle import eos
from oracle import lbm as olbm
from paper_2301_12869_gb300 import inputs, lbm
from test_gpu_column import A, T_C, columns, cuda_lib, run, split  # noqa: F401 (the fixture is used)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision, zh", [("fp32", False), ("fp32", True), ("dd", False), ("dd", True), ("fp64", False)])
@pytest.mark.parametrize("steps", [2, 5, 40])
def test_residual_beyond_the_storage_type(precision, zh, steps):
    """max |rho_t - rho_(t-1)| of a check, against the same from the populations of runs that stop one
    and two steps before, read back in FP64. A column holds its density to 48 bits for it (FP32: the
    value and what its rounding lost), 2e-15 of a density below 0.3 in each of a dozen sums: 5e-14. An FP32
    density alone is off by 1e-8, an FP32 difference by 1e-11 of these changes of 1e-4. Zou-He
    nodes in FP32 take their density from FP32 sums of the known populations: 1e-8."""
    nx, heights = 4, (20, 64, 300)
    states = [run(nx, heights, precision, zh, n)[1] if n else run(nx, heights, precision, zh, 1)[0]
              for n in (steps - 2, steps - 1)]
    _, _, ops, res = run(nx, heights, precision, zh, steps, check_every=steps)
    tol = 1e-8 if zh and precision == "fp32" else 5e-14
    for f0, f1, op, r in zip(*states, ops, res):
        want = olbm.residual(olbm.macroscopic(f1, op).rho, olbm.macroscopic(f0, op).rho)
        assert abs(r - want) <= tol, (op.ny, r, want)


def moments(f):
    g = olbm.stream(f)
    return np.stack([g.sum(axis=0), np.tensordot(olbm.C[:, 0], g, 1), np.tensordot(olbm.C[:, 1], g, 1)])


def extrapolated(states):
    """Minimal polynomial extrapolation of order 4 of six states: their weights, which are those of
    the moments' differences."""
    x = [moments(f).ravel() for f in states]
    u = np.stack([x[j + 1] - x[j] for j in range(5)], axis=1)
    c = np.append(np.linalg.lstsq(u[:, :4], -u[:, 4], rcond=None)[0], 1.0)
    return c / c.sum()


@pytest.mark.parametrize("precision", ["fp32", "dd", "fp64"])
def test_one_extrapolation_cycle(precision):
    """A run of one cycle (six snapshots, one every two checks) ends with the step from the
    estimate, like a run whose cycle ends before its last step. The populations are then the collision of
    the snapshots' weighted mean. Rounding the snapshots' moments (1e-8, 1e-15) moves the estimate by 2e-6
    (FP32) and 3e-13 (double-float) of its distance from the plain state here, storing it by 3e-6 and 3e-13."""
    nx, heights, every, checks = 4, (40, 64, 300), 25, 2
    cols, rhos = columns(nx, heights)
    flat = np.concatenate([r.ravel() for r in rhos])
    p = lbm.make_params(nx, 8, 0.8 * T_C, precision, a=A)
    n = 9 * nx * sum(heights)

    def states(steps, acc):
        b = lbm.lbm_batch_init(p, cols, flat)
        try:
            if acc:
                lbm.lbm_batch_set_acceleration(b, checks)
            lbm.lbm_batch_run(b, 0.0, steps, every)
            f = np.empty(n)
            lbm.lbm_batch_get_state(b, f)
            return split(f, nx, heights)
        finally:
            lbm.lbm_batch_destroy(b)

    last = 6 * checks * every
    plain = [states(k * checks * every - 1, False) for k in range(1, 7)]  # what the snapshots' steps start from
    got, without = states(last, True), states(last, False)
    ops = [olbm.Params(nx=nx, ny=c["ny"], a=A, T=c["T"], g=(c["gx"], c["gy"]), form=c["form"]) for c in cols]
    for j, op in enumerate(ops):
        w = extrapolated([s[j] for s in plain])
        want = olbm.step(sum(wk * s[j] for wk, s in zip(w, plain[:5])), op)
        moved = float(np.max(np.abs(want - without[j])))
        err = float(np.max(np.abs(got[j] - want)))
        assert moved > 1e-4 and err <= TOLERANCE[precision] * moved, (op.ny, err, moved)


# of that distance
TOLERANCE = {"fp32": 1e-4, "dd": 1e-10, "fp64": 1e-11}


def test_double_float_error_over_a_block_of_steps():
    """32 columns of 64 rows, 300 steps, against FP64: 3.0e-14 of the populations' norm in a numpy
    emulation of the kernel's arithmetic over 384 such columns, 4.3e-14 in that of the general kernel and
    5.1e-14 with a constant 1/3 in psi and its stencil; 32 columns spread by 5 %."""
    ncol, nx, ny, steps = 32, 4, 64, 300
    rng = np.random.default_rng(1)
    T, gy = rng.uniform(0.75, 0.9, ncol) * T_C, -(10 ** rng.uniform(-5.5, -4.3, ncol))
    cols, rhos = [], []
    for k in range(ncol):
        rv, rl, _ = eos.maxwell(T[k], A, 4.0, 1.0)
        cols.append(dict(ny=ny, T=float(T[k]), gx=0.0, gy=float(gy[k]), form=1 + k % 2))
        rhos.append(inputs.column_rho0(nx, ny, rl, rv, ny // 2, width=4.0))
    b = lbm.lbm_batch_init(lbm.make_params(nx, 8, 0.8 * T_C, "dd", a=A), cols, np.concatenate([r.ravel() for r in rhos]))
    try:
        lbm.lbm_batch_run(b, 0.0, steps, 1000)
        f = np.empty(9 * nx * ny * ncol)
        lbm.lbm_batch_get_state(b, f)
    finally:
        lbm.lbm_batch_destroy(b)
    want = np.stack([olbm.run(olbm.init_state(r), olbm.Params(nx=nx, ny=ny, a=A, T=c["T"], g=(0.0, c["gy"]), form=c["form"]),
                              steps) for r, c in zip(rhos, cols)])
    got = np.stack(split(f, nx, [ny] * ncol))
    assert np.linalg.norm(got - want) / np.linalg.norm(want) <= 4.0e-14


def test_block_size_of_columns_on_chip():
    """Their block size follows their height: nothing to choose, so one measurement stands for the
    three candidates, and what lbm_batch_set_threads set stays."""
    cols, rhos = columns(4, (40, 64))
    b = lbm.lbm_batch_init(lbm.make_params(4, 8, 0.8 * T_C, "fp32", a=A), cols, np.concatenate([r.ravel() for r in rhos]))
    try:
        lbm.lbm_batch_set_threads(b, 512)
        kept, times = lbm.lbm_batch_autotune(b, 20)
        assert kept == 512 and sorted(times) == [128, 256, 512]
        assert len(set(times.values())) == 1 and times[512] > 0
    finally:
        lbm.lbm_batch_destroy(b)
