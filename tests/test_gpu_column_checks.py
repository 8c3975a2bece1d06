"""What columns on chip do at a residual check: the residual itself, formed in FP64 from the library's
own states."""
import pytest

from oracle import lbm as olbm
from test_gpu_column import cuda_lib, run  # noqa: F401 (the fixture is used)

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
