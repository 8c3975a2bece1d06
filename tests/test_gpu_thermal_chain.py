"""A block of FP64 thermal steps, whose walk and Heun launches overlap at their ends, is not slower than
the same steps with the host waiting between them (1024 x 1024: blocks of the walk that shared an SM
took it from 448 to 628 us a step; the host's wait adds a launch's 10 us)."""
import numpy as np
import pytest

from paper_2301_12869_gb300 import lbm
from test_gpu_walk import T_C, cuda_lib, setup  # noqa: F401 (the fixture is used)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx, ny", [(1024, 1024), (470, 992)])
def test_block_of_thermal_steps(nx, ny):
    import torch

    p, _, rho0, _ = setup(nx, ny, "fp64", 2, False, thermal=1, T_bot=0.9 * T_C, T_top=0.8 * T_C)
    h = lbm.lbm_init(p, rho0, stream=torch.cuda.current_stream().cuda_stream)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def us_a_step(calls, steps):
        times = []
        for _ in range(5):
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(calls):
                lbm.lbm_step(h, steps)
                if steps == 1:
                    torch.cuda.synchronize()
            ev[1].record()
            torch.cuda.synchronize()
            times.append(1e3 * ev[0].elapsed_time(ev[1]) / (calls * steps))
        return float(np.median(times))

    try:
        lbm.lbm_step(h, 8)
        assert us_a_step(1, 8) <= 1.1 * us_a_step(8, 1)
    finally:
        lbm.lbm_destroy(h)
