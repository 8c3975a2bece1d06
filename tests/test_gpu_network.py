"""The fused training pass and the forward kernel's tile layouts at their edges, against the
oracle in its bfloat16-storage mode with the bounds of test_gpu_mlp.py (2^-10 of an element's
magnitude everywhere, 2^-14 on all but 0.1 %)."""
import os

import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2301_12869_gb300 import _build, inputs, lbm
from test_gpu_mlp import assert_elementwise, features, magnitudes, params_for_test, rel_err, to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    if not os.path.exists(lbm.LIB_PATH):
        _build.build()
    lbm.load()


def network_inputs(raw):
    return omlp.normalise(raw.astype(np.float64)).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n", [1, 127, 129, 1000, 152 * 128 + 130])
def test_gradients_over_tiles(n):
    """One row, a tile and its neighbours, several CTAs, and more tiles than SMs (the CTA's
    accumulators carry over from its first tile to its second)."""
    raw, t = features(n, 21)
    h = lbm.lbm_mlp_create(lbm.mlp_pack(params_for_test(6)), 128 * (-(-n // 128)))
    try:
        Pf = lbm.mlp_unpack(lbm.lbm_mlp_get_params(h))
        x, t64 = network_inputs(raw), t.astype(np.float64)
        for _ in range(2):  # a second pass starts from zero gradients again
            loss, g = lbm.lbm_mlp_gradients(h, to_gpu(raw), to_gpu(t))
        G = lbm.mlp_unpack(g)
        l16, g16 = omlp.loss_and_grads(x, t64, Pf, bf16=True)
        S, _ = magnitudes(x, t64, Pf)
        assert loss == pytest.approx(l16, rel=2e-3)
        for k in g16:
            assert_elementwise(G[k], g16[k], S[k], k)
            assert rel_err(G[k], g16[k]) <= 2e-3, k
    finally:
        lbm.lbm_mlp_destroy(h)


def test_losses_of_more_steps_than_are_kept_on_the_device():
    """Losses are read back in blocks of 1024 steps; the first of each run of steps and the last
    follow the oracle's loss of the parameters of the time (lr tiny: the first ones throughout)."""
    raw, t = features(300, 22)
    h = lbm.lbm_mlp_create(lbm.mlp_pack(params_for_test(7)), 128)
    try:
        Pf = lbm.mlp_unpack(lbm.lbm_mlp_get_params(h))
        losses = lbm.lbm_mlp_train(h, to_gpu(raw), to_gpu(t), 100, 1030, 1e-12, 5)
        x = network_inputs(raw)
        for step in (0, 1, 1023, 1024, 1029):
            idx = inputs.minibatch_indices(300, 100, step, 5)
            want = omlp.loss_and_grads(x[idx], t[idx].astype(np.float64), Pf, bf16=True)[0]
            assert losses[step] == pytest.approx(want, rel=5e-3), step
    finally:
        lbm.lbm_mlp_destroy(h)


@pytest.mark.parametrize("n", [1, 100, 128, 129, 128 * 151 + 5, 128 * 152, 128 * 152 + 1, 128 * 608 + 60])
def test_forward_tile_layouts(n):
    """Fewer rows than a tile, tiles up to one a CTA (all warps on a tile) and beyond (four
    pipelines a CTA), and more than one round of those."""
    import torch

    raw, _ = features(n, 23)
    h = lbm.lbm_mlp_create(lbm.mlp_pack(params_for_test(8)), 128)
    try:
        Pf = lbm.mlp_unpack(lbm.lbm_mlp_get_params(h))
        y = torch.full((n,), float("nan"), dtype=torch.float32, device="cuda")
        lbm.lbm_mlp_predict(h, to_gpu(raw), y)
        got = y.cpu().numpy()
        assert np.all(np.isfinite(got))
        rows = np.unique(np.concatenate([np.arange(min(n, 130)), np.arange(max(0, n - 130), n),
                                         np.random.default_rng(4).integers(0, n, 500)]))
        x = network_inputs(raw[rows])
        want, _ = omlp.forward(x, Pf, bf16=True)
        _, aY = magnitudes(x, np.zeros(len(x)), Pf)
        assert_elementwise(got[rows], want, aY, "forward")
    finally:
        lbm.lbm_mlp_destroy(h)
