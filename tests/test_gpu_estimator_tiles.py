"""The estimator's kernels at the edges of their 32-row tiles and of the grid
(two blocks an SM: past that a block takes several tiles), against the
numpy oracle in float64."""

import numpy as np
import pytest

from oracle import mlp
from workloads import mlp_init_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 1000, 152 * 2 * 32 + 1, 40000])
def test_output_and_gradient_at_tile_edges(dspg, n):
    rng = np.random.default_rng(n)
    X = np.log2(1 + rng.integers(0, 5000, (n, 4))).astype(np.float32)
    y = np.log2(1 + rng.integers(0, 5000, n)).astype(np.float32)
    p = mlp_init_params(7).astype(np.float32)
    est = dspg.Estimator(p)
    want, _ = mlp.forward(p, X)
    got = est.predict(X).cpu().numpy()
    # 64 float32 multiply-adds a layer: 2 * 64 * 2^-24 of the magnitudes summed (all below 1e3 here)
    assert np.allclose(got, want, rtol=0, atol=2 * 64 * 2.0 ** -24 * 1e3)
    loss, g = est.grad(X, y)
    wl, wg = mlp.loss_and_grad(p, X, y)
    assert abs(loss - wl) <= 1e-5 * wl
    assert np.all(np.abs(g - wg) <= 1e-3 * np.abs(wg) + 1e-4 * np.abs(wg).max())  # the bound of test_gpu_estimator.py
    loss2, g2 = est.grad(X, y)
    assert loss2 == loss and np.array_equal(g, g2)  # every sum has a fixed order
    est.close()


@pytest.mark.parametrize("at", [0, 1, 3])
def test_outputs_over_their_inputs(dspg, at):
    """dspg_estimator_predict into memory that its inputs lie in: from the
    first row on, inside, and over the last quarter."""
    import torch
    n = 40000
    rng = np.random.default_rng(at)
    X = torch.from_numpy(np.log2(1 + rng.integers(0, 5000, (n, 4))).astype(np.float32)).cuda()
    est = dspg.Estimator(mlp_init_params(7).astype(np.float32))
    want = est.predict(X)
    out = X.reshape(-1)[at * n:][:n]
    torch.cuda.synchronize()
    assert dspg.load().dspg_estimator_predict(est._e, X.data_ptr(), n, out.data_ptr(), None) == 0
    assert torch.equal(out, want)
    est.close()
