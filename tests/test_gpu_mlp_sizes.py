"""The cost model's kernels at the edges of their tiles (32 samples a tile, 304
blocks of gradient sums, 128 samples a prediction block), against the FP64 MLP
oracle with the bound of the other gradient test, 1e-5."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2005_06332_gb300 import mm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 127, 128, 129, 304 * 32 - 1, 304 * 32 + 1, 30000])
def test_loss_gradient_and_prediction(n):
    rng = np.random.default_rng(n)
    theta = rng.normal(scale=0.3, size=omlp.N_PARAMS).astype(np.float32)
    X, y = rng.normal(size=(n, 16)).astype(np.float32), rng.normal(size=n).astype(np.float32)
    mu, sd = rng.normal(size=16).astype(np.float32), rng.uniform(0.5, 2.0, 16).astype(np.float32)
    m = mm.MLP(1)
    try:
        m.set_params(theta)
        m.set_normalisation(mu, sd, 0.25, 1.5)
        loss, g = m.loss_grad(X, y)
        again = m.loss_grad(X, y)
        out = m.predict(X)
    finally:
        m.close()
    Z = (X.astype(np.float64) - mu) / sd
    ref_loss, ref_g = omlp.loss_grad(omlp.bf16(theta), Z, (y.astype(np.float64) - 0.25) / 1.5)
    assert loss == pytest.approx(ref_loss, rel=1e-5)
    assert np.max(np.abs(g - ref_g)) <= 1e-5 * np.max(np.abs(ref_g))
    ref_y = omlp.forward(omlp.bf16(theta), Z)[0] * 1.5 + 0.25
    assert np.max(np.abs(out - ref_y)) <= 1e-5 * np.max(np.abs(ref_y))
    assert again[0] == loss and np.array_equal(again[1], g)  # the sums run in a fixed order
