"""The cost model's prediction at the edges of its blocks (256 samples a block,
1,216 blocks and then a second round), against the FP64 MLP oracle with the
bound of the other prediction test, 1e-5."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2005_06332_gb300 import mm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [255, 256, 257, 511, 512, 513, 1216 * 256 - 1, 1216 * 256, 1216 * 256 + 129])
def test_prediction(n):
    rng = np.random.default_rng(n)
    theta = rng.normal(scale=0.3, size=omlp.N_PARAMS).astype(np.float32)
    X = rng.normal(size=(n, 16)).astype(np.float32)
    mu, sd = rng.normal(size=16).astype(np.float32), rng.uniform(0.5, 2.0, 16).astype(np.float32)
    m = mm.MLP(1)
    try:
        m.set_params(theta)
        m.set_normalisation(mu, sd, 0.25, 1.5)
        out = m.predict(X)
    finally:
        m.close()
    ref = omlp.forward(omlp.bf16(theta), (X.astype(np.float64) - mu) / sd)[0] * 1.5 + 0.25
    assert np.max(np.abs(out - ref)) <= 1e-5 * np.max(np.abs(ref))
