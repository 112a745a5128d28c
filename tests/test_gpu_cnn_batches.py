"""The predictor's one-kernel pass at the edges of its grid: fewer samples than
CTAs, one more than fit at once, several rounds; the forward pass alone against
the logits of the gradient pass."""
import numpy as np
import pytest

from oracle import cnn as ocnn
from paper_2403_15435_gb300 import geoflood, inputs

pytestmark = pytest.mark.gpu


def params():
    rng = np.random.default_rng(21)
    prm = ocnn.init_params(rng)
    for l in range(3):
        prm[l * 2320 + 2304:l * 2320 + 2320] = rng.normal(0, 0.05, 16)
    return prm.astype(np.float32)


@pytest.mark.parametrize("n", [1, 2, 455, 457, 1000])
def test_gradient_of_a_batch_matches_oracle(n):
    rng = np.random.default_rng(n)
    x = rng.normal(0.3, 0.7, (n, 324, 16)).astype(np.float32)
    x = (x.view(np.uint32) >> 16).astype(np.uint16)
    y = (rng.random(n) < 0.3).astype(np.float32)
    g = geoflood.Forest(inputs.Config(mi=1, mj=1, mx=32))
    prm = params()
    g.cnn_set_params(prm)
    z, grad, loss = g.cnn_grad(x, y, pos_weight=3.0)
    l_ref, g_ref, f = ocnn.loss_and_grad(ocnn.bf16_bits_to_float(x), y, prm.astype(np.float64),
                                         3.0, rounding=True)
    # both round to BF16 at the same points; a pixel whose FP32 and FP64 sums
    # fall on two sides of a rounding point moves a logit by 2^-9 / 256 of the
    # pixel's value, which the bound on z holds for a few such pixels
    assert np.abs(z - f["z"]).max() <= 1e-4 * max(1.0, np.abs(f["z"]).max())
    assert abs(loss - l_ref) <= 1e-4 * max(1.0, l_ref)
    for a, b in ((0, 2304), (2304, 2320), (2320, 4624), (4624, 4640), (4640, 6944),
                 (6944, 6960), (6960, 6976), (6976, 6977)):
        # sums of n x 256 terms in FP32 and the rare differing roundings
        assert np.linalg.norm(grad[a:b] - g_ref[a:b]) <= 2e-3 * np.linalg.norm(g_ref[a:b]), a


@pytest.mark.parametrize("mi,mj", [(1, 1), (19, 32), (19, 33)])
def test_prediction_equals_the_gradient_passes_logits(mi, mj):
    cfg = inputs.Config(mi=mi, mj=mj, mx=16, xupper=16.0 * mi, yupper=16.0 * mj, drytol=1e-3)
    g = geoflood.Forest(cfg)
    g.set_state(lambda x, y, b: (1.5 + np.sin(x / 9.0), 0.3 * x / 300.0, 0.2 + 0 * y))
    g.cnn_set_params(params())
    x = g.cnn_features()
    z = g.cnn_predict()
    zg, _, _ = g.cnn_grad(x, np.zeros(len(x), np.float32))
    assert len(z) == mi * mj and np.array_equal(z, zg)
