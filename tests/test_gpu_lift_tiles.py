"""FP32 lifting step: sizes around the edges of both tiles (30 x 14 and 14 x
6 outputs), where planes change from one to the other, against the oracle's
FP64 transform, and element by element in the integer mode."""
import numpy as np
import pytest

import synthetic as S
from oracle import codec as K
from tests._lib import ensure_built

pytestmark = pytest.mark.gpu
ensure_built()


@pytest.fixture(scope="module")
def env():
    import paper_2405_12631_gb300 as pw
    cfg = S.ModelConfig(levels=1, C=32, ll_mode=0)
    blob = S.pack_blob(cfg, S.random_model(cfg, 3))
    c = pw.Codec(0, "fp32")
    m = c.load_model(blob)
    yield c, m, K.Model(blob)
    m.close()
    c.close()


# one level: the steps run on (2h x w) and (h x w) planes of an H x W input
SIZES = [(2, 2), (4, 60), (12, 28), (14, 30), (28, 62), (26, 58), (90, 34),
         (420, 182), (430, 640), (452, 600)]


@pytest.mark.parametrize("H,W", SIZES)
def test_lossy_matches_oracle(env, H, W):
    c, m, om = env
    x = np.random.default_rng(H * 1000 + W).normal(0, 60, (H, W)).astype(np.float32)
    ref = om.lift.forward(x.astype(np.float64), 1, False)
    got = c.lift_forward(m, x)
    # FP32 sums of 2592 products of O(1) weights: the bound of the other lifting tests
    np.testing.assert_allclose(got, np.concatenate([r.reshape(-1) for r in ref]), atol=2e-3)
    np.testing.assert_allclose(c.lift_inverse(m, got, H, W), x, atol=2e-3)


@pytest.mark.parametrize("H,W", SIZES)
def test_integer_mode_exact(env, H, W):
    c, m, om = env
    x = np.random.default_rng(H + W).integers(-2048, 2048, (H, W)).astype(np.float32)
    ref = np.concatenate([r.reshape(-1) for r in om.lift.forward(x, 1, True)])
    got = c.lift_forward(m, x, lossless=True)
    assert np.array_equal(got, ref.astype(np.float32))
    assert np.array_equal(c.lift_inverse(m, got, H, W, lossless=True), x)
