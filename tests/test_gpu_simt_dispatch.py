"""SIMT convolutions: the small blocks that few tiles get and the large ones
of a batch give the same bits (a plane's stream does not depend on the
batch), on sizes around the tile edges and for every channel count."""
import numpy as np
import pytest

from tests._lib import ensure_built

pytestmark = pytest.mark.gpu
ensure_built()


@pytest.mark.parametrize("prec", ["fp32", "int8"])
@pytest.mark.parametrize("C", [32, 64, 128])
@pytest.mark.parametrize("H,W", [(16, 16), (17, 50), (80, 34), (130, 146)])
def test_single_equals_batch(prec, C, H, W):
    import paper_2405_12631_gb300 as pw
    codec = pw.Codec(0, prec)
    model = codec.init_random_model(4, C, 16, 0, seed=2)
    rng = np.random.default_rng(H * W + C)
    imgs = [rng.integers(0, 256, (H, W)).astype(np.uint8) for _ in range(2)]
    one = [codec.encode_image(model, im, q=8.0) for im in imgs]
    # 160 planes put every level of 80 x 34 and more on the large blocks
    many = codec.encode_batch(model, imgs * 80, q=8.0)
    assert all(many[i] == one[i % 2] for i in range(160))
    back = codec.decode_batch(model, many[:160])
    assert np.array_equal(back[0], codec.decode_image(model, one[0]))
    assert np.array_equal(codec.decode_symbols(model, one[1]), codec.analyse(model, imgs[1], q=8.0))
    model.close()
    codec.close()
