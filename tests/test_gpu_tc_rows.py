"""Row kernels of the tensor-core context classes: the short strips that a
single image gets and the long ones of a batch give the same streams (a
plane's stream does not depend on the batch), with strips that end inside
and outside the plane."""
import numpy as np
import pytest

from tests._lib import ensure_built

pytestmark = pytest.mark.gpu
ensure_built()


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("C", [32, 64])
@pytest.mark.parametrize("H,W", [(132, 20), (136, 276), (150, 514)])
def test_single_equals_batch(prec, C, H, W):
    import paper_2405_12631_gb300 as pw
    codec = pw.Codec(0, prec)
    model = codec.init_random_model(2, C, 16, 0, seed=3)
    rng = np.random.default_rng(H * W + C)
    imgs = [rng.integers(0, 256, (H, W)).astype(np.uint8) for _ in range(2)]
    one = [codec.encode_image(model, im, q=8.0) for im in imgs]
    # 150 planes of 66 to 76 rows and more: the long strips at level 1
    many = codec.encode_batch(model, imgs * 75, q=8.0)
    assert all(many[i] == one[i % 2] for i in range(150))
    assert np.array_equal(codec.decode_symbols(model, one[1]),
                          codec.analyse(model, imgs[1], q=8.0, levels=2))
    back = codec.decode_batch(model, many[:150])
    assert np.array_equal(back[1], codec.decode_image(model, one[1]))
    model.close()
    codec.close()
