"""Packed storage, one subtile of 32 channel-blocks per warp: rows of 11, 12, 13 and 31 blocks
(piecewise / bulk pixel loads, stores of short rows), k at which the private fields are packed in
place or beside the public ones and at which either part is empty or nearly so.  Against the
oracle's packed storage, byte for byte."""
import numpy as np
import pytest

from oracle import pack
from paper_1512_02951_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_02951_gb300 import api as _api, build

    build.build()
    _api.init(0)
    return _api


@pytest.mark.parametrize("form", [11, 8])
@pytest.mark.parametrize("w,h", [(88, 8), (96, 24), (104, 56), (248, 40)])
@pytest.mark.parametrize("k", [0, 1, 4, 5, 20, 41, 62, 63])
def test_packed_subtiles(api, form, w, h, k):
    img = np.random.default_rng(w + h + k).integers(0, 256, (h, w, 3), dtype=np.uint8)
    key, iv = synth.make_key(w + k), b"\xff" * 15 + bytes([0xf0 + k % 16])      # the counter's low byte wraps
    pub, priv = api.protect_image_packed(torch.from_numpy(img).to(DEV), key, iv, k, form)
    want_pub, want_priv = pack.protect_packed(img, key, iv, k, form)
    assert pub.cpu().numpy().tobytes() == want_pub
    assert priv.cpu().numpy().tobytes() == want_priv
    back = api.restore_image_packed(pub, priv, w, h, k, key, iv, form).cpu().numpy()
    assert np.array_equal(back, pack.restore_packed(want_pub, want_priv, key, iv, k, form, w, h))
