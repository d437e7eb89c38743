"""Protect of one image, one subtile of 32 channel-blocks per warp: sizes at which its pixel
loads, its last subtile, its AES rounds and its counter windows change form.  Bit-exact against
the CPU oracle, and at sizes the oracle is too slow for against the tensor-core form (a kernel of
its own)."""
import numpy as np
import pytest

from oracle import fds as ofds
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
    _api.counters(reset=True)
    yield _api
    assert _api.counters()[2] == 0


def _check(api, img, k, iv, offset=0):
    h, w, _ = img.shape
    key = synth.make_key(w + h + k)
    buf = torch.zeros(img.size + offset, dtype=torch.uint8, device=DEV)
    buf[offset:] = torch.from_numpy(img.reshape(-1)).to(DEV)
    pub, priv = api.protect_image(buf[offset:].view(h, w, 3), key, iv, k)
    want_pub, want_priv = ofds.protect(img, key, iv, k)
    assert np.array_equal(pub.cpu().numpy(), want_pub)
    assert priv.cpu().numpy().tobytes() == want_priv


# 11 and 12 blocks a row (piecewise / bulk pixel loads), rows that are and are not multiples of 16
# bytes, subtiles across one and several block rows, last subtiles of 3 .. 32 channel-blocks
@pytest.mark.parametrize("w,h", [(8, 8), (8, 264), (88, 24), (96, 8), (96, 64), (104, 40), (248, 16), (256, 8)])
@pytest.mark.parametrize("k", [0, 1, 4, 9, 20, 62, 63])
def test_sizes(api, w, h, k):
    _check(api, synth.make_image(w, h, 3 * w + h), k, synth.make_iv(k))


@pytest.mark.parametrize("w", [88, 120])
def test_pixels_at_an_8_byte_boundary(api, w):
    _check(api, synth.make_image(w, 32, w), 5, synth.make_iv(w), offset=8)


@pytest.mark.parametrize("iv", [bytes(15) + b"\xff", bytes(8) + b"\xff" * 8, b"\xff" * 16, b"\xff" * 15 + b"\x01"])
def test_counter_carries(api, iv):
    _check(api, synth.make_image(320, 72, 9), 5, iv)          # 4050 keystream blocks: 16 windows


def test_noise_image(api):
    img = np.random.default_rng(3).integers(0, 256, (120, 168, 3), dtype=np.uint8)
    _check(api, img, 5, synth.make_iv(4))


# k = 63 at 2600 x 2600: 65 counter windows per CTA, so its warps work on runs of their own
@pytest.mark.parametrize("w,h,k", [(2600, 2600, 63), (4104, 1032, 17)])
def test_large_against_the_tensor_core_form(api, w, h, k):
    img = torch.from_numpy(synth.make_image(w, h, 5)).to(DEV)
    key, iv = synth.make_key(6), b"\xff" * 14 + b"\x12\x34"
    pub, priv = api.protect_image(img, key, iv, k)
    pub2, priv2 = api.protect_image_tc(img, key, iv, k, "bf16")
    assert torch.equal(pub, pub2) and torch.equal(priv, priv2)
