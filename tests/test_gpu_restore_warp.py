"""Restore of one image, one subtile of 32 channel-blocks per warp: sizes at which its last
subtile, its shared blocks, its runs of private parts and its counter windows change form.
Bit-exact against the CPU oracle, and at sizes the oracle is too slow for against the tensor-core
form (a kernel of its own)."""
import numpy as np
import pytest

from oracle import aes as oaes, fds as ofds
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


def _restore(api, pub, priv, w, h, k, key, iv, offset=0):
    out = torch.zeros(3 * w * h + offset, dtype=torch.uint8, device=DEV)
    p = torch.from_numpy(np.ascontiguousarray(pub)).to(DEV)
    v = torch.frombuffer(bytearray(priv), dtype=torch.uint8).to(DEV)
    api.restore_image(p, v, w, h, k, key, iv, out[offset:].view(h, w, 3))
    return out[offset:].view(h, w, 3).cpu().numpy()


# last subtiles of 3 .. 32 channel-blocks, blocks shared by two subtiles in every way, block rows
# shorter than a subtile; k at which runs are 8 .. 1 subtiles long and (42 and above) one buffer
@pytest.mark.parametrize("w,h", [(8, 8), (8, 264), (88, 24), (96, 64), (104, 40), (248, 16)])
@pytest.mark.parametrize("k", [0, 1, 4, 9, 41, 42, 62, 63])
def test_sizes(api, w, h, k):
    img, key, iv = synth.make_image(w, h, 3 * w + h), synth.make_key(w + h), synth.make_iv(k)
    pub, priv = ofds.protect(img, key, iv, k)
    got = _restore(api, pub, priv, w, h, k, key, iv, offset=8 * (k & 1))
    assert np.array_equal(got, ofds.restore(pub, priv, key, iv, k, w, h))


@pytest.mark.parametrize("k", [5, 17])
def test_arbitrary_fragments(api, k):
    w, h, rng = 136, 40, np.random.default_rng(k)
    pub = rng.integers(-32768, 32768, (h // 8, w // 8, 3, 63 - k)).astype(np.int16)
    priv = rng.bytes(h // 8 * (w // 8) * 3 * 2 * (k + 1))
    key, iv = synth.make_key(1), b"\xff" * 16
    got = _restore(api, pub, priv, w, h, k, key, iv)
    assert np.array_equal(got, ofds.restore(pub, priv, key, iv, k, w, h))


@pytest.mark.parametrize("iv", [bytes(15) + b"\xff", bytes(8) + b"\xff" * 8, b"\xff" * 15 + b"\x01"])
def test_counter_carries(api, iv):
    w, h, k = 320, 72, 5                                      # 4050 keystream blocks: 16 windows
    rng, key = np.random.default_rng(2), synth.make_key(3)
    part1 = rng.integers(-200, 200, (h // 8, w // 8, 3, k + 1)).astype("<i2")
    pub = rng.integers(-20, 20, (h // 8, w // 8, 3, 63 - k)).astype(np.int16)
    priv = oaes.ctr_xcrypt(key, iv, part1.tobytes())
    assert np.array_equal(_restore(api, pub, priv, w, h, k, key, iv), ofds.restore(pub, priv, key, iv, k, w, h))


# k = 63 at 2600 x 2600: more counter windows per CTA than its table holds
@pytest.mark.parametrize("w,h,k", [(2600, 2600, 63), (4104, 1032, 17)])
def test_large_against_the_tensor_core_form(api, w, h, k):
    key, iv = synth.make_key(6), b"\xff" * 14 + b"\x12\x34"
    pub, priv = api.protect_image(torch.from_numpy(synth.make_image(w, h, 5)).to(DEV), key, iv, k)
    assert torch.equal(api.restore_image(pub, priv, w, h, k, key, iv),
                       api.restore_image_tc(pub, priv, w, h, k, key, iv))


@pytest.mark.parametrize("k", [0, 5, 62])
def test_public_image_of_ragged_sizes(api, k):
    from oracle import public as opub
    img, w, h = synth.make_image(104, 40, 8), 104, 40
    pub, _ = ofds.protect(img, synth.make_key(1), synth.make_iv(2), k)
    got = api.public_image(torch.from_numpy(pub).to(DEV), w, h, k).cpu().numpy()
    assert np.array_equal(got, opub.public_image(pub, k, w, h))
