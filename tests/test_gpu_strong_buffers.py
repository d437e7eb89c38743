"""Strong protect where the private output lies in memory that the call reads or uses on the way: over
the pixels (which are not needed afterwards), over the plaintext in the scratch buffer, over the
scratch buffer's int16 fragment.  The same bytes as with a buffer of its own."""
import pytest

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


@pytest.mark.parametrize("place", ["pixels", "plaintext", "fragment", "between"])
@pytest.mark.parametrize("w,h,k", [(104, 40, 5), (1600, 1200, 5), (1600, 1200, 31)])
def test_private_output_over_the_calls_own_memory(api, w, h, k, place):
    key, iv = synth.make_key(11), synth.make_iv(12)
    img = torch.from_numpy(synth.make_image(w, h, 13)).to(DEV)
    want_image, want_private = api.protect_image_strong(img, key, iv, k)
    pub16 = (2 * (63 - k) * (w * h // 64) * 3 + 15) // 16 * 16
    n = want_private.numel()
    px, image = img.clone(), torch.empty_like(img)
    scratch = torch.empty(api.sizes_strong(w, h, k)[2], dtype=torch.uint8, device=DEV)
    at = {"pixels": px.view(-1)[:n], "plaintext": scratch[pub16:pub16 + n], "fragment": scratch[:n],
          "between": scratch[pub16 + (n + 15) // 16 * 16:][:n]}[place]    # behind what the call uses: apart
    api.protect_image_strong(px, key, iv, k, scratch=scratch, public=image, private=at)
    assert torch.equal(image, want_image) and torch.equal(at, want_private)
