"""Image statistics at the sizes where the kernel's loads and strips change form: around one strip
of 128 pixels, rows of every alignment, segments shorter and longer than four rows."""
import numpy as np
import pytest

from oracle import public as opub

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


@pytest.mark.parametrize("w", [2, 4, 5, 125, 127, 128, 129, 131, 256, 517])
@pytest.mark.parametrize("h,offset", [(1, 0), (2, 1), (9, 2), (64, 3), (333, 0)])
def test_stats(api, w, h, offset):
    img = np.random.default_rng(w * 1000 + h).integers(0, 256, (h, w, 3), dtype=np.uint8)
    buf = torch.zeros(img.size + offset, dtype=torch.uint8, device=DEV)
    buf[offset:] = torch.from_numpy(img.reshape(-1)).to(DEV)
    hist, sums = api.image_stats(buf[offset:].view(h, w, 3))
    assert np.array_equal(hist.cpu().numpy(), opub.histogram(img))
    assert np.array_equal(sums.cpu().numpy(), opub.pair_sums(img))


def test_stats_of_one_level(api):
    img = np.full((700, 900, 3), 255, dtype=np.uint8)          # every count in one level
    hist, sums = api.image_stats(torch.from_numpy(img).to(DEV))
    assert np.array_equal(hist.cpu().numpy(), opub.histogram(img))
    assert np.array_equal(sums.cpu().numpy(), opub.pair_sums(img))
