"""Image statistics where the strip segments go from one or a few a block of the grid (small images)
to 32 a block: around four a block."""
import numpy as np
import pytest

from oracle import public as opub

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# 128-pixel strips times segments of eight rows: 1, 40, 300, 585, 594, 600 and 1100 of them
@pytest.mark.parametrize("w,h", [(3, 8), (320, 105), (640, 480), (1152, 520), (1152, 528), (1280, 480), (1408, 800)])
def test_stats_of_few_segments(w, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_02951_gb300 import api, build

    build.build()
    api.init(0)
    img = np.random.default_rng(w + h).integers(0, 256, (h, w, 3), dtype=np.uint8)
    hist, sums = api.image_stats(torch.from_numpy(img).to(DEV))
    assert np.array_equal(hist.cpu().numpy(), opub.histogram(img))
    assert np.array_equal(sums.cpu().numpy(), opub.pair_sums(img))
