"""Batches whose tiles are handed out whole, in halves and subtile by subtile in turn: from one
tile a block to a few rounds of tiles a warp, images ending in tiles of one to six subtiles (some
units are empty, a warp's first one too).  Compared with the image-by-image path."""
import numpy as np
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
    _api.counters(reset=True)
    yield _api
    assert _api.counters()[2] == 0


SMALL = [(8, 8), (88, 16), (64, 64), (16, 8), (104, 40), (72, 56), (512, 8)]   # 1 .. 6 subtiles at the end


@pytest.mark.parametrize("k", [0, 5, 20, 63, None])
@pytest.mark.parametrize("sizes", [
    SMALL[:1],                                    # fewer tiles than blocks of the grid
    SMALL * 40,                                   # one or two tiles a block: single subtiles only
    SMALL[:4] * 300,                              # about eight: halves and singles, most units empty
    SMALL[:4] * 1200 + [(1600, 1200)],            # about thirty: whole tiles too
], ids=["1", "280", "1200", "4801"])
def test_units_of_a_batch(api, sizes, k):
    ks = [k if k is not None else 7 * i % 64 for i in range(len(sizes))]
    slots = [api.key_register(synth.make_key(40 + i)) for i in range(3)]
    descs = [api.ImageDesc(w, h, q, slots[i % 3], synth.make_iv(i)) for i, ((w, h), q) in enumerate(zip(sizes, ks))]
    npx, npub, npriv = api.layout(descs)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(len(sizes))
    px = torch.randint(0, 256, (npx,), dtype=torch.uint8, device=DEV, generator=gen)
    pub, priv = (torch.zeros(n, dtype=torch.uint8, device=DEV) for n in (npub, npriv))
    back = torch.zeros_like(px)
    plan = api.Plan(descs)
    plan.protect(px, pub, priv)
    plan.restore(pub, priv, back)
    for i in sorted({*range(min(len(descs), 40)), *range(max(0, len(descs) - 40), len(descs))}):
        d, key = descs[i], synth.make_key(40 + i % 3)
        n = 3 * d.width * d.height
        img = px[d.pixel_offset:d.pixel_offset + n].view(d.height, d.width, 3)
        wpub, wpriv = api.protect_image(img, key, synth.make_iv(i), ks[i])
        want = api.restore_image(wpub, wpriv, d.width, d.height, ks[i], key, synth.make_iv(i))
        a, b = 2 * (63 - ks[i]) * (n // 64), 2 * (ks[i] + 1) * (n // 64)
        assert torch.equal(pub[d.public_offset:d.public_offset + a], wpub.reshape(-1).view(torch.uint8)[:a])
        assert torch.equal(priv[d.private_offset:d.private_offset + b], wpriv.reshape(-1)[:b])
        assert torch.equal(back[d.pixel_offset:d.pixel_offset + n].view_as(want), want)
