"""Buffers that a warp fills by its own stores (or cp.async) and by bulk copies in turn: pixels of
narrow and of wide images in one batch, the 2-byte tails of fragments whose images end in a short
subtile, and the first packed part of a stream that is 8- but not 16-byte aligned.  Every warp gets
several subtiles.  Compared with the image-by-image path and with the restore of a packed stream at an
odd address (kernels of its own)."""
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


SIZES = [(64, 48), (256, 64), (72, 40), (104, 56), (8, 8), (136, 24)]


@pytest.mark.parametrize("dynamic", [False, True])
@pytest.mark.parametrize("k", [0, 5, 20, 62, None])
def test_narrow_and_wide_images_in_turn(api, k, dynamic):
    n = 1500
    ks = [k if k is not None else 7 * i % 64 for i in range(n)]
    slots = [api.key_register(synth.make_key(90 + i)) for i in range(3)]
    descs = [api.ImageDesc(*SIZES[i % 6], ks[i], slots[i % 3], synth.make_iv(i)) for i in range(n)]
    npx, npub, npriv = api.layout(descs)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    px = torch.randint(100, 156, (npx,), dtype=torch.uint8, device=DEV, generator=gen)
    got, want = ([torch.zeros(b, dtype=torch.uint8, device=DEV) for b in (npub, npriv, npx)] for _ in range(2))
    plan = api.Plan(descs)
    plan.set_schedule(0, dynamic, False)
    plan.protect(px, got[0], got[1])
    plan.restore(got[0], got[1], got[2])
    api.protect(px, want[0], want[1], descs)
    api.restore(want[0], want[1], want[2], descs)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    plan.close()
    for s in slots:
        api.key_release(s)


@pytest.mark.parametrize("form", [11, 8])
@pytest.mark.parametrize("k", [0, 5, 41, 62])
def test_packed_stream_whose_first_part_the_lanes_copy(api, form, k):
    w, h = 2600, 2080                                   # 7922 subtiles: three or four a warp
    key, iv = synth.make_key(4), synth.make_iv(9)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(k)
    px = torch.randint(0, 256, (h, w, 3), dtype=torch.uint8, device=DEV, generator=gen)
    pub, priv = api.protect_image_packed(px, key, iv, k, form)
    out = {}
    for offset in (0, 1, 8):
        buf = torch.zeros(pub.numel() + 16, dtype=torch.uint8, device=DEV)
        buf[offset:offset + pub.numel()] = pub
        out[offset] = api.restore_image_packed(buf[offset:offset + pub.numel()], priv, w, h, k, key, iv, form)
    assert torch.equal(out[0], out[1]) and torch.equal(out[8], out[1])
