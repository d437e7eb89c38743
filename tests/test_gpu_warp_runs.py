"""Images of several subtiles a warp, in the kernels that are otherwise tested at one: private parts
collected or loaded in runs, staging areas and landing buffers used again, the last runs handed out
one by one, and the numbers of working warps.  Against kernels of their own: the tensor-core forms, and
for packed storage the int16 fragments packed here."""
import pytest

from paper_1512_02951_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
KEY, IV = synth.make_key(21), b"\xff" * 14 + b"\x7f\xf3"


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


def _image(w, h, seed, offset=0):
    """Ramps with noise (and near ties), at an offset of bytes from an aligned address."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    y, x = torch.arange(h, device=DEV)[:, None, None], torch.arange(w, device=DEV)[None, :, None]
    base = (x // 7 + y // 5 + 40 * torch.arange(3, device=DEV)) % 200 + 20
    buf = torch.zeros(3 * w * h + offset, dtype=torch.uint8, device=DEV)
    img = buf[offset:].view(h, w, 3)
    img.copy_(base + torch.randint(-12, 13, (h, w, 3), device=DEV, generator=gen))
    return img


# runs of 8 to 2 subtiles with two private buffers, and (42) of one with one
@pytest.mark.parametrize("w,h,k", [(4096, 2600, 1), (4096, 2600, 2), (4096, 2600, 4), (4096, 2600, 9), (4096, 2600, 12),
                                   (4096, 2600, 42), (2600, 1400, 9), (3000, 600, 4)])
def test_restore_runs(api, w, h, k):
    pub, priv = api.protect_image_tc(_image(w, h, k), KEY, IV, k)
    assert torch.equal(api.restore_image(pub, priv, w, h, k, KEY, IV), api.restore_image_tc(pub, priv, w, h, k, KEY, IV))


# pixels in 8-byte pieces: rows of fewer than 12 blocks, and an image that is not 16-byte aligned
@pytest.mark.parametrize("w,h,offset", [(88, 40000, 0), (2600, 2080, 8)])
@pytest.mark.parametrize("k", [0, 5, 9, 40])
def test_protect_runs_of_piecewise_pixels(api, w, h, offset, k):
    img = _image(w, h, k, offset)
    pub, priv = api.protect_image(img, KEY, IV, k)
    want_pub, want_priv = api.protect_image_tc(img, KEY, IV, k)
    assert torch.equal(pub, want_pub) and torch.equal(priv, want_priv)


def _bits(values, form, dc):
    """[n, m] coefficients as the bits of their fields, least significant first."""
    v = values.to(torch.int32)
    low = (v.abs().clamp(max=(1 << (form - 1)) - 1)) | ((v < 0).to(torch.int32) << (form - 1))
    cols = [((low[:, 1 if dc else 0:, None] >> torch.arange(form, device=DEV)) & 1).to(torch.uint8).flatten(1)]
    if dc:
        cols.insert(0, ((v[:, :1] >> torch.arange(11, device=DEV)) & 1).to(torch.uint8))
    return torch.cat(cols, 1).reshape(-1)


def _pack(values, form, dc):
    bits = _bits(values, form, dc)
    bits = torch.cat([bits, bits.new_zeros(-bits.numel() % 8)]).view(-1, 8)
    return (bits << torch.arange(8, device=DEV, dtype=torch.uint8)).sum(1).to(torch.uint8)


# per SM about 57, 44, 36, 18 subtiles: several a warp, ragged, and twelve working warps of sixteen
@pytest.mark.parametrize("w,h", [(2600, 2600), (4104, 1032), (2600, 1400), (3000, 600)])
@pytest.mark.parametrize("form", [11, 8])
@pytest.mark.parametrize("k", [0, 1, 5, 9, 41, 63])
def test_packed_runs(api, w, h, form, k):
    ncb = 3 * (w // 8) * (h // 8)
    img = _image(w, h, k)
    pub16, priv16 = api.protect_image(img, KEY, IV, k)
    part1 = api.encrypt_full(priv16, KEY, IV).view(torch.int16).view(ncb, k + 1)
    part2 = pub16.view(ncb, 63 - k)
    plain = _pack(part1, form, True)
    want_pub = _pack(part2, form, False) if k < 63 else None
    want_priv = api.encrypt_full(plain, KEY, IV)
    pub, priv = api.protect_image_packed(img, KEY, IV, k, form)
    assert torch.equal(priv, want_priv)
    if k < 63:
        assert torch.equal(pub, want_pub)
    # what the stored fields say, restored from int16 fragments
    top = (1 << (form - 1)) - 1
    back1 = part1.clamp(-top, top)
    back1[:, 0] = part1[:, 0]
    want = api.restore_image(part2.clamp(-top, top).contiguous(), api.encrypt_full(back1.contiguous(), KEY, IV), w, h, k, KEY, IV)
    for offset in (0, 8):                                # 8: the first part is copied by the lanes
        buf = torch.zeros(pub.numel() + 16, dtype=torch.uint8, device=DEV)
        buf[offset:offset + pub.numel()] = pub
        got = api.restore_image_packed(buf[offset:offset + pub.numel()], priv, w, h, k, KEY, IV, form)
        assert torch.equal(got, want)
