"""The performance cases: what a user of this package has it do, through paper_1512_02951_gb300.api.

A case is a dict of plain values; "op" says which path it takes:

  protect, restore            one image already on the device
  plan_protect, plan_restore  a batch of uneven images as one launch (api.Plan)
  packed                      protect and restore with 11- or 8-bit storage
  strong                      protect and restore at the strong level
  dwt                         protect and restore of any data with the lossless DWT scheme
  publish                     the public fragment as an image, and its statistics
  host                        protect and restore between pinned host buffers

Inputs are smooth seeded scenes with +-8 grey levels of noise (the recipe of the package's
synth module, drawn on the device).
"""
import functools
import math

import numpy as np
import torch

from paper_1512_02951_gb300 import api, synth

DEV = "cuda:0"


def listed():
    return [
        # the smallest request of a serving mix: launches and latency are what count
        dict(name="protect 64x64", op="protect", width=64, height=64, k=5),
        # a thumbnail with only the DC coefficients confidential
        dict(name="restore 512x512", op="restore", width=512, height=512, k=0),
        # the headline image, both directions
        dict(name="protect 4096x4096", op="protect", width=4096, height=4096, k=5),
        dict(name="restore 4096x4096", op="restore", width=4096, height=4096, k=5),
        # a photo whose rows are no multiple of a tile or of 16 bytes, and a selection of its own
        dict(name="protect 3240x2592", op="protect", width=3240, height=2592, k=9),
        # an archive of images of every size in one launch: written, and read back
        dict(name="plan protect 1000", op="plan_protect", images=1000, sizes=7, k=0),
        dict(name="plan restore 300", op="plan_restore", images=300, sizes=8, k=5),
        # where storage is dear: the packed streams
        dict(name="packed 4096x4096", op="packed", width=4096, height=4096, k=5, form=11),
        # where the public fragment must show nothing
        dict(name="strong 4096x4096", op="strong", width=4096, height=4096, k=5),
        # documents and other data, cut into rows of bytes
        dict(name="dwt 4800x4800", op="dwt", width=4800, height=4800),
        # judging a protection: what the public fragment looks like, and how random it is
        dict(name="publish 4096x4096", op="publish", width=4096, height=4096, k=5),
        # a file's pixels in, the fragments out, and the pixels back, all in host memory
        dict(name="host 1600x1200", op="host", width=1600, height=1200, k=5),
    ]


def _log(rng, lo, hi, step):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step))


def draw(rng):
    op = rng.choice(["protect", "protect", "restore", "restore", "plan_protect", "plan_restore", "packed", "strong",
                     "dwt", "publish", "host"])
    if op.startswith("plan"):
        # one selection for all images, or (-1) one of its own for each
        return dict(op=op, images=_log(rng, 8, 1000, 1), sizes=rng.randrange(1 << 20), k=rng.choice([0, 5, 5, -1]))
    case = dict(op=op, width=_log(rng, 64, 4096, 8), height=_log(rng, 64, 4096, 8))
    if op == "dwt":
        return case
    case["k"] = rng.choice([0, 5, 5, rng.randrange(1, 21)])
    if op == "packed":
        case["form"] = rng.choice([11, 8])
    return case


def _ks(case):
    """The selection of every image of a batch."""
    n = case["images"]
    return [case["k"]] * n if case["k"] >= 0 else [(case["sizes"] + 7 * i) % 21 for i in range(n)]


def _image(width, height, gen):
    """A height x width x 3 uint8 scene on the device: 20 Gaussians on mid-grey, and noise."""
    n = synth.N_GAUSSIANS
    u = torch.rand(n, 6, generator=gen, device=DEV, dtype=torch.float64)
    sigma = (0.05 + 0.25 * u[:, 2:3]) * max(width, height)
    xs = torch.arange(width, device=DEV, dtype=torch.float64)
    ys = torch.arange(height, device=DEV, dtype=torch.float64)
    gx = torch.exp(-((xs - width * u[:, 0:1]) ** 2) / (2 * sigma ** 2)).float()
    gy = torch.exp(-((ys - height * u[:, 1:2]) ** 2) / (2 * sigma ** 2)).float()
    amp = (240 * u[:, 3:6] - 120).float()
    img = torch.rand(height, width, 3, generator=gen, device=DEV) * 16 - 8 + 128
    for c in range(3):
        img[:, :, c] += gy.t() @ (amp[:, c:c + 1] * gx)
    return img.round_().clamp_(0, 255).to(torch.uint8)


@functools.lru_cache(maxsize=1)
def _key_slots():
    """The keys of a long-running program, registered once."""
    return [api.key_register(synth.make_key(i)) for i in range(4)]


def _batch(case, gen):
    """Descriptors of the batch, its plan, and its pixels: crops of a few scenes."""
    sizes, ks = synth.batch_sizes(case["images"], case["sizes"]), _ks(case)
    rng = np.random.default_rng(case["sizes"])
    slots = _key_slots()
    descs = [api.ImageDesc(w, h, k, slots[i % 4], rng.bytes(16)) for i, ((w, h), k) in enumerate(zip(sizes, ks))]
    npx, npub, npriv = api.layout(descs)
    scenes = [_image(2048, 2048, gen) for _ in range(4)]
    px = torch.zeros(npx, dtype=torch.uint8, device=DEV)
    for i, d in enumerate(descs):
        n = 3 * d.width * d.height
        px[d.pixel_offset:d.pixel_offset + n].view(d.height, d.width, 3).copy_(scenes[i % 4][:d.height, :d.width])
    frags = [torch.zeros(n, dtype=torch.uint8, device=DEV) for n in (npub, npriv)]
    return api.Plan(descs), px, frags


def prepare(case, seed):
    api.init(0)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    op, rng = case["op"], np.random.default_rng(seed)
    s = dict(case, key=rng.bytes(16), iv=rng.bytes(16))
    if op.startswith("plan"):
        s["plan"], s["px"], (s["pub"], s["priv"]) = _batch(case, gen)
        if op == "plan_restore":
            s["plan"].protect(s["px"], s["pub"], s["priv"])
            s["px"] = torch.zeros_like(s["px"])
        return s
    w, h = case["width"], case["height"]
    if op == "dwt":
        s["data"] = _image(w // 8 * 8, h, gen)[:, :, 0].contiguous()
        return s
    s["px"] = _image(w, h, gen)
    if op in ("restore", "publish"):
        s["pub"], s["priv"] = api.protect_image(s["px"], s["key"], s["iv"], case["k"])
        if op == "publish":
            s["priv"] = None
        s["px"] = None
    elif op == "host":
        npub, npriv = api.sizes(w, h, case["k"])
        s["pub"] = torch.empty(npub // 2, dtype=torch.int16, device=DEV)
        s["priv"] = torch.empty(npriv, dtype=torch.uint8, device=DEV)
        s["back"] = torch.empty_like(s["px"])
        for name, like in (("px", s["px"]), ("pub", s["pub"]), ("priv", s["priv"]), ("back", s["px"])):
            s["h_" + name] = torch.empty(like.shape, dtype=like.dtype, pin_memory=True)
        s["h_px"].copy_(s["px"])
    return s


def run(s):
    op, key, iv = s["op"], s["key"], s["iv"]
    if op == "protect":
        return api.protect_image(s["px"], key, iv, s["k"])
    if op == "restore":
        return api.restore_image(s["pub"], s["priv"], s["width"], s["height"], s["k"], key, iv)
    if op == "plan_protect":
        s["plan"].protect(s["px"], s["pub"], s["priv"])
        return s["pub"].view(torch.int16), s["priv"]
    if op == "plan_restore":
        s["plan"].restore(s["pub"], s["priv"], s["px"])
        return s["px"]
    if op == "packed":
        pub, priv = api.protect_image_packed(s["px"], key, iv, s["k"], s["form"])
        return pub, priv, api.restore_image_packed(pub, priv, s["width"], s["height"], s["k"], key, iv, s["form"])
    if op == "strong":
        pub, priv = api.protect_image_strong(s["px"], key, iv, s["k"])
        return pub, priv, api.restore_image_strong(pub, priv, s["k"], key, iv)
    if op == "dwt":
        levels = api.dwt_protect(s["data"], key, iv)
        return (*levels, api.dwt_restore(*levels, s["width"], s["height"], key, iv))
    if op == "publish":
        image = api.public_image(s["pub"], s["width"], s["height"], s["k"])
        return (image, *api.image_stats(image))
    if op == "host":
        api.protect_image_host(s["h_px"], s["px"], key, iv, s["k"], s["pub"], s["priv"], s["h_pub"], s["h_priv"])
        api.restore_image_host(s["pub"], s["priv"], s["back"], s["h_back"], key, iv, s["k"])
        return s["h_pub"], s["h_priv"], s["h_back"]
    raise ValueError(op)


#: one 8x8 transform of a channel-block: sixteen 8-point passes of at least 34 operations
_BLOCK_FLOPS = 16 * 34


def work(case):
    """Bytes in and out, each once, and the operations of the transforms (hashes and ciphers are
    integer work and are not counted)."""
    op = case["op"]
    if op.startswith("plan"):
        px = sum(3 * w * h for w, h in synth.batch_sizes(case["images"], case["sizes"]))
        return dict(bytes=3 * px, flops=px // 64 * _BLOCK_FLOPS)
    n = case["width"] * case["height"]
    if op == "dwt":      # 64 bytes become 5 + 16 + 60, and back
        return dict(bytes=n // 64 * 2 * (64 + 81), flops=0)
    px, k = 3 * n, case["k"]
    if op in ("protect", "restore"):
        return dict(bytes=3 * px, flops=px // 64 * _BLOCK_FLOPS)
    if op == "packed":   # 11 bits of DC and `form` bits for each other coefficient, out and in
        stored = px // 64 * (11 + 63 * case["form"]) // 8
        return dict(bytes=2 * (px + stored), flops=px // 32 * _BLOCK_FLOPS)
    private = px // 64 * 2 * (k + 1)
    if op == "strong":   # the public image is as large as the pixels; four transforms
        return dict(bytes=2 * (2 * px + private), flops=px // 16 * _BLOCK_FLOPS)
    if op == "publish":  # the fragment in, the image out; the statistics add next to nothing
        return dict(bytes=2 * px - private + px, flops=px // 64 * _BLOCK_FLOPS)
    # host: the pixels cross the link twice, the fragments once
    return dict(bytes=4 * px, flops=px // 32 * _BLOCK_FLOPS)


def exact(case, seed):
    """Every output is whole numbers or bytes, defined bit for bit (rounded from exact values,
    encrypted or hashed), so there is no 64-bit value to be near to."""
    return None
