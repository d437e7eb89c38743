"""Tensors that are not on a CUDA device are refused by the binding before the library sees their
addresses."""
import pytest

torch = pytest.importorskip("torch")
from paper_1512_02951_gb300 import api, build

W = H = 8
K = bytes(16)


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def u8(n):
    return torch.zeros(n, dtype=torch.uint8)


IMG = torch.zeros((H, W, 3), dtype=torch.uint8)
PUB = torch.zeros((1, 1, 3, 58), dtype=torch.int16)
CALLS = {
    "restore_image": lambda: api.restore_image(PUB, u8(36), W, H, 5, K, K),
    "restore_image_tc": lambda: api.restore_image_tc(PUB, u8(36), W, H, 5, K, K),
    "restore_image_packed": lambda: api.restore_image_packed(u8(512), u8(64), W, H, 5, K, K),
    "public_image": lambda: api.public_image(PUB, W, H, 5),
    "image_stats": lambda: api.image_stats(IMG),
    "dwt_restore": lambda: api.dwt_restore(u8(16), u8(16), u8(64), W, H, K, K),
    "encrypt_full": lambda: api.encrypt_full(u8(32), K, K),
    "protect": lambda: api.protect(u8(192), u8(512), u8(64), [api.ImageDesc(W, H, 5, 0, K)]),
    "restore": lambda: api.restore(u8(512), u8(64), u8(192), [api.ImageDesc(W, H, 5, 0, K)]),
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_host_tensors_are_refused(name, monkeypatch):
    # the library must not be reached: its C entry points take addresses and cannot tell them apart
    class NoCalls:
        def __getattr__(self, entry):
            if entry.startswith("fds_sizes"):
                return getattr(lib, entry)

            def reached(*args):
                raise AssertionError(entry + " was called with host addresses")
            return reached

    lib = api._lib.load()
    monkeypatch.setattr(api._lib, "load", lambda: NoCalls())
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 0, raising=False)
    with pytest.raises(ValueError):
        CALLS[name]()
