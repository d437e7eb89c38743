"""The float32 coefficients that the error-guard tests look at (fds_debug_dct_f32) come out of the
functions that the protect kernels transform with, not out of a copy of them."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1512_02951_gb300", "csrc")


def _text(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_export_and_protect_share_their_passes():
    export, protect = _text("fds_protect.cu"), _text("fds_protect_warp.cu")
    for text in (export, protect):
        assert len(re.findall(r"\brow_pass\(", text)) == 1 and len(re.findall(r"\bcolumn_pass\(", text)) == 1
        assert not re.search(r"\bdct8\w*[(<]", text)      # no butterflies of their own
