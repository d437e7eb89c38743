"""Tuning a plan does not choose between schedules that launch the same kernel."""
import pytest

from paper_1512_02951_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_lane_pairs_are_timed_once():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_02951_gb300 import api, build

    build.build()
    api.init(0)
    slot = api.key_register(synth.make_key(3))
    descs = [api.ImageDesc(w, h, 5, slot, synth.make_iv(w)) for w, h in ((256, 64), (512, 512), (104, 80))]
    npx, npub, npriv = api.layout(descs)
    bufs = [torch.zeros(n, dtype=torch.uint8, device=DEV) for n in (npx, npub, npriv, npx)]
    plan = api.Plan(descs)
    got = plan.tune(*bufs, reps=2)
    times = {}
    for c in got["candidates"]:
        times.setdefault((c["direction"], c["largest_first"], c["ctas_per_sm"], c["dynamic"]), []).append((c["aes_pair"], c["ms"]))
    assert len(times) == 2 * (4 + 2) * 2
    for pair in times.values():
        assert [a for a, _ in sorted(pair)] == [0, 1] and len({ms for _, ms in pair}) == 1
    assert got["protect"]["aes_pair"] == 0 and got["restore"]["aes_pair"] == 0
    plan.close()
    api.key_release(slot)
