"""What the launch-shape tuner times and what it remembers; the decoder and the
clock are stand-ins, so this runs without a GPU."""

import pytest

import paper_2402_04834_gb300 as pkg
from paper_2402_04834_gb300 import autotune

torch = pytest.importorskip("torch")


@pytest.fixture
def timed(monkeypatch):
    """Candidates timed, as (batch size, (warps, cosets, messages)); each one's
    time is its place in the order, last first."""
    seen = []

    def shape(p):
        return p.warps, p.cosets, p.messages
    monkeypatch.setattr(autotune, "_cache", {})
    monkeypatch.setattr(autotune, "decode", lambda s, p: seen.append((s.shape[0], shape(p))))
    monkeypatch.setattr(autotune, "decode_mixed", lambda s, o, d, p: seen.append((d.shape[0], shape(p))))

    def clock(fn, reps=3):
        fn()
        return -float(len(seen))
    monkeypatch.setattr(autotune, "_time", clock)
    return seen


def test_a_shape_is_not_carried_over_to_another_batch_size(timed):
    prm = pkg.DecoderParams(d=11, k=4, precision="fp32", algorithm="fused")
    n = len(autotune.candidates(prm))
    for B, more in ((10000, n), (9000, 0), (1, n), (10000, 0), (1, 0)):
        before = len(timed)
        autotune.tune_uniform(torch.zeros(B, prm.m, dtype=torch.uint8), prm)
        assert len(timed) - before == more, B
    odd = pkg.DecoderParams(d=0, k=4, precision="fp32", algorithm="fused")
    for B, again in ((4096, True), (5000, False), (2, True), (4096, False)):
        before = len(timed)
        autotune.tune_mixed(None, None, torch.tensor([7, 9] * (B // 2), dtype=torch.int32), odd, ctas=(0,))
        assert (len(timed) > before) == again, B


def test_register_form_only_shapes_need_a_batch_of_odd_distances(timed):
    # decode_mixed takes messages = 3 as the caller's word that every distance
    # is odd and flags a syndrome of even distance; prm.d says nothing about it.
    for d in (0, 11):
        prm = pkg.DecoderParams(d=d, k=4, precision="fp32", algorithm="fused")
        for ds, lean in (([8, 11], False), ([7, 11], True)):
            del timed[:]
            autotune._cache.clear()
            autotune.tune_mixed(None, None, torch.tensor(ds, dtype=torch.int32), prm, ctas=(0,))
            assert any(shape[2] == 3 for _, shape in timed) == lean, (d, ds)
            assert ((2, (0, 0, 3)) in timed) == lean                # the default's choice among them
            assert len(timed) == len(set(timed))
