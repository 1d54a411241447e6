"""Output buffers of the binding: with `reuse` the same ones on every call, without it fresh ones."""
import pytest


@pytest.fixture
def dev(monkeypatch):
    import torch
    from paper_2511_15618_b200 import binding as B
    d = B.FlashMesh.__new__(B.FlashMesh)
    d.torch, d.device, d.ctx, d.batch, d.D, d.V = torch, torch.device("cpu"), None, 2, 3, 11
    d._before = lambda: None
    d._after = lambda *tensors: None
    for name in ("fm_draft", "fm_verify", "fm_accept"):
        monkeypatch.setattr(B, name, lambda *a: 0)
    return d


def _calls(dev, reuse):
    import torch
    cand = torch.zeros((2, 4), dtype=torch.int32)
    dev._dev = lambda x, dtype: x
    return [t for out in (dev.draft(want_logits=True, reuse=reuse), dev.verify(cand, want_logits=True, reuse=reuse), dev.accept(reuse=reuse))
            for t in out]


@pytest.mark.parametrize("D", [0, 3])
def test_reuse_hands_out_the_same_buffers(dev, D):
    dev.D = D
    first, second = _calls(dev, True), _calls(dev, True)
    assert all(a is b for a, b in zip(first, second))
    assert first[2].shape == (2, D) and first[2].is_contiguous()


def test_without_reuse_every_call_has_its_own(dev):
    first, second = _calls(dev, False), _calls(dev, False)
    assert not {t.data_ptr() for t in first} & {t.data_ptr() for t in second}
