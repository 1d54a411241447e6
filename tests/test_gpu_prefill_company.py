"""What the bits of a prefill depend on, as the header states it: the same call leaves the same bits, other company leaves the
same values to rounding, and repeating a run's prefill and feeding its tokens as drafts continues the run to the bit."""
import numpy as np
import pytest

import fm_synth as S

pytestmark = pytest.mark.gpu


def _config(faces, **kw):
    base = dict(d_model=128, n_heads=2, n_kv_heads=2, head_dim=64, d_ff=256, weight_std=0.1, out_std=0.02)
    base.update(kw)
    return S.toy_config(**base, draft_len=9, layers=(1, 2, 2, 1, 2), max_batch=3, batch=3, gen_faces=2, max_tokens=1 + 9 * (faces + 4) + 11)


# total rows on both sides of every change of form, prompts that together need more than one chunk, rings that only the
# longer prompts overrun
@pytest.mark.parametrize("own,others,kw", [
    (0, ((0, 0), (1, 50)), {}),
    (20, ((0, 0), (5, 61), (120, 3)), {}),
    (20, ((0, 0), (9, 30), (200, 100)), {"n_heads": 16, "n_kv_heads": 16, "d_ff": 2048}),
    (3, ((1, 2), (40, 7)), {"window": (30, 11, 5)}),
    (30, ((2, 2), (150, 90)), {"n_heads": 1, "n_kv_heads": 1, "head_dim": 128, "window": (200, 0, 0)}),
    (500, ((10, 0), (600, 300)), {}),
    (950, ((0, 1), (940, 930)), {"window": (700, 0, 0)}),
])
def test_the_same_call_to_the_bit_and_other_company_to_rounding(own, others, kw):
    import torch
    from paper_2511_15618_b200 import FlashMesh
    cfg = _config(max([own] + [f for o in others for f in o]), **kw)
    dev = FlashMesh(cfg, S.make_weights(cfg))
    conds = np.stack([S.make_condition(cfg, b) for b in range(3)])
    mine = S.fill_prompt(cfg, 1, own) if own else []
    seen = []
    for before, behind in others + others[:1]:
        dev.prefill(conds, [S.fill_prompt(cfg, 0, before) if before else [], mine, S.fill_prompt(cfg, 2, behind) if behind else []])
        cand, draft_logits, _ = dev.draft(want_logits=True)
        if seen:
            cand[1, 1:] = seen[0][0][1:]
        _, logits, _ = dev.verify(cand, want_logits=True)
        seen.append((cand[1].clone(), draft_logits[1].clone(), logits[1].clone()))
        assert dev.device_status() == 0
    for a, b in zip(seen[0], seen[-1]):               # the first call again
        assert torch.equal(a, b)
    # other sums ahead of the bfloat16 roundings of q, k, v and P: a flipped rounding is 2^-8 of a value, and what a row
    # sees of it averages out (1e-4 to 3e-3 over these cases); about four times that
    off = [float((a - b).norm() / b.norm()) for other in seen[1:-1] for a, b in zip(seen[0][1:], other[1:])]
    print(own, others, off)
    assert max(off) <= 1e-2


def test_a_run_is_continued_to_the_bit_from_its_tokens():
    import torch
    from paper_2511_15618_b200 import FlashMesh
    cfg = _config(30)
    dev = FlashMesh(cfg, S.make_weights(cfg))
    conds = np.stack([S.make_condition(cfg, b) for b in range(3)])
    prompts = [S.fill_prompt(cfg, b, f) if f else [] for b, f in enumerate((8, 0, 21))]

    def state(**kw):
        dev.prefill(conds, prompts)
        dev.set_max_faces([3] * 3)
        tok, ln, _ = dev.generate(-1, max_steps=9 if kw else 18, stride=27, plain=not kw, **kw)
        cand, draft_logits, _ = dev.draft(want_logits=True)
        _, logits, _ = dev.verify(cand, want_logits=True)
        return tok.clone(), ln.cpu().tolist(), draft_logits, logits

    tok, ln, dl, lg = state()                         # 18 tokens, one per pass
    assert ln == [18] * 3
    rows = max(len(p) for p in prompts) + 18
    truth = np.zeros((3, rows), np.int32)
    for b, p in enumerate(prompts):
        truth[b, :len(p) + 18] = list(p) + tok[b, :18].cpu().tolist()
    again = state(truth=truth, keep=np.full((1, 3), 1, np.int32))    # the same tokens as drafts, two per pass
    assert again[1] == ln and torch.equal(again[0], tok)
    assert torch.equal(again[2], dl) and torch.equal(again[3], lg)
