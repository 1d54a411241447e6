"""The packed prefill against the oracle at the sizes where it changes form: one query tile and a row more, ragged batches, windows whose ring is shorter
than a chunk (keys of the chunk outside the cache), more positions than one chunk holds."""
import numpy as np
import pytest

import fm_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("faces,window,kw", [
    ((0, 1, 3), (0, 0, 0), {}),
    ((14, 15), (0, 0, 0), {}),                                        # 127 and 136 rows
    ((28, 1), (0, 0, 0), {"n_kv_heads": 1}),                          # 263 rows together
    ((29, 120, 2), (0, 0, 0), {}),
    ((40, 7), (30, 11, 5), {}),                                       # rings shorter than the prompt
    ((100,), (50, 0, 3), {"n_kv_heads": 1}),
    ((90, 20), (0, 0, 0), {"n_heads": 1, "n_kv_heads": 1, "head_dim": 128}),
    ((60,), (20, 9, 0), {"n_heads": 1, "n_kv_heads": 1, "head_dim": 128}),
    ((35, 2), (0, 0, 0), {"d_model": 192, "d_ff": 320}),              # partly empty last tiles
    ((61, 2), (0, 0, 0), {"d_model": 384, "n_heads": 6, "n_kv_heads": 1, "d_ff": 320}),      # pairs of feature tiles: an odd number, a last one half empty
    ((143, 1), (0, 0, 0), {"d_model": 640, "n_heads": 10, "n_kv_heads": 10, "d_ff": 704, "weight_std": 0.04}),
    ((71,), (0, 0, 0), {"n_heads": 16, "n_kv_heads": 16}),            # 640 rows, 5 tiles of 128 on 16 heads: 32 query rows per CTA
    ((71, 0), (30, 0, 0), {"n_heads": 16, "n_kv_heads": 4}),          # a row more, 6 tiles: 128
    ((143,), (0, 0, 0), {"n_heads": 16, "n_kv_heads": 16}),           # 10 tiles and 8 rows more
    ((160, 3), (600, 0, 0), {"n_heads": 16, "n_kv_heads": 2}),        # the same with a ring shorter than the prompt, shared heads
    ((950,), (700, 0, 0), {"n_heads": 16, "n_kv_heads": 16}),         # ... and in two chunks
    ((950, 30), (0, 0, 0), {}),                                       # cut into two chunks
    ((950,), (700, 0, 0), {}),                                        # two chunks and a ring that wraps
])
def test_prefill_lockstep(faces, window, kw):
    from oracle.lockstep import run_lockstep
    from paper_2511_15618_b200 import FlashMesh
    B, D = len(faces), 9
    base = dict(d_model=128, n_heads=2, n_kv_heads=2, head_dim=64, d_ff=256, weight_std=0.1, out_std=0.02)
    base.update(kw)
    cfg = S.toy_config(**base, draft_len=D, layers=(1, 2, 2, 1, 2), window=window, max_batch=B, batch=B, gen_faces=2,
                       max_tokens=1 + 9 * (max(faces) + 4) + D + 2)
    w = S.make_weights(cfg)
    conds = [S.make_condition(cfg, b) for b in range(B)]
    prompts = [S.fill_prompt(cfg, b, f) if f else [] for b, f in enumerate(faces)]
    dev = FlashMesh(cfg, w)
    rep = run_lockstep(cfg, w, conds, prompts, dev, 2, 60, prefill_chunk=512)
    assert rep["done"] and rep["emitted"] == 18 * B and dev.device_status() == 0
    print(faces, {k: rep[k] for k in ("steps", "max_logit_err", "max_draft_err", "overrides")})


@pytest.mark.parametrize("faces,window,kw", [
    ((143,), (0, 0, 0), {}),                                          # 10 tiles and 8 rows more
    ((160, 3), (600, 0, 0), {"n_kv_heads": 2}),                       # a ring shorter than the prompt, shared heads, a tile of few rows
    ((950,), (700, 0, 0), {}),                                        # two chunks, a ring that wraps
])
def test_prefill_lockstep_128_query_rows_per_cta_heads_of_128(faces, window, kw):
    """Heads of 128 take 128 query rows per CTA only where that gives every SM one."""
    import torch
    heads = 16
    rows = [9 * f + 1 for f in faces]
    assert sum(-(-min(r, 8190) // 128) for r in rows) * heads >= torch.cuda.get_device_properties(0).multi_processor_count
    test_prefill_lockstep(faces, window, {"n_heads": heads, "n_kv_heads": heads, "head_dim": 128, **kw})


# The rows on both sides of each change between the split-K and the tiled form: 64 coordinate rows (every projection of d = 128), 481
# (the second FFN matrix with K = 2048), at d = 1024 161 (the output projection) and 193 (QKV in pairs of CTAs).
@pytest.mark.parametrize("faces,kw", [
    ((6, 0, 0, 0, 0, 0, 0, 0, 0), {}), ((7,), {}),                    # 63 and 64 rows
    ((52, 1, 0), {}), ((52, 1, 0, 0), {}),                            # 480 and 481
    ((52, 1, 0, 0), {"d_ff": 2048, "weight_std": 0.05}),
    ((33, 2, 0, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),              # 320 and 321
    ((33, 2, 0, 0, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),
    ((17, 0, 0, 0, 0, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),        # 160 and 161
    ((17, 0, 0, 0, 0, 0, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),
    ((21, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),                    # 192 and 193
    ((21, 0, 0, 0), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),
])
def test_prefill_lockstep_where_projections_change_form(faces, kw):
    test_prefill_lockstep(faces, (0, 0, 0), kw)


# Pairs of CTAs: an even number of 128-feature tiles, an odd one whose last tile is half empty, the conditioning's with an odd one (its second
# CTA repeats the first one's weights and stores nothing).
@pytest.mark.parametrize("faces,projections,kw", [
    ((86,), ("qkv", "out"), {"d_model": 1024, "n_heads": 16, "n_kv_heads": 16, "weight_std": 0.03}),
    ((29,), ("ffn1", "ffn2"), {"d_model": 1088, "n_heads": 4, "n_kv_heads": 1, "d_ff": 2112, "weight_std": 0.03}),
    ((13,), ("ffn2",), {"d_model": 1088, "n_heads": 4, "n_kv_heads": 1, "d_ff": 2112, "weight_std": 0.03}),
    # (so many faces that all 512 conditioning vectors go through one launch)
    ((110,), ("conditioning",), {"d_model": 1024, "n_heads": 6, "n_kv_heads": 3, "n_prefix": 512, "d_ff": 2048, "weight_std": 0.03}),
    ((60, 55), ("conditioning",), {"d_model": 1024, "n_heads": 6, "n_kv_heads": 3, "n_prefix": 256, "d_ff": 2048, "weight_std": 0.03}),
])
def test_prefill_lockstep_pairs_of_ctas(faces, projections, kw):
    from paper_2511_15618_b200 import binding as B
    cfg = B.make_config(S.toy_config(**{"n_heads": 2, "n_kv_heads": 2, "head_dim": 64, "d_ff": 256, "layers": (1, 2, 2, 1, 2), **kw}))
    for p in projections:
        rows = len(faces) * cfg.n_prefix if p == "conditioning" else sum(9 * f + 1 for f in faces)
        assert B.fm_projection_form(cfg, p, rows) == "tiled_pairs"
    test_prefill_lockstep(faces, (0, 0, 0), kw)
