"""The few-row projections against the oracle where they change form: one and two MMA row tiles (up to 8 and 16
rows with two terms each), with more than 8 rows only those with 8 features per CTA or short K, the first row count of the split-K form for all, 16 and 32 features per CTA (long K, many
features), weights too large for a CTA, a last CTA with few features."""
import pytest

import fm_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,batch,kw", [
    (7, 1, {}),                                                       # 8 coordinate rows
    (8, 1, {}),                                                       # 9
    (15, 1, {}),                                                      # 16
    (16, 1, {}),                                                      # 17: split K
    (3, 4, {}),                                                       # 16 rows of four sequences
    (3, 1, {"d_ff": 4096}),                                           # 16 features per CTA, 128 KB of weights; 32 features
    (9, 1, {"d_ff": 4096}),
    (9, 1, {"d_ff": 8192, "n_bins": 133}),                            # weights too large: split K; ragged outputs
    (7, 1, {"d_model": 640, "n_heads": 10, "n_kv_heads": 10, "weight_std": 0.04}),          # 8 rows: all of them; 9: the output projection and the second FFN matrix
    (8, 1, {"d_model": 640, "n_heads": 10, "n_kv_heads": 10, "weight_std": 0.04}),
    (8, 1, {"d_model": 640, "n_heads": 10, "n_kv_heads": 1, "weight_std": 0.04}),           # 9 rows: QKV with 8 features per CTA
    (15, 1, {"d_model": 640, "n_heads": 10, "n_kv_heads": 1, "weight_std": 0.04}),          # 16
    (16, 1, {"d_model": 512, "n_kv_heads": 1, "weight_std": 0.05}),   # 17, QKV with fewer features than the hidden that it keeps for the draft heads
    (9, 2, {"d_model": 640, "n_kv_heads": 1, "weight_std": 0.04}),    # 20
    (15, 1, {"d_model": 640, "n_kv_heads": 1, "weight_std": 0.04}),   # 16, few-row form
])
def test_few_rows_lockstep(D, batch, kw):
    from oracle.lockstep import run_lockstep
    from paper_2511_15618_b200 import FlashMesh
    base = dict(d_model=128, n_heads=2, n_kv_heads=2, head_dim=64, d_ff=256, weight_std=0.1, out_std=0.02)
    base.update(kw)
    if base["d_ff"] > 256:
        base["weight_std"] = 0.03
    cfg = S.toy_config(**base, draft_len=D, layers=(1, 1, 2, 1, 1), max_batch=batch, batch=batch, gen_faces=4, prompt_faces=(1, 1),
                       max_tokens=1 + 9 * 6 + D + 2)
    w = S.make_weights(cfg)
    conds = [S.make_condition(cfg, b) for b in range(batch)]
    prompts = [[int(t) for t in S.make_prompt(cfg, b)] for b in range(batch)]
    dev = FlashMesh(cfg, w)
    rep = run_lockstep(cfg, w, conds, prompts, dev, 4, 60)
    assert rep["done"] and rep["emitted"] == 36 * batch and dev.device_status() == 0
    print(D, batch, {k: rep[k] for k in ("steps", "max_logit_err", "max_draft_err", "overrides")})
