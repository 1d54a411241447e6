"""The GELU of the first FFN matrix's epilogue on the device, in each form of the projection, against 64 bits.

A model whose attention, other layers and levels are zero and whose matrices are exact in bfloat16: a row's logits are two columns of
its embedding plus the GELUs of single pre-activations, scaled by the final norm.  What separates them from 64 bits is the sum of a
pre-activation (fp32, 128 products of together up to 20) and the two bfloat16 terms in which a GELU and a hidden are handed on (2^-17 of
them): 1e-5 of a value, where the tanh form of the GELU would be 4.7e-4 off."""
import math

import numpy as np
import pytest

import fm_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,D,form", [(1, 7, "few_rows"), (1, 15, "split_k"), (7, 8, "split_k"), (16, 3, "tiled")])
def test_gelu_of_the_epilogue(batch, D, form):
    from paper_2511_15618_b200 import FlashMesh, fm_projection_form
    from paper_2511_15618_b200.binding import make_config
    d, dff, V = 128, 256, 64
    cfg = S.toy_config(d_model=d, n_heads=2, n_kv_heads=2, head_dim=64, d_ff=dff, n_bins=V - 3, gain_std=0.0, draft_len=D,
                       max_batch=batch, batch=batch, max_tokens=64)
    assert fm_projection_form(make_config(cfg), "ffn1", batch * (D + 1)) == form
    rng = np.random.default_rng(5)
    w = S.make_weights(cfg)
    for name in ("S_cv", "S_vf", "U_fv", "U_vc"):
        w[name][:] = 0
    for stack in w["stacks"]:
        for layer in stack:
            layer["Wo"][:] = 0
            layer["W2"][:] = 0
    w["E"] = rng.choice(np.array([-1, -0.5, 0.5, 1], dtype=np.float32), size=(V, d))
    ffn = w["stacks"][4][-1]
    ffn["W1"] = S.round_to_bf16(rng.standard_normal((dff, d)).astype(np.float32) * np.float32(3 / math.sqrt(d)))
    ffn["W2"][np.arange(d), np.arange(d)] = 1                          # hidden c takes features c and, by half, d + c
    ffn["W2"][np.arange(d), d + np.arange(d)] = 0.5
    w["W_out"][:] = 0
    w["W_out"][np.arange(V), np.arange(V)] = 1                         # logit v takes hiddens v and V + v
    w["W_out"][np.arange(V), V + np.arange(V)] = 1

    dev = FlashMesh(cfg, w)
    dev.prefill(np.stack([S.make_condition(cfg, b) for b in range(batch)]), [[] for _ in range(batch)])
    cand, _, _ = dev.draft()
    cand[:, 1:] = dev.torch.as_tensor(rng.integers(0, cfg.n_bins, size=(batch, D)), device="cuda")
    _, logits, _ = dev.verify(cand, want_logits=True)
    seen, tokens = logits.double().cpu().numpy().reshape(-1, V), cand.cpu().numpy().reshape(-1)

    x = w["E"].astype(np.float64)[tokens]
    y = x / np.sqrt((x * x).mean(1, keepdims=True) + cfg.norm_eps) @ ffn["W1"].astype(np.float64).T
    g = 0.5 * y * np.vectorize(math.erfc)(-y / math.sqrt(2.0))
    assert np.abs(y).max() > 8 and np.abs(y).min() < 1e-2
    h = x + g[:, :d] + 0.5 * g[:, d:]
    inv = 1 / np.sqrt((h * h).mean(1, keepdims=True) + cfg.norm_eps)
    err = 2.0 ** -17 * (np.abs(g[:, :d]) + 0.5 * np.abs(g[:, d:]) + np.abs(h)) + 2e-5
    ref, bound = inv * (h[:, :V] + h[:, V:]), inv * (err[:, :V] + err[:, V:])
    print(form, "largest error", np.abs(seen - ref).max(), "of its bound", (np.abs(seen - ref) / bound).max())
    assert (np.abs(seen - ref) <= bound).all()
    assert dev.device_status() == 0
