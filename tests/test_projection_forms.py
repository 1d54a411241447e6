"""Which form a projection takes, against times measured on a B200 (chains of launches over the layers, us): the form chosen is
at most a tenth slower than the better one, what the estimates of the choice and the timer leave open."""
import pytest

import fm_synth as S

# width, key/value heads (0: as many as query heads), projection, rows; split-K (None: not measured), tiled in single CTAs, tiled in pairs
MEASURED = [
    (256, 0, "out", 73, 3.7, 3.3, 3.9),
    (256, 0, "ffn2", 73, 3.2, 5.5, 5.4),
    (256, 0, "qkv", 257, 6.0, 3.8, 4.4),
    (256, 0, "ffn1", 480, 5.9, 4.1, 5.2),
    (256, 0, "logits", 640, 6.2, 4.3, 5.5),
    (256, 0, "qkv", 1522, None, 5.1, 6.6),
    (512, 0, "out", 73, 3.2, 4.2, 4.5),
    (512, 0, "ffn1", 160, 5.6, 4.6, 5.4),
    (512, 0, "out", 480, 5.5, 4.3, 4.6),
    (512, 0, "ffn2", 320, 6.7, 8.7, 8.2),
    (512, 0, "logits", 768, 7.4, 5.3, 6.3),
    (512, 0, "ffn1", 1100, 15.9, 7.9, 9.5),
    (512, 1, "qkv", 320, 6.2, 4.4, 4.8),
    (768, 0, "out", 160, 4.8, 5.0, 5.1),
    (768, 0, "out", 384, 9.2, 5.1, 5.2),
    (768, 0, "ffn2", 384, 14.4, 11.7, 10.6),
    (768, 0, "qkv", 257, 10.8, 6.5, 7.0),
    (768, 0, "ffn2", 1522, None, 18.7, 15.4),
    (1024, 0, "qkv", 73, 8.7, 6.0, 6.5),
    (1024, 0, "out", 73, 3.9, 5.7, 5.8),
    (1024, 0, "logits", 73, 4.2, 5.4, 5.5),
    (1024, 0, "ffn2", 160, 9.3, 14.5, 13.1),
    (1024, 0, "out", 320, 7.9, 6.1, 6.6),
    (1024, 0, "ffn1", 257, 10.6, 9.9, 9.5),
    (1024, 0, "ffn2", 520, 15.7, 15.2, 14.0),
    (1024, 0, "qkv", 2334, None, 29.6, 26.6),
    (1024, 0, "ffn2", 6994, None, 92.8, 87.2),
    (1024, 0, "ffn1", 6994, None, 97.7, 91.4),
    (2048, 0, "ffn2", 64, 11.3, 26.2, 24.0),
    (2048, 0, "ffn1", 320, 50.5, 30.0, 26.3),
    (2048, 0, "out", 320, 16.7, 11.5, 11.1),
    (2048, 0, "ffn2", 1100, 116.5, 58.7, 57.9),
]

# 9 to 16 rows; few-row form, split-K (whole passes where a chain of one projection shows no difference)
MEASURED_FEW = [
    (640, 1, "qkv", 10, 608, 625),
    (768, 2, "qkv", 16, 662, 675),
    (896, 1, "qkv", 10, 661, 670),
    (1024, 1, "qkv", 10, 703, 714),
    (512, 0, "qkv", 10, 314, 323),
    (1280, 0, "out", 10, 474, 470),
    (1024, 0, "qkv", 10, 5.3, 4.5),
    (1024, 0, "out", 10, 2.9, 3.1),
    (1024, 0, "ffn1", 10, 5.3, 4.0),
    (1024, 0, "ffn2", 10, 6.7, 6.0),
    (1024, 0, "logits", 10, 3.3, 2.8),
    (256, 0, "qkv", 12, 2.7, 3.2),
    (256, 0, "ffn1", 12, 2.6, 2.3),
    (256, 0, "ffn2", 12, 2.2, 2.7),
    (384, 0, "ffn2", 16, 2.8, 3.0),
    (512, 0, "ffn2", 16, 3.8, 3.4),
]


def _config(d, kv_heads=0):
    from paper_2511_15618_b200 import binding as B
    head_dim = 128 if d == 2048 else 64
    heads = d // head_dim
    return B.make_config(S.get_config("medium").with_(d_model=d, n_heads=heads, n_kv_heads=kv_heads or heads, head_dim=head_dim, d_ff=4 * d))


@pytest.mark.parametrize("d,kv_heads,projection,rows,split,single,pairs", MEASURED)
def test_single_ctas_or_pairs(d, kv_heads, projection, rows, split, single, pairs):
    from paper_2511_15618_b200 import fm_projection_form
    times = {"tiled": single, "tiled_pairs": pairs}
    form = fm_projection_form(_config(d, kv_heads), projection, rows)
    if form in times:
        assert times[form] <= 1.1 * min(single, pairs)


@pytest.mark.parametrize("d,kv_heads,projection,rows,split,single,pairs", [m for m in MEASURED if m[4] is not None])
def test_split_k_or_tiled(d, kv_heads, projection, rows, split, single, pairs):
    from paper_2511_15618_b200 import fm_projection_form
    times = {"split_k": split, "tiled": single, "tiled_pairs": pairs}
    assert times[fm_projection_form(_config(d, kv_heads), projection, rows)] <= 1.1 * min(times.values())


@pytest.mark.parametrize("d,kv_heads,projection,rows,few,split", MEASURED_FEW)
def test_few_rows_or_split_k(d, kv_heads, projection, rows, few, split):
    from paper_2511_15618_b200 import fm_projection_form
    assert fm_projection_form(_config(d, kv_heads), projection, rows) == ("few_rows" if few < split else "split_k")


def test_refuses_what_is_no_projection():
    from paper_2511_15618_b200 import FmError, fm_projection_form, load_library
    import ctypes as C
    with pytest.raises(FmError):
        fm_projection_form(_config(256), "qkv", 0)
    assert load_library().fm_projection_form(C.byref(_config(256)), 6, 8) < 0
    assert load_library().fm_projection_form(None, 0, 8) < 0
