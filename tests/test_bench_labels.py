"""What the benchmark line calls its kernels."""
import os
import re

import bench
import fm_synth as S

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15618_b200", "csrc")


def test_the_projections_are_named_by_the_form_they_take():
    text = open(os.path.join(CSRC, "fm_gemm_rows.cuh")).read()
    assert bench.FEW_ROWS == int(re.search(r"MAX_ROWS = (\d+)", text).group(1))
    for name, kernel in (("tiny", "rg::gemm_rows_kernel"), ("medium", "rg::gemm_rows_kernel")):
        assert bench.gemm_kernels(S.get_config(name)) == kernel
    for name in ("batched", "large"):
        assert "tc::gemm_tc_kernel" in bench.gemm_kernels(S.get_config(name))


def test_merges_do_not_count_as_streaming_launches():
    cfg = S.get_config("medium")                      # 32 layers
    e = bench.attention_entry(cfg, 0.256, 64)
    assert e["launches"] == 64 and e["merges"] == 32 and abs(e["us_per_layer"] - 8.0) < 1e-9
    assert bench.attention_entry(cfg, 0.256, 32)["merges"] == 0
