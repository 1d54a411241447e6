"""What the benchmark line calls its kernels."""
import bench
import fm_synth as S

FEW, SPLIT, TILED = "rg::gemm_rows_kernel", "tc::gemm_tc_kernel", "pf::gemm_kernel"


def test_the_projections_are_named_by_the_form_they_take():
    for name, kernels in (("tiny", [FEW]),                   # 4, 2 and 1 rows
                          ("small", [FEW, SPLIT]),           # 10, 4 and 2: above 8 rows the first FFN matrix is split
                          ("medium", [FEW, SPLIT]),
                          ("batched", [SPLIT, TILED]),       # 160, 64 and 32
                          ("large", [FEW, SPLIT])):          # 52, 20 and 8
        assert bench.gemm_kernels(S.get_config(name)) == ", ".join(kernels)


def test_merges_do_not_count_as_streaming_launches():
    cfg = S.get_config("medium")                      # 32 layers
    e = bench.attention_entry(cfg, 0.256, 64)
    assert e["launches"] == 64 and e["merges"] == 32 and abs(e["us_per_layer"] - 8.0) < 1e-9
    assert bench.attention_entry(cfg, 0.256, 32)["merges"] == 0
