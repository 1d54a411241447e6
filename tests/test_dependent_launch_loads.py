"""How kernels with the programmatic-dependent-launch attribute read what earlier kernels of the chain write, checked on
the sources (no GPU): such a kernel starts while its predecessors still run, so their output is not read-only during its
lifetime, and a `const T* __restrict__` parameter would let the compiler read it through the read-only path."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15618_b200", "csrc")
FILES = ("fm_kernels.cuh", "fm_prefill.cuh", "fm_gemm_rows.cuh", "fm_gemm_tc.cuh", "fm_attention.cuh")
# weights and tables (written when the context is created); maps, prompts and the parameter block of a call (complete
# before its first dependent launch)
CONSTANT = {"E", "g", "gains", "label_g", "label_W", "rope_tab", "segs", "rows", "prompt", "prompt_off", "layers", "gen"}
READ_ONLY = re.compile(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)")


def _functions(text):
    """(name, parameters, body) of every kernel and device function."""
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    for m in re.finditer(r"__(?:global|device)__[^;{(]*?(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(([^{;]*?)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(0).startswith("__global__"), m.group(1), m.group(2), text[m.end():i]


def _all():
    return [(f, *fn) for f in FILES for fn in _functions(open(os.path.join(CSRC, f)).read())]


def test_the_parser_sees_the_kernels_of_a_pass():
    waits = {name for _, is_kernel, name, _, body in _all() if is_kernel and "grid_dep_wait" in body}
    for name in ("embed_kernel", "draft_pick_kernel", "verify_top2_kernel", "accept_kernel", "gemm_rows_kernel", "gemm_tc_kernel",
                 "attn_stream_kernel", "attn_merge_kernel", "gemm_kernel", "gather_kernel", "upsample_kernel", "attn_tc_kernel"):
        assert name in waits, name


def test_no_read_only_qualifier_on_data_of_the_launch_chain():
    bad = []
    for f, is_kernel, name, params, body in _all():
        if is_kernel and "grid_dep_wait" not in body:
            continue                                  # a full barrier in front of it
        bad += [(f, name, p) for p in READ_ONLY.findall(params) if p not in CONSTANT]
    assert not bad, bad


def test_residual_rows_of_earlier_launches_are_read_at_l2():
    """The GEMM epilogues' residual and stash rows (struct members, so the qualifier does not show)."""
    for f in FILES:
        text = open(os.path.join(CSRC, f)).read()
        assert not re.search(r"=\s*e\.stash_x\[", text), f
        assert not re.search(r"(?:=|\?)\s*xr\[\(size_t\)j \* e\.ldx\]", text), f
        assert not re.search(r"(?:=|\?)\s*\*reinterpret_cast<const float2\*>\(xr", text), f


def test_prefill_attention_requests_query_rows_of_its_tile_only():
    """The row expression of attn_kernel's query loads, evaluated for every lane of every tile height."""
    text = open(os.path.join(CSRC, "fm_prefill.cuh")).read()
    first = re.search(r"const int i = (w0 \+ g \+ hr \* 8);\s*const bf16\* qp = a\.q \+ \(\(size_t\)\(r0 \+ \((i < q0 \+ nq) \? (i) : (q0)\)\)", text)
    assert first, "the query loads are not bounded by the tile"
    q0 = 256
    for nq in range(1, 129):
        for w0 in range(q0, q0 + 128, 16):
            for g in range(8):
                for hr in range(2):
                    env = {"w0": w0, "g": g, "hr": hr, "q0": q0, "nq": nq}
                    env["i"] = eval(first.group(1), {}, env)
                    row = eval(first.group(3) if eval(first.group(2), {}, env) else first.group(4), {}, env)
                    assert q0 <= row < q0 + nq
