"""Performance cases of the speculative mesh decoder, through its public Python entry points.

A case names what a user's program does (`do`) and on what: a model (one of the repository's workload
configurations, optionally at another width), a batch, a number of drafts, and prompt lengths in faces.

  pass      one decode pass of a host that sits in the loop, caches already filled: draft, the host's
            own drafts put in (optionally run through the correction stage), verify with logits.  The
            pass is not accepted, so it can be repeated on the same caches.
  prefill   a new request up to its first pass: prefill, draft, verify with logits.
  generate  a whole request on the device: prefill and the decode loop, drafts from a transcript that
            is kept for a seeded number of tokens per pass.
  host      the same request with the host in the loop, one call per pass with pinned host buffers.

The model handle (weights and caches in one workspace) is kept between states, as a serving program
keeps it: a request starts with a prefill, which resets the sequences.  Weights are random but for one
thing: the output matrix is aligned with the embedding so that after token t one successor of t stands
out.  A trained decoder's next-token distributions are peaked like this; with purely random logits the
greedy tokens of a long run would hinge on the last bit of every sum.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import fm_synth as S
from paper_2511_15618_b200 import FlashMesh

LEVELS = ((0, 4), (1, 3), (2,))        # stacks of the coordinate, vertex and face level
KEPT_OF_NINE = 6.7 / 9                 # drafts kept per pass with trained draft modules, of nine
HANDLES_BYTES = 90 << 30               # workspaces kept at a time

_DEFAULTS = {"d_model": 0, "batch": 1, "drafts": 9, "kv_heads": 0, "heads": "reduced", "levels": "three", "average": 0,
             "window": -1, "faces": 0, "faces_to": 0, "new_faces": 0, "corrected": False}


def _case(name, **kw):
    return {"name": name, **_DEFAULTS, **kw}


def listed():
    return [
        # the smallest call: one pass of the smallest model, where the launches are all there is
        _case("tiny pass", do="pass", model="tiny", drafts=3, faces=16),
        # a short request on the smallest model: start-up of a request and many small passes
        _case("tiny request", do="generate", model="tiny", drafts=3, faces=1, new_faces=16),
        # the small model completing a mesh
        _case("small request", do="generate", model="small", faces=8, new_faces=32),
        # three ragged requests at once, one shared key/value head, a long draft, a short window
        _case("small requests, shared head", do="generate", model="small", batch=3, drafts=18, kv_heads=1, window=400, faces=5,
              faces_to=61, new_faces=19),
        # time to the first tokens of an ordinary request
        _case("medium first pass", do="prefill", model="medium", faces=8),
        # completing a large mesh: a prompt of 7000 tokens
        _case("medium long prompt", do="prefill", model="medium", faces=777),
        # sixteen ragged requests starting together
        _case("batched first pass", do="prefill", model="batched", batch=16, faces=8, faces_to=64),
        # the decode pass in the middle of a 4000-face mesh, host in the loop
        _case("medium pass", do="pass", model="medium", faces=2000),
        # the full draft modules and the correction stage
        _case("medium corrected pass", do="pass", model="medium", heads="full", faces=333, corrected=True),
        # a request served with the host in the loop
        _case("medium host loop", do="host", model="medium", faces=8, new_faces=8),
        # serving a batch: ragged caches of 1000 to 2000 faces
        _case("batched pass", do="pass", model="batched", batch=16, faces=1000, faces_to=2000),
        # the largest model
        _case("large pass", do="pass", model="large", batch=4, drafts=12, faces=1000),
    ]


def draw(rng):
    """One more case of these ranges: any width between the tiny and the medium model."""
    def log_int(lo, hi):
        return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))

    do = rng.choice(["pass", "pass", "prefill", "prefill", "generate", "host"])
    d = rng.choice([256, 384, 512, 640, 768, 896, 1024, 1024])
    heads = d // 64
    c = dict(_DEFAULTS, do=do, model="tiny" if d < 512 else ("small" if d < 768 else "medium"), d_model=d)
    c["batch"] = log_int(1, 16)
    c["drafts"] = rng.choice([0, 3, 6, 9, 9, 9, 12, 18, 27])
    c["kv_heads"] = rng.choice([0, 0, 0, 1, 2 if heads % 2 == 0 else 1])
    if c["drafts"] > 0:
        c["heads"] = rng.choice(["reduced", "reduced", "full"])
        c["levels"] = rng.choice(["three", "three", "three", "coord"])
        c["average"] = rng.choice([0, 0, 1]) if c["levels"] == "three" else 0
    c["window"] = rng.choice([-1, -1, 0, rng.randrange(100, 1000)])
    if do == "pass":
        c["faces"] = log_int(1, 1000)
        c["faces_to"] = log_int(c["faces"], 1200)
        c["corrected"] = c["drafts"] >= 3 and rng.random() < 0.4
    elif do == "prefill":
        most = max(8, min(600 // c["batch"], 70 * (c["drafts"] + 1)))
        c["faces"] = log_int(1, most)
        c["faces_to"] = log_int(c["faces"], most)
    else:
        c["faces"] = log_int(1, max(8, 64 // c["batch"]))
        c["faces_to"] = log_int(c["faces"], max(c["faces"], 100 // c["batch"]))
        c["new_faces"] = log_int(2, 16)
    return c


# ------------------------------------------------------------------------------------------
# model handles
# ------------------------------------------------------------------------------------------
def _config(case):
    cfg = S.get_config(case["model"])
    d = case["d_model"] or cfg.d_model
    heads = d // cfg.head_dim
    B, D = case["batch"], case["drafts"]
    most = max(case["faces"], case["faces_to"]) + case["new_faces"]
    window = cfg.window if case["window"] < 0 else (case["window"], 0, 0)
    return cfg.with_(d_model=d, n_heads=heads, n_kv_heads=case["kv_heads"] or heads, d_ff=4 * d, draft_len=D, max_batch=B,
                     batch=B, draft_heads=case["heads"], draft_levels=case["levels"], avg_levels=case["average"], window=window,
                     max_tokens=max(cfg.max_tokens, 1 + 9 * (most + 2) + D + 2))


def _successor(cfg):
    """The token that stands out after each coordinate token, and after BOS (last entry)."""
    rng = np.random.default_rng([cfg.seed, 11])
    return np.append(rng.permutation(cfg.n_bins), rng.integers(cfg.n_bins))


def _weights(cfg):
    """Weights in fm_synth.make_weights' layout, drawn on the GPU (numpy takes a minute for the large model)."""
    gen = torch.Generator(device="cuda").manual_seed(cfg.seed + 1)
    d, dff, hd, V = cfg.d_model, cfg.d_ff, cfg.n_heads * cfg.head_dim, cfg.vocab
    qkv = hd + 2 * cfg.n_kv_heads * cfg.head_dim

    def host(t):
        return t.bfloat16().float().cpu().numpy()

    def mat(o, i, std=0.02):
        return host(torch.randn((o, i), generator=gen, device="cuda") * std)

    def gain():
        return np.ones(d, dtype=np.float32)

    E = torch.randn((V, d), generator=gen, device="cuda") * 2.0
    succ = _successor(cfg)
    out = torch.randn((V, d), generator=gen, device="cuda") * 0.004
    out[torch.as_tensor(succ[:-1], device="cuda")] += 0.01 * E[:cfg.n_bins]
    out[int(succ[-1])] += 0.01 * E[cfg.bos]
    w = {"E": host(E), "W_out": host(out), "g_out": gain(), "stacks": []}
    for s in range(5):
        w["stacks"].append([{"g1": gain(), "Wqkv": mat(qkv, d), "Wo": mat(d, hd), "g2": gain(), "W1": mat(dff, d), "W2": mat(d, dff)}
                            for _ in range(cfg.layers[s])])
    w["S_cv"], w["S_vf"], w["U_fv"], w["U_vc"] = mat(d, 3 * d), mat(d, 3 * d), mat(3 * d, d), mat(3 * d, d)
    three = cfg.draft_levels == "three"
    for name, n in (("heads_c", cfg.n_coord_heads), ("heads_v", 2 if three else 0), ("heads_f", cfg.n_face_heads)):
        w[name] = [{"g": gain(), "A": mat(d, d)} for _ in range(n)]
        if cfg.draft_heads == "full":
            for h in w[name]:
                h.update(ga=gain(), Wq=mat(hd, d), Wo=mat(d, hd))
    w["label"] = {"g": gain(), "W": mat(3, d)}
    if cfg.draft_heads == "full":
        for name, n in (("hf_vc", 6 if three else 0), ("hf_fv", 3 * cfg.n_face_heads), ("hf_fc", 9 * cfg.n_face_heads)):
            w[name] = [{"g": gain(), "Wq": mat(hd, d), "W1": mat(cfg.hf_width, hd), "W2": mat(d, cfg.hf_width)} for _ in range(n)]
    return w


_handles = {}


def _handle(case):
    """The context of a case's model, made once; a `pass` case has one of its own, with filled caches."""
    cfg = _config(case)
    key = (cfg, (case["faces"], case["faces_to"]) if case["do"] == "pass" else None)
    if key not in _handles:
        if sum(h.workspace_bytes for h in _handles.values()) > HANDLES_BYTES:
            _handles.pop(next(iter(_handles))).close()
        dev = FlashMesh(cfg, _weights(cfg))
        if case["do"] == "pass":
            rng = np.random.default_rng([cfg.seed, 13])
            dev.prefill(_condition(cfg, 17), _prompts(case, cfg, rng))
        _handles[key] = dev
    return cfg, _handles[key]


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _condition(cfg, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((cfg.batch, cfg.n_prefix, cfg.d_model), generator=gen, device="cuda")


def _lengths(case, rng):
    lo, hi = case["faces"], max(case["faces"], case["faces_to"])
    n = rng.integers(lo, hi + 1, size=case["batch"])
    n[0] = hi                                            # the longest prompt does not depend on the seed
    return n


def _prompts(case, cfg, rng):
    """Quantised triangles, vertices and faces in ascending (z, y, x) order."""
    out = []
    for n in _lengths(case, rng):
        v = rng.integers(0, cfg.n_bins, size=(int(n), 3, 3))
        key = (v[:, :, 0] * cfg.n_bins + v[:, :, 1]) * cfg.n_bins + v[:, :, 2]
        v = np.take_along_axis(v, np.argsort(key, axis=1)[:, :, None], axis=1)
        out.append(v[np.argsort(key.min(axis=1))].reshape(-1).astype(np.int32))
    return out


def _transcript(cfg, prompts, new_tokens):
    """Prompt and its greedy continuation, per sequence in one row."""
    succ = _successor(cfg)
    rows = np.zeros((len(prompts), max(len(p) for p in prompts) + new_tokens), dtype=np.int32)
    for b, p in enumerate(prompts):
        rows[b, :len(p)] = p
        t = p[-1] if len(p) else cfg.n_bins
        for i in range(new_tokens):
            t = succ[t]
            rows[b, len(p) + i] = t
    return rows


def prepare(case, seed):
    cfg, dev = _handle(case)
    rng = np.random.default_rng([seed, 19])
    B, D = cfg.batch, cfg.draft_len
    st = {"do": case["do"], "dev": dev, "D": D}
    if case["do"] in ("pass", "prefill"):
        st["drafts"] = torch.as_tensor(rng.integers(0, cfg.n_bins, size=(B, D)).astype(np.int32), device="cuda")
    if case["do"] == "pass":
        st["labels"] = torch.as_tensor(rng.integers(0, 3, size=(B, D + 1)).astype(np.int32), device="cuda") if case["corrected"] else None
        return st
    st["cond"], st["prompts"] = _condition(cfg, seed), _prompts(case, cfg, rng)
    if case["do"] in ("generate", "host"):
        st["new_faces"] = case["new_faces"]
        st["truth"] = _transcript(cfg, st["prompts"], 9 * case["new_faces"])
        # the seed does not change how many drafts are kept: every seed is the same amount of work
        st["keep"] = (S.accept_schedule(cfg.seed, B, 256, D, KEPT_OF_NINE * D) - 1).astype(np.int32)
    if case["do"] == "generate":
        st["truth"] = torch.as_tensor(st["truth"], device="cuda")
        st["keep"] = torch.as_tensor(st["keep"], device="cuda")
    if case["do"] == "host":
        st["n_bins"] = cfg.n_bins
        st["cand"], st["n_acc"], st["emitted"], st["kv_len"] = (torch.zeros(s, dtype=torch.int32).pin_memory()
                                                                for s in ((B, D + 1), (B,), (B, D + 1), (B, 3)))
    return st


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
def run(state):
    return {"pass": _run_pass, "prefill": _run_prefill, "generate": _run_generate, "host": _run_host}[state["do"]](state)


def _run_pass(st):
    dev = st["dev"]
    cand, draft_logits, _ = dev.draft(want_logits=True, reuse=True)
    cand[:, 1:].copy_(st["drafts"])
    if st["labels"] is not None:
        dev.correct(cand, st["labels"])
    argmax, logits, margin = dev.verify(cand, want_logits=True, reuse=True)
    return {"candidates": cand, "draft_logits": draft_logits, "argmax": argmax, "logits": logits, "margin": margin}


def _run_prefill(st):
    dev = st["dev"]
    dev.prefill(st["cond"], st["prompts"])
    cand, draft_logits, _ = dev.draft(want_logits=True)
    cand[:, 1:].copy_(st["drafts"])
    argmax, logits, margin = dev.verify(cand, want_logits=True)
    return {"candidates": cand, "draft_logits": draft_logits, "argmax": argmax, "logits": logits, "margin": margin}


def _run_generate(st):
    dev = st["dev"]
    dev.prefill(st["cond"], st["prompts"])
    tokens, lengths, stats = dev.generate(st["new_faces"], truth=st["truth"], keep=st["keep"])
    return {"tokens": tokens, "lengths": lengths, "passes": int(stats.steps)}


def _run_host(st):
    dev, D, truth, keep = st["dev"], st["D"], st["truth"], st["keep"]
    B, new = len(truth), 9 * st["new_faces"]
    tokens = np.full((B, new), -1, dtype=np.int32)
    at = np.array([len(p) for p in st["prompts"]])       # mesh token that is pending, per sequence
    end = at + new
    start = at.copy()
    cand, n_acc, emitted = st["cand"].numpy(), st["n_acc"].numpy(), st["emitted"].numpy()
    dev.prefill(st["cond"], st["prompts"])
    dev.set_max_faces([st["new_faces"]] * B)
    step = 0
    while (at < end).any():
        cand.fill(-1)
        for b in range(B):
            k = min(int(keep[step % len(keep), b]), int(end[b] - at[b]) - 1)
            if k > 0:
                cand[b, 1:1 + k] = truth[b, at[b] + 1:at[b] + 1 + k]
            if 0 <= k < D and at[b] + k + 1 < end[b]:    # the draft after the kept ones is a wrong one
                cand[b, k + 1] = (truth[b, at[b] + k + 1] + 1) % st["n_bins"]
        dev.step_host(st["cand"], st["n_acc"], st["emitted"], st["kv_len"])
        for b in range(B):
            n = int(n_acc[b])
            tokens[b, at[b] - start[b]:at[b] - start[b] + n] = emitted[b, :n]
            at[b] += n
        step += 1
    return {"tokens": tokens, "passes": step}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
def _layer_weights(cfg):
    hd, kv = cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim
    return (hd + 2 * kv) * cfg.d_model + hd * cfg.d_model + 2 * cfg.d_model * cfg.d_ff


def _draft_weights(cfg):
    if cfg.draft_len == 0:
        return 0
    d, hd = cfg.d_model, cfg.n_heads * cfg.head_dim
    n = cfg.n_coord_heads + (2 if cfg.draft_levels == "three" else 0) + cfg.n_face_heads
    w = n * d * d
    if cfg.draft_heads == "full":
        blocks = (6 if cfg.draft_levels == "three" else 0) + 12 * cfg.n_face_heads
        w += n * 2 * d * hd + blocks * (d * hd + cfg.hf_width * hd + d * cfg.hf_width)
    return w


def _forward(cfg, starts, rows):
    """(weight bytes, cache bytes read, cache bytes written, flops) of one forward over `rows` positions per
    sequence behind `starts` earlier ones (numbers of coordinate positions)."""
    hd, kv, P = cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim, cfg.n_prefix
    weights = read = written = flops = 0.0
    for level, stacks in enumerate(LEVELS):
        ratio, W = (1, 3, 9)[level], cfg.window[level]
        layers = sum(cfg.layers[s] for s in stacks)
        n_rows = visible = seen = 0.0
        for s, r in zip(starts, rows):
            lo, hi = -(-s // ratio), (s + r - 1) // ratio
            n = hi - lo + 1
            if n <= 0:
                continue
            n_rows += n
            mean = 0.5 * (lo + hi) + 1
            visible += n * (P + (min(mean, W) if W else mean))
            seen += P + (min(lo, W) if W else lo)        # entries of earlier passes that some row sees
        if n_rows == 0:
            continue
        weights += 2 * layers * _layer_weights(cfg)
        flops += layers * (2 * _layer_weights(cfg) * n_rows + 4 * hd * visible)
        read += layers * seen * 4 * kv
        written += layers * n_rows * 4 * kv
        if level > 0:                                    # shorten into and upsample out of the level
            weights += 2 * 6 * cfg.d_model ** 2
            flops += 12 * cfg.d_model ** 2 * n_rows
    return weights, read, written, flops


def _pass_work(cfg, starts, logits):
    B, D = cfg.batch, cfg.draft_len
    w, r, wr, f = _forward(cfg, starts, [D + 1] * B)
    head = cfg.vocab * cfg.d_model
    by = w + r + wr + 2 * head + 2 * _draft_weights(cfg)
    f += 2 * head * B * (2 * D + 1) + 2 * _draft_weights(cfg) * B
    if logits:
        by += 4 * cfg.vocab * B * (2 * D + 1)
    return by, f


def _prefill_work(cfg, lengths):
    B, P, kv = cfg.batch, cfg.n_prefix, cfg.n_kv_heads * cfg.head_dim
    w, _, wr, f = _forward(cfg, [0] * B, lengths)
    layers = sum(cfg.layers)
    by = w + wr + layers * B * P * 4 * kv + 4 * B * P * cfg.d_model
    return by, f + layers * 4 * B * P * kv * cfg.d_model


def work(case):
    cfg = _config(case)
    lengths = [1 + 9 * 0.5 * (case["faces"] + max(case["faces"], case["faces_to"]))] * cfg.batch
    if case["do"] == "pass":
        by, f = _pass_work(cfg, lengths, True)
        return {"bytes": by, "flops": f}
    by, f = _prefill_work(cfg, lengths)
    if case["do"] == "prefill":
        b2, f2 = _pass_work(cfg, lengths, True)
        return {"bytes": by + b2, "flops": f + f2}
    new = 9 * case["new_faces"]
    passes = math.ceil(new / (1 + KEPT_OF_NINE * cfg.draft_len))
    b2, f2 = _pass_work(cfg, [n + new / 2 for n in lengths], False)
    return {"bytes": by + passes * b2, "flops": f + passes * f2}


def tolerance(case):
    """Generated tokens are exact: every one stands out.  Logits come out of a forward with bfloat16 weights, queries,
    keys and values."""
    return "exact" if case["do"] in ("generate", "host") else {"rel": 1e-2, "max": 8e-2}
