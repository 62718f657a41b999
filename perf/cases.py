"""Workloads of the superposition-prompting hot path, as a serving program issues them.

A case is a plain dict.  `kind` names the part of the path that one pass runs:

  step     the whole path of one layer for a batch of new prompts: rotate Q and K, fork-join prefill, path scores,
           top-k, and one response token over the kept paths
  prefill  the fork-join attention alone, in its variants (rows, encoding, head shapes)
  select   path scores and top-k over the logits of the query copies
  decode   one response token of one layer over the preamble, the kept paths and the tail

Shape fields: `prompts`, `docs` (paths per prompt), `pre` (shared preamble rows), `doc_min`..`doc_max` (document
lengths, uniform), `qry` (rows of every query copy), `joined` (documents of earlier rounds that already belong to
the shared prefix), `heads`, `kv_heads`, `dim`, `dtype`, `vocab`, `keep` (paths kept), `tail` (rows the response
cache has room for), `shape` (seed of the ragged lengths: they belong to the case, the values to prepare()'s seed).
Options: `pos` = how positions reach the attention ("rope": rotated by sp_rope_apply before it or, for a response
token, inside sp_pruned_decode_rope; "fused": Q rotated inside the prefill; "alibi": the bias variants; "given": Q
and K arrive encoded), `rows` = "all" or "query" (path caching: only the query copies are new), `lse` = the
log-sum-exp is wanted too.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2404_06910_b200 as sp

_MOST_VALUES = 1.16e9          # tokens x heads x dim of the largest listed case: drawn ones stay below
_MOST_PAIRS = 2.4e9            # admitted (query, key) pairs x heads, likewise
_MOST_LOGITS = 1.55e9


def _case(name, kind, **fields):
    c = {"name": name, "kind": kind, "prompts": 1, "docs": 20, "pre": 32, "doc_min": 64, "doc_max": 256, "qry": 24,
         "joined": 0, "heads": 32, "kv_heads": 32, "dim": 128, "dtype": "bf16", "vocab": 50432, "keep": 2, "tail": 32,
         "shape": 1, "pos": "rope", "rows": "all", "lse": False}
    c.update(fields)
    return c


def listed():
    return [
        # The smallest whole path: one short prompt in fp32.  Nothing but launches, latency and host time.
        _case("step_tiny_f32", "step", docs=4, pre=16, doc_min=32, doc_max=32, qry=8, heads=4, kv_heads=4, dim=64,
              dtype="f32", vocab=512, keep=1, tail=4),
        # One interactive request of ordinary size.
        _case("step_single", "step", doc_min=96, doc_max=160, tail=64),
        # A full serving batch of ordinary requests: the flagship workload.
        _case("step_batched", "step", prompts=64),
        # The largest prompts: hundreds of documents, about 140 thousand tokens each; Q and K come encoded from the
        # projection.
        _case("prefill_long", "prefill", prompts=2, docs=400, pre=64, doc_min=128, doc_max=512, qry=32, pos="given"),
        # Many documents per prompt, the rotation of Q left to the prefill.
        _case("prefill_fused_rope", "prefill", prompts=8, docs=100, pre=48, qry=32, pos="fused"),
        # The ALiBi model families, with the log-sum-exp for a caller that merges partial results.
        _case("prefill_alibi", "prefill", prompts=32, pos="alibi", lse=True),
        # A later round of iterative superposition: chosen documents have joined the prefix.
        _case("prefill_iterative", "prefill", prompts=64, doc_min=60, doc_max=180, joined=3, pos="given"),
        # Path caching: preamble and documents are cached, only the query copies are new.
        _case("prefill_cached", "prefill", prompts=8, docs=100, pre=48, qry=32, pos="given", rows="query"),
        # Models with half-size heads.
        _case("prefill_head64", "prefill", prompts=8, dim=64, pos="given"),
        # Scoring and pruning of a full serving batch.
        _case("select_batched", "select", prompts=64),
        # A response token of a full serving batch, grouped query heads.
        _case("decode_grouped", "decode", prompts=64, kv_heads=8, tail=64),
        # A response token of two very long prompts: little work, spread over the whole chip.
        _case("decode_long", "decode", prompts=2, docs=400, pre=64, doc_min=128, doc_max=512, qry=32, keep=8, tail=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "prefill", "prefill", "prefill", "select", "decode", "decode"])
    c = _case("", kind)
    del c["name"]
    c["shape"] = rng.randrange(1 << 20)
    c["prompts"] = _log_int(rng, 1, 64)
    c["docs"] = _log_int(rng, 4, 400)
    c["pre"] = rng.randint(8, 128)
    c["doc_min"] = rng.randint(32, 128)
    c["doc_max"] = c["doc_min"] * rng.randint(1, 4)
    c["qry"] = rng.randint(8, 48)
    c["keep"] = min(c["docs"], rng.randint(1, 8))
    c["tail"] = _log_int(rng, 4, 256)
    c["vocab"] = _log_int(rng, 8000, 130000)
    c["heads"] = rng.choice([16, 32, 32, 40])
    c["kv_heads"] = c["heads"] // rng.choice([1, 1, 2, 4, 8])
    c["dim"] = rng.choice([64, 128, 128, 128])
    if kind == "step" and rng.random() < 0.3:           # small fp32 problems: the debugging and reference type
        c.update(dtype="f32", prompts=rng.randint(1, 2), docs=rng.randint(2, 8), doc_min=16, doc_max=64, heads=8,
                 kv_heads=rng.choice([4, 8]), dim=64, vocab=rng.randint(500, 5000))
        c["keep"] = min(c["keep"], c["docs"])
    if kind == "prefill":
        c["pos"] = rng.choice(["given", "given", "alibi", "fused" if c["dim"] == 128 else "given"])
        c["rows"] = "query" if c["pos"] != "fused" and rng.random() < 0.25 else "all"
        c["lse"] = rng.random() < 0.3
        c["joined"] = rng.choice([0, 0, min(c["docs"] // 2, rng.randint(1, 6))])
    if kind == "decode":
        c["pos"] = rng.choice(["rope", "rope", "alibi", "given"])
        if c["pos"] == "rope" and c["heads"] // c["kv_heads"] > 4:
            c["pos"] = "given"                           # the folded rotation serves groups of 1, 2 and 4
    while True:                                          # never more work than the largest listed case
        lay = _layout(c)
        logits = int(lay.qry_len.sum()) * c["vocab"] if kind in ("step", "select") else 0
        if (lay.total_tokens * c["heads"] * c["dim"] <= _MOST_VALUES and _pairs(c, lay) * c["heads"] <= _MOST_PAIRS
                and logits <= _MOST_LOGITS):
            return c
        if c["prompts"] > 1:
            c["prompts"] = max(1, c["prompts"] * 2 // 3)
        else:
            c["docs"] = max(4, c["docs"] * 2 // 3)
            c["keep"], c["joined"] = min(c["keep"], c["docs"]), min(c["joined"], c["docs"] // 2)


# ---- shapes ----------------------------------------------------------------------------------------------------
def _layout(case):
    """The ragged packing: [preamble | doc_0 query_0 | doc_1 query_1 | ...] per prompt, prompts one after another."""
    rng = np.random.default_rng(case["shape"])
    ppo, pre_start, pre_len, path_start, doc_len, row = [0], [], [], [], [], 0
    for _ in range(case["prompts"]):
        docs = rng.integers(case["doc_min"], case["doc_max"] + 1, size=case["docs"])
        prefix = case["pre"] + int(docs[:case["joined"]].sum())
        pre_start.append(row)
        pre_len.append(prefix)
        row += prefix
        for n in docs[case["joined"]:]:
            path_start.append(row)
            doc_len.append(int(n))
            row += int(n) + case["qry"]
        ppo.append(len(path_start))
    i32 = lambda a: np.asarray(a, dtype=np.int32)
    doc_len = i32(doc_len)
    qry_len = np.full(len(doc_len), case["qry"], dtype=np.int32)
    return SimpleNamespace(n_prompts=case["prompts"], n_paths=len(doc_len), prompt_path_off=i32(ppo), pre_start=i32(pre_start),
                           pre_len=i32(pre_len), path_start=i32(path_start), doc_len=doc_len, qry_len=qry_len,
                           total_tokens=row, max_pre_len=max(pre_len), max_path_len=int((doc_len + qry_len).max()))


def _pairs(case, lay):
    """Admitted (query, key) pairs of the prefill."""
    owner = np.repeat(np.arange(lay.n_prompts), np.diff(lay.prompt_path_off))
    pre, doc, qry = lay.pre_len.astype(np.int64), lay.doc_len.astype(np.int64), lay.qry_len.astype(np.int64)
    if case["rows"] == "query":
        return int((qry * (pre[owner] + doc) + qry * (qry + 1) // 2).sum())
    n = doc + qry
    return int((pre * (pre + 1) // 2).sum() + (n * pre[owner] + n * (n + 1) // 2).sum())


def _kept_and_tail(case, lay):
    """The paths a response attends to and how far it has come (part of the shape: they decide the work)."""
    rng = np.random.default_rng(case["shape"] + 1)
    n = case["docs"] - case["joined"]
    kept = np.stack([rng.permutation(n)[:case["keep"]] + lay.prompt_path_off[b] for b in range(lay.n_prompts)])
    return kept.astype(np.int32), rng.integers(1, case["tail"] + 1, size=lay.n_prompts).astype(np.int32)


# ---- inputs ----------------------------------------------------------------------------------------------------
def _positions(case, lay):
    """Equilibrium positions of every packed row, and the first response position of every prompt."""
    pos, nxt = [], []
    for b in range(lay.n_prompts):
        docs = lay.doc_len[lay.prompt_path_off[b]:lay.prompt_path_off[b + 1]]
        p, _, after = sp.sp_positions(int(lay.pre_len[b]), docs, case["qry"])
        pos.append(p)
        nxt.append(after)
    return np.concatenate(pos), np.asarray(nxt)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    randn = lambda *shape, dtype=dt: torch.randn(*shape, generator=gen, device="cuda", dtype=dtype)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    scratch = lambda n: torch.zeros(max(256, n), dtype=torch.uint8, device="cuda")

    lay = _layout(case)
    B, T, H, Hkv, D, kind = lay.n_prompts, lay.total_tokens, case["heads"], case["kv_heads"], case["dim"], case["kind"]
    s = SimpleNamespace(case=case, lay=sp.DeviceLayout.from_host(lay), scale=D ** -0.5)
    pos, nxt = _positions(case, lay)
    if kind in ("step", "prefill"):
        s.q, s.k, s.v = randn(T, H, D), randn(T, Hkv, D), randn(T, Hkv, D)
        s.out = torch.zeros_like(s.q)
        s.lse = torch.zeros((H, T), device="cuda") if case["lse"] else None
        size = sp.sp_prefill_rope_workspace_bytes if case["pos"] == "fused" else sp.sp_prefill_workspace_bytes
        s.ws = scratch(size(s.lay, H, D, sp.dtype_code(s.q)))
    if kind in ("step", "prefill", "decode"):
        s.pos = dev(pos)
        s.slopes = dev(np.exp2(-8.0 * (np.arange(H) + 1) / H).astype(np.float32))
    if kind in ("step", "select"):
        off = np.zeros(lay.n_paths + 1, dtype=np.int32)
        np.cumsum(lay.qry_len, out=off[1:])
        s.logits = randn(int(off[-1]), case["vocab"]).mul_(3.0)
        s.targets = torch.randint(0, case["vocab"], (int(off[-1]),), generator=gen, device="cuda", dtype=torch.int32)
        s.targets[dev(off[1:].astype(np.int64) - 1)] = -1        # the last query token predicts nothing inside its segment
        s.row_off = dev(off)
        s.prior = randn(lay.n_paths, dtype=torch.float32).mul_(0.25).sub_(2.5)
        s.weight = dev((1.0 / lay.qry_len).astype(np.float32))
        s.scores = torch.zeros(lay.n_paths, device="cuda")
        s.row_logp = torch.zeros(int(off[-1]), device="cuda") if kind == "select" else None
        s.score_ws = scratch(sp.sp_path_scores_workspace_bytes(int(off[-1])))
        s.kept = torch.zeros((B, case["keep"]), dtype=torch.int32, device="cuda")
        s.post = torch.zeros((B, case["keep"]), device="cuda")
    if kind in ("step", "decode"):
        kept, tail_len = _kept_and_tail(case, lay)
        if kind == "decode":
            s.k, s.v, s.kept = randn(T, Hkv, D), randn(T, Hkv, D), dev(kept)
        else:
            tail_len[:] = 1                                      # the first token of the response
        s.tok_q = randn(B, H, D)
        s.tail_k, s.tail_v = randn(B, case["tail"], Hkv, D), randn(B, case["tail"], Hkv, D)
        s.tail_len = dev(tail_len)
        s.tok_pos = dev((nxt + tail_len - 1).astype(np.float32))
        s.tail_pos = dev((nxt[:, None] + np.arange(case["tail"])).astype(np.float32))
        s.tok_out = torch.zeros_like(s.tok_q)
        s.tok_lse = torch.zeros((B, H), device="cuda")
        s.dec_ws = scratch(sp.sp_decode_workspace_bytes(B, H, D))
    return s


# ---- one pass --------------------------------------------------------------------------------------------------
def _select(s):
    sp.sp_path_scores(s.logits, s.targets, s.row_off, s.scores, s.prior, s.weight, s.row_logp, s.score_ws)
    sp.sp_prune_topk(s.scores, s.lay.prompt_path_off, s.case["keep"], s.kept, s.post)


def _decode(s):
    c = s.case
    cache = (s.k, s.v, s.lay, s.kept, c["keep"], s.tail_k, s.tail_v, s.tail_len, c["tail"])
    if c["pos"] == "alibi":
        sp.sp_pruned_decode_alibi(s.tok_q, *cache, s.tok_pos, s.pos, s.tail_pos, s.slopes, s.scale, s.tok_out, s.tok_lse,
                                  s.dec_ws)
        return
    if c["pos"] == "rope" and c["heads"] // c["kv_heads"] in (1, 2, 4):
        sp.sp_pruned_decode_rope(s.tok_q, *cache, s.tok_pos, s.scale, s.tok_out, s.tok_lse)
        return
    if c["pos"] == "rope":                                       # larger groups rotate on their own (first token: row 0)
        sp.sp_rope_apply_pair(s.tok_q, c["heads"], s.tail_k, c["kv_heads"], s.tok_pos, c["dim"],
                              ld_k=c["tail"] * c["kv_heads"] * c["dim"])
    sp.sp_pruned_decode(s.tok_q, *cache, s.scale, s.tok_out, s.tok_lse, s.dec_ws)


def run(state):
    s, c = state, state.case
    kind, H, Hkv, D = c["kind"], c["heads"], c["kv_heads"], c["dim"]
    if kind == "select":
        _select(s)
        return [s.scores, s.row_logp, s.kept, s.post]
    if kind == "decode":
        _decode(s)
        return [s.tok_out, s.tok_lse, s.tail_k]
    if kind == "prefill":
        if c["pos"] == "fused":
            sp.sp_superpose_prefill_rope(s.q, s.k, s.v, s.lay, s.pos, 10000.0, sp.SP_ROPE_HALF_SPLIT, s.scale, s.out,
                                         s.lse, s.ws)
        else:
            rows = sp.SP_ROWS_QUERY_ONLY if c["rows"] == "query" else sp.SP_ROWS_ALL
            if c["pos"] == "alibi":
                sp.sp_superpose_prefill_alibi(s.q, s.k, s.v, s.lay, s.pos, s.slopes, s.scale, s.out, s.lse, s.ws, rows=rows)
            else:
                sp.sp_superpose_prefill(s.q, s.k, s.v, s.lay, s.scale, s.out, s.lse, s.ws, rows=rows)
        return [s.out, s.lse]
    sp.sp_rope_apply(s.q, s.pos, H, D)
    sp.sp_rope_apply(s.k, s.pos, Hkv, D)
    sp.sp_superpose_prefill(s.q, s.k, s.v, s.lay, s.scale, s.out, s.lse, s.ws)
    _select(s)
    _decode(s)
    return [s.q, s.k, s.out, s.scores, s.kept, s.post, s.tok_out, s.tok_lse, s.tail_k]


# ---- what a pass cannot do without -----------------------------------------------------------------------------
def work(case):
    lay = _layout(case)
    H, Hkv, D, kind = case["heads"], case["kv_heads"], case["dim"], case["kind"]
    eb = 4 if case["dtype"] == "f32" else 2
    T, R, B = lay.total_tokens, int(lay.qry_len.sum()), lay.n_prompts
    nbytes = flops = 0.0
    if kind in ("step", "prefill"):
        rows = R if case["rows"] == "query" else T
        nbytes += (2.0 * rows * H + 2.0 * T * Hkv) * D * eb + (4.0 * rows * H if case["lse"] else 0.0)
        flops += 4.0 * D * H * _pairs(case, lay)
        if kind == "step":                                       # the rotated Q and K are results too
            nbytes += 1.0 * T * (H + Hkv) * D * eb
    if kind in ("step", "select"):
        nbytes += float(R - lay.n_paths) * case["vocab"] * eb    # rows without a target are not read
        flops += 4.0 * (R - lay.n_paths) * case["vocab"]
    if kind in ("step", "decode"):
        kept, tail_len = _kept_and_tail(case, lay)
        tails = B if kind == "step" else int(tail_len.sum())
        keys = int(lay.pre_len.sum() + (lay.doc_len + lay.qry_len)[kept].sum()) + tails
        nbytes += (2.0 * keys * Hkv + 2.0 * B * H) * D * eb
        flops += 4.0 * keys * H * D
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # bf16 attention: the probabilities and the output are rounded to bf16 once each; against fp64 on the same inputs
    # that is 2e-3 of the output's norm.  fp32: sums of some hundred terms in another order.  Scores: fp32
    # log-sum-exp over the vocabulary with the hardware exponential.  Kept indices are exact.
    if case["kind"] == "select":
        return {"rel": 1e-5, "max": 2e-4, "differ": 0.0}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4, "differ": 0.0}
    return {"rel": 8e-3, "max": 0.1, "differ": 0.0}
