"""The prefill and decode kernels at the sizes where their tiling can go wrong: edges of query tiles, tile pairs, key tiles
and of the preamble's padding, the smallest and largest of each range, and both sides of every dispatch rule, against the
oracle with the tolerances of the parity suite (bf16: rel-L2 1e-2, from one rounding of probabilities and output; per row
twice that; fp32: 1e-5)."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2404_06910_b200 as sp
from helpers import dev, f32, rel_l2, workspace
from workloads import build_layout

pytestmark = pytest.mark.gpu

TOL = {torch.bfloat16: 1e-2, torch.float32: 1e-5}


def _randn(shape, seed, dtype=torch.bfloat16):
    return torch.randn(*shape, generator=torch.Generator().manual_seed(seed)).to(dtype)


def _median_ms(call, n=5):
    times = []
    for _ in range(n):
        begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        begin.record()
        call()
        end.record()
        end.synchronize()
        times.append(begin.elapsed_time(end))
    return sorted(times)[n // 2]


def _prefill(lay, H, Hkv, D, dtype=torch.bfloat16, rows=sp.SP_ROWS_ALL, alibi=False, shift=0, mirror=True, repeats=0):
    """Runs and checks one prefill, and repeats, which have to give the same bits; shift: elements by which the output's address misses 32-byte alignment."""
    T = lay.total_tokens
    q, k, v = _randn((T, H, D), 1, dtype), _randn((T, Hkv, D), 2, dtype), _randn((T, Hkv, D), 3, dtype)
    pos = torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float() if alibi else None
    slopes = np.array([2.0 ** (-8.0 * (h + 1) / H) for h in range(H)], np.float32)
    bias = dict(pos=pos.numpy(), slopes=slopes) if alibi else {}
    ref_o, ref_l = oracle.prefill(f32(q), f32(k), f32(v), lay, 1 / math.sqrt(D), **bias)
    dl = sp.DeviceLayout.from_host(lay, mirror=mirror)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.dtype_code(q)))
    qd, kd, vd, posd, slopesd = dev(q), dev(k), dev(v), dev(pos) if alibi else None, dev(slopes)

    def run():
        out = torch.full((T * H * D + shift,), float("nan"), dtype=dtype, device="cuda")[shift:].view(T, H, D)
        lse = torch.full((H, T), float("nan"), device="cuda")
        if alibi:
            sp.sp_superpose_prefill_alibi(qd, kd, vd, dl, posd, slopesd, 1 / math.sqrt(D), out, lse, ws, rows=rows)
        else:
            sp.sp_superpose_prefill(qd, kd, vd, dl, 1 / math.sqrt(D), out, lse, ws, rows=rows)
        sp.sp_check_status(ws)
        return out, lse

    out, lse = run()
    for _ in range(repeats):
        for a, b in zip(run(), (out, lse)):
            np.testing.assert_array_equal(f32(a), f32(b))
    sel = np.ones(T, bool)
    if rows == sp.SP_ROWS_QUERY_ONLY:
        sel[:] = False
        for s, d, n in zip(lay.path_start, lay.doc_len, lay.qry_len):
            sel[s + d:s + d + n] = True
    got, got_l = f32(out), lse.cpu().numpy()
    assert not np.isnan(got[sel]).any() and np.isnan(got[~sel]).all()
    assert rel_l2(got[sel], ref_o[sel]) <= TOL[dtype]
    num = np.linalg.norm((got - ref_o)[sel].reshape(int(sel.sum()), -1), axis=1)
    assert (num / (np.linalg.norm(ref_o[sel].reshape(int(sel.sum()), -1), axis=1) + 1e-6)).max() <= 2 * TOL[dtype]
    np.testing.assert_allclose(got_l[:, sel], ref_l[:, sel], atol=2e-5 if dtype == torch.float32 else 2e-2)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("pre", [0, 1, 16, 63, 65, 130])
def test_prefill_segment_lengths(D, alibi, pre):
    """One, two and three query tiles and one row on either side of each; preambles around the 16-row padding and the key tile."""
    lens = [1, 31, 33, 127, 128, 129, 191, 255, 256, 257, 385]
    lay = build_layout([pre, 17], [[n - 1 for n in lens], [64, 300]], [[1] * len(lens), [9, 20]])
    _prefill(lay, 4, 2, D, alibi=alibi)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,Hkv", [(3, 1), (6, 1), (4, 1), (12, 1), (16, 2), (16, 1)])
@pytest.mark.parametrize("rows,alibi", [(sp.SP_ROWS_ALL, False), (sp.SP_ROWS_ALL, True), (sp.SP_ROWS_QUERY_ONLY, False)])
def test_prefill_heads_sharing_a_tile(D, H, Hkv, rows, alibi):
    """1, 2, 4 and 8 heads in a tile (128, 64, 32 and 16 rows of each); segments around the tiles' and pairs' edges."""
    lens = [1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 127, 129, 257]
    lay = build_layout([21, 70], [[n - min(n, 33) for n in lens], [40, 150]], [[min(n, 33) for n in lens], [16, 17]])
    _prefill(lay, H, Hkv, D, rows=rows, alibi=alibi)


@pytest.mark.parametrize("n_paths", [20, 63, 64, 79])
@pytest.mark.parametrize("H,Hkv", [(40, 40), (64, 8)])
def test_prefill_sorted_work_list(n_paths, H, Hkv):
    """Lists from a dozen items per block are sorted in runs of 16 records: shorter ones, whole runs and a last run that is
    not full (a record per path and two for the preambles at one head per tile)."""
    rng = np.random.default_rng(n_paths)
    lay = build_layout([33, 5], [rng.integers(0, 180, n_paths), [70]], [[3] * n_paths, [8]])
    _prefill(lay, H, Hkv, 64)


@pytest.mark.parametrize("D", [64, 128])
def test_prefill_output_aligned_to_16_bytes_only(D):
    _prefill(build_layout([20], [[100, 150]], [[24, 24]]), 2, 2, D, shift=8)


def _many_paths(pre, longest, n=46):
    """Enough (path, head) items, with 15 heads, for query rows to go to the warp-level kernel: documents of 0 to 20 rows behind no
    preamble (items of one or two key tiles of 32) among long ones, and ragged ones behind a preamble."""
    rng = np.random.default_rng(11)
    short = [int(x) for x in rng.integers(0, 20, n)]
    short[::7] = [250] * len(short[::7])
    ragged = [int(x) for x in rng.integers(0, 140, n)]
    qry = [int(x) for x in rng.integers(1, 33, n)]
    qry[3] = longest
    return build_layout([0, pre], [short, ragged], [[int(x) for x in rng.integers(1, 12, n)], qry])


@pytest.mark.parametrize("pre,alibi", [(64, True), (65, True), (384, False), (385, False)])
def test_prefill_query_only_either_kernel(pre, alibi):
    """Without a host mirror the preamble decides: both sides of the line."""
    _prefill(_many_paths(pre, 33), 15, 15, 128, rows=sp.SP_ROWS_QUERY_ONLY, alibi=alibi, mirror=False)


@pytest.mark.parametrize("H,Hkv,pre,longest,alibi", [(15, 15, 48, 32, False), (15, 15, 48, 33, False), (15, 5, 385, 32, False),
                                                     (15, 5, 256, 32, True), (15, 15, 257, 32, True), (13, 13, 300, 32, True)])
def test_prefill_query_only_warp_level(H, Hkv, pre, longest, alibi):
    """With one, the number of items (13 heads: few) and the longest query do: 32 and 33 rows, preambles on both sides of the ALiBi
    line for few items, bit-identical repeats."""
    _prefill(_many_paths(pre, longest), H, Hkv, 128, rows=sp.SP_ROWS_QUERY_ONLY, alibi=alibi, repeats=2)


@pytest.mark.parametrize("n,H,Hkv,pre,alibi,low,high", [(4, 6, 6, 48, False, 0.0, 1.8e-3), (4, 6, 2, 64, True, 0.0, 1.8e-3),
                                                        (4, 8, 2, 400, False, 0.0, 1.8e-3), (60, 6, 6, 100, False, 2e-3, 2.4e-3)])
def test_prefill_query_only_precision(n, H, Hkv, pre, alibi, low, high):
    """Distance of the query rows to 64-bit results.  Rounding the output to bf16 alone is 1.66e-3 of its norm for values spread
    over binades (2^-8 / sqrt 3 over a root-mean-square mantissa of 1.36); probabilities carried to 16 bits add 1e-5, rounded to
    bf16 relative to the running maximum (the warp-level kernel, many items) they add 1.4e-3 in quadrature: 2.2e-3."""
    lay = build_layout([pre] * n, [[150, 90, 200, 64]] * n, [[32, 24, 9, 31]] * n)
    T, D = lay.total_tokens, 128
    q, k, v = _randn((T, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3)
    pos = torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float()
    slopes = np.array([2.0 ** (-8.0 * (h + 1) / H) for h in range(H)], np.float32)
    dl = sp.DeviceLayout.from_host(lay)
    out, ws = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))
    args = (dev(q), dev(k), dev(v), dl)
    if alibi:
        sp.sp_superpose_prefill_alibi(*args, dev(pos), dev(slopes), D ** -0.5, out, None, ws, rows=sp.SP_ROWS_QUERY_ONLY)
    else:
        sp.sp_superpose_prefill(*args, D ** -0.5, out, None, ws, rows=sp.SP_ROWS_QUERY_ONLY)
    ref, _ = oracle.prefill(f32(q), f32(k), f32(v), lay, D ** -0.5, **(dict(pos=pos.numpy(), slopes=slopes) if alibi else {}))
    rows = np.concatenate([np.arange(s + d, s + d + n) for s, d, n in zip(lay.path_start, lay.doc_len, lay.qry_len)])
    assert low <= rel_l2(f32(out)[rows], ref[rows]) <= high


@pytest.mark.parametrize("pre,docs", [(48, [160] * 10), (0, [100] * 10), (48, [40] * 20)])
def test_prefill_query_only_alibi_precision_with_many_paths(pre, docs):
    """As above for many items under ALiBi at equilibrium positions: probabilities carried to 16 bits, so no further from 64-bit results
    than the rounding of the output, 1.66e-3, and 2 % for its spread; with one bf16 number it was 1.88e-3."""
    H, D, n = 16, 128, 10
    lay = build_layout([pre] * n, [docs] * n, [[32] * len(docs)] * n)
    T = lay.total_tokens
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    pos = np.concatenate([sp.sp_positions(pre, np.asarray(docs, np.int32), 32)[0]] * n)
    slopes = np.array([2.0 ** (-8.0 * (h + 1) / H) for h in range(H)], np.float32)
    dl = sp.DeviceLayout.from_host(lay)
    out, ws = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))
    sp.sp_superpose_prefill_alibi(dev(q), dev(k), dev(v), dl, dev(pos), dev(slopes), D ** -0.5, out, None, ws, rows=sp.SP_ROWS_QUERY_ONLY)
    ref, _ = oracle.prefill(f32(q), f32(k), f32(v), lay, D ** -0.5, pos=pos, slopes=slopes)
    rows = np.concatenate([np.arange(s + d, s + d + n) for s, d, n in zip(lay.path_start, lay.doc_len, lay.qry_len)])
    assert rel_l2(f32(out)[rows], ref[rows]) <= 1.7e-3


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("alibi", [False, True])
def test_prefill_f32_tiles(D, alibi):
    lay = build_layout([0, 33], [[1, 14, 15, 62], [64, 130]], [[1, 2, 1, 3], [5, 40]])
    _prefill(lay, 4, 2, D, torch.float32, alibi=alibi)
    _prefill(lay, 4, 2, D, torch.float32, rows=sp.SP_ROWS_QUERY_ONLY, alibi=alibi)


@pytest.mark.parametrize("mirror", [False, True])
@pytest.mark.parametrize("H,more", [(4, 0), (1, 600000)])
def test_prefill_f32_loose_bounds(mirror, H, more):
    """max_pre_len / max_path_len are upper bounds: however large, every row is computed and no launch grows with them (with 600 000
    more rows in the tensors the tiles of six segments take two launches of up to 2^17 blocks)."""
    lay = build_layout([40, 3], [[1, 70, 15], [33]], [[4, 1, 2], [9]])
    lay.total_tokens += more
    T, D = lay.total_tokens, 64
    q, k, v = (torch.randn((T, H, D), device="cuda", generator=torch.Generator("cuda").manual_seed(i)) for i in (1, 2, 3))
    dl, ws, out = sp.DeviceLayout.from_host(lay, mirror=mirror), workspace(256), []
    for pre, path in ((lay.max_pre_len, lay.max_path_len), (2 ** 31 - 1, 2 ** 31 - 1)):
        dl.c.max_pre_len, dl.c.max_path_len = pre, path
        for rows in (sp.SP_ROWS_ALL, sp.SP_ROWS_QUERY_ONLY):
            out.append(torch.zeros_like(q))
            sp.sp_superpose_prefill(q, k, v, dl, 0.125, out[-1], None, ws, rows=rows)
            sp.sp_check_status(ws)
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,Hkv", [(5, 1), (8, 1), (9, 1), (16, 1), (64, 32), (24, 8)])
@pytest.mark.parametrize("n_prompts", [1, 60])
def test_decode_group_sizes(D, H, Hkv, n_prompts):
    """Query heads per KV head up to, at and above a block's eight; split over a cluster and unsplit with one to four warps;
    key counts around the 16 keys of a warp's turn."""
    rng = np.random.default_rng(3)
    lay = build_layout([int(x) for x in rng.integers(0, 40, n_prompts)], [[int(x) for x in rng.integers(0, 70, 3)] for _ in range(n_prompts)],
                       [[int(x) for x in rng.integers(1, 9, 3)] for _ in range(n_prompts)])
    T, cap, k = lay.total_tokens, 5, 2
    q, kc, vc = _randn((n_prompts, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3)
    tk, tv = _randn((n_prompts, cap, Hkv, D), 4), _randn((n_prompts, cap, Hkv, D), 5)
    kept = np.stack([lay.prompt_path_off[b] + rng.permutation(3)[:k] for b in range(n_prompts)]).astype(np.int32)
    tl = rng.integers(0, cap + 1, n_prompts).astype(np.int32)
    tl[0] = cap
    ref_o, ref_l = oracle.pruned_decode(f32(q), f32(kc), f32(vc), lay, kept, f32(tk), f32(tv), tl, 1 / math.sqrt(D))
    out = torch.full((n_prompts, H, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((n_prompts, H), float("nan"), device="cuda")
    sp.sp_pruned_decode(dev(q), dev(kc), dev(vc), sp.DeviceLayout.from_host(lay), dev(kept), k, dev(tk), dev(tv), dev(tl), cap,
                        1 / math.sqrt(D), out, lse, workspace(sp.sp_decode_workspace_bytes(n_prompts, H, D)))
    assert rel_l2(f32(out), ref_o) <= TOL[torch.bfloat16]
    fin = np.isfinite(ref_l)
    np.testing.assert_allclose(lse.cpu().numpy()[fin], ref_l[fin], atol=2e-2)
    np.testing.assert_array_equal(lse.cpu().numpy()[~fin], ref_l[~fin])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab,pad", [(1, 0), (7, 0), (8, 0), (9, 4), (129, 0), (2051, 3)])
@pytest.mark.parametrize("n_paths,qry", [(3, 5), (900, 4)])
def test_path_scores_row_alignments(dtype, vocab, pad, n_paths, qry):
    """Rows that start at every offset from a 16-byte boundary, shorter than a vector and longer; few rows (256 threads a row)
    and many (128).  Tolerance: 1e-3 per row as in the parity suite."""
    rows = n_paths * qry
    logits = _randn((rows, vocab + pad), 7, dtype) * 3
    tgt = torch.randint(0, vocab, (rows,), generator=torch.Generator().manual_seed(8), dtype=torch.int32)
    tgt[qry - 1::qry] = -1
    off = np.arange(0, rows + 1, qry, dtype=np.int32)
    ref_s, ref_r = oracle.path_scores(f32(logits[:, :vocab].contiguous()), tgt.numpy(), off, None, None)
    scores, row_logp = torch.empty(n_paths, device="cuda"), torch.empty(rows, device="cuda")
    sp.sp_path_scores(dev(logits)[:, :vocab], dev(tgt), dev(off), scores, None, None, row_logp)
    np.testing.assert_allclose(row_logp.cpu().numpy(), ref_r, atol=1e-3)
    np.testing.assert_allclose(scores.cpu().numpy(), ref_s, atol=1e-3 * qry)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab,pad", [(8, 0), (129, 0), (2051, 3), (2048, 0), (50257, 0)])
@pytest.mark.parametrize("n_paths,qry", [(3, 5), (900, 4)])
@pytest.mark.parametrize("lowest", [False, True])
def test_path_scores_masked_logits(dtype, vocab, pad, n_paths, qry, lowest):
    """Logits of -inf or the type's lowest value at the head of a row, at its end, over a whole range, in every vector of some
    threads, and everywhere but at the target.  Tolerance: 1e-3 per row as in the parity suite."""
    if vocab == 50257 and n_paths == 900:
        n_paths = 300                                        # 1 200 rows suffice where rows are long
    rows = n_paths * qry
    mask = torch.finfo(dtype).min if lowest else float("-inf")
    logits = _randn((rows, vocab + pad), 7, dtype) * 3
    tgt = torch.randint(0, vocab, (rows,), generator=torch.Generator().manual_seed(8), dtype=torch.int32)
    tgt[qry - 1::qry] = -1
    at = torch.arange(vocab + pad)
    banned = [at < 1, at >= vocab - 1, at >= vocab // 2, at // 8 % 256 == 3, at >= 0]
    for r in range(rows):
        keep = logits[r, max(int(tgt[r]), 0)].clone()
        logits[r, banned[r % 5]] = mask
        logits[r, max(int(tgt[r]), 0)] = keep
    off = np.arange(0, rows + 1, qry, dtype=np.int32)
    ref_s, ref_r = oracle.path_scores(f32(logits[:, :vocab].contiguous()), tgt.numpy(), off, None, None)
    assert np.isfinite(ref_r).all()
    scores, row_logp = torch.empty(n_paths, device="cuda"), torch.empty(rows, device="cuda")
    sp.sp_path_scores(dev(logits)[:, :vocab], dev(tgt), dev(off), scores, None, None, row_logp)
    np.testing.assert_allclose(row_logp.cpu().numpy(), ref_r, atol=1e-3)
    np.testing.assert_allclose(scores.cpu().numpy(), ref_s, atol=1e-3 * qry)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("H,D", [(2, 64), (64, 64)])
@pytest.mark.parametrize("waves", [0, 3, 8])
@pytest.mark.parametrize("more", [0, 1])
def test_rope_tokens_per_block(dtype, H, D, waves, more):
    """One, two and four tokens to a block: both sides of each limit (waves of 8 blocks per SM), a last block that is not full.
    Tolerances of the parity suite (fp32: a few roundings of values up to 5; bf16: one rounding more, up to 2^-8 of the value)."""
    T = waves * 8 * torch.cuda.get_device_properties(0).multi_processor_count + more + (1 if waves == 0 else 0)
    x = _randn((T, H, D), 1, dtype)
    pos = torch.rand(T, generator=torch.Generator().manual_seed(2)).mul(700).float()
    got = dev(x)
    sp.sp_rope_apply(got, dev(pos), H, D)
    at = np.unique(np.concatenate([np.arange(min(T, 5)), np.arange(max(T - 5, 0), T), np.arange(0, T, 97)]))
    ref = oracle.rope(f32(x)[at], pos.numpy()[at])
    got = f32(got)
    assert np.isfinite(got).all()
    bound = 4e-6 if dtype == torch.float32 else np.abs(ref) * 2.0 ** -8 * 1.02 + 1e-6
    assert (np.abs(got[at] - ref) <= bound).all()


def _short_paths(pre, n_prompts, n, longest, seed=5):
    """Prompts of many short paths behind a preamble, with paths that fill warps, tiles and pairs of tiles among them."""
    rng = np.random.default_rng(seed)
    docs = [[int(x) for x in rng.integers(0, longest, n)] for _ in range(n_prompts)]
    qry = [[int(x) for x in rng.integers(1, 9, n)] for _ in range(n_prompts)]
    for b, edge in enumerate((31, 32, 33, 127, 128, 129, 255, 256, 257)):
        docs[b % n_prompts][b % n], qry[b % n_prompts][b % n] = edge - 1, 1
    return build_layout([pre] * n_prompts, docs, qry)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("pre,n_prompts,n,longest", [(1, 4, 300, 8), (16, 4, 90, 24), (63, 6, 50, 40), (64, 6, 50, 40), (65, 6, 50, 40),
                                                     (200, 5, 30, 90), (40, 2, 1030, 3)])
def test_prefill_tiles_across_paths(D, alibi, pre, n_prompts, n, longest):
    """Tiles over the rows of consecutive paths: path starts at every row of a warp, more of them than lanes in a tile, preambles
    around the key tile, a last pair that is not full, more paths than the plan has threads; and bit-identical repeats."""
    _prefill(_short_paths(pre, n_prompts, n, longest), 20, 20, D, alibi=alibi, repeats=1)


@pytest.mark.parametrize("how", ["prompts in reverse", "gaps", "an empty path", "no preamble", "paths swapped on the device"])
def test_prefill_tiles_across_paths_conditions(how):
    """What tiles over consecutive paths rest on: other places of the prompts keep it; paths that do not follow each other, one
    without rows, a prompt without a preamble, or device arrays unlike the mirror go segment by segment."""
    import copy
    lay = _short_paths(0 if how == "no preamble" else 40, 4, 90, 24)
    H, D, T = 20, 64, lay.total_tokens
    seen = copy.deepcopy(lay)                                     # what the device arrays say
    if how == "prompts in reverse":
        spans = [lay.prompt_row_range(b) for b in range(4)]
        at = 0
        for b in (3, 2, 1, 0):
            move, paths = at - spans[b][0], slice(lay.prompt_path_off[b], lay.prompt_path_off[b + 1])
            seen.pre_start[b] += move
            seen.path_start[paths] += move
            at += spans[b][1] - spans[b][0]
        lay = seen
    elif how == "gaps":
        seen.path_start = (lay.path_start + 3 * np.arange(lay.n_paths)).astype(np.int32)
        seen.pre_start = (lay.pre_start + 3 * lay.prompt_path_off[:-1]).astype(np.int32)
        T = seen.total_tokens = lay.total_tokens + 3 * lay.n_paths
        lay = seen
    elif how == "an empty path":
        lay.doc_len[17] = lay.qry_len[17] = 0
        seen = lay
    elif how == "paths swapped on the device":
        seen.path_start[100], seen.path_start[101] = lay.path_start[100], lay.path_start[100]
        seen.path_start[100] += int(lay.doc_len[101] + lay.qry_len[101])
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    ref, _ = oracle.prefill(f32(q), f32(k), f32(v), seen, 0.125)
    dl = sp.DeviceLayout.from_host(lay)
    dl.arrays[3].copy_(torch.from_numpy(seen.path_start))
    out, ws = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))
    sp.sp_superpose_prefill(dev(q), dev(k), dev(v), dl, 0.125, out, None, ws)
    sp.sp_check_status(ws)
    rows = np.concatenate([np.arange(s, s + n) for s, n in zip(np.concatenate([seen.pre_start, seen.path_start]),
                                                               np.concatenate([seen.pre_len, seen.doc_len + seen.qry_len]))])
    assert rel_l2(f32(out)[rows], ref[rows]) <= TOL[torch.bfloat16]


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("alibi", [False, True])
def test_prefill_tiles_across_paths_keep_values_to_their_path(D, alibi):
    """NaN and Inf in one path's K and V: every other row is as it was, up to the fp32 arithmetic that computes it again where the
    value shares a tile with it (two roundings of a bf16 result, one of them of P: 2^-7 of the largest value)."""
    lay = _short_paths(40, 4, 90, 24)
    H, T = 20, lay.total_tokens
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    pos, slopes = torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float(), torch.linspace(0.01, 0.5, H)
    dl = sp.DeviceLayout.from_host(lay)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))

    def run(k, v):
        out, lse = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), torch.zeros((H, T), device="cuda")
        if alibi:
            sp.sp_superpose_prefill_alibi(dev(q), dev(k), dev(v), dl, dev(pos), dev(slopes), D ** -0.5, out, lse, ws)
        else:
            sp.sp_superpose_prefill(dev(q), dev(k), dev(v), dl, D ** -0.5, out, lse, ws)
        sp.sp_check_status(ws)
        return f32(out), lse.cpu().numpy()

    out0, lse0 = run(k, v)
    k2, v2, others = k.clone(), v.clone(), np.ones(T, bool)
    for i in (5, 120, 200, 355):
        r = slice(int(lay.path_start[i]), int(lay.path_start[i] + lay.doc_len[i] + lay.qry_len[i]))
        k2[r], v2[r], others[r] = float("inf"), float("nan"), False
        v2[r][::2] = float("-inf")
    out1, lse1 = run(k2, v2)
    np.testing.assert_array_equal(lse0[:, others], lse1[:, others])
    assert np.abs(out0[others] - out1[others]).max() <= 2 ** -7 * np.abs(out0).max()


def _short_path_call(lay, H, D, alibi, q, k, v, mirror=True):
    """A call, over tiles across paths where the layout has its host mirror, and its outputs."""
    T = lay.total_tokens
    pos, slopes = dev(torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float()), dev(torch.linspace(0.01, 0.5, H))
    dl = sp.DeviceLayout.from_host(lay, mirror=mirror)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))
    args, out, lse = (dev(q), dev(k), dev(v), dl), torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), torch.zeros((H, T), device="cuda")

    def call():
        if alibi:
            sp.sp_superpose_prefill_alibi(*args, pos, slopes, D ** -0.5, out, lse, ws)
        else:
            sp.sp_superpose_prefill(*args, D ** -0.5, out, lse, ws)

    call()
    sp.sp_check_status(ws)
    return call, f32(out), lse.cpu().numpy()


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("where", ["a preamble", "everywhere"])
def test_prefill_tiles_across_paths_values_that_rows_see(D, alibi, where):
    """A NaN that every row of a prompt sees, or that fills V: it is each row's own and costs a look at the keys, not the row's
    computation anew (by one thread, at some 300 times the launch).  Every bit that does not depend on it stays."""
    H, n = 20, 60
    rng = np.random.default_rng(6)
    lay = build_layout([700] * 4, [[int(x) for x in rng.integers(8, 60, n)] for _ in range(4)], [[8] * n] * 4)
    q, k, v = (_randn((lay.total_tokens, H, D), i) for i in (1, 2, 3))
    clean, out0, lse0 = _short_path_call(lay, H, D, alibi, q, k, v)
    v2 = v.clone()
    paths = slice(int(lay.path_start[n]), int(lay.path_start[2 * n - 1] + lay.doc_len[2 * n - 1] + lay.qry_len[2 * n - 1]))
    if where == "everywhere":
        v2[:] = float("nan")
    else:
        v2[int(lay.pre_start[1]) + 3, :, 7] = float("nan")
    bad, out1, lse1 = _short_path_call(lay, H, D, alibi, q, k, v2)
    np.testing.assert_array_equal(lse0, lse1)
    if where == "everywhere":
        assert np.isnan(out1).all()
    else:
        assert np.isnan(out1[paths][:, :, 7]).all()
        out0[paths][:, :, 7] = out1[paths][:, :, 7] = 0
        same = np.ones(lay.total_tokens, bool)
        same[int(lay.pre_start[1]):int(lay.pre_start[1] + lay.pre_len[1])] = False
        np.testing.assert_array_equal(out0[same], out1[same])
    assert _median_ms(bad) <= 10 * _median_ms(clean)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("first", [False, True])
def test_prefill_tiles_across_paths_scores_of_minus_infinity(D, first):
    """Rows computed again because of an Inf in another path's V while a key of theirs, the first one or another, scores -Inf: that key has no
    weight.  Tolerance as for other rows that are computed again: 2^-7 of the largest value."""
    lay = _short_paths(40, 4, 90, 24)
    H, T = 20, lay.total_tokens
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    q[:, :, 5] = q[:, :, 5].abs() + 0.125
    k[torch.from_numpy(lay.pre_start).long() + (0 if first else 17), :, 5] = float("-inf")
    _, out0, lse0 = _short_path_call(lay, H, D, False, q, k, v)
    others, v2 = np.ones(T, bool), v.clone()
    for b in range(4):                                       # a preamble's rows in front of that key see nothing else
        others[int(lay.pre_start[b]):int(lay.pre_start[b]) + 18] = False
    for i in (5, 120, 200, 355):
        r = slice(int(lay.path_start[i]), int(lay.path_start[i] + lay.doc_len[i] + lay.qry_len[i]))
        v2[r], others[r] = float("inf"), False
    _, out1, lse1 = _short_path_call(lay, H, D, False, q, k, v2)
    assert np.isfinite(out0[others]).all()
    np.testing.assert_array_equal(lse0[:, others], lse1[:, others])
    assert np.abs(out0[others] - out1[others]).max() <= 2 ** -7 * np.abs(out0[others]).max()


@pytest.mark.parametrize("alibi", [False, True])
def test_prefill_short_paths_with_the_output_in_place_of_the_queries(alibi):
    """Output over the queries, with values that are not finite: nothing reads a row of queries again once its result is stored, so the
    bits are those of tiles segment by segment (which a layout without its host mirror always gets) into a buffer of their own."""
    lay = _short_paths(40, 4, 90, 24)
    H, D, T = 20, 128, lay.total_tokens
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    v[int(lay.path_start[120])] = float("inf")
    pos, slopes = torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float(), torch.linspace(0.01, 0.5, H)

    def run(in_place):
        dl = sp.DeviceLayout.from_host(lay, mirror=in_place)
        ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))
        qd, lse = dev(q), torch.zeros((H, T), device="cuda")
        out = qd if in_place else torch.zeros_like(qd)
        if alibi:
            sp.sp_superpose_prefill_alibi(qd, dev(k), dev(v), dl, dev(pos), dev(slopes), D ** -0.5, out, lse, ws)
        else:
            sp.sp_superpose_prefill(qd, dev(k), dev(v), dl, D ** -0.5, out, lse, ws)
        sp.sp_check_status(ws)
        return f32(out), lse.cpu().numpy()

    for a, b in zip(run(True), run(False)):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("H,Hkv", [(10, 10), (8, 2)])
def test_prefill_head64_values_that_rows_see(alibi, H, Hkv):
    """Tiles of one segment, head_dim 64: a NaN in a preamble, which every row of a prompt sees, is no reason to compute rows again; an Inf
    is, for the rows in front of it, and keys that score -Inf, the first one among them, then have no weight."""
    rng = np.random.default_rng(6)
    lay = build_layout([300] * 4, [[int(x) for x in rng.integers(8, 200, 12)] for _ in range(4)], [[8] * 12] * 4)
    T, D = lay.total_tokens, 64
    q, k, v = _randn((T, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3)
    q[:, :, 5] = q[:, :, 5].abs() + 0.125
    k[torch.from_numpy(lay.pre_start).long(), :, 5] = float("-inf")
    clean, out0, lse0 = _short_path_call(lay, H, D, alibi, q, k, v, mirror=False)
    v2 = v.clone()
    v2[int(lay.pre_start[1]) + 3, :, 7] = float("nan")
    bad, out1, lse1 = _short_path_call(lay, H, D, alibi, q, k, v2, mirror=False)
    assert _median_ms(bad) <= 10 * _median_ms(clean)
    np.testing.assert_array_equal(lse0, lse1)
    rows = slice(int(lay.path_start[12]), int(lay.path_start[23] + lay.doc_len[23] + lay.qry_len[23]))
    assert np.isnan(out1[rows][:, :, 7]).all()
    v2 = v.clone()
    r = int(lay.path_start[12]) + 13
    v2[r, :, 7] = float("inf")
    _, out2, _ = _short_path_call(lay, H, D, alibi, q, k, v2, mirror=False)
    first = slice(int(lay.path_start[12]), r)
    assert np.abs(out2[first] - out0[first]).max() <= 2 ** -7 * np.abs(out0[first]).max()


QRY_EDGES = [1, 8, 15, 16, 17, 31, 32, 33, 47, 48]


@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("longest", [32, 48])
@pytest.mark.parametrize("pre", [0, 1, 16, 17, 127, 128, 129, 300])
@pytest.mark.parametrize("H,Hkv,n", [(3, 1, 2), (29, 29, 6)])
def test_prefill_query_rows_key_tiles(alibi, longest, pre, H, Hkv, n):
    """Keys on the M side: 1 to 48 query rows, documents and preambles around the 128 keys of a tile, items of one key to several
    tiles; few items (P as two numbers) and many (with at most 32 rows and 128 of preamble: for the first keys); bit-identical repeats."""
    docs = [0, 1, 15, 95, 96, 97, 127, 128, 129, 260]
    qry = [x for x in QRY_EDGES if x <= longest]
    qry = (qry * 2)[:len(docs)]
    lay = build_layout([pre] * n, [docs] * n, [qry[i:] + qry[:i] for i in range(n)])
    _prefill(lay, H, Hkv, 128, rows=sp.SP_ROWS_QUERY_ONLY, alibi=alibi, repeats=1)


@pytest.mark.parametrize("alibi", [False, True])
@pytest.mark.parametrize("pre,longest", [(21, 32), (200, 32), (21, 48)])
def test_prefill_query_rows_key_tiles_keep_values_to_their_path(alibi, pre, longest):
    """NaN and Inf in every third path, which the padding behind preambles and paths reaches into: the others keep their bits."""
    rng = np.random.default_rng(7)
    docs, qry = ([[int(x) for x in rng.integers(lo, hi, n)] for n in (50, 45)] for lo, hi in ((0, 60), (1, longest + 1)))
    qry[0][1] = longest
    lay = build_layout([pre, pre], docs, qry)
    T, H, D = lay.total_tokens, 15, 128
    q, k, v = (_randn((T, H, D), i) for i in (1, 2, 3))
    pos, slopes = torch.rand(T, generator=torch.Generator().manual_seed(4)).mul(300).float(), torch.linspace(0.01, 0.5, H)
    dl = sp.DeviceLayout.from_host(lay)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))

    def run():
        out, lse = torch.zeros((T, H, D), dtype=torch.bfloat16, device="cuda"), torch.zeros((H, T), device="cuda")
        args = (dev(q), dev(k), dev(v), dl)
        if alibi:
            sp.sp_superpose_prefill_alibi(*args, dev(pos), dev(slopes), D ** -0.5, out, lse, ws, rows=sp.SP_ROWS_QUERY_ONLY)
        else:
            sp.sp_superpose_prefill(*args, D ** -0.5, out, lse, ws, rows=sp.SP_ROWS_QUERY_ONLY)
        sp.sp_check_status(ws)
        return f32(out), lse.cpu().numpy()

    out0, lse0 = run()
    others = np.ones(T, bool)
    for i in range(0, lay.n_paths, 3):
        r = slice(int(lay.path_start[i]), int(lay.path_start[i] + lay.doc_len[i] + lay.qry_len[i]))
        q[r], k[r], v[r], others[r] = float("nan"), float("inf"), float("nan"), False
    out1, lse1 = run()
    np.testing.assert_array_equal(out0[others], out1[others])
    np.testing.assert_array_equal(lse0[:, others], lse1[:, others])


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("k", [1, 2, 3, 6, 7])
@pytest.mark.parametrize("H,Hkv,n_prompts,longest", [(8, 8, 1, 70), (32, 32, 3, 300), (8, 4, 40, 70), (16, 2, 60, 40), (40, 40, 30, 30), (12, 4, 9, 400), (64, 64, 20, 20)])
def test_decode_keys_through_a_ring(D, k, H, Hkv, n_prompts, longest):
    """Segment tables of odd and even size in front of the rings, single and grouped heads, from few units, each split over a cluster, to
    more than there are warps; turns of 16 keys within a segment and across its end, prompts with fewer keys than warps."""
    rng = np.random.default_rng(k)
    lay = build_layout([int(x) for x in rng.integers(0, 40, n_prompts)], [[int(x) for x in rng.integers(0, longest, 8)] for _ in range(n_prompts)],
                       [[int(x) for x in rng.integers(1, 9, 8)] for _ in range(n_prompts)])
    T, cap = lay.total_tokens, 5
    q, kc, vc = _randn((n_prompts, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3)
    tk, tv = _randn((n_prompts, cap, Hkv, D), 4), _randn((n_prompts, cap, Hkv, D), 5)
    kept = np.stack([lay.prompt_path_off[b] + rng.permutation(8)[:k] for b in range(n_prompts)]).astype(np.int32)
    tl = rng.integers(0, cap + 1, n_prompts).astype(np.int32)
    ref_o, ref_l = oracle.pruned_decode(f32(q), f32(kc), f32(vc), lay, kept, f32(tk), f32(tv), tl, 1 / math.sqrt(D))
    args = (dev(q), dev(kc), dev(vc), sp.DeviceLayout.from_host(lay), dev(kept), k, dev(tk), dev(tv), dev(tl), cap, 1 / math.sqrt(D))
    ws = workspace(sp.sp_decode_workspace_bytes(n_prompts, H, D))
    outs = []
    for _ in range(2):
        out, lse = torch.full((n_prompts, H, D), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((n_prompts, H), float("nan"), device="cuda")
        sp.sp_pruned_decode(*args, out, lse, ws)
        outs.append((f32(out), lse.cpu().numpy()))
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    assert rel_l2(outs[0][0], ref_o) <= TOL[torch.bfloat16]
    fin = np.isfinite(ref_l)
    np.testing.assert_allclose(outs[0][1][fin], ref_l[fin], atol=2e-2)
    np.testing.assert_array_equal(outs[0][1][~fin], ref_l[~fin])


@pytest.mark.parametrize("H,D", [(32, 128), (40, 64)])
@pytest.mark.parametrize("alibi", [False, True])
def test_decode_single_heads_in_fp32_arithmetic(H, D, alibi):
    """Scores, probabilities and sums of single heads in bf16 are fp32 numbers.  An error of 2^-22 puts an output on the other side of a
    rounding boundary, bf16 numbers being 2^-8 apart, in one of 2^13 cases, 0.012 %; four times that are allowed.  Probabilities cut off behind 16
    bits came to 0.27 and 0.31 %."""
    rng = np.random.default_rng(0)
    lay = build_layout([64, 64], [[int(x) for x in rng.integers(128, 513, 8)] for _ in range(2)], [[24] * 8] * 2)
    T, cap, k = lay.total_tokens, 256, 8
    q, kc, vc, tk, tv = _randn((2, H, D), 1), _randn((T, H, D), 2), _randn((T, H, D), 3), _randn((2, cap, H, D), 4), _randn((2, cap, H, D), 5)
    kept, tl = np.arange(16, dtype=np.int32).reshape(2, 8), np.array([200, 31], np.int32)
    q_pos, pos, tail_pos = torch.tensor([700.0, 650.0]), torch.rand(T, generator=torch.Generator().manual_seed(6)) * 600, torch.full((2, cap), 640.0)
    slopes = torch.exp2(-8.0 * (torch.arange(H) + 1) / H).float()
    out, lse = torch.zeros((2, H, D), dtype=torch.bfloat16, device="cuda"), torch.zeros((2, H), device="cuda")
    args = (dev(q), dev(kc), dev(vc), sp.DeviceLayout.from_host(lay), dev(kept), k, dev(tk), dev(tv), dev(tl), cap)
    ws = workspace(sp.sp_decode_workspace_bytes(2, H, D))
    if alibi:
        sp.sp_pruned_decode_alibi(*args, dev(q_pos), dev(pos), dev(tail_pos), dev(slopes), D ** -0.5, out, lse, ws)
    else:
        sp.sp_pruned_decode(*args, D ** -0.5, out, lse, ws)
    wrong = 0
    for b in range(2):
        (lo, hi), n = lay.prompt_row_range(b), int(tl[b])
        keys, values = torch.cat([kc[lo:hi], tk[b, :n]]).double(), torch.cat([vc[lo:hi], tv[b, :n]]).double()
        s = torch.einsum("hd,khd->hk", q[b].double(), keys) * D ** -0.5
        if alibi:
            s -= slopes.double()[:, None] * (q_pos[b].double() - torch.cat([pos[lo:hi], tail_pos[b, :n]]).double()).abs()
        wrong += int((out[b].cpu() != torch.einsum("hk,khd->hd", torch.softmax(s, 1), values).float().bfloat16()).sum())
    assert wrong <= 5e-4 * 2 * H * D


@pytest.mark.parametrize("H,Hkv", [(8, 1), (8, 4)])
def test_decode_thousands_of_kept_paths(H, Hkv):
    """The table of 4 096 kept paths, 112 KB, leaves shared memory for little else: twice the keys of 2 048 paths, and not above three times
    their time (six where rings were kept at the cost of splits)."""
    D, cap, n = 128, 4, 4096
    rng = np.random.default_rng(3)
    lay = build_layout([9], [[int(x) for x in rng.integers(1, 9, n)]], [[1] * n])
    T = lay.total_tokens
    q, kc, vc, tk, tv = _randn((1, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3), _randn((1, cap, Hkv, D), 4), _randn((1, cap, Hkv, D), 5)
    tl, dl, ws = np.array([3], np.int32), sp.DeviceLayout.from_host(lay), workspace(sp.sp_decode_workspace_bytes(1, H, D))
    cache, took = (dev(q), dev(kc), dev(vc), dl), []
    for k in (n, n // 2):
        kept = rng.permutation(n)[:k].astype(np.int32)[None]
        args = (*cache, dev(kept), k, dev(tk), dev(tv), dev(tl), cap, D ** -0.5)
        out, lse = torch.full((1, H, D), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((1, H), float("nan"), device="cuda")
        sp.sp_pruned_decode(*args, out, lse, ws)
        ref_o, ref_l = oracle.pruned_decode(f32(q), f32(kc), f32(vc), lay, kept, f32(tk), f32(tv), tl, D ** -0.5)
        assert rel_l2(f32(out), ref_o) <= TOL[torch.bfloat16]
        np.testing.assert_allclose(lse.cpu().numpy(), ref_l, atol=2e-2)
        took.append(_median_ms(lambda: [sp.sp_pruned_decode(*args, out, lse, ws) for _ in range(20)], 9))
    assert took[0] <= 3 * took[1]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lens,vocab", [([1], 5), ([4, 5], 700), ([8, 9, 16, 17, 33], 1001), ([100, 0, 1], 64), ([33] * 7, 2051), ([250, 6], 4096), ([257], 64),
                                        ([27], 300), ([25, 1, 1, 0], 64), ([0, 26, 0, 1], 1000), ([1] * 27, 129), ([2, 0, 1], 2051), ([25, 1, 1, 1], 64)])
def test_path_scores_in_one_launch(dtype, lens, vocab):
    """The rows of a path over one to eight blocks of a cluster, four a block at a time; paths without rows, rows in front of the first and
    behind the last path; one path with nearly all rows, as many blocks as fit; a row more than one launch takes.  Bit-identical repeats; tolerance 1e-3 per row as in the parity suite."""
    before, behind = 3, 2
    off = np.concatenate([[before], before + np.cumsum(lens)]).astype(np.int32)
    rows = int(off[-1]) + behind
    logits = _randn((rows, vocab), 7, dtype) * 3
    tgt = torch.randint(-1, vocab, (rows,), generator=torch.Generator().manual_seed(8), dtype=torch.int32)
    prior, weight = _randn((len(lens),), 9, torch.float32), torch.full((len(lens),), 0.125)
    ref_s, ref_r = oracle.path_scores(f32(logits), tgt.numpy(), off, prior.numpy(), weight.numpy())
    got = []
    for _ in range(2):
        scores, row_logp = torch.full((len(lens),), float("nan"), device="cuda"), torch.full((rows,), float("nan"), device="cuda")
        sp.sp_path_scores(dev(logits), dev(tgt), dev(off), scores, dev(prior), dev(weight), row_logp)
        got.append((scores.cpu().numpy(), row_logp.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    want = torch.log_softmax(logits.double(), 1).gather(1, tgt.clamp(min=0).long()[:, None])[:, 0].masked_fill(tgt < 0, 0).numpy()
    np.testing.assert_allclose(got[0][1], want, atol=1e-3)
    np.testing.assert_allclose(got[0][0], ref_s, atol=1e-3 * max(max(lens), 1))


@pytest.mark.parametrize("rows,paths,vocab,more_rows,more_paths", [(8, 65535, 512, 0, 1), (8, 4096, 512, 512, 0), (256, 1, 8000, 4, 0), (128, 1, 8000, 132, 0),
                                                                   (32, 4, 60000, 228, 0)])
def test_path_scores_of_few_rows_take_no_longer_than_of_more(rows, paths, vocab, more_rows, more_paths):
    """Paths without rows by the thousand, one path with all rows, long rows: not above what a call with more rows or paths takes, which
    always goes through two launches.  Half as much again for what timing on a shared machine varies; it was 1.9 to 28 times."""
    def call(rows, paths):
        logits, tgt = torch.randn(rows, vocab, device="cuda").bfloat16(), torch.zeros(rows, dtype=torch.int32, device="cuda")
        off = torch.full((paths + 1,), rows, dtype=torch.int32, device="cuda")
        off[:2] = torch.tensor([0, rows if paths == 1 else rows // 2])
        scores, row_logp = torch.empty(paths, device="cuda"), torch.empty(rows, device="cuda")

        def many():
            for _ in range(20):
                sp.sp_path_scores(logits, tgt, off, scores, None, None, row_logp)
        many()
        return _median_ms(many, 9)

    assert call(rows, paths) <= 1.5 * call(rows + more_rows, paths + more_paths)
