"""Path independence on the device (Section 3.2: a path sees its prompt's preamble and itself,
never another path).  The oracle has this property by construction (pinned on the CPU); here
the CUDA kernels are held to it bit for bit: changing one document's Q / K / V, even to Inf or
NaN, must leave every other path's and the preamble's rows of `out` and `lse` unchanged."""
import math

import numpy as np
import pytest
import torch

import paper_2404_06910_b200 as sp
from helpers import dev, workspace
from workloads import build_layout

pytestmark = pytest.mark.gpu

TDT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _randn(shape, dtype, seed, std=1.0):
    g = torch.Generator()
    g.manual_seed(seed)
    return (torch.randn(*shape, generator=g) * std).to(TDT[dtype])


def _layout():
    # ragged on purpose: document ends fall inside 16-key MMA steps and inside TMA boxes, so the
    # rows that follow a path's last key in shared memory belong to its neighbour
    return build_layout([21, 40],
                        [[37, 130, 9, 77], [150, 3, 61]],
                        [[5, 7, 3, 11], [9, 2, 6]])


def _path_rows(lay, i):
    return np.arange(lay.path_start[i], lay.path_start[i] + lay.doc_len[i] + lay.qry_len[i])


def _run_prefill(q, k, v, lay, rows):
    dl = sp.DeviceLayout.from_host(lay)
    T, H, D = q.shape
    out = torch.zeros((T, H, D), dtype=q.dtype, device="cuda")
    lse = torch.zeros((H, T), device="cuda")
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.dtype_code(q)))
    sp.sp_superpose_prefill(dev(q), dev(k), dev(v), dl, 1 / math.sqrt(D), out, lse, ws, rows=rows)
    sp.sp_check_status(ws)
    return out.cpu(), lse.cpu()


# tcgen05 kernel (bf16), SIMT kernel (fp32); the warp-level kernel for query rows has a test of its own below
@pytest.mark.parametrize("dtype,D,rows", [("bf16", 128, sp.SP_ROWS_ALL), ("bf16", 128, sp.SP_ROWS_QUERY_ONLY),
                                          ("f32", 64, sp.SP_ROWS_ALL), ("bf16", 64, sp.SP_ROWS_ALL)])
@pytest.mark.parametrize("kind", ["finite", "non_finite"])
def test_prefill_paths_do_not_see_each_other(dtype, D, rows, kind):
    lay = _layout()
    T, H, Hkv = lay.total_tokens, 4, 2
    q, k, v = _randn((T, H, D), dtype, 900), _randn((T, Hkv, D), dtype, 901), _randn((T, Hkv, D), dtype, 902)
    out0, lse0 = _run_prefill(q, k, v, lay, rows)
    for j in (1, 2, 5):                                   # a path of each prompt, one of them tiny
        q2, k2, v2 = q.clone(), k.clone(), v.clone()
        r = torch.from_numpy(_path_rows(lay, j))
        if kind == "finite":
            q2[r], k2[r], v2[r] = q2[r] * -1.5 + 0.25, k2[r] * 2.0 - 0.5, v2[r] * -3.0 + 1.0
        else:
            q2[r], k2[r] = float("nan"), float("inf")
            v2[r] = float("nan")
            v2[r[::2]] = float("-inf")
        out1, lse1 = _run_prefill(q2, k2, v2, lay, rows)
        keep = np.ones(T, dtype=bool)
        keep[r.numpy()] = False
        assert torch.equal(out0[keep], out1[keep]), f"path {j} ({kind}) leaked into another path's output"
        assert torch.equal(lse0[:, keep], lse1[:, keep])


@pytest.mark.parametrize("kind", ["finite", "non_finite"])
def test_query_rows_on_the_warp_level_kernel_do_not_see_other_paths(kind):
    """Query rows, an odd number of heads and more than 9 items per SM: the warp-level kernel."""
    rng = np.random.default_rng(7)
    lay = build_layout([21, 400], [[int(x) for x in rng.integers(0, 60, n)] for n in (50, 45)],
                       [[int(x) for x in rng.integers(1, 33, n)] for n in (50, 45)])
    T, H, D = lay.total_tokens, 15, 128
    q, k, v = _randn((T, H, D), "bf16", 940), _randn((T, H, D), "bf16", 941), _randn((T, H, D), "bf16", 942)
    out0, lse0 = _run_prefill(q, k, v, lay, sp.SP_ROWS_QUERY_ONLY)
    rows = np.concatenate([_path_rows(lay, j) for j in range(0, lay.n_paths, 3)])
    r = torch.from_numpy(rows)
    if kind == "finite":
        q[r], k[r], v[r] = q[r] * -1.5 + 0.25, k[r] * 2.0 - 0.5, v[r] * -3.0 + 1.0
    else:
        q[r], k[r], v[r] = float("nan"), float("inf"), float("nan")
    out1, lse1 = _run_prefill(q, k, v, lay, sp.SP_ROWS_QUERY_ONLY)
    keep = np.ones(T, dtype=bool)
    keep[rows] = False
    assert torch.equal(out0[keep], out1[keep]) and torch.equal(lse0[:, keep], lse1[:, keep])


def test_prefill_ignores_rows_outside_every_segment():
    """Packed rows that belong to no segment (gaps between segments) may hold anything."""
    base = build_layout([16], [[45, 70]], [[6, 9]])
    # the same segments with 5 unused rows after each of them
    gap = 5
    import copy
    lay = copy.deepcopy(base)
    lay.path_start = (base.path_start + gap * (1 + np.arange(base.n_paths))).astype(np.int32)
    lay.total_tokens = base.total_tokens + gap * (base.n_paths + 1)
    T, H, D = lay.total_tokens, 2, 128
    used = np.zeros(T, dtype=bool)
    used[:16] = True
    for i in range(lay.n_paths):
        used[_path_rows(lay, i)] = True
    q, k, v = _randn((T, H, D), "bf16", 910), _randn((T, H, D), "bf16", 911), _randn((T, H, D), "bf16", 912)
    out0, lse0 = _run_prefill(q, k, v, lay, sp.SP_ROWS_ALL)
    q2, k2, v2 = q.clone(), k.clone(), v.clone()
    q2[~used], k2[~used], v2[~used] = float("nan"), float("nan"), float("nan")
    out1, lse1 = _run_prefill(q2, k2, v2, lay, sp.SP_ROWS_ALL)
    assert torch.equal(out0[used], out1[used]) and torch.equal(lse0[:, used], lse1[:, used])


@pytest.mark.parametrize("dtype,D,rows", [("f32", 64, sp.SP_ROWS_ALL), ("f32", 64, sp.SP_ROWS_QUERY_ONLY), ("f32", 128, sp.SP_ROWS_ALL),
                                          ("f32", 128, sp.SP_ROWS_QUERY_ONLY), ("bf16", 64, sp.SP_ROWS_ALL),
                                          ("bf16", 64, sp.SP_ROWS_QUERY_ONLY)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_prefill_rows_in_front_of_a_key_do_not_see_it(dtype, D, rows, bad):
    """Causality with a value that is not finite: the rows in front of it keep theirs, the rows behind it have it in its column
    and keep the other columns (probabilities of a few hundred keys do not underflow).  Bit for bit, except that bf16 may have
    computed the column of the rows in front another way: one rounding of the output."""
    lay = _layout()
    T, H, Hkv = lay.total_tokens, 4, 2
    q, k, v = _randn((T, H, D), dtype, 930), _randn((T, Hkv, D), dtype, 931), _randn((T, Hkv, D), dtype, 932)
    out0, lse0 = _run_prefill(q, k, v, lay, rows)
    own = _path_rows(lay, 1)                              # 137 rows, the last seven are query rows
    for at in (0, 1, 62, 63, 64, 127, 131, 135, 136):
        v2 = v.clone()
        v2[own[at], :, 5] = bad
        out1, lse1 = _run_prefill(q, k, v2, lay, rows)
        behind = own[at:] if rows == sp.SP_ROWS_ALL else own[max(at, 130):]
        keep = torch.ones(T, dtype=torch.bool)
        keep[torch.from_numpy(behind)] = False
        cols = torch.arange(D) != 5
        front0, front1 = out0[keep].float(), out1[keep].float()
        assert torch.equal(front0[..., cols], front1[..., cols]) and torch.equal(lse0, lse1), at
        off = (front0[..., 5] - front1[..., 5]).abs()
        assert bool((off <= (0.0 if dtype == "f32" else 2.0 ** -7 * front0[..., 5].abs() + 1e-6)).all()), at
        assert torch.equal(out0[behind][..., cols], out1[behind][..., cols]), at
        got = out1[behind][..., 5]
        assert bool(torch.isnan(got).all() if bad != bad else (got == bad).all()), at


@pytest.mark.parametrize("dtype,D", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("kind", ["finite", "non_finite"])
def test_decode_sees_only_kept_paths(dtype, D, kind):
    """The decode attention reads the preamble, the kept paths and the tail: a path that was
    pruned may change (or hold Inf / NaN) without any effect, bit for bit."""
    lay = _layout()
    B, T, H, Hkv, cap = lay.n_prompts, lay.total_tokens, 4, 2, 3
    kc, vc = _randn((T, Hkv, D), dtype, 920), _randn((T, Hkv, D), dtype, 921)
    q = _randn((B, H, D), dtype, 922)
    tk, tv = _randn((B, cap, Hkv, D), dtype, 923), _randn((B, cap, Hkv, D), dtype, 924)
    kept = np.array([[3, 0], [4, -1]], np.int32)           # pruned: paths 1, 2 (prompt 0) and 5, 6 (prompt 1)
    tl = np.array([2, 3], np.int32)
    dl = sp.DeviceLayout.from_host(lay)

    def run(kc_, vc_):
        out = torch.zeros((B, H, D), dtype=TDT[dtype], device="cuda")
        lse = torch.zeros((B, H), device="cuda")
        ws = workspace(sp.sp_decode_workspace_bytes(B, H, D))
        sp.sp_pruned_decode(dev(q), dev(kc_), dev(vc_), dl, dev(kept), 2, dev(tk), dev(tv), dev(tl), cap,
                            1 / math.sqrt(D), out, lse, ws)
        sp.sp_check_status(ws)
        return out.cpu(), lse.cpu()

    out0, lse0 = run(kc, vc)
    for j in (1, 2, 5, 6):
        k2, v2 = kc.clone(), vc.clone()
        r = torch.from_numpy(_path_rows(lay, j))
        if kind == "finite":
            k2[r], v2[r] = k2[r] * 2.0 - 0.5, v2[r] * -3.0 + 1.0
        else:
            k2[r], v2[r] = float("inf"), float("nan")
        out1, lse1 = run(k2, v2)
        assert torch.equal(out0, out1) and torch.equal(lse0, lse1), f"pruned path {j} ({kind}) reached the decode output"


@pytest.mark.parametrize("dtype,D,Hkv", [("bf16", 128, 1), ("bf16", 128, 2), ("bf16", 128, 4), ("bf16", 64, 1), ("bf16", 64, 2),
                                         ("f32", 64, 1)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("rope", [False, True])
def test_decode_values_that_are_not_finite_stay_in_their_column(dtype, D, Hkv, bad, rope):
    """An Inf in V is an Inf of the output and no NaN, in its column alone, wherever the key lies: preamble, kept paths, the last
    key of a split, the tail's older rows and the newest one.  The other columns keep their bits."""
    lay = build_layout([21], [[37, 130, 9, 77]], [[5, 7, 3, 11]])
    T, H, cap, k = lay.total_tokens, 4, 3, 2
    kc, vc = _randn((T, Hkv, D), dtype, 970), _randn((T, Hkv, D), dtype, 971)
    q, tk, tv = dev(_randn((1, H, D), dtype, 972)), _randn((1, cap, Hkv, D), dtype, 973), _randn((1, cap, Hkv, D), dtype, 974)
    dl, kept, tl, pos = sp.DeviceLayout.from_host(lay), dev(np.array([[3, 0]], np.int32)), dev(np.array([3], np.int32)), torch.full((1,), 9.0, device="cuda")

    def run(vc_, tv_):
        out = torch.zeros((1, H, D), dtype=TDT[dtype], device="cuda")
        args = (q, dev(kc), dev(vc_), dl, kept, k, dev(tk), dev(tv_), tl, cap)
        if rope:
            sp.sp_pruned_decode_rope(*args, pos, D ** -0.5, out)
        else:
            sp.sp_pruned_decode(*args, D ** -0.5, out, None, workspace(sp.sp_decode_workspace_bytes(1, H, D)))
        return out.cpu()

    out0, cols = run(vc, tv), torch.arange(D) != 5
    rows = [("cache", r) for r in (0, 15, 20, int(_path_rows(lay, 0)[-1]), int(_path_rows(lay, 3)[0]), int(_path_rows(lay, 3)[-1]))]
    for where, r in rows + [("tail", 0), ("tail", 2)]:
        v2, t2 = vc.clone(), tv.clone()
        (v2 if where == "cache" else t2[0])[r, :, 5] = bad
        out1 = run(v2, t2)
        assert torch.equal(out0[..., cols], out1[..., cols]), (where, r)
        got = out1[..., 5].float()
        assert bool(torch.isnan(got).all() if bad != bad else (got == bad).all()), (where, r, got)


@pytest.mark.parametrize("D,Hkv", [(128, 4), (128, 2), (64, 4)])
def test_prefills_in_a_row_through_one_workspace(D, Hkv):
    """Launches may start before the one in front of them has finished: each reads the work list of its own layout.  Layouts of
    different lengths through one workspace, nothing waited for in between, against runs on their own."""
    lays = [build_layout([21, 40], [[37, 130, 9, 77], [150, 3, 61]], [[5, 7, 3, 11], [9, 2, 6]]),
            build_layout([300], [[400, 20]], [[30, 1]]),
            build_layout([0, 5, 16] * 8, [[60, 1], [200, 31, 8], [90]] * 8, [[8, 2], [32, 1, 9], [40]] * 8)]
    H, runs = 4, []
    for n, lay in enumerate(lays):
        q, k, v = (dev(_randn((lay.total_tokens, h, D), "bf16", 950 + 3 * n + i)) for i, h in enumerate((H, Hkv, Hkv)))
        runs.append((sp.DeviceLayout.from_host(lay), q, k, v, torch.arange(lay.total_tokens, device="cuda", dtype=torch.float32)))
    size = sp.sp_prefill_rope_workspace_bytes if D == 128 else sp.sp_prefill_workspace_bytes
    ws = workspace(max(size(r[0], H, D, sp.SP_BF16) for r in runs))

    def call(r, form):
        dl, q, k, v, pos = r
        out = torch.zeros_like(q)
        if form == 2 and D == 128:
            sp.sp_superpose_prefill_rope(q, k, v, dl, pos, 10000.0, sp.SP_ROPE_HALF_SPLIT, D ** -0.5, out, None, ws)
        else:
            sp.sp_superpose_prefill(q, k, v, dl, D ** -0.5, out, None, ws, rows=sp.SP_ROWS_QUERY_ONLY if form == 1 else sp.SP_ROWS_ALL)
        return out

    alone = []
    for r in runs:
        for form in range(3):
            alone.append(call(r, form))
            torch.cuda.synchronize()
    order = np.random.default_rng(1).integers(0, len(alone), 120)
    got = [call(runs[i // 3], i % 3) for i in order]
    sp.sp_check_status(ws)
    for i, o in zip(order, got):
        assert torch.equal(o, alone[i]), (i // 3, i % 3)


@pytest.mark.parametrize("H,Hkv", [(4, 4), (8, 2)])
def test_a_chain_reads_what_the_call_before_wrote(H, Hkv):
    """Rotation -> decode on inputs that change from step to step, scores -> top-k -> decode: what one kernel writes the next one
    reads, nothing waited for in between, against the same steps one by one."""
    lay, D, V, k, steps = _layout(), 128, 600, 2, 24
    dl = sp.DeviceLayout.from_host(lay)
    B, T, R = lay.n_prompts, lay.total_tokens, int(lay.qry_len.sum())
    off = dev(np.concatenate([[0], np.cumsum(lay.qry_len)]).astype(np.int32))
    kc, vc = dev(_randn((T, Hkv, D), "bf16", 960)), dev(_randn((T, Hkv, D), "bf16", 961))
    tk, tv = dev(_randn((steps, B, 1, Hkv, D), "bf16", 962)), dev(_randn((steps, B, 1, Hkv, D), "bf16", 963))
    qs, logits = dev(_randn((steps, B, H, D), "bf16", 964)), dev(_randn((steps, R, V), "bf16", 965))
    tgt = dev(torch.randint(0, V, (R,), generator=torch.Generator().manual_seed(966), dtype=torch.int32))
    tl, ws, sws = dev(np.ones(B, np.int32)), workspace(sp.sp_decode_workspace_bytes(B, H, D)), workspace(sp.sp_path_scores_workspace_bytes(R))
    q, key, scores = torch.empty_like(qs[0]), torch.empty_like(tk[0]), torch.empty(lay.n_paths, device="cuda")
    kept = torch.empty((B, k), dtype=torch.int32, device="cuda")

    def run(wait):
        outs = []
        for i in range(steps):
            pos = torch.full((B,), 100.0 + i, device="cuda")
            out = torch.empty_like(q)
            q.copy_(qs[i])
            key.copy_(tk[i])
            for f in (lambda: sp.sp_path_scores(logits[i], tgt, off, scores, None, None, None, sws),
                      lambda: sp.sp_prune_topk(scores, dl.prompt_path_off, k, kept),
                      lambda: sp.sp_rope_apply_pair(q, H, key, Hkv, pos, D),
                      lambda: sp.sp_pruned_decode(q, kc, vc, dl, kept, k, key, tv[i], tl, 1, D ** -0.5, out, None, ws)):
                f()
                if wait:
                    torch.cuda.synchronize()
            outs.append((out, kept.clone()))
        return outs

    for (a, ka), (b, kb) in zip(run(True), run(False)):
        assert torch.equal(ka, kb) and torch.equal(a, b)
