"""The decode with K and V rows through rings in shared memory (bf16, more than 24 units of a prompt and a KV head, or 1 024 keys and
more): the ALiBi bias, the folded rotation and values that are not finite, single heads and groups of 2 and 4, prompts without
preamble, kept paths or tail, splits that end within a turn of 16 keys.  Oracle and tolerances of the parity suite."""
import numpy as np
import pytest
import torch

import oracle
import paper_2404_06910_b200 as sp
from helpers import dev, f32, rel_l2, workspace
from workloads import build_layout

pytestmark = pytest.mark.gpu

TOL = 1e-2
SHAPES = [(32, 32, 3, 300), (8, 4, 40, 70), (16, 4, 10, 200), (40, 40, 30, 30), (8, 8, 2, 900), (8, 2, 2, 900)]      # H, Hkv, prompts, longest document


def _randn(shape, seed):
    return torch.randn(*shape, generator=torch.Generator().manual_seed(seed)).bfloat16()


class Problem:
    def __init__(self, H, Hkv, B, longest, D, k=3, cap=5):
        rng = np.random.default_rng(H + B)
        self.B, self.H, self.Hkv, self.D, self.k, self.cap, self.scale = B, H, Hkv, D, k, cap, D ** -0.5
        pre = [int(x) for x in rng.integers(0, 50, B)]
        pre[0] = 0
        self.lay = lay = build_layout(pre, [[longest] + [int(x) for x in rng.integers(0, longest, 4)] for _ in range(B)], [[int(x) for x in rng.integers(1, 9, 5)] for _ in range(B)])
        T = lay.total_tokens
        self.q, self.kc, self.vc = _randn((B, H, D), 1), _randn((T, Hkv, D), 2), _randn((T, Hkv, D), 3)
        self.tk, self.tv = _randn((B, cap, Hkv, D), 4), _randn((B, cap, Hkv, D), 5)
        self.kept = np.stack([lay.prompt_path_off[b] + rng.permutation(5)[:k] for b in range(B)]).astype(np.int32)
        self.tl = rng.integers(1, cap + 1, B).astype(np.int32)
        self.kept[0] = -1                                    # the newest key is the only one
        self.tl[0] = 1
        self.kept[-1], self.tl[-1] = lay.prompt_path_off[B - 1] + np.arange(k), 0
        self.dl = sp.DeviceLayout.from_host(lay)

    def cache(self, kc=None, vc=None, tk=None, tv=None, tl=None):
        pick = lambda new, old: dev(old if new is None else new)
        return (pick(kc, self.kc), pick(vc, self.vc), self.dl, dev(self.kept), self.k, pick(tk, self.tk), pick(tv, self.tv), pick(tl, self.tl), self.cap)

    def outputs(self):
        return torch.full((self.B, self.H, self.D), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((self.B, self.H), float("nan"), device="cuda")

    def check(self, out, lse, ref_o, ref_l):
        assert rel_l2(f32(out), ref_o) <= TOL
        fin = np.isfinite(ref_l)
        np.testing.assert_allclose(lse.cpu().numpy()[fin], ref_l[fin], atol=2e-2)
        np.testing.assert_array_equal(lse.cpu().numpy()[~fin], ref_l[~fin])

    def kept_rows(self):
        """Cache rows that some prompt attends to."""
        rows = [np.arange(s, s + n) for s, n in zip(self.lay.pre_start, self.lay.pre_len)]
        rows += [np.arange(s, s + d + n) for i in self.kept.ravel() if i >= 0 for s, d, n in [(self.lay.path_start[i], self.lay.doc_len[i], self.lay.qry_len[i])]]
        return np.concatenate(rows).astype(np.int64)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("shape", SHAPES)
def test_ring_with_alibi(D, shape):
    p = Problem(*shape, D)
    g = torch.Generator().manual_seed(9)
    pos, tail_pos, q_pos = torch.rand(p.lay.total_tokens, generator=g) * 300, 300 + torch.rand(p.B, p.cap, generator=g) * 9, torch.full((p.B,), 310.5)
    slopes = torch.exp2(-8.0 * (torch.arange(p.H) + 1) / p.H).float() * 4
    out, lse = p.outputs()
    sp.sp_pruned_decode_alibi(dev(p.q), *p.cache(), dev(q_pos), dev(pos), dev(tail_pos), dev(slopes), p.scale, out, lse, workspace(sp.sp_decode_workspace_bytes(p.B, p.H, D)))
    tensors = (f32(p.q), f32(p.kc), f32(p.vc), p.lay, p.kept, f32(p.tk), f32(p.tv), p.tl, p.scale)
    ref = oracle.pruned_decode(*tensors, q_pos=q_pos.numpy(), cache_pos=pos.numpy(), tail_pos=tail_pos.numpy(), slopes=slopes.numpy())
    assert rel_l2(oracle.pruned_decode(*tensors)[0], ref[0]) > 0.05          # the bias matters here
    p.check(out, lse, *ref)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("pairing", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_ring_with_the_rotation_folded_in(D, pairing, shape):
    """Three steps, whose keys are written back and read again; written rows as the stand-alone rotation stores them, others untouched."""
    p = Problem(*shape, D, cap=7)
    first = np.minimum(p.tl, p.cap - 2)
    tk, sep, ref_tk = dev(p.tk), dev(p.tk), f32(p.tk).copy()
    rnd = lambda a: torch.from_numpy(np.ascontiguousarray(a)).bfloat16().float().numpy()
    for step in range(3):
        tl = (first + step).astype(np.int32)
        q, pos = _randn((p.B, p.H, D), 20 + step), (101.25 + 3.5 * np.arange(p.B) + step).astype(np.float32)
        out, lse = p.outputs()
        kc, vc, dl, kept, k, _, tv, tld, cap = p.cache(tl=tl)
        sp.sp_pruned_decode_rope(dev(q), kc, vc, dl, kept, k, tk, tv, tld, cap, dev(pos), p.scale, out, lse, pairing=pairing)
        for b in np.flatnonzero(tl > 0):
            r = tl[b] - 1
            ref_tk[b, r] = rnd(oracle.rope(np.ascontiguousarray(ref_tk[b, r][None]), pos[b:b + 1], pairing=pairing))[0]
            sp.sp_rope_apply(sep[b, r], dev(pos[b:b + 1]), p.Hkv, D, n_tokens=1, pairing=pairing)
        q_ref = rnd(oracle.rope(f32(q), pos, pairing=pairing))
        p.check(out, lse, *oracle.pruned_decode(q_ref, f32(p.kc), f32(p.vc), p.lay, p.kept, ref_tk, f32(p.tv), tl, p.scale))
        got, want = f32(tk), f32(sep)
        assert (np.abs(got - want) <= np.abs(want) * 2.0 ** -7 + 2e-6).all()          # one rounding of the last place
        for b in range(p.B):
            np.testing.assert_array_equal(got[b, tl[b]:], f32(p.tk)[b, tl[b]:])


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_ring_sees_nothing_but_its_keys(D, rope, shape):
    """Inf and NaN in every row that no prompt attends to, directly behind preambles, kept paths and tails too: the same bits.  An Inf or
    NaN in one column of a row that prompt 1 attends to is in that column of its heads alone."""
    p = Problem(*shape, D)
    seen = np.zeros(p.lay.total_tokens, bool)
    seen[p.kept_rows()] = True

    def run(kc, vc, tk, tv):
        out, lse = p.outputs()
        if rope:
            sp.sp_pruned_decode_rope(dev(p.q), *p.cache(kc, vc, tk, tv), dev(torch.full((p.B,), 9.0)), p.scale, out, lse)
        else:
            sp.sp_pruned_decode(dev(p.q), *p.cache(kc, vc, tk, tv), p.scale, out, lse, workspace(sp.sp_decode_workspace_bytes(p.B, p.H, D)))
        return f32(out), lse.cpu().numpy()

    out0, lse0 = run(p.kc, p.vc, p.tk, p.tv)
    hidden = torch.from_numpy(~seen)
    unused = torch.arange(p.cap)[None] >= torch.from_numpy(p.tl)[:, None]
    kc, vc, tk, tv = p.kc.clone(), p.vc.clone(), p.tk.clone(), p.tv.clone()
    kc[hidden], vc[hidden], tk[unused], tv[unused] = float("nan"), float("inf"), float("inf"), float("nan")
    for a, b in zip(run(kc, vc, tk, tv), (out0, lse0)):
        np.testing.assert_array_equal(a, b)
    i = int(p.kept[1, 0])
    cols = np.arange(D) != 5
    # a kept path's first and last row, the newest key
    for at in [0, int(p.lay.doc_len[i] + p.lay.qry_len[i]) - 1] + [-1] * int(p.tl[1] > 0):
        for bad in (float("inf"), float("-inf"), float("nan")):
            vc, tv = p.vc.clone(), p.tv.clone()
            if at < 0:
                tv[1, int(p.tl[1]) - 1, :, 5] = bad
            else:
                vc[int(p.lay.path_start[i]) + at, :, 5] = bad
            out, lse = run(p.kc, vc, p.tk, tv)
            np.testing.assert_array_equal(lse, lse0)
            np.testing.assert_array_equal(out[..., cols], out0[..., cols])
            np.testing.assert_array_equal(np.delete(out, 1, 0), np.delete(out0, 1, 0))
            assert (np.isnan(out[1, :, 5]) if bad != bad else out[1, :, 5] == bad).all()
