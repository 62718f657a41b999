"""Failure detection without a GPU fault: the producer of the tensor-core prefill is told (on
the host, through a test-only symbol) to load nothing, so every device-side wait runs into its limit.  The kernel must
unwind by itself, report SP_ERR_TIMEOUT through the workspace status word, and leave the
context usable: the next ordinary call gives the same result as before."""
import ctypes
import math
import os
import subprocess
import threading

import numpy as np
import pytest
import torch

import paper_2404_06910_b200 as sp
from helpers import dev, workspace
from workloads import build_layout

pytestmark = pytest.mark.gpu


def test_prefill_bounded_waits_report_timeout_and_context_survives():
    lay = build_layout([32], [[100, 40]], [[24, 24]])
    H, D = 2, 128
    g = torch.Generator().manual_seed(5)
    q, k, v = (torch.randn(lay.total_tokens, H, D, generator=g).bfloat16() for _ in range(3))
    dl = sp.DeviceLayout.from_host(lay)
    qd, kd, vd = dev(q), dev(k), dev(v)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))

    def run():
        out = torch.zeros_like(qd)
        sp.sp_superpose_prefill(qd, kd, vd, dl, 1 / math.sqrt(D), out, None, ws)
        return out

    good = run()
    sp.sp_check_status(ws)

    sp.lib.sp_test_stall_producer(1)            # test-only symbol: the producer loads nothing from now on
    try:
        run()
        with pytest.raises(sp.SpError) as e:
            sp.sp_check_status(ws)
        assert e.value.code == sp.SP_ERR_TIMEOUT
    finally:
        sp.lib.sp_test_stall_producer(0)

    again = run()
    sp.sp_check_status(ws)                      # status word is cleared by the next call
    torch.cuda.synchronize()
    assert torch.equal(good, again)


REPEAT = r"""
#include "sp.h"
int repeat(__typeof__(&sp_pruned_decode) f, int n, const void *q, const void *k, const void *v, const sp_layout *lay, const int32_t *kept,
           const void *tail_k, const void *tail_v, const int32_t *tail_len, int n_heads, void *out, void *ws, size_t ws_bytes, void *stream)
{
    int rc = 0;
    for (int i = 0; i < n && !rc; ++i)
        rc = f(q, k, v, lay, kept, 2, tail_k, tail_v, tail_len, 4, 40 + 2 * 708 + 4, n_heads, n_heads, 128, 0.0883883f, out, 0, ws, ws_bytes, SP_BF16, stream);
    return rc;
}
"""


def test_decode_shapes_that_differ_from_two_threads(tmp_path):
    """Two threads with a stream each launch the same kernel as fast as the host can, with 100 KB (few prompts: four warps a block) and
    50 KB of shared memory (many: two): neither's launch is refused for what the other has set, and both have their results."""
    include = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "include")
    (tmp_path / "repeat.c").write_text(REPEAT)
    subprocess.check_call(["gcc", "-O2", "-shared", "-fPIC", "-I", include, str(tmp_path / "repeat.c"), "-o", str(tmp_path / "repeat.so")])
    repeat = ctypes.CDLL(str(tmp_path / "repeat.so")).repeat          # releases the interpreter's lock for all of its calls
    H, D, cap, failed = 20, 128, 4, []

    def prepare(n):
        g = torch.Generator().manual_seed(n)
        randn = lambda *s: dev(torch.randn(*s, generator=g).bfloat16())
        lay = build_layout([40] * n, [[700, 600]] * n, [[8, 8]] * n)
        T = lay.total_tokens
        dl, out, ws = sp.DeviceLayout.from_host(lay), torch.zeros((n, H, D), dtype=torch.bfloat16, device="cuda"), workspace(sp.sp_decode_workspace_bytes(n, H, D))
        tensors = [randn(n, H, D), randn(T, H, D), randn(T, H, D), dev(np.arange(2 * n, dtype=np.int32)), randn(n, cap, H, D), randn(n, cap, H, D),
                   dev(np.full(n, cap, np.int32)), out, ws]
        p = [ctypes.c_void_p(t.data_ptr()) for t in tensors]
        stream = torch.cuda.Stream()
        call = lambda m: repeat(sp.lib.sp_pruned_decode, m, *p[:3], ctypes.byref(dl.c), *p[3:7], H, *p[7:], ctypes.c_size_t(ws.numel()), ctypes.c_void_p(stream.cuda_stream))
        assert call(1) == 0
        torch.cuda.synchronize()
        return call, stream, out, out.clone(), (tensors, dl)

    def work(call, stream, out, want, keep):
        for _ in range(10):
            rc = call(400)
            stream.synchronize()
            if rc or not torch.equal(out, want):
                failed.append((rc, sp.lib.sp_last_error()))
                return

    threads = [threading.Thread(target=work, args=prepare(n)) for n in (3, 24)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("rows", [32, 48])
def test_query_rows_bounded_waits_report_timeout_and_context_survives(rows):
    lay = build_layout([32], [[100, 40]], [[24, rows]])
    H, D = 2, 128
    g = torch.Generator().manual_seed(5)
    qd, kd, vd = (dev(torch.randn(lay.total_tokens, H, D, generator=g).bfloat16()) for _ in range(3))
    dl = sp.DeviceLayout.from_host(lay)
    ws = workspace(sp.sp_prefill_workspace_bytes(dl, H, D, sp.SP_BF16))

    def run():
        out = torch.zeros_like(qd)
        sp.sp_superpose_prefill(qd, kd, vd, dl, 1 / math.sqrt(D), out, None, ws, rows=sp.SP_ROWS_QUERY_ONLY)
        return out

    good = run()
    sp.sp_check_status(ws)
    sp.lib.sp_test_stall_producer(1)
    try:
        run()
        with pytest.raises(sp.SpError) as e:
            sp.sp_check_status(ws)
        assert e.value.code == sp.SP_ERR_TIMEOUT
    finally:
        sp.lib.sp_test_stall_producer(0)
    again = run()
    sp.sp_check_status(ws)
    assert torch.equal(good, again)
