"""CPU-only checks of the C-ABI library: it loads, exports every symbol the header
declares, rejects bad arguments before any launch, and its host-side position
assignment agrees with the oracle.  No compute call needs a GPU here."""
import ctypes
import os
import re

import numpy as np
import pytest

import oracle
import paper_2404_06910_b200 as sp
from workloads import CONFIGS, draw_lengths
from helpers import positions_for

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "sp.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(sp_[a-z_0-9]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    names = _declared_functions()
    assert len(names) >= 12
    raw = ctypes.CDLL(sp.LIB_PATH)
    for n in names:
        assert hasattr(raw, n), f"{n} declared in include/sp.h but not exported"
    assert set(names) == set(sp.EXPORTS)
    assert sp.sp_version().startswith("sp-b200")


def test_binding_has_a_function_per_symbol():
    for n in _declared_functions():
        if n != "sp_last_error":
            assert callable(getattr(sp, n)), n


@pytest.mark.parametrize("cfg", CONFIGS[:4], ids=lambda c: c.name)
def test_host_positions_match_oracle(cfg):
    lay = draw_lengths(cfg, n_prompts=min(cfg.n_prompts, 4))
    got, nxt = positions_for(lay, lambda P, L, Q: sp.sp_positions(P, L, Q))
    ref, nref = positions_for(lay, lambda P, L, Q: oracle.positions(P, L, Q))
    np.testing.assert_array_equal(got, ref)            # both round the fp64 value once to fp32
    np.testing.assert_allclose(nxt, nref, rtol=1e-15)


def test_host_positions_variants_match_oracle():
    L = [7, 0, 33, 12]
    for scheme, name in ((sp.SP_POS_EQUILIBRIUM, "equilibrium"), (sp.SP_POS_LEFT_ALIGNED, "left")):
        for q_mode in (0, 1):
            got, S, nxt = sp.sp_positions(5, L, 3, scheme=scheme, q_mode=q_mode)
            ref, Sr, nr = oracle.positions(5, L, 3, scheme=name, q_mode=q_mode)
            np.testing.assert_array_equal(got, ref.astype(np.float32))
            assert S == pytest.approx(Sr, rel=1e-15) and nxt == pytest.approx(nr, rel=1e-15)
    got, S, _ = sp.sp_positions(0, [], 0)
    assert got.size == 0 and S == 0.0


def _rc(fn, *args):
    return fn(*args)


def test_invalid_arguments_are_rejected_on_the_host():
    lib = sp.lib
    # sp_positions
    L = np.array([3, -1], np.int32)
    pos = np.zeros(16, np.float32)
    assert lib.sp_positions(0, 0, 2, 2, L.ctypes.data, 1, pos.ctypes.data, None, None) == sp.SP_ERR_INVALID_ARG
    assert b"doc_len" in lib.sp_last_error()
    assert lib.sp_positions(7, 0, 2, 0, None, 1, pos.ctypes.data, None, None) == sp.SP_ERR_INVALID_ARG
    # sp_rope_apply: odd rot_dim, bad dtype, short stride (all before any launch)
    assert lib.sp_rope_apply(256, 256, 4, 64, 1, 64, 63, 10000.0, 0, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_rope_apply(256, 256, 4, 64, 1, 64, 64, 10000.0, 0, 9, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_rope_apply(256, 256, 4, 32, 1, 64, 64, 10000.0, 0, 0, None) == sp.SP_ERR_INVALID_ARG
    # sp_prune_topk: k <= 0
    assert lib.sp_prune_topk(256, 256, 1, 0, 256, None, None) == sp.SP_ERR_INVALID_ARG
    assert b"k must be" in lib.sp_last_error()
    # sp_path_scores: vocab > ld, missing workspace
    assert lib.sp_path_scores(256, 8, 256, 256, 4, 1, 16, None, None, 256, None, None, 0, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_path_scores(256, 16, 256, 256, 4, 1, 16, None, None, 256, None, None, 0, 0, None) == sp.SP_ERR_WORKSPACE
    # layouts
    lay = sp.binding._CLayout(1, 1, 256, 256, 256, 256, 256, 256, 10, 2, 8)
    ref = ctypes.byref(lay)
    # head_dim unsupported / heads not divisible / NULL layout / missing workspace
    assert lib.sp_superpose_prefill(256, 256, 256, ref, 4, 4, 96, 1.0, 0, 256, None, None, 0, 0, None) == sp.SP_ERR_UNSUPPORTED
    assert lib.sp_superpose_prefill(256, 256, 256, ref, 4, 3, 64, 1.0, 0, 256, None, None, 0, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_superpose_prefill(256, 256, 256, None, 4, 4, 64, 1.0, 0, 256, None, None, 0, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_superpose_prefill(256, 256, 256, ref, 4, 4, 64, 1.0, 0, 256, None, None, 0, 0, None) == sp.SP_ERR_WORKSPACE
    assert lib.sp_superpose_prefill(264, 256, 256, ref, 4, 4, 64, 1.0, 0, 256, None, 256, 1 << 20, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_superpose_prefill(256, 256, 256, ref, 4, 4, 64, 1.0, 5, 256, None, 256, 1 << 20, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_pruned_decode(256, 256, 256, ref, 256, 1, None, None, None, 0, 0, 4, 4, 64, 1.0, 256, None,
                                None, 0, 0, None) == sp.SP_ERR_WORKSPACE
    assert lib.sp_pruned_decode(256, 256, 256, ref, None, 1, None, None, None, 0, 0, 4, 4, 64, 1.0, 256, None,
                                256, 1 << 20, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_pruned_decode(256, 256, 256, ref, 256, 1, None, None, None, 4, 0, 4, 4, 64, 1.0, 256, None,
                                256, 1 << 20, 0, None) == sp.SP_ERR_INVALID_ARG   # tail_cap > 0, NULL tail
    bad = sp.binding._CLayout(-1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0)
    assert lib.sp_pruned_decode(256, 256, 256, ctypes.byref(bad), 256, 1, None, None, None, 0, 0, 4, 4, 64, 1.0,
                                256, None, 256, 1 << 20, 0, None) == sp.SP_ERR_INVALID_ARG
    assert lib.sp_check_status(None, None) == sp.SP_ERR_INVALID_ARG


def test_workspace_sizes_are_sane():
    lib = sp.lib
    assert lib.sp_path_scores_workspace_bytes(1000) >= 256 + 4000
    assert lib.sp_decode_workspace_bytes(1, 32, 128) % 256 == 0
    assert lib.sp_decode_workspace_bytes(64, 32, 128) >= 256
    assert lib.sp_prefill_workspace_bytes(1, 20, 32, 184, 32, 128, sp.SP_BF16) >= 256


def test_next_round_layout_moves_kept_documents_into_the_prefix():
    import numpy as np
    from workloads import build_layout, next_round_layout
    lay = build_layout([3, 0], [[10, 20, 30], [5, 6]], [[4, 4, 4], [2, 2]])
    nxt = next_round_layout(lay, np.array([[2, 0], [4, -1]]))
    assert list(nxt.pre_len) == [3 + 30 + 10, 6]
    assert list(nxt.doc_len) == [20, 5] and list(nxt.qry_len) == [4, 2]
    assert list(nxt.prompt_path_off) == [0, 1, 2]
    assert nxt.total_tokens == 43 + 24 + 6 + 7


def test_kernels_read_coherently():
    """Every kernel may start while the one before it still writes (programmatic dependent launch), so none may read through the
    non-coherent path or promise the compiler that its pointers do not alias: such loads are not ordered by the wait."""
    src = os.path.join(os.path.dirname(sp.LIB_PATH), "csrc")
    for name in sorted(os.listdir(src)):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(src, name)).read(), flags=re.S)
        found = re.findall(r"__ldg|__restrict__|ld\.global\.nc|__ldcs", text)
        assert not found, (name, found)


def test_tensor_memory_is_taken_between_the_wait_and_the_trigger():
    """A block that holds tensor memory while it waits for the kernel in front of it, or lets the next kernel's blocks in before
    it has its own, can deadlock with a neighbour on the SM (nothing to run: this is the order of the statements).  Where shared
    memory leaves no room for a neighbour the order is free."""
    body = open(os.path.join(os.path.dirname(sp.LIB_PATH), "csrc", "prefill_tc.cu")).read()
    assert "ALONE = SMEM + 3 * 1024 > 228 * 1024;" in body
    body = body[body.index(") prefill_tc_kernel("):]
    assert body.index("tmem_alloc(") < body.index("pdl_trigger();") < body.index("pdl_wait(); take_tmem();")
    assert "if (C::ALONE) { take_tmem(); pdl_wait(); } else { pdl_wait(); take_tmem(); }" in body
    assert body.count("tmem_alloc(") == body.count("pdl_trigger();") - 1 == 1          # the rotation of Q has the other trigger


@pytest.mark.parametrize("old,new", [("", ""), ("int k, const void *tail_k", "const int32_t *k, const void *tail_k"),
                                     ("int n_prompts, int k,\n                  int32_t *kept_idx", "int n_prompts, int32_t *kept_idx"),
                                     ("float *lse, int dtype", "float *lse, int more, int dtype"),
                                     ("int64_t ld_token, int n_heads", "const void *ld_token, int n_heads")])
def test_marshalling_is_compiled_against_the_header(old, new, tmp_path):
    """A parameter that sp.h declares otherwise than the marshalling passes it does not compile."""
    import importlib.util
    import shutil
    import subprocess
    pkg = os.path.dirname(sp.LIB_PATH)
    spec = importlib.util.spec_from_file_location("sp_build", os.path.join(pkg, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    (tmp_path / "include").mkdir()
    (tmp_path / "pkg" / "csrc").mkdir(parents=True)
    text = re.sub(r",\s*", ", ", open(os.path.join(ROOT, "include", "sp.h")).read())
    old, new = (re.sub(r",\s*", ", ", x) for x in (old, new))
    assert old in text
    (tmp_path / "include" / "sp.h").write_text(text.replace(old, new) if old else text)
    shutil.copy(os.path.join(pkg, "csrc", "marshal.c"), tmp_path / "pkg" / "csrc")
    rc = subprocess.run(["gcc", *build.MARSHAL_FLAGS, "-fsyntax-only", str(tmp_path / "pkg" / "csrc" / "marshal.c")], capture_output=True).returncode
    assert (rc == 0) == (old == "")
