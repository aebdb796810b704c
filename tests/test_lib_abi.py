"""The C-ABI library loads on a machine without a GPU and exports every declared symbol; host-side
argument validation rejects bad calls before anything is launched."""
import ctypes
import os
import re

import pytest

from paper_2508_16201_b200 import specvlm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    src = open(os.path.join(ROOT, "include", "specvlm.h")).read()
    return sorted(set(re.findall(r"\b(specvlm_[a-z0-9_]+)\s*\(", src)))


def test_library_exports_every_declared_symbol():
    if not os.path.exists(specvlm.LIB_PATH):
        from paper_2508_16201_b200 import build
        build.build()
    L = specvlm.lib()
    names = _declared()
    assert len(names) >= 11
    for n in names:
        assert hasattr(L, n), n
    assert set(names) == set(specvlm.EXPORTS)
    assert "sm_100a" in specvlm.version()
    assert specvlm.status_string(0) == "ok"
    assert specvlm.status_string(-3) == "workspace too small"


def test_host_validation_without_gpu():
    L = specvlm.lib()
    kv = specvlm.KvStruct()
    # null cache pointers
    rc = L.specvlm_draft_decode_attn(ctypes.byref(kv), None, 1, 4, 0.1, None, None, None, 0, None, None)
    assert rc == specvlm.ERR_INVALID_ARG
    # unsupported head_dim
    kv.k = kv.v = 0x1000
    kv.seq_lens = 0x1000
    kv.n_layers = kv.n_kv_heads = kv.n_blocks = 1
    kv.block_tokens = kv.max_seq_len = 128
    kv.head_dim = 96
    kv.stride_token = 96
    kv.stride_head = kv.stride_block = kv.stride_layer = 96 * 128
    rc = L.specvlm_draft_decode_attn(ctypes.byref(kv), 0x1000, 1, 4, 0.1, 0x1000, None, None, 0, None, None)
    assert rc == specvlm.ERR_UNSUPPORTED_SHAPE
    # bad stride alignment
    kv.head_dim = 64
    kv.stride_token = 68
    rc = L.specvlm_draft_decode_attn(ctypes.byref(kv), 0x1000, 1, 4, 0.1, 0x1000, None, None, 0, None, None)
    assert rc == specvlm.ERR_INVALID_ARG
    # gamma out of range
    kv.stride_token = 64
    kv.stride_head = kv.stride_block = kv.stride_layer = 64 * 128
    rc = L.specvlm_verify_attn(ctypes.byref(kv), 0x1000, 1, 4, 9, 0.1, 0x1000, None, None, 0, None, None)
    assert rc == specvlm.ERR_UNSUPPORTED_SHAPE
    # select: k_stage1 > k_total
    i32 = lambda *a: (ctypes.c_int32 * len(a))(*a)
    rc = L.specvlm_select(0x1000, i32(0, 100), i32(1), 100, i32(20), i32(10), i32(0, 10), 1, 0x1000, None, None)
    assert rc == specvlm.ERR_INVALID_ARG
    # select: too many tokens for one CTA
    rc = L.specvlm_select(0x1000, i32(0, 80000), i32(800), 100, i32(10), i32(20), i32(0, 20), 1, 0x1000, None, None)
    assert rc == specvlm.ERR_UNSUPPORTED_SHAPE
    # accept: workspace too small
    rc = L.specvlm_accept(0x1000, 0x1000, 1, 4, 1024, 0x1000, 0x1000, None, 0x1000, 8, None)
    assert rc == specvlm.ERR_WORKSPACE_TOO_SMALL
    assert L.specvlm_accept_workspace_bytes(1, 4, 1024) >= 5 * 8
    # rating a range of layers: a range outside the cache's layers is refused before anything runs
    kv.head_dim = 128
    kv.stride_token = 128
    kv.stride_head = kv.stride_block = kv.stride_layer = 128 * 128
    kv.n_layers = 4
    common = (ctypes.byref(kv), 0x1000, i32(0, 8), i32(64), i32(0), i32(64), i32(0, 64), 1, 4, 0.1, None, 0x1000,
              0x1000, 1 << 30)
    assert L.specvlm_stage1_scores_layers(*common, 3, 5, 0, None, None) == specvlm.ERR_INVALID_ARG
    assert L.specvlm_stage1_scores_layers(*common, 2, 1, 0, None, None) == specvlm.ERR_INVALID_ARG
    # tree verification: more nodes than the ancestor masks hold
    rc = L.specvlm_verify_tree_attn(ctypes.byref(kv), 0x1000, 0x1000, 1, 4, 65, 0.1, 0x1000, None, 0x1000, 1 << 30,
                                    None, None)
    assert rc == specvlm.ERR_UNSUPPORTED_SHAPE


def _cache_of(layers, kv_heads, head_dim, max_seq_len):
    kv = specvlm.KvStruct()
    kv.n_layers, kv.n_kv_heads, kv.head_dim, kv.max_seq_len, kv.block_tokens = layers, kv_heads, head_dim, max_seq_len, 64
    return kv


@pytest.mark.parametrize("layers,group,n_q", [(1, 8, 3), (1, 8, 6), (2, 8, 9), (1, 8, 16), (1, 8, 26), (3, 16, 60), (80, 8, 6)])
def test_a_workspace_for_the_largest_verification_serves_every_smaller_one(layers, group, n_q):
    """The size query never falls as the batch or the sequences grow (chain up to nine tokens, tree beyond)."""
    def size(batch, tokens):
        kv = ctypes.byref(_cache_of(layers, 8, 128, tokens))
        if n_q <= 9:
            return specvlm.lib().specvlm_attn_workspace_bytes(kv, batch, 8 * group, n_q - 1)
        return specvlm.lib().specvlm_verify_tree_workspace_bytes(kv, batch, 8 * group, n_q)

    lengths = [1, 64, 65, 128, 129, 256, 257, 384, 385, 640, 1000, 2048, 2049, 6400, 50000]
    sizes = [[size(batch, tokens) for tokens in lengths] for batch in range(1, 41)]
    for batch, row in enumerate(sizes):
        assert row[0] > 0 and row == sorted(row), (batch, row)
        if batch:
            assert all(a <= b for a, b in zip(sizes[batch - 1], row)), (batch, sizes[batch - 1], row)


@pytest.mark.parametrize("layers,kv_heads,head_dim", [(1, 4, 128), (1, 1, 64), (2, 4, 64), (8, 4, 128), (16, 4, 128), (28, 4, 128)])
@pytest.mark.parametrize("batch", [1, 3, 16])
def test_a_decode_workspace_for_the_longest_sequences_serves_shorter_ones(layers, kv_heads, head_dim, batch):
    """As the lengths grow a cluster of CTAs per item and slices take turns, and the slices' scratch comes and goes; the size
    query never falls."""
    table = (ctypes.c_int32 * 1)()
    for paged in (False, True):
        last = 256
        for tokens in sorted({*range(64, 4096, 64), *range(4096, 60000, 256), *range(8704, 9344, 64)}):
            kv = _cache_of(layers, kv_heads, head_dim, tokens)
            kv.block_table = ctypes.addressof(table) if paged else None
            size = specvlm.lib().specvlm_attn_workspace_bytes(ctypes.byref(kv), batch, 7 * kv_heads, 0)
            assert size >= last, (paged, tokens, last, size)
            last = size


def test_decode_asks_for_scratch_only_where_slices_beat_a_cta_per_item():
    """64 items of 2560 tokens (d = 128): no slices, and a call without a workspace is accepted."""
    kv = _cache_of(16, 4, 128, 2560)
    assert specvlm.lib().specvlm_attn_workspace_bytes(ctypes.byref(kv), 1, 28, 0) == 256


def test_missing_library_raises_and_package_is_oracle_free(monkeypatch, tmp_path):
    """No fallback: with the library file absent every call through the binding raises; and the
    package's sources neither import nor include anything of the oracle."""
    monkeypatch.setattr(specvlm, "_lib", None)
    monkeypatch.setattr(specvlm, "LIB_PATH", str(tmp_path / "libspecvlm.so"))
    with pytest.raises(RuntimeError, match="missing"):
        specvlm.lib()
    with pytest.raises(RuntimeError, match="missing"):
        specvlm.accept_workspace_bytes(1, 4, 1024)
    pkg = os.path.dirname(specvlm.__file__)
    for root, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h", ".cpp")):
                with open(os.path.join(root, f)) as fh:
                    src = fh.read()
                assert not re.search(r"^\s*(import|from)\s+oracle|#include[^\n]*oracle|oracle[./]", src, re.M), f


def test_rating_kernels_compile_without_heavy_spills():
    """The rating kernels run under tight register caps (two CTAs of 320 threads, or 576 threads, per
    SM) and which exponentials take the polynomial decides whether ptxas fits the loop in them: a
    choice that spills a few hundred bytes runs two to four times slower.  The build keeps ptxas's
    report; this reads the spill figures of the two kernels from it."""
    from paper_2508_16201_b200 import build
    build.build()
    log = os.path.join(ROOT, "paper_2508_16201_b200", "_build", "scores.ptxas.log")
    if not os.path.exists(log):
        pytest.skip("no ptxas report (the objects were not compiled by this checkout)")
    text = open(log).read()
    seen = 0
    for m in re.finditer(r"Function properties for (\S*scores_(?:lse|colsum)_tc_kernel\S*)\s*\n\s*(\d+) bytes stack frame, "
                         r"(\d+) bytes spill stores, (\d+) bytes spill loads", text):
        seen += 1
        assert int(m.group(3)) <= 64 and int(m.group(4)) <= 64, m.group(0)
    assert seen >= 4


def test_kernels_with_tensor_memory_release_their_successor_after_the_allocation():
    """A kernel may let its successor start only once each of its CTAs has its tensor memory: a successor's CTA that
    took the columns first and then waited for that kernel would leave both waiting.  In the sources: every allocation
    is the helper that releases after it, and no kernel that calls it releases anywhere else."""
    csrc = os.path.join(ROOT, "paper_2508_16201_b200", "csrc")
    seen = 0
    for f in sorted(os.listdir(csrc)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, f)).read())
        if f == "common.cuh":
            body = src[src.index("void tmem_alloc_launch_next("):]
            assert body.index("tmem_alloc(smem_dst") < body.index("pdl_launch_next();") < body.index("}")
            continue
        assert not re.search(r"\btmem_alloc\(|tcgen05\.alloc|griddepcontrol\.launch_dependents", src), f
        for kernel in src.split("__global__")[1:]:
            if "tmem_alloc_launch_next(" in kernel:
                seen += 1
                # up to the kernel's end: the first line that is a closing brace alone
                assert "pdl_launch_next()" not in kernel[:kernel.index("\n}\n")], (f, kernel[:80])
    assert seen == 4


def test_a_tree_without_the_module_counts_as_not_built(monkeypatch, tmp_path):
    """The module carries the interpreter's suffix, so that another one does not load it; a tree that has the library
    alone is built before the tests run."""
    import sysconfig
    from paper_2508_16201_b200 import _binding, build
    assert build.BINDING == _binding.__file__ and build.BINDING.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert build.is_built()
    for name in ("LIB", "BINDING"):
        with monkeypatch.context() as m:
            m.setattr(build, name, str(tmp_path / "not built"))
            assert not build.is_built()


def test_binding_takes_what_ctypes_took():
    """The CPython module: device pointers as tensors or None, host arrays as any sequence, integers modulo
    2^32; a wrong number or type of arguments is refused.  Every call here is one that the library rejects on the host."""
    import numpy as np
    import torch
    from paper_2508_16201_b200 import _binding
    bad = specvlm.ERR_INVALID_ARG
    _binding.init(lambda: 0, lambda device: 0)
    try:
        kv = specvlm.KvStruct()
        assert _binding.draft_decode_attn(ctypes.addressof(kv), None, 1, 4, 0.1, None, None, None, 0, None) == bad
        t = torch.zeros(16)
        for one, cu in (([5], [0, 10]), ((5,), (0, 10)), (np.array([5]), torch.tensor([0, 10])), ([5.0], ["0", 10])):
            # k_stage1 = 5 > k_total = 3
            assert _binding.select(t, cu, [2], 5, one, [3], [0, 3], 1, t, None) == bad
        many = list(range(1, 200))                             # longer than the array on the stack
        assert _binding.select(t, [0] + many, many, 1, [5] * 199, [3] * 199, [0] + many, 199, t, None) == bad
        assert _binding.rollback_kv(t, t, 1, -1, None) == bad   # gamma < 0
        assert _binding.rollback_kv(t, t, 1, (1 << 32) - 1, None) == bad
        for minus_one in (np.int64(-1), np.int8(-1), torch.tensor(-1)):     # whatever has __index__
            assert _binding.rollback_kv(t, t, 1, minus_one, None) == bad
        class Empties:
            """An element whose conversion empties the list that it is in."""
            def __int__(self):
                outer.clear()
                return 5
        for n in (1, 60, 199):                                 # on the stack and beyond it
            outer = [Empties()] + [3] * (n - 1)
            assert _binding.select(t, [0, 10], [2], 5, outer, [3], [0, 3], 1, t, None) == bad and outer == []
        for call, args in ((_binding.rollback_kv, (t, t, 1)), (_binding.rollback_kv, (t, t, 1.5, 0, None)),
                           (_binding.select, (t, 7, [2], 5, [5], [3], [0, 3], 1, t, None)),
                           (_binding.select, (t, None, [2], 5, [5], [3], [0, 3], 1, t, None))):
            with pytest.raises(TypeError):
                call(*args)
        for no_tensor in ("no tensor", 0x1000, True, 0):         # a number is not taken for an address either
            with pytest.raises(AttributeError):
                _binding.rollback_kv(no_tensor, t, 1, -1, None)
            with pytest.raises(AttributeError):
                _binding.rollback_kv(t, t, 1, -1, no_tensor)
        with pytest.raises(TypeError):
            _binding.draft_decode_attn(t, None, 1, 4, 0.1, None, None, None, 0, None)   # a cache is its descriptor's address
    finally:
        _binding.init(torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream)
