"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, answers its host-only calls, and rejects bad arguments before any launch."""
import ctypes
import os
import re
import subprocess
import sys

import pytest

from paper_1911_02150_b200 import binding
from paper_1911_02150_b200.build import build_library

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    build_library()
    return binding.lib()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "mqa_decode.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"^\s*#.*$", "", text, flags=re.M)          # preprocessor lines
    return sorted(set(re.findall(r"\b(\w+)\s*\([^;{}]*\)\s*;", text)))


def test_header_and_binding_agree(L):
    names = declared_functions()
    assert "mqa_decode_step" in names and "mha_decode_step" in names and "kv_cache_append" in names
    assert sorted(binding.EXPORTS) == names
    for n in names:
        assert hasattr(L, n), f"{n} is declared in include/mqa_decode.h but not exported"


def test_header_constants_and_binding_agree():
    text = open(os.path.join(ROOT, "include", "mqa_decode.h")).read()
    defines = {m.group(1): int(m.group(2), 0) for m in re.finditer(r"^#define\s+(MQA_\w+)\s+\(?(\d+|0x[0-9a-fA-F]+)u?\)?\s*$", text, flags=re.M)}
    assert defines["MQA_STEP_ADVANCE"] == binding.STEP_ADVANCE == 1
    assert defines["MQA_STEP_CHAINED"] == binding.STEP_CHAINED == 2
    assert defines["MQA_STEP_TEST_WRONG_GUESS"] == binding.STEP_TEST_WRONG_GUESS == 4
    assert binding._step_flags(True, False) == 1 and binding._step_flags(False, True) == 2
    assert binding._step_flags(True, "wrong-guess") == 7
    assert defines["MQA_STEP_TEST_WITHHOLD_COPY"] == binding.STEP_TEST_WITHHOLD_COPY == 8
    assert binding._step_flags(False, False, True) == 8


def test_step_flags_are_checked_before_any_launch(L):
    vp = ctypes.c_void_p
    a = vp(0x1000)
    # an unknown flag bit: refused on the host, nothing dereferenced
    rc = L.mqa_decode_append_step(a, a, a, a, a, a, 16, a, a, 1 << 30, None, 4, 8, 256, 128, 128, None)
    assert rc == binding.ERR_INVALID_ARG


def test_layer_cut(L):
    for b, h, d in ((1, 1, 128), (128, 8, 1024), (256, 128, 2048), (65, 32, 256)):
        for columns, ctas in binding.layer_cut(b, h, d):
            assert columns in (16, 32, 64, 128) and ctas in (1, 2, 4, 8)
    for bad in ((0, 8, 128), (1, 0, 128), (1, 8, 0), (1, 8, 100)):
        with pytest.raises(binding.MqaError):
            binding.layer_cut(*bad)


def test_status_strings(L):
    seen = {binding.status_string(c) for c in range(0, 5)}
    assert len(seen) == 5
    assert "unknown" in binding.status_string(99)


def test_plan_and_workspace_are_consistent(L):
    for mq in (True, False):
        for (b, h, m) in [(1, 8, 128), (128, 8, 128), (32, 32, 8192), (256, 16, 2048), (1, 16, 32768), (256, 16, 32768)]:
            n, chunk = binding.plan_splits(mq, b, h, m)
            assert n >= 1 and chunk >= 1
            need = binding.workspace_bytes(b, h, m)
            if n > 1:
                assert need >= h * n * (128 + 2) * 4
    assert binding.workspace_bytes(0, 8, 128) == 0
    assert binding.workspace_bytes(1, 8, 128, k=64, v=64) == 0
    assert binding.plan_splits(True, 1, 8, 0) == (0, 0)


def test_sizes_that_take_no_workspace(L):
    """Short caches, and many sequences of a few hundred rows, are whole splits and take no scratch, on either variant."""
    for (b, h, m) in [(1, 8, 200), (30, 32, 255), (100, 17, 129), (384, 8, 256), (600, 4, 300)]:
        assert binding.plan_splits(True, b, h, m)[0] == 1
    for (b, h, m) in [(1, 1, 511), (3, 8, 300), (20, 4, 500)]:
        assert binding.plan_splits(False, b, h, m)[0] == 1


@pytest.mark.parametrize("h,m_max,b", [(32, 1024, 128), (4, 300, 64), (16, 2048, 300), (8, 200, 5000), (40, 900, 160), (24, 33000, 50)])
def test_a_workspace_for_every_batch_up_to_the_largest(L, h, m_max, b):
    """The need does not grow evenly with the batch (32 heads x 1024 rows: 49 sequences need some, 128 none)."""
    each = [binding.workspace_bytes(i, h, m_max) for i in range(1, b + 1)]
    assert L.mqa_workspace_bytes_up_to(b, h, m_max, 128, 128) == max(each)
    assert L.mqa_workspace_bytes_up_to(0, h, m_max, 128, 128) == L.mqa_workspace_bytes_up_to(b, h, m_max, 64, 128) == 0
    for d in (128, 1024):        # the layer step's: all but the attention step's part grows with the batch
        largest = binding.layer_workspace_bytes(b, h, d, m_max) + max(each)
        assert all(binding.layer_workspace_bytes(i, h, d, m_max) <= largest for i in range(1, b + 1))


def test_sizes_whose_clusters_do_not_fit_keep_the_second_pass(L):
    """Where the device has no room for a cluster (a part of a card), the splits of a sequence are merged by a second launch."""
    sizes = [(1, 16, 512), (4, 16, 1000), (1, 32, 600), (8, 16, 4096), (30, 8, 900)]
    try:
        assert [binding.append_step_launches(*s) for s in sizes] == [1] * 5
        binding.set_test_cluster_room(0)
        assert [binding.append_step_launches(*s) for s in sizes] == [2] * 5
        binding.set_test_cluster_room(4)
        assert [binding.append_step_launches(*s) for s in sizes[:3]] == [1] * 3 and binding.append_step_launches(30, 8, 900) == 2
    finally:
        binding.set_test_cluster_room(-1)
    assert [binding.append_step_launches(*s) for s in sizes] == [1] * 5


def test_plans_of_the_longest_caches(L):
    """Host-only questions about caches of hundreds of millions of rows are answered, and at once (in a process of its own: one that
    overflows takes it down)."""
    # (a plan first: it asks the device, where there is one, for a millisecond or so.  Walking such a cache takes 11 to 80 ms a plan)
    code = ("import time; from paper_1911_02150_b200 import binding as m\n"
            "for h in (16, 32): m.workspace_bytes(1, h, 4096)\n"
            "t = time.perf_counter()\n"
            "for rows in (1 << 28, 1_073_741_825, 1_500_000_000, 2_000_000_000, 2_147_483_646):\n"
            "    for h in (1, 16, 32, 64): assert m.plan_splits(True, 1, h, rows)[0] > 1 and m.workspace_bytes(1, h, rows) > 0\n"
            "assert time.perf_counter() - t < 1e-2")
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT)


def test_bad_arguments_are_rejected_before_any_launch(L):
    vp = ctypes.c_void_p
    a = vp(0x1000)          # plausible, 16-byte aligned, never dereferenced on the host
    odd = vp(0x1004)
    step = L.mqa_decode_step
    ok_tail = (1, 8, 128, 128, 128, None)
    assert step(None, a, a, a, a, None, 0, None, *ok_tail) == binding.ERR_INVALID_ARG
    assert step(a, a, a, a, None, None, 0, None, *ok_tail) == binding.ERR_INVALID_ARG
    assert step(odd, a, a, a, a, None, 0, None, *ok_tail) == binding.ERR_INVALID_ARG
    assert step(a, a, odd, a, a, None, 0, None, *ok_tail) == binding.ERR_INVALID_ARG
    assert step(a, a, a, a, a, None, 0, None, 0, 8, 128, 128, 128, None) == binding.ERR_INVALID_ARG
    assert step(a, a, a, a, a, None, 0, None, 1, 8, -5, 128, 128, None) == binding.ERR_INVALID_ARG
    assert step(a, a, a, a, a, None, 0, None, 1, 8, 128, 64, 128, None) == binding.ERR_UNSUPPORTED
    assert L.mha_decode_step(a, a, a, a, a, None, 0, None, 1, 8, 128, 128, 96, None) == binding.ERR_UNSUPPORTED
    # a plan with several splits needs a workspace of the advertised size
    n, _ = binding.plan_splits(True, 1, 16, 32768)
    assert n > 1
    need = binding.workspace_bytes(1, 16, 32768)
    big = (1, 16, 32768, 128, 128, None)
    assert step(a, a, a, a, a, None, 0, None, *big) == binding.ERR_INVALID_ARG
    assert step(a, a, a, a, a, a, need - 1, None, *big) == binding.ERR_WORKSPACE_TOO_SMALL
    assert L.mqa_decode_step_combine(a, a, a, need - 1, 1, 16, 32768, 128, 128, None) == binding.ERR_WORKSPACE_TOO_SMALL
    app = L.kv_cache_append
    assert app(None, a, a, a, a, 1, None, 1, 1, 128, 128, 128, None) == binding.ERR_INVALID_ARG
    assert app(a, a, a, odd, a, 1, None, 1, 1, 128, 128, 128, None) == binding.ERR_INVALID_ARG
    assert app(a, a, a, a, a, 1, None, 1, 0, 128, 128, 128, None) == binding.ERR_INVALID_ARG
    assert app(a, a, a, a, a, 1, None, 1, 1, 128, 32, 128, None) == binding.ERR_UNSUPPORTED


def test_binding_type_checks():
    import torch
    q = torch.zeros(1, 8, 128, dtype=torch.bfloat16)
    with pytest.raises(TypeError):
        binding.mqa_decode_step(q, q, q, torch.zeros(1, dtype=torch.int32), torch.zeros(1, 8, 128))


def test_the_native_half_belongs_to_one_torch(L, monkeypatch):
    """Under a torch that it was not built for it is not loaded, the wrappers go by their own checks, and the build is out of date."""
    import torch
    from paper_1911_02150_b200 import build
    assert os.path.exists(binding.checked_call_path()) and not build._stale()
    monkeypatch.setattr(torch, "__version__", "0.0+other")
    monkeypatch.setattr(binding, "_native", None)
    assert build._stale()
    q = torch.zeros(1, 8, 128, dtype=torch.bfloat16)
    with pytest.warns(UserWarning), pytest.raises(TypeError):
        binding.mqa_decode_step(q, q, q, torch.zeros(1, dtype=torch.int32), torch.zeros(1, 8, 128))
    for name in ("kv_cache_append", "mqa_decode_step", "mha_decode_step", "mqa_prefill_attention"):
        assert getattr(binding._native, name)(q, q, None) is None


def test_which_kernel_takes_the_batched_form(L):
    """Calls of few tiles go one tile to a CTA or to a cluster of them, as far as those fit; many, or ones that a CTA has done before it
    would be shared out, stay with two tiles to a CTA."""
    kernel = binding.prefill_plan_kernel
    assert kernel(32, 32, 4096, 4096, False) == kernel(20, 1, 380, 380, False) == kernel(5, 16, 471, 471, False) == ("mqa_prefill_kernel", 1)
    assert kernel(5, 9, 333, 3000, True) == kernel(2, 1, 132, 132, False) == ("mqa_prefill_tile_kernel", 1)
    assert kernel(14, 1, 88, 1707, True) == ("mqa_prefill_tile_kernel", 8) and kernel(15, 1, 88, 1707, True)[1] == 4
    assert kernel(2, 8, 512, 256, False) == ("", 0)


def test_plans_of_many_query_rows_and_of_the_batched_form(L):
    """More than 32 query rows per sequence are planned on the kernel with the query rows as tile rows, and the batched
    form's workspace and refusals are answered on the host (the plan assumes the 148 SMs of a B200 without a GPU)."""
    assert binding.plan_kernel_name(True, False, 32, 128, 8192) == "mqa_decode_wide_kernel"       # 65 .. 128 rows: rows as tile rows
    assert binding.plan_kernel_name(True, False, 32, 192, 8192) == "mqa_decode_wide_kernel"       # beyond: tiles of 128 rows
    assert binding.plan_kernel_name(True, True, 32, 32, 8192) == "mqa_decode_stream_umma_kernel<32, fused, guess>"
    assert binding.plan_kernel_name(False, False, 32, 32, 8192) == "decode_split_simt_kernel"
    assert binding.plan_kernel_name(True, False, 0, 32, 8192) == ""
    assert binding.append_step_launches(32, 128, 8192) == 2
    assert binding.append_step_launches(256, 128, 8192) == 1
    assert binding.append_step_launches(32, 192, 8192) == 2
    assert binding.workspace_bytes(32, 128, 8192) >= binding.workspace_bytes(32, 64, 8192)
    need = binding.prefill_workspace_bytes(2, 8, 128, 256)
    assert need > 0
    assert binding.prefill_workspace_bytes(2, 8, 100, 256) > 0           # any number of positions
    assert binding.prefill_workspace_bytes(2, 8, 512, 256) == 0          # the queries' positions must fit the memory
    assert binding.prefill_workspace_bytes(2, 8, 128, 256, k=64) == 0
    a = ctypes.c_void_p(0x1000)
    pf = L.mqa_prefill_attention
    assert pf(a, a, a, None, a, a, need, None, 2, 8, 512, 256, 128, 128, None) == binding.ERR_UNSUPPORTED
    assert pf(a, a, a, None, a, a, need - 1, None, 2, 8, 128, 256, 128, 128, None) == binding.ERR_WORKSPACE_TOO_SMALL
    assert pf(None, a, a, None, a, a, need, None, 2, 8, 128, 256, 128, 128, None) == binding.ERR_INVALID_ARG
    assert pf(a, a, a, ctypes.c_void_p(0x1002), a, a, need, None, 2, 8, 128, 256, 128, 128, None) == binding.ERR_INVALID_ARG
