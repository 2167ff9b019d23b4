"""A bounded wait that runs out.  No kernel of the library waits without a limit: when a copy it waits for does not
arrive, the kernel flags MQA_STATUS_PIPELINE_TIMEOUT, lets its other copies land, frees its tensor memory and
returns by itself.  Here the limit is shortened to about a millisecond and a testing flag keeps one copy of the
first CTA from ever being started; afterwards the limit is restored and an ordinary call on the same workspace and
the same GPU must be correct again (nothing was left behind: no held tensor memory, no stale bookkeeping)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1911_02150_b200 as mqa
from paper_1911_02150_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ABS_TOL, REL_TOL = 4e-3, 1e-2
SHORT_LIMIT = 2_000_000          # SM clock cycles: about a millisecond


def check_close(got, ref, what):
    assert np.all(np.isfinite(got)), f"{what}: non-finite output"
    err = np.abs(got.astype(np.float64) - ref)
    assert err.max() <= ABS_TOL, f"{what}: max abs err {err.max():.3e}"
    assert np.all(err.max(-1) <= REL_TOL * np.abs(ref).max(-1)), f"{what}: row-relative error"


@pytest.mark.parametrize("b,h,m_max,chained,kernel,launches", [
    (40, 32, 2048, False, "stream_umma_kernel<32", 1),      # persistent kernel, pieces merged through global memory
    (100, 16, 3000, False, "stream_umma_kernel<16", 1), (100, 16, 3000, True, "stream_umma_kernel<16", 1),
    (32, 32, 2048, True, "stream_umma_kernel<32", 1),       # persistent kernel launched as clusters, copies started on a guess
    (64, 16, 4096, True, "stream_umma_kernel<16", 1),
    (40, 16, 2048, False, "split_mma_kernel<1>", 1),        # fixed splits, a cluster to a sequence
    (6, 8, 300, False, "split_mma_kernel<1>", 1),
    (200, 8, 200, False, "split_mma_kernel<1>", 1),         # ... and one CTA to a sequence
    (20, 96, 2048, False, "wide_kernel", 2),                # many query rows: the kernel with the query rows as tile rows, pieces and a second pass
    (160, 40, 700, False, "wide_kernel", 1),                # the same kernel, one split per sequence
    (20, 96, 2048, True, "wide_kernel", 2), (160, 40, 700, True, "wide_kernel", 1),                     # ... with a stage fetched ahead of the wait
    # fixed splits, one and several, with tiles ahead of the wait and without
    (6, 8, 300, True, "split_mma_kernel<1>", 1), (8, 24, 1000, True, "split_mma_kernel<2>", 1), (8, 24, 1000, False, "split_mma_kernel<2>", 1),
    (200, 8, 200, True, "split_mma_kernel<1>", 1), (4, 9, 7909, True, "split_mma_kernel<1>", 2),
])
def test_a_wait_that_runs_out_is_reported_and_leaves_nothing_behind(b, h, m_max, chained, kernel, launches):
    assert kernel in mqa.plan_kernel_name(True, chained, b, h, m_max) and mqa.append_step_launches(b, h, m_max) == launches
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=77, device=DEV)
    lens0 = np.full(b, m_max - 1, np.int32)
    lens0[1::3] = np.random.default_rng(7).integers(m_max // 2, m_max - 1, size=len(lens0[1::3]))
    wl.poison_tail(inp["K"], lens0); wl.poison_tail(inp["V"], lens0)
    Kh, Vh, lens_h = wl.bits(inp["K"]), wl.bits(inp["V"]), lens0.copy()
    oracle.kv_cache_append(Kh, Vh, wl.bits(inp["k_new"]), wl.bits(inp["v_new"]), lens_h, True)
    ref = oracle.mqa_decode_step(wl.bits(inp["q"]), Kh, Vh, lens_h)
    lens = torch.from_numpy(lens0).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    o = torch.zeros(b, h, 128, dtype=torch.float32, device=DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    try:
        mqa.set_wait_limit_cycles(SHORT_LIMIT)
        mqa.mqa_decode_append_step(inp["q"], inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens, o, ws, status,
                                   advance=False, chained=chained, withhold_copy=True)
        torch.cuda.synchronize()                     # the kernel came back by itself
    finally:
        mqa.set_wait_limit_cycles(0)
    assert int(status.item()) & binding.STATUS_PIPELINE_TIMEOUT
    assert np.array_equal(lens.cpu().numpy(), lens0)
    # the same step again, as it should be: same workspace, nothing cleared
    for rnd in range(2):
        status.zero_()
        o.fill_(float("nan"))
        lens.copy_(torch.from_numpy(lens0))
        mqa.mqa_decode_append_step(inp["q"], inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens, o, ws, status,
                                   advance=True, chained=chained and rnd > 0)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert np.array_equal(lens.cpu().numpy(), lens_h)
        check_close(o.cpu().numpy(), ref, f"call {rnd} after the timed-out one")
    assert np.array_equal(wl.bits(inp["K"]), Kh) and np.array_equal(wl.bits(inp["V"]), Vh)


@pytest.mark.parametrize("b,h,m_max", [(6, 8, 300), (8, 24, 1000), (20, 96, 2048), (160, 40, 700)])
def test_copies_ahead_of_the_wait_behind_the_host_inputs_that_run_out(b, h, m_max):
    """The same flag through the host-buffer step, where the attention kernel fetches all that its stages hold before its wait."""
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=78, device=DEV)
    lens0 = np.full(b, m_max - 1, np.int32)
    Kh, Vh, lens_h = wl.bits(inp["K"]).copy(), wl.bits(inp["V"]).copy(), lens0.copy()
    oracle.kv_cache_append(Kh, Vh, wl.bits(inp["k_new"]), wl.bits(inp["v_new"]), lens_h, True)
    ref = oracle.mqa_decode_step(wl.bits(inp["q"]), Kh, Vh, lens_h)
    lens = torch.from_numpy(lens0).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    host = [inp[n].cpu().pin_memory() for n in ("q", "k_new", "v_new")]
    o = torch.zeros(b, h, 128, dtype=torch.float32).pin_memory()
    staging = torch.empty(mqa.host_staging_bytes(b, h), dtype=torch.uint8, device=DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    args = list(binding._host_step_args(*host, o, inp["K"], inp["V"], lens, staging, ws, status, False, None, False))
    flags = 7                                        # (the position of `advance` in mqa_decode_append_step_host)
    assert args[flags] == 0
    args[flags] = binding.STEP_TEST_WITHHOLD_COPY
    try:
        mqa.set_wait_limit_cycles(SHORT_LIMIT)
        assert binding.lib().mqa_decode_append_step_host(*args) == 0
        torch.cuda.synchronize()
    finally:
        mqa.set_wait_limit_cycles(0)
    assert int(status.item()) & binding.STATUS_PIPELINE_TIMEOUT
    status.zero_()
    o.fill_(float("nan"))
    mqa.mqa_decode_append_step_host(*host, o, inp["K"], inp["V"], lens, staging, ws, status, advance=True)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and np.array_equal(lens.cpu().numpy(), lens_h)
    check_close(o.numpy(), ref, "the call after the timed-out one")


@pytest.mark.parametrize("b,h,n,m_max,starts,kernel,ctas", [
    (3, 4, 512, 600, [88, 0, 31], "mqa_prefill_tile_kernel", 1),                 # one tile to a CTA
    (1, 4, 16, 2064, [2048], "mqa_prefill_tile_kernel", 8),                      # a cluster of CTAs per tile: the others go on to the merge
    (5, 9, 333, 3000, [2667, 0, 100, 1300, 700], "mqa_prefill_tile_kernel", 1),
    (20, 16, 128, 700, [(37 * i + 300) % 570 for i in range(20)], "mqa_prefill_kernel", 1),       # two tiles to a CTA, several units to each (the first has several stages)
])
def test_the_batched_form_reports_a_wait_that_runs_out_and_is_correct_again_afterwards(b, h, n, m_max, starts, kernel, ctas):
    assert mqa.prefill_plan_kernel(b, h, n, m_max, True) == (kernel, ctas)
    gen = torch.Generator(device=DEV).manual_seed(4)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array(starts, np.int32)
    start = torch.from_numpy(st).to(DEV)
    O = torch.zeros(b, h, n, 128, dtype=torch.float32, device=DEV)
    ws = torch.empty(max(16, mqa.prefill_workspace_bytes(b, h, n, m_max)), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    try:
        mqa.set_wait_limit_cycles(SHORT_LIMIT)
        mqa.set_test_withhold_copy(True)
        mqa.mqa_prefill_attention(Q, K, V, O, ws, start, status)
        torch.cuda.synchronize()                     # the kernel came back by itself
    finally:
        mqa.set_test_withhold_copy(False)
        mqa.set_wait_limit_cycles(0)
    assert int(status.item()) & binding.STATUS_PIPELINE_TIMEOUT
    status.zero_()
    O.fill_(float("nan"))
    mqa.mqa_prefill_attention(Q, K, V, O, ws, start, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle.mqa_batched_attention(wl.bits(Q), wl.bits(K), wl.bits(V), st)
    check_close(O.cpu().numpy(), ref, "the call after the timed-out one")


@pytest.mark.parametrize("b,h,window", [(320, 8, 100), (310, 20, 33), (150, 40, 32)])
def test_the_local_step_reports_a_wait_that_runs_out(b, h, window):
    """A warp per sequence, the copy of its second tile (or of its second pass over the only one) never complete."""
    inp = wl.make_inputs(b, h, window, "mqa", seed=5, device=DEV)
    pos0 = np.full(b, window + 3, np.int32)
    pos = torch.from_numpy(pos0).to(DEV)
    o = torch.zeros(b, h, 128, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    step = lambda: mqa.mqa_decode_local_step(inp["q"], inp["K"], inp["V"], inp["k_new"], inp["v_new"], pos, o, status)
    try:
        mqa.set_wait_limit_cycles(SHORT_LIMIT)
        mqa.set_test_withhold_copy(True)
        step()
        torch.cuda.synchronize()                     # the kernel came back by itself
    finally:
        mqa.set_test_withhold_copy(False)
        mqa.set_wait_limit_cycles(0)
    assert int(status.item()) == binding.STATUS_PIPELINE_TIMEOUT
    assert np.array_equal(pos.cpu().numpy(), pos0 + (np.arange(b) > 0))          # (the sequence that gave up stays where it was)
    status.zero_()
    pos.copy_(torch.from_numpy(pos0))
    step()
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check_close(o.cpu().numpy(), oracle.mqa_decode_step(wl.bits(inp["q"]), wl.bits(inp["K"]), wl.bits(inp["V"]), np.full(b, window, np.int32)), "the call after it")


@pytest.mark.parametrize("b,h,window", [(300, 8, 32), (5, 16, 20)])
def test_the_local_step_of_one_tile_reports_a_wait_that_runs_out(b, h, window):
    test_the_local_step_reports_a_wait_that_runs_out(b, h, window)


@pytest.mark.parametrize("b,h,d,m_max", [(17, 5, 640, 130), (128, 8, 1024, 64), (3, 1, 1024, 130)])
def test_the_projections_report_sums_that_do_not_come(b, h, d, m_max):
    gen = torch.Generator(device=DEV).manual_seed(b)
    x, P_q, P_k, P_v, P_o, K, V = (wl.bf16_normal(s, std, gen, DEV) for s, std in (
        ((b, d), 1.0), ((h, d, 128), (d * 128) ** -0.5), ((d, 128), d ** -0.5), ((d, 128), d ** -0.5), ((h, d, 128), (h * 128) ** -0.5),
        ((b, m_max, 128), 1.0), ((b, m_max, 128), 1.0)))
    lens = torch.full((b,), m_max // 2, dtype=torch.int32, device=DEV)
    ws, status = mqa.alloc_layer_workspace(b, h, d, m_max, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    results = []
    for withhold in (False, True, False):
        y = torch.full((b, d), float("nan"), dtype=torch.float32, device=DEV)
        status.zero_()
        try:
            if withhold:
                mqa.set_wait_limit_cycles(SHORT_LIMIT)
                mqa.set_test_withhold_copy(True)
            mqa.mqa_layer_decode_step(x, P_q, P_k, P_v, P_o, K, V, lens, y, ws, status, advance=False)
            torch.cuda.synchronize()                 # every kernel came back by itself
        finally:
            mqa.set_test_withhold_copy(False)
            mqa.set_wait_limit_cycles(0)
        assert int(status.item()) == (binding.STATUS_PIPELINE_TIMEOUT if withhold else 0)
        results.append(y)
    assert bool(torch.isfinite(results[0]).all()) and torch.equal(results[0], results[2])
