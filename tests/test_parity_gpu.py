"""GPU parity: the CUDA path, called through the C ABI, against the fp64 CPU oracle on the
same seeded bf16 inputs.

Tolerance (from the build's stated target, bf16 inputs with fp32 accumulation):
  * every element: |gpu - oracle| <= 4e-3;
  * every (sequence, head) row: max_c |gpu - oracle| <= 1e-2 * max_c |oracle|  (relative to the
    row's scale -- at long context the outputs are ~1e-2 and element-wise relative error is
    ill-posed near zero crossings).
The cache append is compared bit for bit.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_1911_02150_b200 as mqa
from guards import Guarded
from paper_1911_02150_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu

ABS_TOL = 4e-3
REL_TOL = 1e-2
DEV = "cuda:0"


def check_close(got: np.ndarray, ref: np.ndarray, what: str = ""):
    assert got.shape == ref.shape
    assert np.all(np.isfinite(got)), f"{what}: non-finite output"
    err = np.abs(got.astype(np.float64) - ref)
    assert err.max() <= ABS_TOL, f"{what}: max abs err {err.max():.3e}"
    row_err = err.max(axis=-1)
    row_ref = np.abs(ref).max(axis=-1)
    bad = row_err > REL_TOL * row_ref
    assert not bad.any(), f"{what}: {bad.sum()} rows over relative tolerance, worst {np.max(row_err / np.maximum(row_ref, 1e-300)):.3e}"


def oracle_step(variant, q, K, V, lens_np, idx=None):
    """Oracle on all sequences, or on the sampled ones in idx."""
    if idx is not None:
        sel = torch.as_tensor(idx, device=q.device)
        q, K, V, lens_np = q[sel], K[sel], V[sel], lens_np[idx]
    fn = oracle.mqa_decode_step if variant == "mqa" else oracle.mha_decode_step
    return fn(wl.bits(q), wl.bits(K), wl.bits(V), lens_np.astype(np.int32))


def check_against_oracle(variant, q, K, V, lens_np, o, what, idx=None, chunk_bytes=1 << 30):
    """Every sequence (or those in idx) against the oracle, read back a slice of sequences at a time so that the host
    never holds more than about chunk_bytes of one cache tensor (the largest caches here are tens of GiB)."""
    b = q.shape[0]
    seqs = list(range(b)) if idx is None else list(idx)
    per_seq = K[0].numel() * 2
    step = max(1, chunk_bytes // per_seq)
    for at in range(0, len(seqs), step):
        part = seqs[at:at + step]
        ref = oracle_step(variant, q, K, V, lens_np, part)
        check_close(o[torch.as_tensor(part, device=o.device)].cpu().numpy(), ref, f"{what} sequences {part[0]}..{part[-1]}")


def gpu_step(variant, q, K, V, lens_t, expect_status=0):
    """One step through the C ABI.  The output, the workspace, the queries and lens sit between guard regions (a
    pattern either side, checked after the kernels have run): a write beyond any of them fails the test even where
    it would not fault."""
    b, h, _ = q.shape
    og = Guarded((b, h, V.shape[-1]), torch.float32, q.device)
    og.t.fill_(float("nan"))
    wsg = Guarded((max(16, mqa.workspace_bytes(b, h, K.shape[-2])),), torch.uint8, q.device)
    wsg.t.fill_(0xFF)                                  # stale NaN bit patterns in the scratch
    qg = Guarded(tuple(q.shape), q.dtype, q.device, like=q)
    lg = Guarded(tuple(lens_t.shape), lens_t.dtype, q.device, like=lens_t)
    sg = Guarded((1,), torch.int32, q.device)
    sg.t.zero_()
    fn = mqa.mqa_decode_step if variant == "mqa" else mqa.mha_decode_step
    fn(qg.t, K, V, lg.t, og.t, wsg.t, sg.t)
    torch.cuda.synchronize()
    for g, name in ((og, "o"), (wsg, "workspace"), (qg, "q"), (lg, "lens"), (sg, "status")):
        g.check(f"{variant} b={b} h={h}: {name}")
    assert torch.equal(qg.t, q) and torch.equal(lg.t, lens_t)
    assert int(sg.t.item()) == expect_status
    return og.t


def run_case(variant, b, h, m_max, lens_np, seed=0, sample=None):
    inp = wl.make_inputs(b, h, m_max, variant, seed=seed, device=DEV)
    lens_np = np.asarray(lens_np, dtype=np.int32)
    wl.poison_tail(inp["K"], lens_np)
    wl.poison_tail(inp["V"], lens_np)
    lens_t = torch.from_numpy(lens_np).to(DEV)
    o = gpu_step(variant, inp["q"], inp["K"], inp["V"], lens_t)
    check_against_oracle(variant, inp["q"], inp["K"], inp["V"], lens_np, o, f"{variant} b={b} h={h} m_max={m_max}", sample)
    return inp, o


SMALL = [
    # b, h, m_max, lens
    (1, 1, 1, [1]),
    (1, 8, 128, [128]),                       # the single-step configuration
    (3, 8, 300, [300, 1, 77]),                # ragged, several tiles, odd tails
    (2, 16, 1000, [999, 513]),
    (2, 32, 700, [700, 65]),
    (4, 5, 257, [257, 256, 255, 2]),          # a head count outside {8, 16, 32}
    (2, 40, 600, [600, 31]),                  # more heads than two tensor-core tiles: general kernel
    (3, 17, 95, [95, 32, 33]),                # 17 heads: second head tile nearly empty
    (2, 12, 4096, [4096, 3000]),              # several splits
    (5, 16, 64, [64, 63, 33, 17, 16]),
    (1, 16, 20000, [19999]),                  # many splits of one sequence
]


@pytest.mark.parametrize("variant", ["mqa", "mha"])
@pytest.mark.parametrize("b,h,m_max,lens", SMALL)
def test_small_cases_match_oracle(variant, b, h, m_max, lens):
    run_case(variant, b, h, m_max, lens, seed=b * 1000 + h)


def _mixed_lens(b, m_max, seed):
    r = np.random.default_rng(seed)
    lens = r.integers(1, m_max + 1, size=b).astype(np.int32)
    lens[r.integers(0, b, size=max(1, b // 10))] = 0          # some empty sequences
    lens[r.integers(0, b, size=max(1, b // 10))] = m_max       # some full ones
    lens[0], lens[-1] = 0, m_max
    return lens


# Batches large enough for the persistent kernel (caches of 1024 rows or more, two 32-row tiles per SM or more),
# shaped so that one SM's share spans several sequences, starts and ends mid-sequence and meets empty sequences;
# and batches just outside it (short caches, too many sequences), which take the fixed-split kernels.
STREAM = [
    (200, 8, 1100, 21),     # ~50 tiles per SM over 1.4 sequences: every SM crosses a sequence
    (90, 16, 1800, 22),
    (40, 16, 1500, 22),     # (four fixed splits in a cluster)
    (150, 17, 1030, 23),    # 17..32 heads: two 16-head groups, the second nearly empty
    (1024, 4, 1024, 24),    # the most sequences the persistent kernel indexes
    (1100, 8, 64, 25),      # more than that: fixed-split kernel
    (37, 32, 4000, 26),
    (70, 32, 3000, 27),
    (60, 24, 1300, 27),     # (a CTA per sequence of the kernel with the query rows as tile rows)
    (40, 48, 1500, 28),     # 33..64 heads
    (33, 64, 2100, 29),
    (300, 17, 200, 30),     # short caches: fixed-split kernel
    (160, 32, 333, 31),
    (3, 16, 9000, 32),      # few long sequences: cut into many pieces, merged by the second-pass kernel
    (1, 8, 20000, 33),
    # 33 .. 128 query rows per sequence (many heads, or beams x heads over one shared memory): the query rows are the tile rows
    (32, 128, 2048, 34),    # 4 beams x 32 heads
    (40, 96, 1500, 35),
    (16, 65, 1100, 37),     # one warp of the tile holds a single row of the sequence
    (150, 33, 700, 40),     # more sequences than SMs: one split each, short caches (two roundings of the weights)
    (1, 127, 20000, 41),    # one sequence in many splits
    (7, 100, 127, 42),      # less than one stage
    # more than 128: row tiles of 128 on the same kernel
    (3, 200, 9000, 36),     # few long sequences, two tiles (the second of 72 rows)
    (80, 160, 600, 43),     # one split per sequence, two tiles
    (4, 385, 2100, 44),     # four tiles, the last of one row
    # batches that divide the grid are launched as clusters (16 and 8 CTAs here); with mixed lengths the clusters
    # change nothing and one CTA merges a sequence's many pieces
    (8, 16, 20000, 38),
    (16, 32, 5000, 39),
]


@pytest.mark.parametrize("b,h,m_max,seed", STREAM)
def test_persistent_kernel_shapes(b, h, m_max, seed):
    run_case("mqa", b, h, m_max, _mixed_lens(b, m_max, seed), seed=seed)


def test_persistent_kernel_all_empty_but_one():
    b, h, m_max = 64, 16, 1024
    lens = np.zeros(b, np.int32)
    lens[17] = 1000
    run_case("mqa", b, h, m_max, lens, seed=31)


@pytest.mark.parametrize("variant", ["mqa", "mha"])
@pytest.mark.parametrize("edge", range(60, 70))
def test_every_length_around_a_tile_edge(variant, edge):
    """lens = 60..69 crosses the 64-row boundary the kernels tile by."""
    run_case(variant, 2, 8, 256, [edge, 256 - edge], seed=edge)


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_long_context_configuration(variant):
    """b=32, h=32, m_max=8192: 8191 rows resident, the step appends row 8191 and attends over 8192."""
    w = wl.WORKLOADS["long_context"]
    inp = wl.make_inputs(w.b, w.h, w.m_max, variant, seed=0, device=DEV)
    lens0 = wl.initial_lens(w)
    lens_t = torch.from_numpy(lens0).to(DEV)
    Kbefore = inp["K"].clone() if variant == "mqa" else None
    mqa.kv_cache_append(inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens_t, advance=True)
    o = gpu_step(variant, inp["q"], inp["K"], inp["V"], lens_t)
    assert torch.equal(lens_t.cpu(), torch.from_numpy(lens0 + 1))
    if Kbefore is not None:                            # only the appended row changed
        same = (Kbefore.view(torch.int16) == inp["K"].view(torch.int16)).all(dim=-1)
        assert bool(same[:, : w.m_max - 1].all())
        assert torch.equal(inp["K"][:, w.m_max - 1].view(torch.int16), inp["k_new"].view(torch.int16))
    # every sequence and head, also of the 4 GiB multi-head cache
    check_against_oracle(variant, inp["q"], inp["K"], inp["V"], lens0 + 1, o, f"long_context {variant}")


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_ragged_configuration(variant):
    """b=256, h=16, m_max=2048, valid lengths uniform on [1, 2048], dead rows NaN-poisoned."""
    w = wl.WORKLOADS["ragged"]
    lens = wl.ragged_lens(w.b, w.m_max, seed=0)
    assert lens.min() >= 1 and lens.max() <= w.m_max
    run_case(variant, w.b, w.h, w.m_max, lens, seed=0)


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_paper_incremental_decoding(variant):
    """b=128, h=8: the cache grows from 1 to 128 rows over 128 steps (append, then attend over the
    prefix); each step's output is checked against the oracle on the cache as it then stands."""
    w = wl.WORKLOADS["paper_incremental"]
    b, h, m_max = w.b, w.h, w.m_max
    base = wl.make_inputs(b, h, m_max, variant, seed=0, device=DEV)
    K, V = base["K"], base["V"]
    nan = torch.tensor(wl.NAN_BITS, dtype=torch.int16, device=DEV)
    K.view(torch.int16).fill_(nan)                     # nothing is valid before the first append
    V.view(torch.int16).fill_(nan)
    lens_t = torch.zeros(b, dtype=torch.int32, device=DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    step_fn = mqa.mqa_decode_step if variant == "mqa" else mqa.mha_decode_step
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1234)
    new_shape = (b,) if variant == "mqa" else (b, h)
    outs, qs = [], []
    for t in range(w.steps):
        q = wl.bf16_normal((b, h, 128), 128 ** -0.5, gen, DEV)
        k_new = wl.bf16_normal(new_shape + (128,), 1.0, gen, DEV)
        v_new = wl.bf16_normal(new_shape + (128,), 1.0, gen, DEV)
        mqa.kv_cache_append(K, V, k_new, v_new, lens_t, advance=True, status=status)
        o = torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
        step_fn(q, K, V, lens_t, o, ws, status)
        outs.append(o)
        qs.append(q)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(lens_t.cpu(), torch.full((b,), w.steps, dtype=torch.int32))
    Kb, Vb = wl.bits(K), wl.bits(V)                    # rows are immutable once written
    ofn = oracle.mqa_decode_step if variant == "mqa" else oracle.mha_decode_step
    for t in range(w.steps):
        ref = ofn(wl.bits(qs[t]), Kb, Vb, np.full(b, t + 1, np.int32))
        check_close(outs[t].cpu().numpy(), ref, f"{variant} step {t + 1}")


@pytest.mark.parametrize("variant", ["mqa", "mha"])
@pytest.mark.parametrize("m", wl.SWEEP_M)
@pytest.mark.parametrize("b", wl.SWEEP_B)
def test_sweep_points(variant, b, m):
    """All 24 points of the bandwidth sweep (h = 16, full-length caches, both variants).  Every sequence is compared
    with the oracle; only the two multi-head caches of 16 GiB and more (b=64 and b=256 at 32768 rows: the latter is
    2^35 elements per tensor pair, beyond 32-bit indexing) are compared on the first, the last and six seeded
    sequences, all heads."""
    h = 16
    cache = 2 * b * (h if variant == "mha" else 1) * m * 256
    free, _ = torch.cuda.mem_get_info()
    if cache + 8 * 2 ** 30 > free:
        pytest.skip(f"a cache of {cache >> 30} GiB does not fit this GPU")
    sample = None
    if cache >= 16 * 2 ** 30:
        rng = np.random.default_rng(b * 7 + m)
        sample = sorted({0, b - 1, *rng.integers(0, b, size=6).tolist()})
    run_case(variant, b, h, m, np.full(b, m, np.int32), seed=m + b, sample=sample)
    torch.cuda.empty_cache()


# ----------------------------------------------------------------------------- properties
@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_dead_rows_never_contribute_bitwise(variant):
    b, h, m_max = 6, 16, 1500
    lens = np.array([1, 64, 65, 700, 1499, 1500], np.int32)
    inp = wl.make_inputs(b, h, m_max, variant, seed=3, device=DEV)
    lens_t = torch.from_numpy(lens).to(DEV)
    outs = []
    for pattern in (0x0000, wl.NAN_BITS, 0x7F80, 0xFF80, 0x7F7F):    # zeros, NaN, +inf, -inf, huge
        K, V = inp["K"].clone(), inp["V"].clone()
        wl.poison_tail(K, lens, pattern)
        wl.poison_tail(V, lens, pattern)
        outs.append(gpu_step(variant, inp["q"], K, V, lens_t))
    for o in outs[1:]:
        assert torch.equal(o.view(torch.int32), outs[0].view(torch.int32))


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_two_runs_are_bit_identical(variant):
    b, h, m_max = 16, 16, 5000
    lens = wl.ragged_lens(b, m_max, seed=4)
    inp = wl.make_inputs(b, h, m_max, variant, seed=4, device=DEV)
    lens_t = torch.from_numpy(lens).to(DEV)
    a = gpu_step(variant, inp["q"], inp["K"], inp["V"], lens_t)
    c = gpu_step(variant, inp["q"], inp["K"], inp["V"], lens_t)
    assert torch.equal(a.view(torch.int32), c.view(torch.int32))


@pytest.mark.parametrize("b,h,m_max", [(96, 16, 512), (40, 32, 2048), (8, 16, 4096)])
def test_a_thousand_launches_are_bit_identical(b, h, m_max):
    """Races show up as rare differences between identical launches (a refilled pipeline stage read a moment too late
    was one): fixed-split kernel with reused stages, persistent kernel with in-kernel merge, persistent kernel with the
    second-pass kernel."""
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=41, device=DEV)
    lens = np.random.default_rng(41).integers(3 * m_max // 4, m_max + 1, size=b).astype(np.int32)
    wl.poison_tail(inp["K"], lens); wl.poison_tail(inp["V"], lens)
    lens_t = torch.from_numpy(lens).to(DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    first = None
    for _ in range(50):
        outs = []
        for _ in range(20):
            o = torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
            mqa.mqa_decode_step(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
            outs.append(o)
        torch.cuda.synchronize()
        first = outs[0] if first is None else first
        for o in outs:
            assert torch.equal(o.view(torch.int32), first.view(torch.int32))
    ref = oracle.mqa_decode_step(wl.bits(inp["q"]), wl.bits(inp["K"]), wl.bits(inp["V"]), lens)
    check_close(first.cpu().numpy(), ref, f"b={b} h={h} m_max={m_max}")


def test_multiquery_equals_multihead_on_replicated_cache():
    """Section 3: multi-query is multi-head whose heads share one K and V."""
    b, h, m_max = 3, 16, 900
    lens = np.array([900, 450, 3], np.int32)
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=5, device=DEV)
    lens_t = torch.from_numpy(lens).to(DEV)
    o_q = gpu_step("mqa", inp["q"], inp["K"], inp["V"], lens_t)
    Krep = inp["K"][:, None].expand(b, h, m_max, 128).contiguous()
    Vrep = inp["V"][:, None].expand(b, h, m_max, 128).contiguous()
    o_h = gpu_step("mha", inp["q"], Krep, Vrep, lens_t)
    assert float((o_q - o_h).abs().max()) <= 2e-5


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_dominant_logit_returns_that_row_exactly(variant):
    b, h, m_max, star = 1, 8, 333, 201
    inp = wl.make_inputs(b, h, m_max, variant, seed=6, device=DEV)
    q = torch.zeros_like(inp["q"]); q[..., 0] = 1.0
    K = torch.zeros_like(inp["K"]); K[..., star, 0] = 200.0
    lens_t = torch.full((b,), m_max, dtype=torch.int32, device=DEV)
    o = gpu_step(variant, q, K, inp["V"], lens_t)
    want = inp["V"][..., star, :].float()
    want = want.expand(b, h, 128) if variant == "mqa" else want
    assert torch.equal(o, want.contiguous())


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_identical_keys_give_the_mean(variant):
    b, h, m_max = 2, 8, 512
    inp = wl.make_inputs(b, h, m_max, variant, seed=7, device=DEV)
    K = inp["K"].clone()
    K[..., :, :] = K[..., :1, :]
    lens = np.array([512, 100], np.int32)
    o = gpu_step(variant, inp["q"], K, inp["V"], torch.from_numpy(lens).to(DEV))
    for s in range(b):
        mean = inp["V"][s, ..., : lens[s], :].double().mean(dim=-2)
        ref = mean.expand(h, 128) if variant == "mqa" else mean
        assert float((o[s].double() - ref).abs().max()) <= 1e-5


@pytest.mark.parametrize("variant", ["mqa", "mha"])
def test_empty_and_out_of_range_lengths(variant):
    b, h, m_max = 4, 8, 200
    inp = wl.make_inputs(b, h, m_max, variant, seed=8, device=DEV)
    lens = np.array([0, 200, -3, 999], np.int32)        # empty, full, negative (-> 0), too long (-> 200)
    o = gpu_step(variant, inp["q"], inp["K"], inp["V"], torch.from_numpy(lens).to(DEV),
                 expect_status=binding.STATUS_LEN_CLAMPED)
    ref = oracle_step(variant, inp["q"], inp["K"], inp["V"], np.array([0, 200, 0, 200], np.int32))
    check_close(o.cpu().numpy()[[1, 3]], ref[[1, 3]], "clamped")
    assert float(o[0].abs().max()) == 0.0 and float(o[2].abs().max()) == 0.0
    # a batch made only of empty sequences, at a size that uses several splits
    b2, m2 = 2, 8192
    inp2 = wl.make_inputs(b2, h, m2, variant, seed=9, device=DEV)
    o2 = gpu_step(variant, inp2["q"], inp2["K"], inp2["V"], torch.zeros(b2, dtype=torch.int32, device=DEV))
    assert float(o2.abs().max()) == 0.0


@pytest.mark.parametrize("b,h,m_max", [(40, 32, 2048), (90, 16, 1800), (40, 16, 1500), (24, 96, 2048), (6, 8, 300), (4, 9, 7909), (3, 200, 2100)])
def test_split_and_combine_phases_equal_the_step_on_every_plan(b, h, m_max):
    """The pass and the second pass on their own give the step's bits on the streaming kernel (whose step merges inside
    the kernel), on the kernel with the query rows as tile rows (one and two row tiles) and on the fixed-split kernel."""
    lens = _mixed_lens(b, m_max, seed=b + h)
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=12, device=DEV)
    lens_t = torch.from_numpy(lens).to(DEV)
    whole = gpu_step("mqa", inp["q"], inp["K"], inp["V"], lens_t)
    o = torch.full_like(whole, float("nan"))
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    mqa.mqa_decode_step_split(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
    mqa.mqa_decode_step_combine(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
    torch.cuda.synchronize()
    check_against_oracle("mqa", inp["q"], inp["K"], inp["V"], lens, o, f"split + combine b={b} h={h} m_max={m_max}", None)
    if not mqa.plan_kernel_name(True, False, b, h, m_max).startswith("mqa_decode_stream_umma"):
        assert torch.equal(o.view(torch.int32), whole.view(torch.int32))      # (the streaming step merges in another order)


def test_split_and_combine_phases_equal_the_step():
    b, h, m_max = 4, 16, 9000
    lens = np.array([9000, 1, 4500, 8999], np.int32)
    for variant in ("mqa", "mha"):
        inp = wl.make_inputs(b, h, m_max, variant, seed=10, device=DEV)
        lens_t = torch.from_numpy(lens).to(DEV)
        whole = gpu_step(variant, inp["q"], inp["K"], inp["V"], lens_t)
        o = torch.full_like(whole, float("nan"))
        ws = mqa.alloc_workspace(b, h, m_max, DEV)
        split = mqa.mqa_decode_step_split if variant == "mqa" else mqa.mha_decode_step_split
        comb = mqa.mqa_decode_step_combine if variant == "mqa" else mqa.mha_decode_step_combine
        split(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
        comb(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
        torch.cuda.synchronize()
        assert torch.equal(o.view(torch.int32), whole.view(torch.int32))


# --------------------------------------------------------------------------------- append
@pytest.mark.parametrize("kvh", [1, 8, 40])
def test_append_is_bit_exact_and_touches_one_row(kvh):
    b, m_max = 5, 37
    g = torch.Generator(device="cpu"); g.manual_seed(11)
    shape = (b, m_max, 128) if kvh == 1 else (b, kvh, m_max, 128)
    new = (b, 128) if kvh == 1 else (b, kvh, 128)
    rnd = lambda s: torch.randint(-32768, 32768, s, generator=g, dtype=torch.int16)
    K, V, k_new, v_new = rnd(shape), rnd(shape), rnd(new), rnd(new)
    k_new[..., :6] = torch.tensor([-32768, 1, 0x7FC1, -1, 0x7F80, -128], dtype=torch.int16)  # -0.0, subnormal, NaNs, infs
    lens = np.array([0, 36, 37, 5, -1], np.int32)       # full and negative sequences are skipped
    Kd, Vd = K.to(DEV).view(torch.bfloat16), V.to(DEV).view(torch.bfloat16)
    lens_t = torch.from_numpy(lens).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.kv_cache_append(Kd, Vd, k_new.to(DEV).view(torch.bfloat16), v_new.to(DEV).view(torch.bfloat16), lens_t,
                        advance=True, status=status)
    torch.cuda.synchronize()
    Kh, Vh, lens_h = K.numpy().view(np.uint16).copy(), V.numpy().view(np.uint16).copy(), lens.copy()
    skipped = oracle.kv_cache_append(Kh, Vh, k_new.numpy().view(np.uint16), v_new.numpy().view(np.uint16), lens_h, True)
    assert skipped == 2
    assert int(status.item()) == binding.STATUS_APPEND_CACHE_FULL | binding.STATUS_APPEND_NEGATIVE_LEN
    assert np.array_equal(wl.bits(Kd), Kh) and np.array_equal(wl.bits(Vd), Vh)
    assert np.array_equal(lens_t.cpu().numpy(), lens_h)
    # advance = 0 leaves lens alone
    keep = lens_t.clone()
    mqa.kv_cache_append(Kd, Vd, k_new.to(DEV).view(torch.bfloat16), v_new.to(DEV).view(torch.bfloat16), lens_t,
                        advance=False)
    torch.cuda.synchronize()
    assert torch.equal(lens_t, keep)


def test_errors_leave_outputs_untouched():
    b, h, m_max = 1, 16, 32768
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=12, device=DEV)
    lens_t = torch.full((b,), m_max, dtype=torch.int32, device=DEV)
    o = torch.full((b, h, 128), 7.0, dtype=torch.float32, device=DEV)
    n, _ = mqa.plan_splits(True, b, h, m_max)
    assert n > 1
    small = torch.empty(64, dtype=torch.uint8, device=DEV)
    with pytest.raises(mqa.MqaError) as e:
        mqa.mqa_decode_step(inp["q"], inp["K"], inp["V"], lens_t, o, small)
    assert e.value.code == binding.ERR_WORKSPACE_TOO_SMALL
    torch.cuda.synchronize()
    assert bool((o == 7.0).all())


def test_runs_on_a_side_stream():
    b, h, m_max = 8, 16, 3000
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=13, device=DEV)
    lens_t = torch.full((b,), m_max, dtype=torch.int32, device=DEV)
    ref = gpu_step("mqa", inp["q"], inp["K"], inp["V"], lens_t)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    o = torch.zeros_like(ref)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    with torch.cuda.stream(s):
        mqa.mqa_decode_step(inp["q"], inp["K"], inp["V"], lens_t, o, ws)
    s.synchronize()
    assert torch.equal(o.view(torch.int32), ref.view(torch.int32))


def test_wrappers_by_their_native_half_and_by_their_own_checks():
    """A tensor that is not plainly one (a subclass) goes through the wrapper's own checks, with the same result; what they refuse
    stays refused, with nothing written."""
    class Odd(torch.Tensor):
        pass

    b, h, m = 3, 5, 600
    inp = wl.make_inputs(b, h, m, "mha", seed=3, device=DEV)
    lens = torch.tensor([0, 599, 64], dtype=torch.int32, device=DEV)
    ws, status = mqa.alloc_workspace(b, h, m, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    outs = []
    for odd, stream in ((False, None), (True, None), (False, side)):
        n, o = lens.clone(), torch.full((b, h, 128), float("nan"), dtype=torch.float32, device=DEV)
        torch.cuda.synchronize()
        q = inp["q"].as_subclass(Odd) if odd else inp["q"]
        mqa.kv_cache_append(inp["K"], inp["V"].as_subclass(Odd) if odd else inp["V"], inp["k_new"], inp["v_new"], n, status=status, stream=stream)
        assert mqa.mha_decode_step(q, inp["K"], inp["V"], n, o, ws, status, stream) is o
        torch.cuda.synchronize()
        assert n.tolist() == [1, 600, 65]
        outs.append(o.view(torch.int32))
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2]) and int(status.item()) == 0
    o = torch.zeros(b, h, 128, dtype=torch.float32, device=DEV)
    for bad, error in ((inp["q"].float(), TypeError), (inp["q"].cpu(), TypeError), (inp["q"].transpose(0, 1).contiguous().transpose(0, 1), ValueError),
                       (inp["q"][:2], ValueError)):
        with pytest.raises(error):
            mqa.mha_decode_step(bad, inp["K"], inp["V"], lens, o, ws, status)
    with pytest.raises(mqa.MqaError):
        mqa.mha_decode_step(inp["q"], inp["K"], inp["V"], lens, o, torch.empty(16, dtype=torch.uint8, device=DEV), status)
    torch.cuda.synchronize()
    assert float(o.abs().max()) == 0.0


def test_a_stream_whose_handle_is_no_integer_is_refused():
    class Odd:
        cuda_stream = 1.5

    b, h, m = 2, 3, 64
    inp = wl.make_inputs(b, h, m, "mqa", seed=1, device=DEV)
    lens, o, status = torch.full((b,), 5, dtype=torch.int32, device=DEV), torch.zeros(b, h, 128, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    before = inp["K"].clone()
    with pytest.raises(TypeError):
        mqa.kv_cache_append(inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens, status=status, stream=Odd())
    with pytest.raises(TypeError):
        mqa.mqa_decode_step(inp["q"], inp["K"], inp["V"], lens, o, None, status, Odd())
    torch.cuda.synchronize()
    assert torch.equal(inp["K"], before) and float(o.abs().max()) == 0.0 and lens.tolist() == [5, 5]
