"""mqa_decode_append_step (append + attention + merge in one call, one kernel launch for large
batches) against the oracle: oracle append, then oracle multi-query step on the grown cache."""
import numpy as np
import pytest
import torch

import oracle
import paper_1911_02150_b200 as mqa
from guards import Guarded
from paper_1911_02150_b200 import binding, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ABS_TOL, REL_TOL = 4e-3, 1e-2


def check_close(got, ref, what):
    assert np.all(np.isfinite(got)), f"{what}: non-finite output"
    err = np.abs(got.astype(np.float64) - ref)
    assert err.max() <= ABS_TOL, f"{what}: max abs err {err.max():.3e}"
    assert np.all(err.max(-1) <= REL_TOL * np.abs(ref).max(-1)), f"{what}: row-relative error"


def run(b, h, m_max, lens0, advance, seed, chained=False):
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=seed, device=DEV)
    lens0 = np.asarray(lens0, np.int32)
    wl.poison_tail(inp["K"], np.clip(lens0, 0, m_max))
    wl.poison_tail(inp["V"], np.clip(lens0, 0, m_max))
    Kh, Vh, lens_h = wl.bits(inp["K"]), wl.bits(inp["V"]), lens0.copy()
    skipped = oracle.kv_cache_append(Kh, Vh, wl.bits(inp["k_new"]), wl.bits(inp["v_new"]), lens_h, True)
    ref = oracle.mqa_decode_step(wl.bits(inp["q"]), Kh, Vh, lens_h)
    # everything small that the step reads or writes sits between guard regions, checked after the kernels have run
    lens_g = Guarded((b,), torch.int32, DEV, like=torch.from_numpy(lens0).to(DEV))
    lens_t = lens_g.t
    o_g = Guarded((b, h, 128), torch.float32, DEV)
    o = o_g.t
    o.fill_(float("nan"))
    ws_g = Guarded((max(16, mqa.workspace_bytes(b, h, m_max)),), torch.uint8, DEV)
    ws = ws_g.t
    ws.fill_(0xFF)
    status_g = Guarded((1,), torch.int32, DEV)
    status = status_g.t
    status.zero_()
    q_g, kn_g, vn_g = (Guarded(tuple(inp[n].shape), torch.bfloat16, DEV, like=inp[n]) for n in ("q", "k_new", "v_new"))
    mqa.mqa_decode_append_step(q_g.t, inp["K"], inp["V"], kn_g.t, vn_g.t, lens_t, o, ws, status,
                               advance=advance, chained=chained)
    torch.cuda.synchronize()
    for g, name in ((lens_g, "lens"), (o_g, "o"), (ws_g, "workspace"), (status_g, "status"), (q_g, "q"), (kn_g, "k_new"), (vn_g, "v_new")):
        g.check(f"append_step b={b} h={h} m_max={m_max}: {name}")
    assert torch.equal(q_g.t, inp["q"]) and torch.equal(kn_g.t, inp["k_new"]) and torch.equal(vn_g.t, inp["v_new"])
    check_close(o.cpu().numpy(), ref, f"append_step b={b} h={h} m_max={m_max}")
    assert np.array_equal(wl.bits(inp["K"]), Kh) and np.array_equal(wl.bits(inp["V"]), Vh)   # the append, bit for bit
    assert np.array_equal(lens_t.cpu().numpy(), lens_h if advance else lens0)
    want_status = 0
    if (lens0 >= m_max).any():
        want_status |= binding.STATUS_APPEND_CACHE_FULL
    if (lens0 < 0).any():
        want_status |= binding.STATUS_APPEND_NEGATIVE_LEN | binding.STATUS_LEN_CLAMPED
    assert int(status.item()) == want_status, (int(status.item()), want_status, skipped)
    return inp, o


def lens_mix(b, m_max, seed):
    r = np.random.default_rng(seed)
    lens = r.integers(0, m_max, size=b).astype(np.int32)
    lens[r.integers(0, b, size=max(1, b // 8))] = 0          # first token of a sequence
    lens[r.integers(0, b, size=max(1, b // 8))] = m_max - 1  # fills the cache
    return lens


CASES = [
    # b, h, m_max: plans with the append inside the pass (persistent kernels) ...
    (40, 16, 1500), (160, 32, 333), (300, 8, 200), (37, 32, 4000), (64, 5, 777),
    # ... 33 .. 128 query rows per sequence: the kernel with the query rows as tile rows (fixed splits; the CTA whose rows
    # hold the new one stores it; one split per sequence moves lens on itself, else the second pass does) ...
    (40, 48, 1500), (33, 64, 2100), (24, 128, 2048), (20, 96, 1500), (150, 33, 700), (1, 127, 20000), (5, 65, 129),
    # ... more query rows than that: row tiles of 128 over the same cache rows, each CTA of the row's split storing the
    # new row; with one split per sequence lens is moved on by a kernel of its own ...
    (6, 200, 3000), (80, 160, 600), (2, 129, 5000), (3, 300, 1500),
    # ... and plans that run as separate launches (small batches)
    (4, 8, 300), (1, 16, 20000), (2, 40, 600),
]


@pytest.mark.parametrize("advance", [True, False])
@pytest.mark.parametrize("b,h,m_max", CASES)
def test_append_step_matches_oracle(b, h, m_max, advance):
    run(b, h, m_max, lens_mix(b, m_max, seed=b + h), advance, seed=b * 7 + h)


@pytest.mark.parametrize("chained", [True, "wrong-guess"])
@pytest.mark.parametrize("b,h,m_max", CASES + [(300, 16, 1500), (1024, 8, 1024)])
def test_append_step_with_the_chained_promise_matches_oracle(b, h, m_max, chained):
    """Every plan accepts the promise (most ignore it); nothing but the set-up copies precedes the step here, so it holds."""
    run(b, h, m_max, lens_mix(b, m_max, seed=b + h + 1), True, seed=b * 5 + h, chained=chained)


@pytest.mark.parametrize("chained", [False, True])
@pytest.mark.parametrize("h,m_max", [(8, 128), (16, 700), (32, 130), (17, 900)])
def test_new_row_at_the_edges_of_tiles_and_splits(h, m_max, chained):
    """The fixed-split kernel puts the new row into the landed tile itself: rows either side of every edge of a 32-row tile,
    of four tiles and of a split, one and two head tiles, one split and several."""
    lens = sorted({min(m_max - 1, max(0, e + x)) for e in (0, 32, 64, 128, 160, 256, 320, 448, 512, 640, m_max) for x in (-2, -1, 0, 1)})
    run(len(lens), h, m_max, lens, True, seed=h + m_max, chained=chained)


@pytest.mark.parametrize("chained", [False, True, "wrong-guess"])
@pytest.mark.parametrize("h,m_max", [(40, 700), (96, 2600), (130, 1500), (33, 260)])
def test_new_row_at_the_edges_of_stages_and_splits_with_many_query_rows(h, m_max, chained):
    """The many-rows kernel does so in stages of 128 rows: rows either side of every edge of a stage and of a split, with one row
    tile and two, several splits and one."""
    chunk = mqa.plan_splits(True, 32, h, m_max)[1]
    edges = {0, 128, 256, m_max, *(chunk * i for i in range(1, 5)), chunk + 128}
    lens = sorted({min(m_max - 1, max(0, e + x)) for e in edges for x in (-2, -1, 0, 1)})[:32]
    lens = (lens + [m_max - 1] * 32)[:32]
    assert mqa.plan_splits(True, len(lens), h, m_max)[1] == chunk
    run(len(lens), h, m_max, lens, True, seed=h + m_max, chained=chained)


def test_append_step_full_and_negative_sequences_take_no_row():
    b, h, m_max = 48, 16, 1024
    lens = lens_mix(b, m_max, seed=5)
    lens[3] = m_max          # full: no row, attends over m_max rows
    lens[7] = -2             # negative: no row, empty prefix -> zeros
    run(b, h, m_max, lens, True, seed=77)


def test_incremental_decoding_with_append_steps():
    """A decoding loop of 40 steps on a batch large enough for the persistent kernel (append inside the pass): every step's
    output against the oracle on the cache as it then stands, and two runs bit-identical."""
    b, h, m_max, steps = 96, 16, 512, 40
    gen = torch.Generator(device=DEV)
    outs = []
    for rep in range(2):
        gen.manual_seed(321)
        K = torch.zeros(b, m_max, 128, dtype=torch.bfloat16, device=DEV)
        V = torch.zeros_like(K)
        nan = torch.tensor(wl.NAN_BITS, dtype=torch.int16, device=DEV)
        K.view(torch.int16).fill_(nan); V.view(torch.int16).fill_(nan)
        start = np.random.default_rng(3).integers(380, 470, size=b).astype(np.int32)     # prefill of different lengths
        for s in range(b):
            K[s, : start[s]] = wl.bf16_normal((int(start[s]), 128), 1.0, gen, DEV)
            V[s, : start[s]] = wl.bf16_normal((int(start[s]), 128), 1.0, gen, DEV)
        lens_t = torch.from_numpy(start.copy()).to(DEV)
        ws = mqa.alloc_workspace(b, h, m_max, DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        run_outs, qs = [], []
        for t in range(steps):
            q = wl.bf16_normal((b, h, 128), 128 ** -0.5, gen, DEV)
            k_new = wl.bf16_normal((b, 128), 1.0, gen, DEV)
            v_new = wl.bf16_normal((b, 128), 1.0, gen, DEV)
            o = torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
            mqa.mqa_decode_append_step(q, K, V, k_new, v_new, lens_t, o, ws, status)
            run_outs.append(o); qs.append(q)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        assert np.array_equal(lens_t.cpu().numpy(), start + steps)
        outs.append(run_outs)
        if rep == 0:
            Kb, Vb = wl.bits(K), wl.bits(V)
            for t in (0, 1, 17, steps - 1):
                ref = oracle.mqa_decode_step(wl.bits(qs[t]), Kb, Vb, (start + t + 1).astype(np.int32))
                check_close(run_outs[t].cpu().numpy(), ref, f"step {t}")
    for a, c in zip(*outs):
        assert torch.equal(a.view(torch.int32), c.view(torch.int32))


def test_host_buffer_entry_point_matches_the_device_one():
    b, h, m_max = 40, 16, 1500
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=21, device=DEV)
    lens0 = lens_mix(b, m_max, seed=21)
    wl.poison_tail(inp["K"], lens0); wl.poison_tail(inp["V"], lens0)
    K2, V2 = inp["K"].clone(), inp["V"].clone()
    lens_a, lens_b = torch.from_numpy(lens0).to(DEV), torch.from_numpy(lens0.copy()).to(DEV)
    o_dev = torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    mqa.mqa_decode_append_step(inp["q"], inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens_a, o_dev, ws)
    # host side: once as three separate pinned tensors, once packed back to back (one copy)
    for packed in (False, True):
        Kc, Vc, lens_c = K2.clone(), V2.clone(), lens_b.clone()
        if packed:
            parts = [inp[n].cpu().contiguous() for n in ("q", "k_new", "v_new")]
            buf = torch.empty(sum(t.numel() * 2 for t in parts), dtype=torch.uint8).pin_memory()
            views, at = [], 0
            for t in parts:
                n = t.numel() * 2
                buf[at : at + n].copy_(t.view(torch.uint8).view(-1))
                views.append(buf[at : at + n].view(torch.bfloat16).view(t.shape))
                at += n
            qh, kh, vh = views
        else:
            qh, kh, vh = (inp[n].cpu().pin_memory() for n in ("q", "k_new", "v_new"))
        o_host = torch.full((b, h, 128), float("nan"), dtype=torch.float32).pin_memory()
        staging = torch.empty(mqa.host_staging_bytes(b, h), dtype=torch.uint8, device=DEV)
        if packed:
            mqa.HostStep(qh, kh, vh, o_host, Kc, Vc, lens_c, staging, ws)()      # bound once, then the bare C call
        else:
            mqa.mqa_decode_append_step_host(qh, kh, vh, o_host, Kc, Vc, lens_c, staging, ws)
        torch.cuda.synchronize()
        assert torch.equal(o_host, o_dev.cpu())
        assert torch.equal(Kc.view(torch.int16), inp["K"].view(torch.int16)) and torch.equal(lens_c, lens_a)


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("b,h,m_max", [(32, 32, 2048), (40, 16, 1500), (6, 48, 700), (4, 8, 100), (3, 130, 300), (150, 8, 1100)])
def test_host_buffer_steps_in_a_loop_against_the_oracle(b, h, m_max, pinned):
    """Five consecutive steps through the host-buffer entry point, bound once, the same host buffers refilled before each
    step (pinned: the inputs are fetched by a kernel and o is stored to the host by the kernels; pageable: copies either
    side): every step is the oracle's append and step on the grown cache, lens moves on, the cache holds the new rows."""
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=31, device=DEV)
    lens0 = np.minimum(lens_mix(b, m_max, seed=31), m_max - 5).clip(0).astype(np.int32)
    wl.poison_tail(inp["K"], lens0); wl.poison_tail(inp["V"], lens0)
    Kh, Vh, lens_h = wl.bits(inp["K"]), wl.bits(inp["V"]), lens0.copy()
    lens_t = torch.from_numpy(lens0).to(DEV)
    hold = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    qh, kh, vh = (hold(torch.empty(tuple(inp[n].shape), dtype=torch.bfloat16)) for n in ("q", "k_new", "v_new"))
    o_host = hold(torch.empty(b, h, 128, dtype=torch.float32))
    staging = torch.empty(mqa.host_staging_bytes(b, h), dtype=torch.uint8, device=DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    step = mqa.HostStep(qh, kh, vh, o_host, inp["K"], inp["V"], lens_t, staging, ws, status)
    for t in range(5):
        new = wl.make_inputs(b, h, 1, "mqa", seed=100 + t, device="cpu")
        qh.copy_(new["q"]); kh.copy_(new["k_new"]); vh.copy_(new["v_new"])
        o_host.fill_(float("nan"))
        step()
        torch.cuda.synchronize()
        oracle.kv_cache_append(Kh, Vh, wl.bits(kh), wl.bits(vh), lens_h, True)
        check_close(o_host.numpy(), oracle.mqa_decode_step(wl.bits(qh), Kh, Vh, lens_h), f"host step {t}")
        assert np.array_equal(lens_t.cpu().numpy(), lens_h)
    assert int(status.item()) == 0
    assert np.array_equal(wl.bits(inp["K"]), Kh) and np.array_equal(wl.bits(inp["V"]), Vh)


def test_bound_step_gives_what_the_call_gives():
    b, h, m_max = 40, 16, 1500
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=22, device=DEV)
    lens0 = lens_mix(b, m_max, seed=22)
    wl.poison_tail(inp["K"], lens0); wl.poison_tail(inp["V"], lens0)
    K2, V2 = inp["K"].clone(), inp["V"].clone()
    lens_a, lens_b = torch.from_numpy(lens0).to(DEV), torch.from_numpy(lens0.copy()).to(DEV)
    o_a, o_b = (torch.empty(b, h, 128, dtype=torch.float32, device=DEV) for _ in range(2))
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    for _ in range(3):                                        # three tokens each way (the same q and rows: only lens moves)
        mqa.mqa_decode_append_step(inp["q"], inp["K"], inp["V"], inp["k_new"], inp["v_new"], lens_a, o_a, ws)
    step = mqa.AppendStep(inp["q"], K2, V2, inp["k_new"], inp["v_new"], lens_b, o_b, ws)
    for _ in range(3):
        assert step() is o_b
    torch.cuda.synchronize()
    assert torch.equal(o_a.view(torch.int32), o_b.view(torch.int32)) and torch.equal(lens_a, lens_b)
    assert torch.equal(inp["K"].view(torch.int16), K2.view(torch.int16)) and torch.equal(inp["V"].view(torch.int16), V2.view(torch.int16))
    with pytest.raises(TypeError):
        mqa.AppendStep(inp["q"].float(), K2, V2, inp["k_new"], inp["v_new"], lens_b, o_b, ws)


@pytest.mark.parametrize("b,h,m_max", [(5, 40, 700), (3, 96, 2600), (160, 33, 600), (2, 130, 1500)])
def test_logits_of_minus_infinity_weigh_nothing_with_many_query_rows(b, h, m_max):
    """Key rows whose logit is -inf for every query row: whole 128-row stages of them, the first, the second (the other softmax
    warps' first) and all but the last rows."""
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=m_max, device=DEV)
    inp["q"][..., 0] = inp["q"][..., 0].abs() + 0.125
    lens = torch.full((b,), m_max - 1, dtype=torch.int32, device=DEV)
    ws, status = mqa.alloc_workspace(b, h, m_max, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    for rows in (slice(128, 256), slice(0, 128), slice(0, 384), slice(130, 500), slice(0, m_max - 2)):
        K, o = inp["K"].clone(), torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
        K[:, rows, 0] = -float("inf")
        mqa.mqa_decode_append_step(inp["q"], K, inp["V"], inp["k_new"], inp["v_new"], lens, o, ws, status, advance=False)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        ref = torch.softmax(inp["q"].double() @ K.double().transpose(1, 2), -1) @ inp["V"].double()    # (the new row is in K and V by now)
        check_close(o.cpu().numpy(), ref.cpu().numpy(), f"rows {rows}")


@pytest.mark.parametrize("b,h,m_max", [
    (70, 8, 128), (40, 16, 1000), (8, 32, 600),        # fixed splits: one, and several
    (64, 40, 300), (9, 100, 2000),                     # many rows: one split, several
    (40, 16, 1500),                                    # fixed splits in clusters
    (40, 32, 2048), (90, 16, 1800), (300, 8, 1024),   # the streaming kernel, most sequences cut and few
])
def test_a_loop_of_steps_back_to_back_equals_steps_one_at_a_time(b, h, m_max):
    """60 tokens, each step behind the one before with nothing waited for, its inputs put into the same buffers; 32
    sequences' lengths share a line of memory and every step moves them all.  The caches and lengths are the same, o to the last bit."""
    steps = 60
    inp = wl.make_inputs(b, h, m_max, "mqa", seed=b + m_max, device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(h)
    q, kn, vn = (wl.bf16_normal((steps, *s), std, gen, DEV) for s, std in (((b, h, 128), 128 ** -0.5), ((b, 128), 1.0), ((b, 128), 1.0)))
    lens0 = torch.from_numpy(np.random.default_rng(b).integers(0, m_max - steps // 2, size=b).astype(np.int32)).to(DEV)
    results = []
    for apart in (False, True):
        K, V, lens = inp["K"].clone(), inp["V"].clone(), lens0.clone()
        ws, status = mqa.alloc_workspace(b, h, m_max, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        o = torch.full((steps, b, h, 128), float("nan"), dtype=torch.float32, device=DEV)
        qb, kb, vb = q[0].clone(), kn[0].clone(), vn[0].clone()
        torch.cuda.synchronize()
        for t in range(steps):
            for buf, src in ((qb, q), (kb, kn), (vb, vn)):
                buf.copy_(src[t])
            mqa.mqa_decode_append_step(qb, K, V, kb, vb, lens, o[t], ws, status, chained=not apart and t > 0)
            if apart:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        results.append((o, K, V, lens, status))
    for name, x, y in zip(("o", "K", "V", "lens", "status"), *results):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), name
    assert bool(torch.isfinite(results[0][0]).all())


@pytest.mark.parametrize("variant,b,h,m_max", [
    ("mqa", 70, 8, 128), ("mqa", 40, 16, 1000), ("mqa", 8, 32, 600),            # fixed splits: one, and several
    ("mqa", 64, 40, 300), ("mqa", 9, 100, 2000), ("mqa", 2, 130, 1500), ("mqa", 1, 16, 20000),   # many rows: one split, several, dozens
    ("mqa", 40, 16, 1500), ("mqa", 4, 9, 7909),                                 # fixed splits: a cluster, a second pass
    ("mqa", 40, 32, 2048), ("mqa", 100, 16, 3000), ("mqa", 32, 32, 2048), ("mqa", 64, 16, 4096), ("mqa", 300, 8, 1024),    # streaming: merged in the kernel, by clusters, mostly whole
    ("mha", 3, 4, 700), ("mha", 1, 2, 40000),
])
def test_a_prefix_whose_rows_are_partly_nan_gives_nan(variant, b, h, m_max):
    """Whatever pieces the prefix is cut into, and where all the logits of some of them, or of all, are NaN: never a finite
    result made of the others, nor the empty prefix's zeros."""
    inp = wl.make_inputs(b, h, m_max, variant, seed=m_max + h, device=DEV)
    L = m_max - 3
    lens = torch.full((b,), L, dtype=torch.int32, device=DEV)
    ws, status = mqa.alloc_workspace(b, h, m_max, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    step = mqa.mqa_decode_step if variant == "mqa" else mqa.mha_decode_step
    for rows in (slice(0, L), slice(L // 2, L), slice(0, L // 2), slice(L // 3, 2 * L // 3), slice(L - 1, L), slice(7, 8)):
        K, o = inp["K"].clone(), torch.zeros(b, h, 128, dtype=torch.float32, device=DEV)
        K[..., rows, :] = float("nan")
        step(inp["q"], K, inp["V"], lens, o, ws, status)
        torch.cuda.synchronize()
        assert bool(torch.isnan(o).all()), f"step, rows {rows}: {int((~torch.isnan(o)).sum())} elements are not NaN"
        if variant == "mqa":
            o.zero_()
            mqa.mqa_decode_append_step(inp["q"], K, inp["V"], inp["k_new"], inp["v_new"], lens, o, ws, status, advance=False)
            torch.cuda.synchronize()
            assert bool(torch.isnan(o).all()), f"append step, rows {rows}: {int((~torch.isnan(o)).sum())} elements are not NaN"
    assert int(status.item()) == 0


@pytest.mark.parametrize("variant,b,h,m_max", [
    ("mqa", 3, 8, 100), ("mqa", 12, 16, 1000), ("mqa", 20, 32, 1500), ("mqa", 8, 16, 4096), ("mqa", 4, 9, 7909),      # fixed splits: one, clusters, a second pass
    ("mqa", 64, 16, 4096), ("mqa", 40, 32, 2100), ("mqa", 20, 24, 9000),                                             # the streaming kernel
    ("mqa", 5, 40, 1500), ("mqa", 96, 16, 1586),                                                                     # query rows as tile rows
    ("mha", 3, 4, 700), ("mha", 2, 16, 100),
])
def test_logits_of_minus_infinity_weigh_nothing(variant, b, h, m_max):
    """Key rows whose logit is -inf for every head: single tiles and stages of them, the first ones, later ones, the last;
    and where there are no others, 0 / 0."""
    inp = wl.make_inputs(b, h, m_max, variant, seed=m_max, device=DEV)
    inp["q"][..., 0] = inp["q"][..., 0].abs() + 0.125
    lens = torch.full((b,), m_max - 1, dtype=torch.int32, device=DEV)
    lens[b // 2] = m_max // 2
    ws, status = mqa.alloc_workspace(b, h, m_max, DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    valid = torch.arange(m_max, device=DEV) <= lens[:, None]
    for rows in (slice(0, 32), slice(0, 128), slice(32, 96), slice(0, m_max // 4), slice(m_max // 3, m_max), slice(0, m_max)):
        K, V, o = inp["K"].clone(), inp["V"].clone(), torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
        K[..., rows, 0] = -float("inf")
        k_new = inp["k_new"].clone()
        if rows == slice(0, m_max):
            k_new[..., 0] = -float("inf")
        if variant == "mqa":
            mqa.mqa_decode_append_step(inp["q"], K, V, k_new, inp["v_new"], lens, o, ws, status, advance=False)
        else:
            mqa.kv_cache_append(K, V, k_new, inp["v_new"], lens, advance=False, status=status)
            mqa.mha_decode_step(inp["q"], K, V, lens + 1, o, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        if rows == slice(0, m_max):
            assert bool(torch.isnan(o).all())
            continue
        q = inp["q"].double() if variant == "mqa" else inp["q"].double().unsqueeze(2)
        s = q @ K.double().transpose(-1, -2)                         # (the new row is in K and V by now)
        seen = valid[:, None] if variant == "mqa" else valid[:, None, None]
        ref = torch.softmax(s.masked_fill(~seen, -float("inf")), -1) @ V.double()
        check_close(o.cpu().numpy(), ref.reshape(b, h, 128).cpu().numpy(), f"rows {rows}")
