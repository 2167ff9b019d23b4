"""mqa_prefill_attention (Section 3, the attention lines of the batched multi-query function under the autoregressive
mask of Section 2.3) against the fp64 oracle on the same bf16 bits.  Tolerance as for the decode step: every element
within 4e-3, every (sequence, head, position) row within 1e-2 of its own scale."""
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
    bad = err.max(-1) > REL_TOL * np.abs(ref).max(-1)
    assert not bad.any(), f"{what}: {bad.sum()} rows over the relative tolerance"


def run(b, h, n, m_max, start=None, seed=0, sample=None):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.zeros(b, np.int32) if start is None else np.asarray(start, np.int32)
    wl.poison_tail(K, st + n)                              # rows after a sequence's last query position are never read
    wl.poison_tail(V, st + n)
    Og = Guarded((b, h, n, 128), torch.float32, DEV)
    Og.t.fill_(float("nan"))
    wsg = Guarded((max(16, mqa.prefill_workspace_bytes(b, h, n, m_max)),), torch.uint8, DEV)
    wsg.t.fill_(0xFF)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    start_t = None if start is None else torch.from_numpy(st).to(DEV)
    mqa.mqa_prefill_attention(Q, K, V, Og.t, wsg.t, start_t, status)
    torch.cuda.synchronize()
    Og.check("O"); wsg.check("workspace")
    assert int(status.item()) == 0
    O = Og.t
    assert bool(torch.isfinite(O).all())                   # every row was written, sampled or not
    if sample is None:
        ref = oracle.mqa_batched_attention(wl.bits(Q), wl.bits(K), wl.bits(V), st)
        check_close(O.cpu().numpy(), ref, f"b={b} h={h} n={n}")
    else:
        for s, heads in sample:
            hs = torch.as_tensor(heads, device=DEV)
            ref = oracle.mqa_batched_attention(wl.bits(Q[s:s + 1, hs]), wl.bits(K[s:s + 1]), wl.bits(V[s:s + 1]), st[s:s + 1])
            check_close(O[s:s + 1, hs].cpu().numpy(), ref, f"b={b} h={h} n={n} sequence {s} heads {heads}")
    return O


SMALL = [
    # b, h, n, m_max, start
    (1, 1, 64, 64, None),                       # one group: every column has its own last row
    (2, 8, 128, 128, None),
    (3, 4, 192, 512, [0, 100, 320]),            # a chunk of a longer prompt: queries begin at start[b]
    (2, 3, 256, 300, [44, 0]),                  # a head count that does not divide 64
    (1, 32, 128, 1100, [900]),                  # long memory in front of few queries
    (5, 16, 64, 2048, [1984, 0, 63, 64, 1000]),
    (2, 5, 100, 260, [160, 0]),                 # n is no multiple of anything: the last tile of a head is partly filled
    (3, 2, 1, 700, [0, 699, 350]),              # one position: a decoding step
    (1, 3, 129, 129, None),                     # one position in a tile of its own
    (2, 4, 333, 1200, [867, 5]),
]


@pytest.mark.parametrize("b,h,n,m_max,start", SMALL)
def test_small_cases_match_oracle(b, h, n, m_max, start):
    run(b, h, n, m_max, start, seed=b * 100 + h)


@pytest.mark.parametrize("b,h", [(128, 8), (32, 32)])
@pytest.mark.parametrize("n", [128, 1024, 4096])
def test_prompt_lengths_of_the_decode_configurations(b, h, n):
    """n = m in {128, 1024, 4096} for the batch and head counts of the paper-shaped and the long-context
    configurations.  The oracle is the plain fp64 definition (n^2 / 2 pairs per head): checked in full at n = 128, on
    seeded (sequence, heads) samples beyond (all positions of those heads)."""
    r = np.random.default_rng(n + b)
    if n == 128:
        sample = None
    else:
        seqs = sorted({0, b - 1, *r.integers(0, b, size=2).tolist()})
        per = 4 if n == 1024 else 1
        sample = [(s, sorted(set(r.integers(0, h, size=per).tolist()) | ({0} if s == 0 else {h - 1}))) for s in seqs]
    run(b, h, n, n, None, seed=n + h, sample=sample)


def test_rows_are_the_decode_steps():
    """Position t of the batched form is the incremental step over start + t + 1 rows (Section 2.4: up to and
    including its own position): the two entry points agree to within the two paths' rounding."""
    b, h, n, m_max = 2, 16, 128, 1300
    start = np.array([1000, 1172], np.int32)
    O = run(b, h, n, m_max, start, seed=5)
    gen = torch.Generator(device=DEV).manual_seed(5)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    ws = mqa.alloc_workspace(b, h, m_max, DEV)
    for t in (0, 1, 63, 64, 127):
        o = torch.empty(b, h, 128, dtype=torch.float32, device=DEV)
        mqa.mqa_decode_step(Q[:, :, t].contiguous(), K, V, torch.from_numpy(start + t + 1).to(DEV), o, ws)
        torch.cuda.synchronize()
        assert float((o - O[:, :, t]).abs().max()) <= 2e-3


WHOLE_TILES = [
    # b, h, n, m_max, start: n a multiple of 128 (the kernel of the batched form: two heads per CTA)
    (2, 5, 384, 700, [300, 17]),                # an odd head count: the last CTA of a position tile holds one head
    (1, 2, 1152, 1300, [100]),                  # memories on both sides of 1024 rows (two roundings of the weights below it)
    (3, 7, 256, 1000, [744, 0, 511]),           # start + n = m_max exactly; a stage that ends inside the next sequence's rows
    (2, 1, 128, 128, None),                     # a single head
    (1, 4, 512, 2049, [1537]),                  # one row of the memory in a stage of its own
]


@pytest.mark.parametrize("b,h,n,m_max,start", WHOLE_TILES)
def test_whole_tiles_match_oracle(b, h, n, m_max, start):
    run(b, h, n, m_max, start, seed=7 * b + h)


@pytest.mark.parametrize("b,h,n,m_max,start", [
    # tiles of several heads: rows past the last position, past the last head, a tile alone in its unit, more heads than rows
    (2, 9, 45, 400, [0, 355]), (3, 20, 16, 1100, [1084, 0, 500]), (1, 33, 7, 64, [3]), (2, 128, 3, 40, [0, 37]), (1, 130, 2, 20, None),
    (1, 6, 130, 130, None), (2, 7, 21, 1030, [1003, 1009]),
    # few units: 2, 4 and 8 CTAs share a unit's stages; stages that some rows, or some CTAs, see nothing of
    (5, 9, 333, 3000, [0, 2667, 100, 1300, 700]), (8, 16, 64, 2000, [0, 1, 63, 64, 127, 900, 1935, 1936]), (1, 4, 16, 2064, [2048]),
    (1, 4, 16, 2064, [0]), (2, 3, 100, 1500, [1400, 130]), (1, 1, 1500, 1500, None), (3, 2, 128, 4096, [3968, 0, 895]),
])
def test_tile_shapes_and_shared_units(b, h, n, m_max, start):
    run(b, h, n, m_max, start, seed=b + 3 * h + n)


@pytest.mark.parametrize("b,h,n,m_max,start", [
    # one tile to a CTA, its stages in turn between the warpgroups and between 1, 2, 4 and 8 CTAs: one stage and two, an odd number, CTAs
    # that get none, rows that see nothing of a CTA's run, a last stage of one row, tiles of several heads partly filled
    (2, 5, 129, 257, [128, 0]), (6, 20, 100, 640, [540, 0, 28, 412, 413, 29]), (1, 3, 1, 3000, [2999]),
    (30, 4, 128, 1500, list(range(0, 1350, 45))), (9, 8, 256, 513, [257, 256, 0, 1, 100, 127, 128, 129, 200]), (1, 2, 640, 4000, [3200]),
    (20, 2, 64, 1500, list(range(0, 1400, 70))), (60, 1, 128, 2000, list(range(0, 1800, 30))),
])
def test_one_tile_to_a_cta(b, h, n, m_max, start):
    assert mqa.prefill_plan_kernel(b, h, n, m_max, start is not None)[0] == "mqa_prefill_tile_kernel"
    run(b, h, n, m_max, start, seed=2 * b + h + n)


@pytest.mark.parametrize("b,h,n,m_max,start", [
    # two tiles to a CTA: one stage, one tile alone in its unit; several units to a CTA, memories of one to eight stages in any order
    (3, 9, 128, 128, None), (1, 1, 1, 1, None), (1, 148, 2, 64, [62]), (20, 16, 128, 1100, [(251 * i) % 973 for i in range(20)]),
    (30, 12, 200, 900, [(301 * i) % 701 for i in range(30)]), (80, 5, 130, 420, [(97 * i) % 291 for i in range(80)]),
])
def test_two_tiles_to_a_cta(b, h, n, m_max, start):
    assert mqa.prefill_plan_kernel(b, h, n, m_max, start is not None)[0] == "mqa_prefill_kernel"
    run(b, h, n, m_max, start, seed=2 * b + h + n)


def test_starts_of_all_kinds_with_two_tiles_to_a_cta():
    """Many tiles: a negative start in the middle of the batch gives zeros, memories that would pass m_max are cut there, and the
    sequences beside them, on the same CTAs, are not affected."""
    b, h, n, m_max = 20, 16, 128, 600
    assert mqa.prefill_plan_kernel(b, h, n, m_max, True)[0] == "mqa_prefill_kernel"
    gen = torch.Generator(device=DEV).manual_seed(43)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K, V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV), wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array([(83 * i) % 473 for i in range(b)], np.int32)
    st[[3, 10]] = -1, -700
    st[[5, 11, 19]] = m_max - 1, m_max - n + 3, m_max + 40
    O = torch.full((b, h, n, 128), float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, torch.empty(16, dtype=torch.uint8, device=DEV), torch.from_numpy(st).to(DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == binding.STATUS_LEN_CLAMPED
    assert bool((O[[3, 10]] == 0).all())
    keep = [i for i in range(b) if i not in (3, 10)]
    for t in (0, 1, 63, 64, 100, 126, 127):
        lens = np.clip(st + t + 1, 0, m_max).astype(np.int32)
        ref = oracle.mqa_decode_step(wl.bits(Q[:, :, t].contiguous()), wl.bits(K), wl.bits(V), lens)
        check_close(O[keep, :, t].cpu().numpy(), ref[keep], f"position {t}")


def test_shared_units_with_a_negative_start_and_one_past_the_memory():
    """The same units shared by a cluster: nothing to look at gives zeros, a memory that would pass m_max is cut there."""
    b, h, n, m_max = 3, 4, 16, 2064
    gen = torch.Generator(device=DEV).manual_seed(41)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array([-5, m_max - 3, 1000], np.int32)
    O = torch.full((b, h, n, 128), float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, torch.empty(16, dtype=torch.uint8, device=DEV), torch.from_numpy(st).to(DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == binding.STATUS_LEN_CLAMPED
    assert bool((O[0] == 0).all())
    for t in range(n):
        lens = np.clip(st + t + 1, 0, m_max).astype(np.int32)
        ref = oracle.mqa_decode_step(wl.bits(Q[:, :, t].contiguous()), wl.bits(K), wl.bits(V), lens)
        check_close(O[1:, :, t].cpu().numpy(), ref[1:], f"position {t}")


def test_a_logit_far_above_every_earlier_one_in_a_long_memory():
    """A key row 300 times larger than the others, deep in a memory of more than 1024 rows, makes logits hundreds of
    units above (and below) everything before it: the rows' reference maxima move late and by a lot, and their
    accumulated outputs are rescaled by factors that underflow."""
    b, h, n, m_max = 2, 3, 256, 1536
    gen = torch.Generator(device=DEV).manual_seed(21)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array([1280, 1100], np.int32)
    K[0, 1400] *= 300
    K[1, 1290] *= 300
    K[1, 5] *= 40                                           # (and one in the first stage, for comparison)
    O = torch.full((b, h, n, 128), float("nan"), dtype=torch.float32, device=DEV)
    ws = torch.empty(max(16, mqa.prefill_workspace_bytes(b, h, n, m_max)), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, ws, torch.from_numpy(st).to(DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle.mqa_batched_attention(wl.bits(Q), wl.bits(K), wl.bits(V), st)
    check_close(O.cpu().numpy(), ref, "a dominant key row late in the memory")


def test_a_negative_start_gives_zeros_and_a_flag():
    """start[b] < 0 is an empty memory for that sequence (zeros, LEN_CLAMPED); the other sequences are not affected."""
    b, h, n, m_max = 3, 4, 256, 512
    gen = torch.Generator(device=DEV).manual_seed(11)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array([5, -1, 100], np.int32)
    O = torch.full((b, h, n, 128), float("nan"), dtype=torch.float32, device=DEV)
    ws = torch.empty(max(16, mqa.prefill_workspace_bytes(b, h, n, m_max)), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, ws, torch.from_numpy(st).to(DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == binding.STATUS_LEN_CLAMPED
    assert bool((O[1] == 0).all())
    keep = [0, 2]
    ref = oracle.mqa_batched_attention(wl.bits(Q[keep]), wl.bits(K[keep]), wl.bits(V[keep]), st[keep])
    check_close(O[keep].cpu().numpy(), ref, "sequences beside a bad start")


def test_two_runs_are_bit_identical():
    a = run(4, 8, 256, 700, [0, 400, 444, 13], seed=9)
    c = run(4, 8, 256, 700, [0, 400, 444, 13], seed=9)
    assert torch.equal(a.view(torch.int32), c.view(torch.int32))


def test_what_is_not_supported_is_refused_before_any_launch():
    b, h, n, m_max = 2, 4, 300, 256                        # more positions than the memory holds
    assert mqa.prefill_workspace_bytes(b, h, n, m_max) == 0
    Q = torch.zeros(b, h, n, 128, dtype=torch.bfloat16, device=DEV)
    K = torch.zeros(b, m_max, 128, dtype=torch.bfloat16, device=DEV)
    O = torch.full((b, h, n, 128), 7.0, dtype=torch.float32, device=DEV)
    with pytest.raises(mqa.MqaError) as e:
        mqa.mqa_prefill_attention(Q, K, K, O, torch.empty(1 << 20, dtype=torch.uint8, device=DEV))
    assert e.value.code == binding.ERR_UNSUPPORTED
    torch.cuda.synchronize()
    assert bool((O == 7.0).all())


def test_a_memory_that_would_pass_m_max_is_cut_there_and_flagged():
    """start[b] + n > m_max: the positions past the end of the memory attend over all m_max rows (there is no row of
    their own to add), LEN_CLAMPED is flagged, nothing outside K and V is read; the other sequences are not affected.
    Checked row by row against the decoding step's oracle over min(start + t + 1, m_max) rows."""
    b, h, n, m_max = 2, 4, 256, 600
    gen = torch.Generator(device=DEV).manual_seed(31)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    st = np.array([m_max - n + 70, 100], np.int32)          # the first sequence's last 70 positions have no row
    O = torch.full((b, h, n, 128), float("nan"), dtype=torch.float32, device=DEV)
    ws = torch.empty(max(16, mqa.prefill_workspace_bytes(b, h, n, m_max)), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, ws, torch.from_numpy(st).to(DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == binding.STATUS_LEN_CLAMPED
    Oh = O.cpu().numpy()
    assert np.all(np.isfinite(Oh))
    for t in (0, 100, 185, 186, 200, 255):
        lens = np.minimum(st + t + 1, m_max).astype(np.int32)
        ref = oracle.mqa_decode_step(wl.bits(Q[:, :, t].contiguous()), wl.bits(K), wl.bits(V), lens)
        check_close(Oh[:, :, t], ref, f"position {t}")


def attend(Q, K, V, start):
    """O of the batched form as it comes, whatever the inputs hold."""
    b, h, n, _ = Q.shape
    O = torch.empty(b, h, n, 128, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    mqa.mqa_prefill_attention(Q, K, V, O, torch.empty(16, dtype=torch.uint8, device=DEV),
                              None if start is None else torch.tensor(start, dtype=torch.int32, device=DEV), status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return O


@pytest.mark.parametrize("b,h,n,m_max,start,positions", [
    # the two tiles of a unit begin at different positions: an odd number of tiles side by side at each position
    (1, 1, 256, 256, None, 128), (300, 1, 256, 260, None, 128), (3, 1, 500, 900, [0, 37, 399], 128), (1, 1, 256, 2048, [1003], 128),
    (2, 9, 333, 1000, [100, 3], 42), (40, 9, 84, 84, None, 42), (1, 9, 333, 3000, [2001], 42), (60, 9, 333, 340, None, 42),
])
def test_rows_of_later_positions_do_not_reach_the_tiles_before_them(b, h, n, m_max, start, positions):
    """NaN and Inf in V rows from the first position of a tile on: the tiles before it are the same to the last bit, those
    positions themselves are not finite where the row is not."""
    gen = torch.Generator(device=DEV).manual_seed(n + h)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    clean = attend(Q, K, V, start)
    assert bool(torch.isfinite(clean).all())
    at = torch.tensor([0] * b if start is None else start, device=DEV)[:, None]
    for first in range(positions, n, positions):
        bad = V.clone()
        later = torch.arange(m_max, device=DEV)[None] >= at + first
        bad[..., ::2].masked_fill_(later[..., None], float("nan"))
        bad[..., 1::2].masked_fill_(later[..., None], float("inf"))
        O = attend(Q, K, bad, start)
        assert torch.equal(O[:, :, :first].view(torch.int32), clean[:, :, :first].view(torch.int32)), f"rows from position {first} on"
        assert bool(torch.isnan(O[:, :, first:, ::2]).all()) and not bool(torch.isfinite(O[:, :, first:]).any())


@pytest.mark.parametrize("b,h,n,m_max,start", [
    (1, 4, 16, 2064, 2048), (1, 4, 16, 2064, 1500), (2, 9, 100, 1500, 1400), (1, 3, 128, 1000, 700), (200, 4, 128, 512, 384),
])
def test_a_memory_whose_rows_are_partly_nan_gives_nan(b, h, n, m_max, start):
    """A position that sees a key row of NaN has no finite output, wherever the row lies: also where all that one of several
    CTAs sees of the memory is such rows (and where a position sees nothing else at all)."""
    gen = torch.Generator(device=DEV).manual_seed(m_max)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    for rows in (slice(start // 2, start), slice(0, start // 2), slice(0, start), slice(0, start + n), slice(start // 3, start // 3 + 1)):
        bad = K.clone()
        bad[:, rows] = float("nan")
        assert bool(torch.isnan(attend(Q, bad, V, [start] * b)).all()), f"rows {rows}"
    bad = K.clone()
    bad[:, start + n // 2] = float("nan")                  # a row that only the later positions see
    O, clean = attend(Q, bad, V, [start] * b), attend(Q, K, V, [start] * b)
    assert bool(torch.isnan(O[:, :, n // 2:]).all())
    assert torch.equal(O[:, :, : n // 2].view(torch.int32), clean[:, :, : n // 2].view(torch.int32))


@pytest.mark.parametrize("b,h,n,m_max,start", [
    (1, 4, 16, 2064, 2048), (2, 9, 100, 1500, 1400), (200, 2, 128, 640, 512), (150, 4, 128, 1300, 1172),
])
def test_logits_of_minus_infinity_weigh_nothing(b, h, n, m_max, start):
    """Key rows whose logit is -inf for every query: whole stages of them, first, in the middle and last."""
    gen = torch.Generator(device=DEV).manual_seed(m_max)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    Q[..., 0] = Q[..., 0].abs() + 0.125
    K = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    for rows in (slice(0, 128), slice(0, 300), slice(128, 384), slice(start // 2, start), slice(128, start)):
        K2 = K.clone()
        K2[:, rows, 0] = -float("inf")
        O = attend(Q, K2, V, [start] * b)
        s = Q[0].double() @ K2[0].double().T
        hidden = torch.arange(m_max, device=DEV)[None] > start + torch.arange(n, device=DEV)[:, None]
        ref = torch.softmax(s.masked_fill(hidden, -float("inf")), -1) @ V[0].double()
        check_close(O[0].cpu().numpy(), ref.cpu().numpy(), f"rows {rows}")
    K2 = K.clone()
    K2[..., 0] = -float("inf")                             # nothing else: 0 / 0
    assert bool(torch.isnan(attend(Q, K2, V, [start] * b)).all())


@pytest.mark.parametrize("b,h,n,m_max,start", [
    (1, 1, 1024, 1024, 0), (2, 1, 384, 1100, 640), (3, 1, 300, 1400, 800), (5, 9, 333, 1400, 600), (40, 1, 1024, 1024, 0), (70, 3, 250, 1100, 700),
])
def test_two_roundings_of_the_weights_up_to_the_same_position_on_either_kernel(b, h, n, m_max, start):
    """Positions whose tile's pair begins in a block of 128 that sees fewer than 1024 rows have weights in two bf16 parts: 2^-17 of each,
    1e-6 to 1e-5 of a row of O; one part (2^-9 of each) leaves 5e-4 and more."""
    gen = torch.Generator(device=DEV).manual_seed(n)
    Q = wl.bf16_normal((b, h, n, 128), 128 ** -0.5, gen, DEV)
    K, V = wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV), wl.bf16_normal((b, m_max, 128), 1.0, gen, DEV)
    O = attend(Q, K, V, [start] * b).double()
    hidden = torch.arange(m_max, device=DEV)[None] > start + torch.arange(n, device=DEV)[:, None]
    two = torch.zeros(h, n, dtype=torch.bool)
    # the tiles: of all heads x positions with up to 128 rows the fewest tiles, among equals the most positions; heads' blocks within positions'
    heads = min(range(1, min(h, 128) + 1), key=lambda g: (-(-n // min(128 // g, n)) * -(-h // g), g))
    positions, blocks = min(128 // heads, n), -(-h // heads)
    for tile in range(-(-n // positions) * blocks):
        first = (tile & ~1) // blocks * positions // 128 * 128
        p, g = tile // blocks * positions, tile % blocks * heads
        two[g:g + heads, p:p + positions] = start + min(first + 128, n) < 1024
    assert bool(two.any())
    for i in {0, b - 1}:
        ref = torch.softmax((Q[i].double() @ K[i].double().T).masked_fill(hidden, -float("inf")), -1) @ V[i].double()
        rel = ((O[i] - ref).norm(dim=-1) / ref.norm(dim=-1)).cpu()
        assert float(rel[two].max()) < 1e-4
        assert bool(two.all()) or float(rel[~two].mean()) > 3e-4      # (the border is where it is meant to be)
