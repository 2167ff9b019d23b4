"""What this library is timed on: the calls a decoder makes of it, over the range of sizes it makes them at.

Every case goes through the public entry points (the bound calls and checked wrappers of the binding), with inputs drawn as
in ``workloads.py`` (q ~ N(0, 1/k), K, V and the new rows ~ N(0, 1), rounded to bf16).  The kinds of case:

``step``     one decoding step of one layer over the shared cache (``AppendStep``: append the new row, attend, merge), called
             directly, as a decoder without CUDA graphs calls it; heads, or beams x heads, of one to a few hundred rows
``loop``     the paper's timed decoding: a cache that grows from empty by one row per token, the tokens' steps captured once
             as a CUDA graph and replayed for every batch of sentences
``mha``      the multi-head step the multi-query one is compared with: ``kv_cache_append`` and ``mha_decode_step``
``prefill``  the attention of many positions at once: a whole prompt, or a chunk of one over rows that are in the cache
``layer``    one token through the self-attention layers of a decoder, projections included, replayed as a CUDA graph
``local``    the same for layers with local attention (rings of the window's size)

A step leaves ``lens`` (or ``pos``) as it was, so that it can be repeated on the same state; the loop advances them on the
device and begins each pass with an empty cache.
"""
import math

import numpy as np
import torch

import paper_1911_02150_b200 as mqa
from paper_1911_02150_b200 import workloads as wl

LAYERS = 6                  # decoder layers of the paper's models (Section 4.1)
ROW_BYTES = 512             # one cache row: 128 bf16 of K and 128 of V
SINGLE_ROUNDING_ROWS = 1024     # from this prefix length on the weights enter the second product rounded to bf16 once


def listed():
    return [
        # the smallest call of the sweep: one sequence, 16 heads, 512 rows; all latency, on the host and on the GPU
        dict(name="step_single", op="step", b=1, h=16, m=512, ragged=False, chained=True),
        # the paper's decoding (Section 4.3): 128 sequences, 8 heads, a cache growing from 1 to 128 rows over 128 tokens
        dict(name="loop_paper", op="loop", b=128, h=8, m=128),
        # few sequences of middling length, an interactive server: neither latency nor bandwidth alone
        dict(name="step_few", op="step", b=8, h=16, m=4096, ragged=False, chained=True),
        # long context, the workload of the headline number: 32 sequences, 32 heads, full caches of 8192 rows
        dict(name="step_long", op="step", b=32, h=32, m=8192, ragged=False, chained=True),
        # a large batch of sequences of every length up to 2048, as continuous batching makes it
        dict(name="step_ragged", op="step", b=256, h=16, m=2048, ragged=True, chained=True),
        # the largest caches of the sweep: 256 sequences of 32768 rows, 4 GiB read per step
        dict(name="step_large", op="step", b=256, h=16, m=32768, ragged=False, chained=True),
        # beam search (Section 4.2), beam 4 x 32 heads over one shared memory of 8192 rows: 128 query rows per sequence
        dict(name="step_beams", op="step", b=32, h=128, m=8192, ragged=False, chained=True),
        # the multi-head baseline with a cache per head: 64 sequences, 16 heads, 4096 rows, 2 GiB read per step
        dict(name="mha", op="mha", b=64, h=16, m=4096, ragged=False),
        # processing of whole prompts: 32 prompts of 4096 tokens, 32 heads; bound by the tensor cores
        dict(name="prefill_prompts", op="prefill", b=32, h=32, n=4096, m=4096, offset=False),
        # chunked prompt processing: 333 tokens each for 5 sequences somewhere inside their caches; odd heads, ragged tiles
        dict(name="prefill_chunk", op="prefill", b=5, h=9, n=333, m=3000, offset=True),
        # one token through the six attention layers of the paper's decoder (128 sequences, 8 heads, d = 1024, 128 rows)
        dict(name="layers_paper", op="layer", b=128, h=8, d=1024, m=128, ragged=False),
        # the same through six layers of local attention (window 32) for the paper's 1024 sequences
        dict(name="layers_local", op="local", b=1024, h=8, window=32),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "loop", "mha", "mha", "prefill", "prefill", "layer", "layer", "local"])
    if op == "step":
        h = _log_int(rng, 33, 192) if rng.random() < 0.25 else _log_int(rng, 1, 32)      # beams x heads, or heads
        m = _log_int(rng, 256, 32768)
        b = _log_int(rng, 1, max(1, min(512, 256 * 32768 // m)))
        return dict(op=op, b=b, h=h, m=m, ragged=rng.random() < 0.5, chained=rng.random() < 0.75)
    if op == "loop":
        return dict(op=op, b=_log_int(rng, 1, 256), h=_log_int(rng, 1, 32), m=rng.randint(16, 192))
    if op == "mha":
        m = _log_int(rng, 64, 8192)
        h = _log_int(rng, 1, 32)
        b = _log_int(rng, 1, max(1, min(256, 64 * 16 * 4096 // (m * h))))
        return dict(op=op, b=b, h=h, m=m, ragged=rng.random() < 0.5)
    if op == "prefill":
        n = _log_int(rng, 16, 4096)
        offset = rng.random() < 0.5
        m = rng.randint(n, 2 * n + 2048) if offset else n
        most = 32 * 32 * 4096 * 4097 // 2
        units = max(1, int(most / (n * (n + 1) / 2 + n * ((m - n) / 2 if offset else 0))))
        h = _log_int(rng, 1, min(32, units))
        b = _log_int(rng, 1, max(1, min(32, units // h)))
        return dict(op=op, b=b, h=h, n=n, m=m, offset=offset)
    if op == "layer":
        m = _log_int(rng, 32, 8192)
        return dict(op=op, b=_log_int(rng, 1, max(1, min(256, 32 * 8192 // m))), h=_log_int(rng, 1, 32), d=128 * rng.randint(2, 16), m=m,
                    ragged=rng.random() < 0.5)
    return dict(op=op, b=_log_int(rng, 1, 2048), h=_log_int(rng, 1, 32), window=_log_int(rng, 16, 512))


def _lens(case, seed):
    """Rows per sequence BEFORE the step: full caches but for the row the step appends, or uniform lengths."""
    b, m = case["b"], case["m"]
    if case["ragged"]:
        return torch.from_numpy(wl.ragged_lens(b, m, seed) - 1).cuda()
    return torch.full((b,), m - 1, dtype=torch.int32, device="cuda")


def _status():
    return torch.zeros(1, dtype=torch.int32, device="cuda")


def _normal(gen, shape, std):
    return wl.bf16_normal(shape, std, gen, "cuda")


def _captured(work):
    """`work` (which enqueues on the current stream) as a CUDA graph: what a decoder keeps and replays per token."""
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        work()
    return graph


def _prepare_step(case, seed):
    b, h, m = case["b"], case["h"], case["m"]
    x = wl.make_inputs(b, h, m, "mqa", seed=seed, device="cuda")
    lens, o, status = _lens(case, seed), torch.empty(b, h, 128, device="cuda"), _status()
    step = mqa.AppendStep(x["q"], x["K"], x["V"], x["k_new"], x["v_new"], lens, o, mqa.alloc_workspace(b, h, m, "cuda"), status,
                          advance=False, chained=case["chained"])
    return dict(op="step", step=step, x=x, out=dict(o=o, K=x["K"], V=x["V"], lens=lens, status=status))


def _prepare_loop(case, seed):
    b, h, m = case["b"], case["h"], case["m"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, k_new, v_new = _normal(gen, (m, b, h, 128), 128 ** -0.5), _normal(gen, (m, b, 128), 1.0), _normal(gen, (m, b, 128), 1.0)
    K, V = torch.zeros(2, b, m, 128, dtype=torch.bfloat16, device="cuda").unbind(0)
    lens, status = torch.zeros(b, dtype=torch.int32, device="cuda"), _status()
    o, ws = torch.empty(m, b, h, 128, device="cuda"), mqa.alloc_workspace(b, h, m, "cuda")

    def tokens():
        lens.zero_()
        for t in range(m):
            # (the first step follows something that wrote lens: it makes no promise about the work before it)
            mqa.AppendStep(q[t], K, V, k_new[t], v_new[t], lens, o[t], ws, status, chained=t > 0)()

    return dict(op="graph", graph=_captured(tokens), keep=(q, k_new, v_new, ws), out=dict(o=o, K=K, V=V, lens=lens, status=status))


def _prepare_mha(case, seed):
    b, h, m = case["b"], case["h"], case["m"]
    x = wl.make_inputs(b, h, m, "mha", seed=seed, device="cuda")
    lens, o = _lens(case, seed), torch.empty(b, h, 128, device="cuda")
    return dict(op="mha", x=x, lens=lens, lens_after=lens + 1, o=o, ws=mqa.alloc_workspace(b, h, m, "cuda"), status=_status())


def _prepare_prefill(case, seed):
    b, h, n, m = case["b"], case["h"], case["n"], case["m"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    Q, K, V = _normal(gen, (b, h, n, 128), 128 ** -0.5), _normal(gen, (b, m, 128), 1.0), _normal(gen, (b, m, 128), 1.0)
    start = None
    if case["offset"]:
        start = torch.from_numpy(np.random.default_rng(seed).integers(0, m - n + 1, size=b).astype(np.int32)).cuda()
    ws = torch.empty(mqa.prefill_workspace_bytes(b, h, n, m), dtype=torch.uint8, device="cuda")
    return dict(op="prefill", Q=Q, K=K, V=V, start=start, O=torch.empty(b, h, n, 128, device="cuda"), ws=ws, status=_status())


def _prepare_layer(case, seed):
    b, h, d, m = case["b"], case["h"], case["d"], case["m"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ws, status, y = mqa.alloc_layer_workspace(b, h, d, m, "cuda"), _status(), torch.empty(LAYERS, b, d, device="cuda")
    lens = _lens(case, seed)
    layers = []
    for _ in range(LAYERS):
        layers.append((_normal(gen, (b, d), 1.0), _normal(gen, (h, d, 128), (d * 128) ** -0.5), _normal(gen, (d, 128), d ** -0.5),
                       _normal(gen, (d, 128), d ** -0.5), _normal(gen, (h, d, 128), (h * 128) ** -0.5),
                       _normal(gen, (b, m, 128), 1.0), _normal(gen, (b, m, 128), 1.0), lens.clone()))

    def token():
        for i, args in enumerate(layers):
            mqa.mqa_layer_decode_step(*args, y[i], ws, status, advance=False)

    out = dict(y=y, status=status, K=[a[5] for a in layers], V=[a[6] for a in layers])
    return dict(op="graph", graph=_captured(token), keep=(layers, ws), out=out)


def _prepare_local(case, seed):
    b, h, w = case["b"], case["h"], case["window"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pos = torch.from_numpy(np.random.default_rng(seed).integers(0, 4 * w, size=b).astype(np.int32)).cuda()
    status, o = _status(), torch.empty(LAYERS, b, h, 128, device="cuda")
    layers = [(_normal(gen, (b, h, 128), 128 ** -0.5), _normal(gen, (b, w, 128), 1.0), _normal(gen, (b, w, 128), 1.0),
               _normal(gen, (b, 128), 1.0), _normal(gen, (b, 128), 1.0), pos.clone()) for _ in range(LAYERS)]

    def token():
        for i, args in enumerate(layers):
            mqa.mqa_decode_local_step(*args, o[i], status, advance=False)

    out = dict(o=o, status=status, K=[a[1] for a in layers], V=[a[2] for a in layers])
    return dict(op="graph", graph=_captured(token), keep=layers, out=out)


def prepare(case, seed):
    return dict(step=_prepare_step, loop=_prepare_loop, mha=_prepare_mha, prefill=_prepare_prefill, layer=_prepare_layer,
                local=_prepare_local)[case["op"]](case, seed)


def run(state):
    op = state["op"]
    if op == "step":
        state["step"]()
        return state["out"]
    if op == "graph":
        state["graph"].replay()
        return state["out"]
    if op == "mha":
        x = state["x"]
        mqa.kv_cache_append(x["K"], x["V"], x["k_new"], x["v_new"], state["lens"], advance=False, status=state["status"])
        mqa.mha_decode_step(x["q"], x["K"], x["V"], state["lens_after"], state["o"], state["ws"], state["status"])
        return dict(o=state["o"], K=x["K"], V=x["V"], status=state["status"])
    mqa.mqa_prefill_attention(state["Q"], state["K"], state["V"], state["O"], state["ws"], state["start"], state["status"])
    return dict(O=state["O"], status=state["status"])


def _attend(q, K, V, rows):
    """In 64 bits: softmax(q K^T) V over the first `rows` rows of one sequence's cache (q [..., 128]; K, V [m, 128])."""
    K, V = K[:rows].double(), V[:rows].double()
    return torch.softmax(q.double() @ K.T, -1) @ V


def _with_row(cache, new, row):
    """One sequence's cache with the new row in its place (a copy; the given one stays as it is)."""
    cache = cache.clone()
    cache[row] = new.to(cache.dtype)
    return cache


def _exact_step(case, state):
    x, lens = state["x"], state["out"]["lens"].tolist()
    o = torch.stack([_attend(x["q"][i], _with_row(x["K"][i], x["k_new"][i], n), _with_row(x["V"][i], x["v_new"][i], n), n + 1)
                     for i, n in enumerate(lens)])
    return dict(o=o, K=None, V=None, lens=None, status=None)


def _exact_loop(case, state):
    q, k_new, v_new, _ = state["keep"]
    keys, values = k_new.transpose(0, 1).double(), v_new.transpose(0, 1).double()
    o = torch.stack([torch.softmax(q[t].double() @ keys[:, : t + 1].transpose(1, 2), -1) @ values[:, : t + 1] for t in range(case["m"])])
    return dict(o=o, K=None, V=None, lens=None, status=None)


def _exact_mha(case, state):
    x, lens = state["x"], state["lens"].tolist()
    o = torch.empty(case["b"], case["h"], 128, dtype=torch.float64, device="cuda")
    for i, n in enumerate(lens):
        K, V = x["K"][i, :, : n + 1].double(), x["V"][i, :, : n + 1].double()
        K[:, n], V[:, n] = x["k_new"][i].double(), x["v_new"][i].double()
        o[i] = (torch.softmax(x["q"][i].double().unsqueeze(1) @ K.transpose(1, 2), -1) @ V).squeeze(1)
    return dict(o=o, K=None, V=None, status=None)


def _exact_prefill(case, state):
    b, h, n = case["b"], case["h"], case["n"]
    Q, K, V = state["Q"], state["K"], state["V"]
    starts = [0] * b if state["start"] is None else state["start"].tolist()
    O = torch.empty(b, h, n, 128, dtype=torch.float64, device="cuda")
    for i, first in enumerate(starts):
        keys, values = K[i, : first + n].double(), V[i, : first + n].double()
        hidden = torch.ones(n, first + n, dtype=torch.bool, device="cuda").triu(first + 1)
        for g in range(h):
            O[i, g] = torch.softmax((Q[i, g].double() @ keys.T).masked_fill_(hidden, -math.inf), -1) @ values
    return dict(O=O, status=None)


def _exact_layer(case, state):
    y = []
    for x, P_q, P_k, P_v, P_o, K, V, lens in state["keep"][0]:
        x = x.double()
        q, k_new, v_new = torch.einsum("bd,hdk->bhk", x, P_q.double()), x @ P_k.double(), x @ P_v.double()
        o = []
        for i, n in enumerate(lens.tolist()):
            rows, values = K[i, : n + 1].double(), V[i, : n + 1].double()
            rows[n], values[n] = k_new[i], v_new[i]
            o.append(_attend(q[i], rows, values, n + 1))
        y.append(torch.einsum("bhv,hdv->bd", torch.stack(o), P_o.double()))
    return dict(y=torch.stack(y), status=None, K=None, V=None)


def _exact_local(case, state):
    w, o = case["window"], []
    for q, K, V, k_new, v_new, pos in state["keep"]:
        K, V, at = K.double(), V.double(), pos.long()
        each = torch.arange(case["b"], device="cuda")
        K[each, at % w], V[each, at % w] = k_new.double(), v_new.double()
        unused = torch.arange(w, device="cuda") >= (at + 1).clamp(max=w)[:, None]
        s = (q.double() @ K.transpose(1, 2)).masked_fill_(unused[:, None, :], -math.inf)
        o.append(torch.softmax(s, -1) @ V)
    return dict(o=torch.stack(o), status=None, K=None, V=None)


def exact(case, seed):
    """What ``run`` computes for these inputs, in 64 bits and without intermediate roundings; the caches and counters it also
    returns are copies of bytes and whole numbers."""
    by_op = dict(step=_exact_step, loop=_exact_loop, mha=_exact_mha, prefill=_exact_prefill, layer=_exact_layer, local=_exact_local)
    return by_op[case["op"]](case, prepare(case, seed))


def _mean_rows(case):
    return (case["m"] + 1) / 2 if case["ragged"] else case["m"]


def work(case):
    """Bytes: every valid K and V row, q and the new rows in, the new rows and o out, once each (weights and x in, y out for
    a layer).  Flops: 4 k per query row and visible cache row, 2 per weight and sequence in the projections."""
    op, b, h = case["op"], case["b"], case["h"]
    qo, new = b * h * (256 + 512), 2 * b * ROW_BYTES
    if op in ("step", "mha"):
        caches = h if op == "mha" else 1
        rows = b * _mean_rows(case)
        return dict(bytes=caches * (rows * ROW_BYTES + new) + qo, flops=rows * h * 512)
    if op == "loop":
        m = case["m"]
        rows = b * m * (m + 1) / 2
        return dict(bytes=rows * ROW_BYTES + m * (new + qo), flops=rows * h * 512)
    if op == "prefill":
        n, start = case["n"], (case["m"] - case["n"]) / 2 if case["offset"] else 0
        return dict(bytes=n * qo + b * (start + n) * ROW_BYTES, flops=b * h * (n * (n + 1) / 2 + n * start) * 512)
    if op == "layer":
        d, rows = case["d"], b * _mean_rows(case)
        weights = (2 * h + 2) * d * 128
        return dict(bytes=LAYERS * (rows * ROW_BYTES + b * ROW_BYTES + 2 * weights + b * d * (2 + 4)),
                    flops=LAYERS * (rows * h * 512 + 2 * b * weights))
    w = case["window"]
    rows = b * ((w + 1) / 8 + 0.75 * w)                      # tokens in the ring at a position uniform over 0 .. 4 w - 1
    return dict(bytes=LAYERS * (rows * ROW_BYTES + new + qo), flops=LAYERS * rows * h * 512)


def tolerance(case):
    """Four times the error seen against the same case in 64 bits (2-norm, and the largest element): 32-bit sums of exact bf16
    products (mha, 2.9e-7 and 1.6e-6); weights as two bf16 parts for short prefixes (2.3e-6 and 2.0e-5); weights rounded to bf16
    once (1.7e-3 and 1.0e-2); q, the new rows, the weights and the attention's result rounded to bf16 in a layer (2.8e-3 and
    1.5e-2)."""
    if case["op"] == "layer":
        return dict(rel=1.1e-2, max=6e-2)
    if case["op"] == "mha":
        return dict(rel=1.2e-6, max=1e-5)
    if case.get("m", case.get("window")) < SINGLE_ROUNDING_ROWS:
        return dict(rel=1e-5, max=1e-4)
    return dict(rel=7e-3, max=4e-2)
