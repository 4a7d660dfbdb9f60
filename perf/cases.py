"""What a user of the decode-path library has it do, as measurable cases.

A case names a `kind` and its sizes:

  layer       one layer of a model's forward pass at one decode step: the new row joins the cache
              and the layer's queries attend over it (lg_append, lg_decode_attend)
  step        one whole guarded decode step of a cache at its budget (lg_begin_step, appends,
              attention, lg_detect_prune; a budget cut every 65 steps or so)
  prune       the retained set and its compaction on sequences over their budget, half of them
              on a trigger with a repetitive span (lg_prune_compact)
  prefill     the monitor's sketches of a prompt's rows, after a prefill (Cache.prepare)
  comparator  one whole decode step of the H2O or StreamingLLM policy at its budget
  cut         the comparators' first cut of a prompt to the budget (lg_h2o_evict,
              lg_streaming_evict), with the scores a prefill accumulated
  token       the token-level monitor with its retained set (lg_token_detect_prune)

Keys and values are normal with a scale per (layer, kv-head) drawn from U(0.5, 2), as in the
repository's synthetic workloads; queries are normal, so the attention is neither flat nor
collapsed and the loop votes stay quiet on `step`, whose decode is a healthy one.
"""
import math

import numpy as np
import torch

from paper_2604_10044_gb300 import lg

DEV = "cuda:0"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one layer of the 1.7B-class model at one sequence and the paper's
        # budget of 1024 rows; launches and latency are all of it
        dict(name="layer_b1", kind="layer", H_q=16, H_kv=8, d=128, dtype="bf16", batch=1,
             n=1024, ragged=False),
        # an ordinary serving layer: 8B-class heads, 8 sequences at a budget of 4096
        dict(name="layer_b8", kind="layer", H_q=32, H_kv=8, d=128, dtype="bf16", batch=8,
             n=4096, ragged=False),
        # continuous batching: 64 sequences of log-uniform lengths, odd ones among them
        dict(name="layer_ragged_b64", kind="layer", H_q=32, H_kv=8, d=128, dtype="bf16",
             batch=64, n=16381, ragged=True),
        # long context, 8 query heads to a kv-head, two sequences
        dict(name="layer_long_b2", kind="layer", H_q=64, H_kv=8, d=128, dtype="bf16", batch=2,
             n=131071, ragged=False),
        # a caller that keeps its cache in fp32
        dict(name="layer_f32_b4", kind="layer", H_q=32, H_kv=8, d=128, dtype="f32", batch=4,
             n=8191, ragged=False),
        # the paper's setting as an engine runs it: 28 layers called one by one at one sequence,
        # the whole step captured as a CUDA graph and replayed
        dict(name="step_b1_graph", kind="step", L=28, H_q=16, H_kv=8, d=128, dtype="bf16",
             batch=1, n=1024, ragged=False, per_layer=True, graph=True),
        # the 8B-class model's step over a batch of 8, every layer in one attention call: the
        # largest case
        dict(name="step_b8", kind="step", L=32, H_q=32, H_kv=8, d=128, dtype="bf16", batch=8,
             n=4096, ragged=False, per_layer=False, graph=False),
        # prompts of 32768 rows brought to a budget of 8192 (small model, 2 kv-heads)
        dict(name="prune_32k", kind="prune", L=14, H_kv=2, d=128, dtype="bf16", batch=8,
             n=32769, budget=8192, ragged=False),
        # the sketches of eight prompts of 32768 rows
        dict(name="prefill_32k", kind="prefill", H_kv=8, d=128, dtype="bf16", batch=8, n=32768,
             ragged=False),
        # the H2O comparator's decode step on a ragged batch
        dict(name="step_h2o_b16", kind="comparator", policy="h2o", L=4, H_q=32, H_kv=8, d=128,
             dtype="bf16", batch=16, n=8191, ragged=True),
        # the H2O comparator's cut of eight prompts to half their length
        dict(name="cut_h2o_8k", kind="cut", policy="h2o", L=8, H_kv=8, d=128, dtype="bf16",
             batch=8, n=8193, budget=4096, ragged=False),
        # the token-level monitor over a batch of 32 sequences, half of them in a loop
        dict(name="token_b32", kind="token", L=4, H_kv=8, d=128, dtype="bf16", batch=32,
             budget=1024),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


CAP = 2 << 30  # K/V bytes of a drawn case at most


def _fit(batch, n, row_bytes, lo=1):
    """batch and rows brought under CAP"""
    while batch * n * row_bytes > CAP:
        if batch > 1:
            batch = (batch + 1) // 2
        else:
            n = max(lo, n // 2)
    return batch, n


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "step", "prune", "prefill", "comparator",
                       "cut", "token"])
    H_kv = rng.choice([2, 4, 8])
    d = rng.choice([64, 128, 128])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    row = 2 * H_kv * d * (2 if dtype == "bf16" else 4)  # K and V bytes of a row of one layer
    ragged = rng.random() < 0.5
    if kind == "layer":
        batch, n = _fit(_logint(rng, 1, 64), _logint(rng, 33, 131071), row)
        return dict(kind=kind, H_q=H_kv * rng.randint(1, 8), H_kv=H_kv, d=d, dtype=dtype,
                    batch=batch, n=n, ragged=ragged)
    L = rng.randint(1, 16)
    if kind == "step":
        batch, n = _fit(_logint(rng, 1, 16), _logint(rng, 160, 16384), row * L, 160)
        return dict(kind=kind, L=L, H_q=H_kv * rng.randint(1, 8), H_kv=H_kv, d=d, dtype=dtype,
                    batch=batch, n=n, ragged=False, per_layer=rng.random() < 0.5,
                    graph=rng.random() < 0.5)
    if kind == "comparator":
        batch, n = _fit(_logint(rng, 1, 32), _logint(rng, 160, 16384), row * L, 160)
        return dict(kind=kind, policy=rng.choice(["h2o", "h2o", "streaming"]), L=L,
                    H_q=H_kv * rng.randint(1, 8), H_kv=H_kv, d=d, dtype=dtype, batch=batch, n=n,
                    ragged=ragged)
    if kind == "prefill":
        batch, n = _fit(_logint(rng, 1, 32), _logint(rng, 128, 65536), row)
        return dict(kind=kind, H_kv=H_kv, d=d, dtype=dtype, batch=batch, n=n, ragged=ragged)
    if kind == "token":
        return dict(kind=kind, L=rng.randint(1, 4), H_kv=8, d=128, dtype="bf16",
                    batch=_logint(rng, 1, 32), budget=rng.choice([512, 1024, 2048]))
    batch, n = _fit(_logint(rng, 1, 16), _logint(rng, 512, 65536), row * L, 512)
    budget = max(256, int(n * rng.uniform(0.2, 0.9)))
    c = dict(kind=kind, L=L, H_kv=H_kv, d=d, dtype=dtype, batch=batch, n=n, budget=budget,
             ragged=ragged)
    if kind == "cut":
        c["policy"] = rng.choice(["h2o", "h2o", "streaming"])
    return c


# ------------------------------------------------------------------ inputs

def _lengths(case):
    """rows of each sequence: all n, or spread log-uniformly over [n / 16, n]"""
    n, b = case["n"], case["batch"]
    if not case["ragged"]:
        return np.full(b, n, dtype=np.int32)
    lo = max(1, n // 16)
    u = (np.arange(b) * 0.6180339887498949 + 0.9999) % 1.0
    return np.floor(lo * (n / lo) ** u + 1e-9).astype(np.int32)


def _esize(case):
    return 2 if case["dtype"] == "bf16" else 4


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(g, shape, case):
    return torch.randn(shape, generator=g, device=DEV,
                       dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)


def _kv(g, case, L, S):
    """K and V [L][H_kv][S][d] with a scale per (layer, kv-head)"""
    kv = []
    for _ in range(2):
        x = _normal(g, (L, case["H_kv"], S, case["d"]), case)
        x *= torch.rand((L, case["H_kv"], 1, 1), generator=g, device=DEV).mul_(1.5).add_(
            0.5).to(x.dtype)
        kv.append(x)
    return kv


def _rows(case):
    """(lengths in the cache before the pass, slots of each sequence, first slot of each)"""
    n = _lengths(case)
    if case["kind"] in ("layer", "step"):
        held, cap = n - 1, n + 1          # the pass adds a row
    else:
        held, cap = n, n + 1
    if case["kind"] == "step":
        held = held - min(20, case["n"] // 8)  # some steps before the next budget cut
    return held, cap, np.concatenate([[0], np.cumsum(cap.astype(np.int64))[:-1]])


def _step_inputs(g, case, L):
    b = case["batch"]
    return (_normal(g, (L, b, case["H_q"], case["d"]), case),
            _normal(g, (L, b, case["H_kv"], case["d"]), case),
            _normal(g, (L, b, case["H_kv"], case["d"]), case))


def _attention_inputs(case, seed):
    """everything the attention of one pass reads, from the seed"""
    g = _gen(seed)
    L = case.get("L", 1)
    held, cap, off = _rows(case)
    k, v = _kv(g, case, L, int(cap.sum()))
    q, kn, vn = _step_inputs(g, case, L)
    scores = None
    if case["kind"] == "comparator":
        scores = torch.rand((L, case["H_kv"], int(cap.sum())), generator=g, device=DEV) * 8.0
    return held, cap, off, k, v, q, kn, vn, scores


class _State:
    pass


def _cache(case, L, held, cap, off, k, v, policy="loopguard"):
    return lg.Cache(L, case["H_kv"], case["d"], case["dtype"], off, cap, held, DEV, policy, k, v)


def _prepare_attention(case, seed):
    s = _State()
    s.case, kind, L = case, case["kind"], case.get("L", 1)
    held, cap, off, k, v, s.q, s.kn, s.vn, scores = _attention_inputs(case, seed)
    policy = case.get("policy", "loopguard")
    c = s.cache = _cache(case, L, held, cap, off, k, v, policy)
    s.p = lg.lg_default_params()
    c.prepare(int(held.max()), s.p)
    one_by_one = kind == "layer" or case.get("per_layer")
    s.g = lg.Guard(c, case["H_q"], s.p, policy=policy, n_layers_per_call=1 if one_by_one else L)
    s.budget = torch.as_tensor(_lengths(case), device=DEV)
    if kind == "layer":
        lg.lg_begin_step(c)  # the step has reserved the new row's slot
    if kind == "comparator":
        c.h2o.copy_(scores)
        s.pos = torch.as_tensor(held - 1, device=DEV)
    if case.get("graph"):
        side = torch.cuda.Stream(device=DEV)
        with torch.cuda.stream(side):
            held_d = c.len.clone()
            _guarded_step(s)          # loads every kernel before the capture
            c.len.copy_(held_d)
            s.g.dstate.zero_()
            lg.lg_state_init(c, s.g.state, 64)
            side.synchronize()
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph, stream=side, capture_error_mode="thread_local"):
                _guarded_step(s)
            side.synchronize()
    return s


def _guarded_step(s):
    c, g, case = s.cache, s.g, s.case
    if not case["per_layer"]:
        g.step(s.q, s.kn, s.vn, s.budget)
        return
    lg.lg_begin_step(c)
    for l in range(c.L):
        lg.lg_append(c, l, 1, s.kn[l], s.vn[l], None, s.p)
        lg.lg_decode_attend(c, l, 1, s.q[l], case["H_q"], g.scale, g.out[l], g.stats[l],
                            s.p.suffix_w, 0, g.max_len, g.ws)
    lg.lg_detect_prune(c, g.stats, case["H_q"], g.state, s.budget, s.p, g.flags, g.spans, None,
                       g.dstate, g.kept_idx, g.kept_count, g.max_keep, g.max_len)


def _span(n):
    """rows of the repetitive tail of a sequence of n rows that triggered"""
    return np.clip(n // 16, 16, 3072).astype(np.int32)


def _moved(n, B, span):
    """rows of the retained set that change their slot (a budget cut with span 0)"""
    top = min(B // 2, n - 32)                        # W^recent: the last rows
    between = max(0, n - 32 - top)                   # the lattice's rows
    lattice = min(between, B - min(64, B // 4) - 32 - B // 4)
    j = np.arange(lattice, dtype=np.int64)
    rows = j * between // max(lattice, 1) if between > lattice else j
    recent = min(B // 4, top - min(span, top))
    first = n - span - recent                        # slot of the first recent row kept
    return int((rows != j).sum()) + (recent if first != 32 + lattice else 0)


def _prepare_prune(case, seed):
    s = _State()
    s.case = case
    g = _gen(seed)
    n, cap, off = _rows(case)
    k, v = _kv(g, case, case["L"], int(cap.sum()))
    c = s.cache = _cache(case, case["L"], n, cap, off, k, v)
    s.p = lg.lg_default_params()
    c.prepare(int(n.max()), s.p)
    s.n = c.len.clone()
    b = case["batch"]
    s.flags = torch.zeros(b, dtype=torch.int32, device=DEV)
    s.spans = torch.zeros((b, 2), dtype=torch.int32, device=DEV)
    s.flags[::2] = 1
    s.spans[::2, 0] = s.n[::2] - torch.as_tensor(_span(n[::2]), device=DEV)
    s.spans[::2, 1] = s.n[::2]
    s.state = torch.zeros((b, lg.STATE_BYTES // 4), dtype=torch.int32, device=DEV)
    lg.lg_state_init(c, s.state)
    s.budget = torch.full((b,), case["budget"], dtype=torch.int32, device=DEV)
    s.max_len = int(n.max())
    s.kept_idx = torch.zeros((b, s.max_len), dtype=torch.int32, device=DEV)
    s.kept_count = torch.zeros(b, dtype=torch.int32, device=DEV)
    return s


def _prepare_prefill(case, seed):
    s = _State()
    s.case = case
    n, cap, off = _rows(case)
    k, v = _kv(_gen(seed), case, 1, int(cap.sum()))
    s.cache = _cache(case, 1, n, cap, off, k, v)
    s.p = lg.lg_default_params()
    s.max_len = int(n.max())
    return s


def _prepare_cut(case, seed):
    s = _State()
    s.case = case
    g = _gen(seed)
    n, cap, off = _rows(case)
    k, v = _kv(g, case, case["L"], int(cap.sum()))
    c = s.cache = _cache(case, case["L"], n, cap, off, k, v, case["policy"])
    # accumulated attention of a prefill: heavy-tailed over the rows
    s.scores = torch.randn(c.h2o.shape, generator=g, device=DEV).mul_(1.5).exp_()
    s.n = c.len.clone()
    s.budget = torch.as_tensor(np.minimum(n, case["budget"]).astype(np.int32), device=DEV)
    s.pos_now = s.n - 1
    s.max_len = int(n.max())
    return s


TOKEN_STEPS = 509  # token bank: as many steps, then the same again


def _prepare_token(case, seed):
    s = _State()
    s.case = case
    g = _gen(seed)
    b, B = case["batch"], case["budget"]
    cap = np.full(b, B + 1, dtype=np.int32)
    off = np.arange(b, dtype=np.int64) * (B + 1)
    # sequences come to their budgets at different steps
    held = (B - 1 - (np.arange(b) * 37) % 64).astype(np.int32)
    k, v = _kv(g, case, case["L"], int(cap.sum()))
    c = s.cache = _cache(case, case["L"], held, cap, off, k, v)
    s.p = lg.lg_default_params()
    s.tp = lg.lg_default_token_params()
    c.prepare(int(held.max()), s.p)
    tok = torch.randint(0, 50000, (TOKEN_STEPS, b), generator=g, device=DEV, dtype=torch.int32)
    pm = torch.rand((TOKEN_STEPS, b), generator=g, device=DEV) * 0.6 + 0.2
    t = torch.arange(TOKEN_STEPS, device=DEV)
    for i in range(0, b, 2):  # every other sequence repeats a period of 16 to 64 tokens
        P = 16 + (i * 29) % 49
        tok[:, i] = tok[t % P, i]
        pm[:, i] = 0.95
    s.tok, s.pm, s.t = tok, pm, 0
    s.state = torch.zeros((b, lg.STATE_BYTES // 4), dtype=torch.int32, device=DEV)
    lg.lg_state_init(c, s.state, 0)
    s.tstate = torch.zeros(lg.lg_token_state_size(c, s.p, s.tp) // 4, dtype=torch.int32,
                           device=DEV)
    s.flags = torch.zeros(b, dtype=torch.int32, device=DEV)
    s.spans = torch.zeros((b, 2), dtype=torch.int32, device=DEV)
    s.budget = torch.full((b,), B, dtype=torch.int32, device=DEV)
    s.kept_idx = torch.zeros((b, B + 1), dtype=torch.int32, device=DEV)
    s.kept_count = torch.full((b,), -1, dtype=torch.int32, device=DEV)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("layer", "step", "comparator"):
        return _prepare_attention(case, seed)
    return {"prune": _prepare_prune, "prefill": _prepare_prefill, "cut": _prepare_cut,
            "token": _prepare_token}[kind](case, seed)


# ------------------------------------------------------------------ one pass

def run(s):
    case, c = s.case, s.cache
    kind = case["kind"]
    if kind == "layer":
        g = s.g
        lg.lg_append(c, 0, 1, s.kn, s.vn, None, s.p)
        lg.lg_decode_attend(c, 0, 1, s.q, case["H_q"], g.scale, g.out, g.stats, s.p.suffix_w, 0,
                            g.max_len, g.ws)
        return dict(out=g.out, stats=g.stats, k=c.k, v=c.v, sketch=c.sketch, len=c.len)
    if kind == "step":
        g = s.g
        if case["graph"]:
            s.graph.replay()
        else:
            _guarded_step(s)
        return dict(out=g.out, stats=g.stats, k=c.k, v=c.v, sketch=c.sketch, len=c.len,
                    flags=g.flags, spans=g.spans, state=g.state, kept_idx=g.kept_idx,
                    kept_count=g.kept_count)
    if kind == "prune":
        c.len.copy_(s.n)  # the sequences are over their budgets again
        lg.lg_prune_compact(c, s.flags, s.spans, s.state, s.budget, s.p, s.kept_idx,
                            s.kept_count, s.max_len, s.max_len)
        return dict(k=c.k, v=c.v, sketch=c.sketch, len=c.len, kept_idx=s.kept_idx,
                    kept_count=s.kept_count)
    if kind == "prefill":
        c.prepare(s.max_len, s.p)
        return dict(sketch=c.sketch)
    if kind == "comparator":
        s.pos.add_(1)
        s.g.step(s.q, s.kn, s.vn, s.budget, s.pos)
        return dict(out=s.g.out, stats=s.g.stats, k=c.k, v=c.v, len=c.len, h2o=c.h2o, pos=c.pos)
    if kind == "cut":
        c.len.copy_(s.n)  # prompts of full length again, positions in order, prefill scores
        c.prepare(s.max_len)
        c.h2o.copy_(s.scores)
        if case["policy"] == "h2o":
            lg.lg_h2o_evict(c, s.budget, s.pos_now, s.max_len)
        else:
            lg.lg_streaming_evict(c, s.budget, s.pos_now, lg.N_SINK, s.max_len)
        return dict(k=c.k, v=c.v, len=c.len, h2o=c.h2o, pos=c.pos)
    t = s.t
    s.t = (t + 1) % TOKEN_STEPS
    lg.lg_begin_step(c)
    lg.lg_token_detect_prune(c, s.tok[t], s.pm[t], s.state, s.budget, s.p, s.tp, s.flags,
                             s.spans, None, s.tstate, s.kept_idx, s.kept_count, case["budget"] + 1,
                             case["budget"] + 1)
    return dict(k=c.k, v=c.v, sketch=c.sketch, len=c.len, flags=s.flags, spans=s.spans,
                state=s.state, tstate=s.tstate, kept_count=s.kept_count)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind, L, H_kv, d, b = case["kind"], case.get("L", 1), case["H_kv"], case["d"], case["batch"]
    row = 2 * H_kv * d * _esize(case)  # K and V of one row of one layer
    if kind in ("layer", "step", "comparator"):
        held, _, _ = _rows(case)
        rows = int((held + 1).sum()) if kind != "comparator" else int(held.sum()) + b
        head = d * _esize(case)
        byt = L * (rows * row + 2 * b * row + b * case["H_q"] * (2 * head + 16))
        if kind == "comparator" and case["policy"] == "h2o":
            byt += L * H_kv * rows * (4 + 4 + 4)   # score read and written, position read
        if kind == "step":
            byt += b * 256 * H_kv * d // 8         # the monitor's window of sketches
        return dict(bytes=byt, flops=4 * L * rows * case["H_q"] * d)
    if kind == "token":
        return dict(bytes=b * (2 * 256 + 129) * 4, flops=0)
    n = _lengths(case).astype(np.int64)
    if kind == "prefill":
        return dict(bytes=int(n.sum()) * (row // 2 + H_kv * d // 8), flops=0)
    B = case["budget"]
    if kind == "prune":
        kept = sum(_moved(int(x), B, int(_span(x)) if i % 2 == 0 else 0)
                   for i, x in enumerate(n) if i % 2 == 0 or x > B)
        return dict(bytes=2 * kept * (L * row + H_kv * d // 8), flops=0)
    over = n > B
    kept = B * int(over.sum())
    # kept rows, scores and positions read and written, the other scores and positions read
    return dict(bytes=L * (2 * kept * (row + 8 * H_kv) + int((n[over] - B).sum()) * 8 * H_kv),
                flops=0)


def tolerance(case):
    if case["kind"] in ("prune", "prefill", "cut", "token"):
        return "exact"  # copies, bits and counts
    if case["dtype"] == "bf16":
        # sums in another order, the output rounded to bf16: a flipped last bit is 2^-8 of a value
        return dict(rel=1e-3, max=1e-2, differ=1e-4)
    return dict(rel=4e-6, max=1e-4, differ=1e-4)


# ------------------------------------------------------------------ the same in 64 bits

def exact(case, seed):
    if case["kind"] not in ("layer", "step", "comparator"):
        return None
    L, b, H_kv, H_q, d = case.get("L", 1), case["batch"], case["H_kv"], case["H_q"], case["d"]
    held, cap, off, k, v, q, kn, vn, scores = _attention_inputs(case, seed)
    g, scale, W = H_q // H_kv, 1.0 / math.sqrt(d), lg.lg_default_params().suffix_w
    out = torch.empty((L, b, H_q, d), dtype=torch.float64, device=DEV)
    stats = torch.empty((L, b, H_q, 4), dtype=torch.float64, device=DEV)
    h2o = None
    if case.get("policy") == "h2o":
        h2o = scores.double()
    for l in range(L):
        for s in range(b):
            o, n = int(off[s]), int(held[s]) + 1
            K = torch.cat([k[l, :, o:o + n - 1], kn[l, s][:, None]], 1).double()
            V = torch.cat([v[l, :, o:o + n - 1], vn[l, s][:, None]], 1).double()
            z = q[l, s].double().view(H_kv, g, d) @ K.transpose(1, 2) * scale  # [H_kv][g][n]
            m = z.max(-1, keepdim=True).values
            e = torch.exp(z - m)
            tot = e.sum(-1, keepdim=True)
            a = e / tot
            out[l, s] = (a @ V).view(H_q, d)
            H = torch.log(tot[..., 0]) - (a * (z - m)).sum(-1)
            stats[l, s] = torch.stack([m[..., 0], tot[..., 0], H, a[..., -min(W, n):].sum(-1)],
                                      -1).view(H_q, 4)
            if h2o is not None:
                h = h2o[l, :, o:o + n]
                h[:, n - 1] = 0.0
                h += a.sum(1)
                # the lowest score older than the recent half leaves; the last row takes its slot
                B = n - 1
                old = h[:, :n - B // 2]
                x = old.argmin(-1)
                h[torch.arange(H_kv, device=DEV), x] = h[:, n - 1]
    res = dict(out=out, stats=stats, k=None, v=None, len=None)
    if case["kind"] == "comparator":
        return dict(res, h2o=h2o, pos=None)
    res.update(sketch=None)
    if case["kind"] == "step":
        res.update(flags=None, spans=None, state=None, kept_idx=None, kept_count=None)
    return res
