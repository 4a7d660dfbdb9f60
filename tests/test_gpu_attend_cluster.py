"""The cluster pass of lg_decode_attend (batch up to 64) against a plain fp64 attention and against
the general pass on the same cache: empty sequences appended until the batch passes the cluster
pass's limit send the same call there.

Lengths around its 128-row tiles, empty and one-row sequences, equal lengths (the clusters' runs
known before the lengths) and uneven ones, groups within one CTA, shared by two, by a whole
cluster, and several groups a CTA, every GQA group, both head sizes, several layers a call, and
the H2O logits it leaves for the score update."""
import numpy as np
import pytest
import torch

from paper_2604_10044_gb300 import lg

pytestmark = pytest.mark.gpu

LIMIT = 64  # kClusterSeqs in csrc/lg_attend_cluster.cuh


def _run(k, v, q, lens, layer0, n_layers, suffix_w, h2o, pad, ran="cluster"):
    """out, stats (and scores) of layers [layer0, layer0 + n_layers) over cache rows k, v
    [L][H_kv][S][d]; pad: empty sequences after the real ones; ran: the pass that the call is to run"""
    L, H_kv, S, d = k.shape
    b, H_q = len(lens), q.shape[2]
    cap = np.concatenate([np.asarray(lens) + 1, np.ones(pad, np.int64)]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(cap)[:-1]]).astype(np.int64)
    extra = int(cap.sum()) - S
    kk, vv = (torch.cat([x, torch.full((L, H_kv, extra, d), 3.0, dtype=x.dtype, device=x.device)],
                        2) for x in (k, v))
    n = np.concatenate([lens, np.zeros(pad, np.int64)]).astype(np.int32)
    c = lg.Cache(L, H_kv, d, "bf16" if k.dtype == torch.bfloat16 else "f32", off, cap, n, k.device,
                 "h2o" if h2o else "loopguard", kk, vv)
    g = lg.Guard(c, H_q, policy="h2o" if h2o else "loopguard", n_layers_per_call=n_layers)
    qq = torch.cat([q, torch.ones((n_layers, pad, H_q, d), dtype=q.dtype, device=q.device)], 1)
    out = torch.full((n_layers, b + pad, H_q, d), 7.0, dtype=k.dtype, device=k.device)
    st = torch.full((n_layers, b + pad, H_q, 4), 7.0, dtype=torch.float32, device=k.device)
    ws = _Workspace(c, H_q, n_layers, int(cap.max()), g.ws)
    lg.lg_decode_attend(c, layer0, n_layers, qq.contiguous(), H_q, g.scale, out, st, suffix_w,
                        1 if h2o else 0, int(cap.max()), g.ws)
    assert lg.lg_read_device_status(c) == 0
    if sum(lens):
        assert ws.ran() == ran
    sc = c.h2o[layer0:layer0 + n_layers, :, :S].clone() if h2o else None
    return out[:, :b], st[:, :b], sc, off


class _Workspace:
    """Which pass a call ran, from what it left in its workspace: the general passes write split-K
    partials, its first part, the cluster pass none."""

    MARK = -12345

    def __init__(self, cache, H_q, n_layers, max_len, ws):
        counters = (2 + n_layers * cache.batch * cache.H_kv) * 4
        self.partials = lg.lg_workspace_size(cache, H_q, n_layers, max_len) - -(-counters // 256) * 256
        self.ws = ws.view(torch.int32)
        self.ws.fill_(self.MARK)

    def ran(self):
        part = self.ws[:self.partials // 4]
        return "cluster" if bool((part == self.MARK).all()) else "general"


def _exact(k, v, q, lens, off, layer0, n_layers, suffix_w):
    H_kv, d = k.shape[1], k.shape[3]
    H_q = q.shape[2]
    out = torch.zeros((n_layers, len(lens), H_q, d), dtype=torch.float64, device=k.device)
    st = torch.zeros((n_layers, len(lens), H_q, 4), dtype=torch.float64, device=k.device)
    st[..., 0] = -float("inf")
    for l in range(n_layers):
        for b, n in enumerate(lens):
            if n == 0:
                continue
            rows = slice(int(off[b]), int(off[b]) + int(n))
            K, V = k[layer0 + l, :, rows].double(), v[layer0 + l, :, rows].double()
            z = q[l, b].double().view(H_kv, -1, d) @ K.transpose(1, 2) / np.sqrt(d)
            m = z.amax(-1, keepdim=True)
            e = torch.exp(z - m)
            t = e.sum(-1, keepdim=True)
            a = e / t
            out[l, b] = (a @ V).reshape(H_q, d)
            H = torch.log(t[..., 0]) - (a * (z - m)).sum(-1)
            S = a[..., -min(suffix_w, int(n)):].sum(-1)
            st[l, b] = torch.stack([m[..., 0], t[..., 0], H, S], -1).reshape(H_q, 4)
    return out, st


def _close(got, want, rtol, atol, what):
    got, want = got.double(), want.double()
    fine = torch.isfinite(want)
    assert torch.equal(fine, torch.isfinite(got)), what
    off = (got - want).abs()[fine] - (atol + rtol * want.abs()[fine])
    assert off.numel() == 0 or off.max().item() <= 0, (what, off.max().item())


CASES = [  # lengths, H_kv, G, d, layers of the call
    ([1], 1, 1, 128, 1), ([127], 2, 2, 128, 1), ([128], 8, 2, 128, 1), ([129], 8, 3, 128, 1),
    ([1024], 8, 2, 128, 1), ([1025], 8, 4, 128, 2), ([5000], 1, 8, 128, 1), ([4096], 2, 5, 128, 3),
    ([9000], 8, 8, 128, 1), ([300] * 5, 8, 4, 128, 1), ([640] * 16, 8, 6, 128, 2),
    ([130] * 64, 2, 7, 128, 1), ([0], 8, 2, 128, 1), ([0, 0, 0], 2, 4, 128, 2),
    ([0, 1, 2, 127, 128, 129, 0, 4000, 3], 4, 4, 128, 2), ([4000] + [1] * 63, 8, 4, 128, 1),
    (list(range(0, 1280, 20)), 2, 6, 128, 1), ([2047, 60, 0, 513], 8, 8, 128, 2),
    ([1024], 8, 2, 64, 1), ([777] * 3, 2, 4, 64, 3), ([0, 1500, 64, 63], 4, 8, 64, 2),
    ([3000, 10], 2, 1, 64, 1),
]


@pytest.mark.parametrize("dtype,h2o", [("bf16", False), ("bf16", True), ("f32", False),
                                       ("f32", True)])
@pytest.mark.parametrize("lens,H_kv,G,d,nl", CASES)
def test_cluster_pass(cuda, lens, H_kv, G, d, nl, dtype, h2o):
    assert len(lens) <= LIMIT
    g = torch.Generator(device=cuda)
    g.manual_seed(len(lens) * 1000 + G * 10 + d)
    L, S = nl + 1, int(sum(lens)) + len(lens)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    k, v = (torch.randn((L, H_kv, S, d), generator=g, device=cuda).to(tdt) for _ in range(2))
    k *= 1.5
    q = torch.randn((nl, len(lens), H_kv * G, d), generator=g, device=cuda).to(tdt)
    got, st, sc, off = _run(k, v, q, lens, 1, nl, 50, h2o, 0)
    want, ws = _exact(k, v, q, lens, off, 1, nl, 50)
    # the parity tests' bounds: bf16 output rounding, fp32 sums
    _close(got, want, *((2e-2, 1e-3) if dtype == "bf16" else (1e-4, 1e-5)), "out")
    _close(st, ws, 1e-4, 1e-6, "stats")
    gen, gst, gsc, _ = _run(k, v, q, lens, 1, nl, 50, h2o, LIMIT + 1 - len(lens), "general")
    # bf16: both within 2^-8 of the same value, so they differ by one step at most
    _close(got, gen, 2.0 ** -7 if dtype == "bf16" else 2e-5, 1e-5, "out against the general pass")
    _close(st, gst, 2e-5, 1e-6, "stats against the general pass")
    if h2o:
        _close(sc, gsc, 2e-5, 1e-9, "scores against the general pass")
        # every non-empty sequence adds G to its kv-head's scores
        total, all_ = sc.double().sum(-1), float(G * sum(n > 0 for n in lens))
        assert torch.allclose(total, torch.full_like(total, all_), rtol=1e-5)


@pytest.mark.parametrize("dtype,n0,b,H_kv,G,nl", [
    ("bf16", 126, 1, 8, 2, 1), ("bf16", 254, 3, 2, 4, 2), ("bf16", 1022, 1, 8, 2, 1),
    ("f32", 62, 2, 8, 2, 1), ("f32", 127, 1, 2, 8, 1), ("f32", 190, 1, 4, 3, 2)])
def test_lengths_that_move_beside_the_call(cuda, dtype, n0, b, H_kv, G, nl):
    """The pass looks at the lengths before its dependency wait and copies the tiles it then
    expects; here lg_begin_step, still in flight beside it in a graph, moves the lengths past a
    tile boundary, so that the expectation is dropped on one of the steps."""
    steps, d = 5, 128
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device=cuda)
    gen.manual_seed(n0)
    cap = n0 + steps + 1
    k, v = (torch.randn((nl, H_kv, b * cap, d), generator=gen, device=cuda).to(tdt)
            for _ in range(2))
    q = torch.randn((nl, b, H_kv * G, d), generator=gen, device=cuda).to(tdt)
    off = np.arange(b, dtype=np.int64) * cap
    c = lg.Cache(nl, H_kv, d, dtype, off, [cap] * b, [n0] * b, cuda, k=k, v=v)
    g = lg.Guard(c, H_kv * G, n_layers_per_call=nl)
    out = torch.zeros((steps, nl, b, H_kv * G, d), dtype=tdt, device=cuda)
    st = torch.zeros((steps, nl, b, H_kv * G, 4), device=cuda)

    def run():
        for s in range(steps):
            lg.lg_begin_step(c)
            lg.lg_decode_attend(c, 0, nl, q, H_kv * G, g.scale, out[s], st[s], 64, 0, cap, g.ws)

    side = torch.cuda.Stream(device=cuda)
    with torch.cuda.stream(side):
        run()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
            run()
        for _ in range(3):
            out.zero_()
            c.len.fill_(n0)
            graph.replay()
            side.synchronize()
            assert lg.lg_read_device_status(c) == 0
            for s in range(steps):
                want, ws = _exact(k, v, q, [n0 + s + 1] * b, off, 0, nl, 64)
                _close(out[s], want, *((2e-2, 1e-3) if dtype == "bf16" else (1e-4, 1e-5)), "out")
                _close(st[s], ws, 1e-4, 1e-6, "stats")


@pytest.mark.parametrize("lens,H_kv,G,d", [([40000], 1, 8, 128), ([30001], 2, 4, 128),
                                           ([20000, 9000], 2, 1, 128), ([33000], 2, 6, 64),
                                           ([50000], 2, 2, 64)])
def test_long_fp32_segments_keep_their_precision(cuda, lens, H_kv, G, d):
    """Segments of many times the 32 rows a lane adds up before it puts its sums away: their
    error against 64 bits stays that of short chains.  A sum of n random terms in a chain is off
    by about 2^-24.8 sqrt(n / 2) of its size (a rounding is 2^-24.8 of its value on average), so
    1.4e-7 for each of the 32-row chains, the chain of put-away sums (a dozen to 60 long) and the
    merges of 8 warps and 8 CTAs, 2.4e-7 together with the products' roundings; unbroken chains of
    400 to 2000 rows would give 4.8e-7 to 1.1e-6."""
    g = torch.Generator(device=cuda)
    g.manual_seed(sum(lens))
    S = int(sum(lens)) + len(lens)
    k, v = (torch.randn((1, H_kv, S, d), generator=g, device=cuda) for _ in range(2))
    q = torch.randn((1, len(lens), H_kv * G, d), generator=g, device=cuda)
    got, st, _, off = _run(k, v, q, lens, 0, 1, 64, False, 0)
    want, ws = _exact(k, v, q, lens, off, 0, 1, 64)
    assert ((got.double() - want).norm() / want.norm()).item() < 4e-7
    assert ((st.double() - ws).norm() / ws.norm()).item() < 4e-7


@pytest.mark.parametrize("lens,H_kv,G,d", [([131071, 131071], 8, 8, 128),
                                           ([131071, 131071], 8, 8, 64)])
def test_long_bf16_segments_keep_their_precision(cuda, lens, H_kv, G, d):
    """Segments of some 340 blocks of 16 rows a warp: how far the sums are off 64 bits before the
    output's rounding shows in the share of outputs that are not the correctly rounded 64-bit value.
    For normal values with an error of 4e-6 of their norm, twice what P's two bf16 parts leave, it is
    0.39 % (2.4e-6: 0.25 %, 1.28e-5, as with unbroken chains of matrix products: 1.06 %; by
    simulation); 2.5 standard deviations of 8192 outputs are 0.17 % more.  The statistics stay in
    fp32: chains of 700 rounded additions, 2^-24.8 sqrt(700 / 2) = 6.5e-7."""
    g = torch.Generator(device=cuda)
    g.manual_seed(d)
    S = int(sum(lens)) + len(lens)
    k, v = (torch.randn((1, H_kv, S, d), generator=g, device=cuda, dtype=torch.bfloat16)
            for _ in range(2))
    q = torch.randn((1, len(lens), H_kv * G, d), generator=g, device=cuda, dtype=torch.bfloat16)
    got, st, _, off = _run(k, v, q, lens, 0, 1, 64, False, 0)
    want, ws = _exact(k, v, q, lens, off, 0, 1, 64)
    assert (got != want.bfloat16()).double().mean().item() < 5.6e-3
    for i in range(4):
        assert ((st[..., i].double() - ws[..., i]).norm() / ws[..., i].norm()).item() < 6.5e-7, i


@pytest.mark.parametrize("lens,H_kv,G,d,dtype,h2o,ran", [
    # few long groups, with 8 CTAs each in the cluster pass: the general pass is the faster
    ([131071], 2, 1, 128, "bf16", False, "general"),
    ([60000, 500, 800, 3], 2, 1, 128, "bf16", True, "general"),
    # a CTA's arithmetic bounds the cluster pass over fp32 rows with many heads a group
    ([9036] * 6, 8, 6, 64, "f32", False, "general"),
    ([20000, 700, 0, 5000], 2, 8, 128, "f32", True, "general"),
    # beside them, calls that the cluster pass keeps
    ([9036] * 6, 8, 6, 64, "bf16", False, "cluster"),
    ([20000, 700, 0, 5000], 2, 1, 128, "f32", True, "cluster")])
def test_either_side_of_the_choice(cuda, lens, H_kv, G, d, dtype, h2o, ran):
    g = torch.Generator(device=cuda)
    g.manual_seed(sum(lens) + G)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    S = int(sum(lens)) + len(lens)
    k, v = (torch.randn((1, H_kv, S, d), generator=g, device=cuda).to(tdt) for _ in range(2))
    q = torch.randn((1, len(lens), H_kv * G, d), generator=g, device=cuda).to(tdt)
    got, st, sc, off = _run(k, v, q, lens, 0, 1, 64, h2o, 0, ran)
    want, ws = _exact(k, v, q, lens, off, 0, 1, 64)
    # the parity tests' bounds: bf16 output rounding, fp32 sums
    _close(got, want, *((2e-2, 1e-3) if dtype == "bf16" else (1e-4, 1e-5)), "out")
    _close(st, ws, 1e-4, 1e-6, "stats")
    if h2o:
        total, all_ = sc.double().sum(-1), float(G * sum(n > 0 for n in lens))
        assert torch.allclose(total, torch.full_like(total, all_), rtol=1e-5)


@pytest.mark.parametrize("h2o", [False, True])
@pytest.mark.parametrize("dtype,b,slot,H_kv,G,d,nl", [
    ("bf16", 8, 36000, 4, 6, 64, 1), ("bf16", 8, 46500, 2, 1, 128, 1), ("f32", 4, 15000, 2, 6, 64, 2),
    ("f32", 4, 30001, 1, 5, 128, 1)])
def test_lengths_in_equal_slots_choose_the_pass(cuda, dtype, b, slot, H_kv, G, d, nl, h2o):
    """Few long groups in equal slots: the call gets both passes, of which the one that is the
    faster for the lengths runs, here in one graph whose lengths change from replay to replay (one
    workspace, so that each pass finds what the other left)."""
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device=cuda)
    gen.manual_seed(slot)
    off = np.arange(b, dtype=np.int64) * slot
    k, v = (torch.randn((nl, H_kv, b * slot, d), generator=gen, device=cuda).to(tdt)
            for _ in range(2))
    q = torch.randn((nl, b, H_kv * G, d), generator=gen, device=cuda).to(tdt)
    c = lg.Cache(nl, H_kv, d, dtype, off, [slot] * b, [slot - 1] * b, cuda,
                 "h2o" if h2o else "loopguard", k, v)
    g = lg.Guard(c, H_kv * G, policy="h2o" if h2o else "loopguard", n_layers_per_call=nl)
    out = torch.zeros((nl, b, H_kv * G, d), dtype=tdt, device=cuda)
    st = torch.zeros((nl, b, H_kv * G, 4), device=cuda)
    side = torch.cuda.Stream(device=cuda)
    ws = _Workspace(c, H_kv * G, nl, slot, g.ws)

    def run():
        lg.lg_decode_attend(c, 0, nl, q, H_kv * G, g.scale, out, st, 64, int(h2o), slot, g.ws)

    with torch.cuda.stream(side):
        run()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
            run()
        for lens, ran in [([slot - 1] * b, "cluster"), ([slot - 1] + [100] * (b - 1), "general"),
                          ([0, 1] + [100] * (b - 3) + [slot - 1], "general"),
                          ([slot // 2] * b, "cluster"), ([0, slot] + [3] * (b - 2), "general"),
                          ([0] * b, "none"), ([100] * (b - 1) + [slot], "general")]:
            ws.ws[:ws.partials // 4].fill_(ws.MARK)
            out.fill_(7.0)
            st.fill_(7.0)
            c.len.copy_(torch.as_tensor(np.asarray(lens, np.int32), device=cuda))
            if h2o:
                c.h2o.zero_()
            graph.replay()
            side.synchronize()
            assert lg.lg_read_device_status(c) == 0
            if ran != "none":
                assert ws.ran() == ran, lens
            want, wst = _exact(k, v, q, lens, off, 0, nl, 64)
            _close(out, want, *((2e-2, 1e-3) if dtype == "bf16" else (1e-4, 1e-5)), "out")
            _close(st, wst, 1e-4, 1e-6, "stats")
            if h2o:
                total, all_ = c.h2o.double().sum(-1), float(G * sum(n > 0 for n in lens))
                assert torch.allclose(total, torch.full_like(total, all_), rtol=1e-5)
