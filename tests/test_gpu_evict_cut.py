"""The comparators' cut of several rows (lg_h2o_evict, lg_streaming_evict) against a sort in
numpy: every row width, lengths around the kernel's windows of 2048 rows and its tiles, budgets
from two rows over to a few rows, scores that tie (within the recent bound's digits and exactly,
so that positions decide), negative, infinite and zero scores, and slots in another order than
their positions.  Rows, scores and positions move byte for byte; slots past the budget stay."""
import numpy as np
import pytest
import torch

from paper_2604_10044_gb300 import lg

pytestmark = pytest.mark.gpu


def _kept(score, pos, n, B, now, policy):
    """slots kept, ascending: the protected ones and, for H2O, the highest (score, position)"""
    thr = now - (B // 2 if policy == "h2o" else B - lg.N_SINK)
    keep = pos[:n] > thr
    if policy != "h2o":
        return np.flatnonzero(keep | (pos[:n] < lg.N_SINK))
    k = B - int(keep.sum())
    old = np.flatnonzero(~keep)
    if k > 0:
        order = np.lexsort((pos[old], score[old]))
        keep[old[order[len(old) - k:]]] = True
    return np.flatnonzero(keep)


@pytest.mark.parametrize("policy", ["h2o", "streaming"])
@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("bf16", 128), ("f32", 64), ("f32", 128)])
@pytest.mark.parametrize("scores", ["spread", "ties", "zero"])
def test_cut(cuda, policy, dtype, d, scores):
    rng = np.random.default_rng(d + len(scores))
    n = np.array([10, 64, 2047, 2048, 2049, 4100, 6145], dtype=np.int32)
    B = np.array([7, 62, 1024, 2040, 130, 4098, 600], dtype=np.int32)
    cap = n + 3
    off = np.concatenate([[0], np.cumsum(cap)[:-1]]).astype(np.int64)
    S, L, H = int(cap.sum()), 2, 2
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device=cuda)
    g.manual_seed(3)
    k = torch.randn((L, H, S, d), generator=g, device=cuda).to(tdt)
    v = torch.randn((L, H, S, d), generator=g, device=cuda).to(tdt)
    c = lg.Cache(L, H, d, dtype, off, cap, n, cuda, policy=policy, k=k, v=v)
    sc = rng.lognormal(0.0, 2.0, (L, H, S)).astype(np.float32)
    sc[0, 0] *= rng.choice([-1.0, 1.0], S)
    sc[0, 0, ::17] = np.inf
    if scores == "ties":
        sc = np.round(sc * 2).astype(np.float32) / 2 + 0.0
    elif scores == "zero":
        sc[:] = 0.0
    ps = np.full((L, H, S), -1, dtype=np.int32)
    for b in range(len(n)):
        for l in range(L):
            ps[l, 0, off[b]:off[b] + n[b]] = np.arange(n[b]) * 3
            ps[l, 1, off[b]:off[b] + n[b]] = rng.permutation(n[b]) * 3
    if policy == "streaming":
        ps //= 3
    now = np.array([ps[0, 0, o + m - 1] for o, m in zip(off, n)], dtype=np.int32)
    c.h2o.copy_(torch.from_numpy(sc))
    c.pos.copy_(torch.from_numpy(ps))
    k0, v0 = k.cpu().view(torch.uint8), v.cpu().view(torch.uint8)
    bd, nd = torch.from_numpy(B).to(cuda), torch.from_numpy(now).to(cuda)
    if policy == "h2o":
        lg.lg_h2o_evict(c, bd, nd, int(n.max()))
    else:
        lg.lg_streaming_evict(c, bd, nd, lg.N_SINK, int(n.max()))
    assert lg.lg_read_device_status(c) == 0
    assert np.array_equal(c.lengths(), B)
    k1, v1 = c.k.cpu().view(torch.uint8), c.v.cpu().view(torch.uint8)
    s1, p1 = c.h2o.cpu().numpy(), c.pos.cpu().numpy()
    for b in range(len(n)):
        o = int(off[b])
        for l in range(L):
            for h in range(H):
                kept = _kept(sc[l, h, o:o + n[b]], ps[l, h, o:o + n[b]], n[b], B[b],
                             int(now[b]), policy)
                src = np.arange(o, o + cap[b])
                src[:len(kept)] = o + kept
                src = torch.from_numpy(src)
                rows = slice(o, o + int(cap[b]))
                tag = (b, l, h)
                assert torch.equal(k1[l, h, rows], k0[l, h, src]), tag
                assert torch.equal(v1[l, h, rows], v0[l, h, src]), tag
                np.testing.assert_array_equal(s1[l, h, rows], sc[l, h, src.numpy()])
                np.testing.assert_array_equal(p1[l, h, rows], ps[l, h, src.numpy()])
