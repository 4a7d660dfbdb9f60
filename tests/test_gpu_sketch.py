"""lg_sketch_build against the sign bits of the guard layer's V rows, word by word: every row
width of the kernel's loads, kv-head counts around its eight loads a warp, lengths around its
rows a load and a second CTA, and no word touched past a sequence's length."""
import numpy as np
import pytest
import torch

from paper_2604_10044_gb300 import lg

pytestmark = pytest.mark.gpu

LENS = [0, 1, 2, 3, 5, 31, 64, 129, 1031]


@pytest.mark.parametrize("dtype,d,H_kv", [("bf16", 128, 1), ("bf16", 128, 8), ("bf16", 128, 5),
                                          ("bf16", 64, 2), ("bf16", 64, 6), ("f32", 128, 3),
                                          ("f32", 128, 8), ("f32", 64, 2), ("f32", 64, 10)])
def test_sketch_build(cuda, dtype, d, H_kv):
    cap = np.array([n + 2 for n in LENS], dtype=np.int32)
    off = np.concatenate([[0], np.cumsum(cap)[:-1]]).astype(np.int64)
    g = torch.Generator(device=cuda)
    g.manual_seed(H_kv * d)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    v = torch.randn((2, H_kv, int(cap.sum()), d), generator=g, device=cuda).to(tdt)
    v[1, :, :, 3] = -0.0  # the raw sign bit counts
    cache = lg.Cache(2, H_kv, d, dtype, off, cap, np.array(LENS, dtype=np.int32), cuda,
                     k=torch.zeros_like(v), v=v)
    cache.sketch.fill_(-7)
    lg.lg_sketch_build(cache, lg.lg_default_params(guard_layer=1), max(LENS))
    assert lg.lg_read_device_status(cache) == 0
    got = cache.sketch.cpu().numpy().view(np.uint32)
    rows = v[1].permute(1, 0, 2).reshape(int(cap.sum()), H_kv * d)
    bits = torch.signbit(rows).cpu().numpy().astype(np.uint64)
    want = (bits.reshape(len(rows), -1, 32) << np.arange(32, dtype=np.uint64)).sum(-1)
    for o, n, c in zip(off, LENS, cap):
        np.testing.assert_array_equal(got[o:o + n], want[o:o + n].astype(np.uint32))
        assert (got[o + n:o + c].view(np.int32) == -7).all()
