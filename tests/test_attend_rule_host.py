"""The choice of lg_decode_attend's pass (csrc/lg_attend_rule.cuh), compiled for the host: which
pass the host chooses from a call's sizes, and which one runs for its lengths where it launches
both."""
import os
import random
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2604_10044_gb300", "csrc")
RESIDENT = "15, 23, 36, 76, 152"  # clusters of each size on a GB300

MAIN = r'''
#include <cstdio>
#include <vector>
#include "lg_attend_rule.cuh"
using namespace lg;
int main() {  // bf16 d g H_kv layers batch max_len S_total chunk_rows lengths...
  int b16, d, g, H, nl, batch, max_len, chunk; long long S;
  const int resident[kNumSizes] = {%s};
  while (std::scanf("%%d %%d %%d %%d %%d %%d %%d %%lld %%d", &b16, &d, &g, &H, &nl, &batch, &max_len, &S,
                    &chunk) == 9) {
    const PassKind kind = {b16 != 0, d, g, b16 ? 128 : g <= 4 ? 64 : 32};
    const int groups = nl * batch * H, chunks = (max_len + chunk - 1) / chunk;
    const float fill = fminf(1.f, (float)S / ((float)batch * (float)max_len));
    const AttendChoice ch = attend_choose(call_shape(kind, groups, max_len, chunk, chunks, 152), batch, fill,
                                          resident);
    std::vector<int> n(batch);
    int rows = 0, total = 0;
    for (int &x : n) {
      if (std::scanf("%%d", &x) != 1) return 1;
      rows = x > rows ? x : rows;
      total += (x + kind.tile_rows - 1) / kind.tile_rows;
    }
    const CallShape s = call_shape(kind, groups, rows, chunk, chunks, 152);
    const bool equal = total == s.tiles * batch;
    const float mean = s.tiles ? (float)total / ((float)batch * (float)s.tiles) : 1.f;
    std::printf("%%d %%d %%d %%d %%g %%g\n", (int)ch.pass, ch.ctas, ch.clusters,
                (int)(general_gains_us(s, batch, total, equal, ch.ctas, ch.clusters) > 0.f),
                cluster_us(s, ch.ctas, ch.clusters, equal, mean), general_us(s, mean, chunks));
  }
}
'''


def _chunk_rows(bf16, d, H, nl, batch, max_len):
    """attend_chunk_rows in csrc/lg_api.cu"""
    tile, target = (128, 152 * 8) if bf16 else (8192 // (d * 4), 152 * 12)
    ch = -(-(-(-max_len * batch * H * nl // target)) // tile) * tile
    return max(tile, min(ch, 4096)) if bf16 else max(2 * tile, min(ch, 2048 // tile * tile))


@pytest.fixture(scope="module")
def rule():
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    with tempfile.TemporaryDirectory() as tmp:
        cpp, exe = os.path.join(tmp, "r.cpp"), os.path.join(tmp, "r")
        open(cpp, "w").write(MAIN % RESIDENT)
        subprocess.run(["g++", "-x", "c++", "-O2", "-std=c++17", "-I" + CSRC, cpp, "-o", exe],
                       check=True)

        def ask(calls):
            """[(dtype, d, g, H_kv, layers, max_len, S_total, lengths)] -> [(pass, CTAs a cluster,
            clusters, whether the general pass runs where both are launched, estimates of both)]"""
            text = []
            for dt, d, g, H, nl, max_len, S, n in calls:
                bf16 = dt == "bf16"
                text.append(" ".join(str(int(x)) for x in [
                    bf16, d, g, H, nl, len(n), max_len, S,
                    _chunk_rows(bf16, d, H, nl, len(n), max_len), *n]))
            out = subprocess.run([exe], input="\n".join(text), capture_output=True, text=True,
                                 check=True).stdout
            rows = [r.split() for r in out.splitlines()]
            assert len(rows) == len(calls)
            return [(["cluster", "general", "either"][int(r[0])], int(r[1]), int(r[2]), r[3] == "1",
                     float(r[4]), float(r[5])) for r in rows]

        yield ask


def _tight(n):
    """a call over sequences without spare rows but one each"""
    return int(max(n)) + 1, int(sum(n)) + len(n), list(n)


def _slots(slot, n):
    return slot, slot * len(n), list(n)


def _ragged(n, b):
    lo = max(1, n // 16)
    return [int(lo * (n / lo) ** ((i * 0.6180339887498949 + 0.9999) % 1.0)) for i in range(b)]


def test_sizes_decide_where_lengths_cannot_matter(rule):
    for want, call in [
            ("cluster", ("bf16", 128, 2, 8, 1, *_tight([1024]))),
            ("cluster", ("bf16", 128, 4, 8, 1, *_tight([4096] * 8))),
            ("cluster", ("bf16", 128, 4, 8, 1, *_slots(4097, [4096, 1, 0, 5, 9, 100, 3, 7]))),
            ("cluster", ("bf16", 128, 4, 8, 1, *_tight(_ragged(16381, 64)))),
            ("cluster", ("bf16", 128, 4, 8, 32, *_tight([4096] * 8))),
            ("cluster", ("f32", 128, 4, 8, 1, *_tight([8191] * 4))),
            ("general", ("bf16", 128, 1, 2, 1, *_tight([131071]))),
            ("general", ("f32", 128, 8, 8, 1, *_tight([9036] * 6)))]:
        got = rule([call])[0]
        assert got[0] == want or (got[0] == "either" and want == "cluster" and not got[3]), \
            (call, got)


def test_lengths_decide_in_equal_slots(rule):
    """one full slot of eight leaves two groups of 1024 tiles, 8 of 2048 in fp32: the general pass is
    the faster, 85 against 110 and 280 against 391 us, and for eight full ones the cluster pass"""
    for dt, g, H in (("bf16", 4, 2), ("f32", 4, 8)):
        full = rule([(dt, 128, g, H, 1, *_slots(131072, [131000] * 8))])[0]
        one = rule([(dt, 128, g, H, 1, *_slots(131072, [131000] + [300] * 7))])[0]
        assert full[:3] == one[:3] and full[0] == "either" and full[1] == 6
        assert not full[3] and one[3], (full, one)


def test_no_lengths_make_the_chosen_pass_much_the_slower(rule):
    """Over random calls in equal or tight slots and random lengths within them, by the estimates: a
    call left to the cluster pass alone is not slower than by the general pass by more than 5 % and
    the 15 us that both would be launched for (2 us on top: the choice looks at 1, 2, 4, ... full
    slots, the lengths here fall between), but for one in a thousand; of both, the faster one runs."""
    rng = random.Random(5)
    li = lambda lo, hi: int(round(np.exp(rng.uniform(np.log(lo), np.log(hi)))))  # noqa: E731
    calls = []
    for _ in range(3000):
        dt, d, H, g = rng.choice(["bf16", "f32"]), rng.choice([64, 128]), rng.choice([1, 2, 4, 8]), \
            rng.randint(1, 8)
        b, n, nl = li(2, 64), li(33, 131071), rng.choice([1, 1, 1, 4])
        for _ in range(6):
            kind = rng.random()
            lens = [n if i < rng.randint(1, b) else li(1, n) for i in range(b)] if kind < .3 else \
                [n] + [li(1, n) if kind < .6 else li(1, min(n, 200)) for _ in range(b - 1)]
            calls.append((dt, d, g, H, nl, *_slots(n, lens)))
        calls.append((dt, d, g, H, nl, *_tight(_ragged(n, b))))
    slower = either = 0
    for call, (which, _, _, general, cl, gen) in zip(calls, rule(calls)):
        if which == "cluster":
            slower += 0.95 * cl > gen + 17
        elif which == "either":
            ran, other = (gen, cl) if general else (cl, gen)
            either += 1
            assert ran < 1.06 * other, (call, cl, gen)
    assert slower <= len(calls) // 1000 and either > 500, (slower, either)
