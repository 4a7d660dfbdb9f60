"""The cluster pass's bookkeeping (quick_div, TileSpace, run_bound in csrc/lg_attend_cluster.cuh),
compiled for the host from the kernel's own source text, over random batches with empty and
uneven sequences: quotients exact over their range with the float division off by two units in
the last place either way; tiles found in their groups; clusters' runs and their CTAs' ranges that cover
every tile once, runs of whole groups."""
import os
import re
import shutil
import subprocess
import tempfile

import pytest

from test_attend_geometry_host import _block

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2604_10044_gb300", "csrc", "lg_attend_cluster.cuh")

HARNESS = r'''
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <algorithm>
#include <random>
#include <vector>
#define __device__
#define __forceinline__ inline
using std::max; using std::min;
constexpr int kClusterSeqs = 64, kMaxCluster = 8;
static int g_ulp = 0;  // error of the float division, units in the last place
static inline float __fdividef(float a, float b) {
  float q = a / b;
  for (int i = 0; i < std::abs(g_ulp); ++i) q = std::nextafter(q, g_ulp > 0 ? INFINITY : -INFINITY);
  return q < 0 ? 0 : q;
}
%(code)s
static int fails = 0;
#define CHECK(c, ...) do { if (!(c) && fails++ < 10) { std::printf(__VA_ARGS__); std::printf("\n"); } } while (0)
int main() {
  std::mt19937_64 rng(1);
  auto pick = [&](long long lo, long long hi) { return lo + (long long)(rng() %% (unsigned long long)(hi - lo + 1)); };
  for (g_ulp = -2; g_ulp <= 2; ++g_ulp)
    for (int it = 0; it < 400000; ++it) {
      const int d = (int)pick(1, it %% 2 ? 200 : 1 << 20);
      const long long x = pick(0, std::min((1LL << 24) - 1, ((long long)d << 20) - 1));
      CHECK(quick_div((int)x, d) == x / d, "quick_div %%lld / %%d", x, d);
    }
  for (int it = 0; it < 4000; ++it) {
    g_ulp = (int)pick(-2, 2);
    const int batch = (int)pick(1, 64), H_kv = (int)pick(1, 8), L = (int)pick(1, 6);
    std::vector<int> len(batch), pre(batch);
    int total = 0;
    const int rows = it %% 2 ? 128 : 32;
    const int top = (int)pick(1, it %% 3 ? 3000 : 60000);
    for (int b = 0; b < batch; ++b) {
      len[b] = pick(0, 3) ? (int)pick(0, top) : 0;
      pre[b] = total;
      total += (len[b] + rows - 1) / rows;
    }
    TileSpace ts{len.data(), pre.data(), batch, H_kv, L, total, rows};
    const int T = total * H_kv * L;
    if (T == 0 || T >= 1 << 20) continue;
    TileGroup g = ts.find(0);
    std::vector<int> starts;  // group starts, walked
    for (int t = 0; t < T;) {
      CHECK(g.start == t && g.tiles > 0 && g.tiles == ts.tiles(g.b), "walk at %%d", t);
      for (int x : {t, t + g.tiles / 2, t + g.tiles - 1}) {
        const TileGroup f = ts.find(x);
        CHECK(f.start == g.start && f.lloc == g.lloc && f.b == g.b && f.kvh == g.kvh, "find %%d", x);
      }
      starts.push_back(t);
      t += g.tiles;
      if (t < T) ts.next(g);
    }
    const int n_cl = (int)pick(1, std::min(152, L * batch * H_kv)), ctas = (int)pick(1, 8);
    int at = 0;
    for (int k = 0; k < n_cl; ++k) {
      const int c0 = run_bound(ts, T, k, n_cl), c1 = run_bound(ts, T, k + 1, n_cl);
      CHECK(c0 == at && c1 >= c0, "runs %%d: %%d %%d", k, c0, c1);
      CHECK(c1 == T || std::binary_search(starts.begin(), starts.end(), c1), "run end %%d", c1);
      at = c1;
      int u = c0;
      for (int r = 0; r < ctas; ++r) {
        const int u0 = c0 + quick_div((c1 - c0) * r, ctas), u1 = c0 + quick_div((c1 - c0) * (r + 1), ctas);
        CHECK(u0 == u && u1 >= u0, "cta ranges");
        u = u1;
      }
      CHECK(u == c1, "cta cover");
    }
    CHECK(at == T, "cluster cover %%d of %%d", at, T);
  }
  std::printf("mismatches %%d\n", fails);
  return fails != 0;
}
'''


def test_cluster_bookkeeping():
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    text = open(SRC).read()
    assert re.search(r"kClusterSeqs = 64;", text)
    assert "kMaxCluster = 8;" in open(SRC.replace("cluster", "rule")).read()
    assert "groups <= 1 << 16 && tiles < 1 << 20" in open(SRC[:-1]).read()  # the ranges checked here
    code = "\n".join([_block(text, r"^__device__ __forceinline__ int quick_div\("),
                      _block(text, r"^struct TileGroup \{"), _block(text, r"^struct TileSpace \{"),
                      _block(text, r"^__device__ __forceinline__ int run_bound\(")])
    with tempfile.TemporaryDirectory() as d:
        cpp, exe = os.path.join(d, "c.cpp"), os.path.join(d, "c")
        open(cpp, "w").write(HARNESS % dict(code=code))
        subprocess.run(["g++", "-O2", "-std=c++17", cpp, "-o", exe], check=True)
        r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def _kernel():
    """the cluster pass's producer and consumers, without comments"""
    text = open(SRC).read()
    body = re.sub(r"//[^\n]*", "", text[text.index("attend_cluster_kernel(const"):])
    body = body[:body.index("\n}\n") + 2]  # to the kernel's own closing brace
    at = body.index("pdl_enter();\n  named_sync")
    return body[:at], body[at:]


def test_nothing_of_a_warp_branches_on_a_lanes_wait():
    """What follows a wait uses shuffles and matrix instructions of all lanes, and at the time limit a
    warp's lanes may see the barrier differently: so a wait that ran out sets a flag of the CTA and
    the warp goes on together.  After that no copy is waited for, and the barriers that hand stages and
    query buffers back are held before the warp arrives on them, so that the producer arms none again."""
    producer, code = _kernel()
    landed = re.search(r"auto landed = [^{]*\{(.*?)\n  \};", code, re.S).group(1)
    assert re.sub(r"\s+", " ", landed).strip() == \
        "if (!mbar_try_wait(bar, parity) && !stopped() && !mbar_wait(bar, parity)) ran_out();"
    ran_out = re.search(r"auto ran_out = [^{]*\{(.*?)\n  \};", code, re.S).group(1)
    assert "s_stop, 2" in ran_out
    assert "s < Cl::kStages; ++s) mbar_hold(&empty_bar[s])" in ran_out
    assert "s < 2; ++s) mbar_hold(&q_empty[s])" in ran_out
    for use in re.finditer(r"[^;{}]*(pass\.begin|pass\.update|landed)\(&?[^;]*;", code):
        assert "if (" not in use.group(0) or "P::" in use.group(0), use.group(0)
    skip = code[code.index("if (s_skip > 0)"):code.index("for (int t = u0;")]
    assert "in = in && mbar_wait(&full_bar[it], 0);" in skip and "if (!in) ran_out();" in skip
    # (those two, the one in landed() and the one of the pieces)
    assert len(re.findall(r"\bmbar_wait(?:_cluster)?\(", code)) == 4
    # the wait for a stage's copy, then its work, then the arrival that hands it back
    tile = code[code.index("for (; t < stop;"):]
    assert tile.index("landed(&full_bar[st]") < tile.index("pass.update(") < \
        tile.index("mbar_arrive(&empty_bar[st])")
    assert skip.index("ran_out();") < skip.index("mbar_arrive(&empty_bar[it])")
    for bar in ("empty_bar", "q_empty"):
        assert re.search(r"timed_out\(&%s\[" % bar, producer)
    text = open(SRC).read()
    hold = text[text.index("void mbar_hold("):]
    assert "mbarrier.expect_tx" in hold[:hold.index("}")]


def test_a_cta_outlives_what_is_sent_to_it():
    """A CTA leaves when the pieces for it have arrived, or, once a wait ran out, when every thread
    of the cluster has ended or met it at a barrier and what is in flight has had time to land.
    Every CTA reaches its sends whatever became of its own copies, so that the barrier is met."""
    _, code = _kernel()
    assert re.search(r"__syncwarp\(\);\s*if \(stopped\(\) & 2\) \{\s*cluster_arrive\(\);\s*"
                     r"cluster_wait\(\);\s*linger\(\);\s*\}\s*\}$", code), code[-300:]
    lambdas = re.sub(r"auto \w+ = \[&\].*?\n  \};", "", code, flags=re.S)
    assert not re.search(r"\breturn\b", re.sub(r"if \(whole\) return;", "", lambdas))
    sends = code[code.index("for (int task = warp;"):code.index("slot0 : slot1) = Slot")]
    whole, shared = sends.split("} else {")
    assert "if (!bad) finish" in whole and "peer_st(" in shared and "if (lane == 0) peer_st4" in shared
    # a CTA that owns units waits for their pieces with the status set, too
    merge = code[code.index("for (int slot = 0;"):]
    assert "if (!mbar_wait_cluster(&recv_bar[slot], 0)) ran_out();" in merge[:merge.index("if (bad")]


def test_the_general_passes_waits_have_one_answer_a_warp():
    """The same in the persistent pass, whose consumer and merger warps end together after a wait that
    ran out, and in the chunk kernel, whose warps go on and all end after the CTA's next barrier
    (a warp that left before it would leave the others waiting at the one after)."""
    src = os.path.dirname(SRC)
    mma = re.sub(r"//[^\n]*", "", open(os.path.join(src, "lg_attend_mma.cu")).read())
    for bar in ("full_bar", "tfull"):
        waits = re.findall(r"(mbar_wait\w*)\(&%s\[" % bar, mma)
        assert waits == ["mbar_wait_warp"], (bar, waits)
    assert re.search(r"mbar_wait_warp\(&full_bar[^{]*\{[^}]*linger\(\);\s*return;", mma)
    common = open(os.path.join(src, "lg_common.cuh")).read()
    assert "return __all_sync(0xffffffffu, mbar_wait(bar, parity));" in common
    chunk = re.sub(r"//[^\n]*", "", open(os.path.join(src, "lg_attend.cu")).read())
    chunk = chunk[chunk.index("attend_partial_kernel(AttendArgs a)"):chunk.index("attend_combine_kernel")]
    loop, rest = chunk[chunk.index("const int suffix_lo"):].split("bar.sync 1", 1)
    assert "break" not in loop and "ok" not in re.findall(r"\b\w+\b", loop)
    assert re.search(r"^[^}]*?if \(stopped\(\)\) \{\s*linger\(\);\s*return;\s*\}", rest)
