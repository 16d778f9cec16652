"""The kernel's header compiled for the host: the walk that takes two heads' whole units of one row tile at a time (every pair that the
ranges allow, and no other), and the schedule of batches of up to 32 in 32 bits against the general one, with a warp's 32 lanes emulated."""
import os
import subprocess

import numpy as np
import pytest

from tests.harness import stream_k_shares
from tests.test_attn_schedule import SHAPES, _cfg

_SHIM = r"""
#include <ucontext.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <functional>
#include <vector>
using std::min; using std::max;
// A warp: 32 contexts in turn.  A collective writes its lane's value, lets the others run up to the same point and reads theirs; the
// next one uses the other set, so that nobody overwrites what a lane has yet to read.
constexpr int kLanes = 32;
static int lane_now, ops[kLanes];
static unsigned long long vals[2][kLanes];
static ucontext_t ctxs[kLanes], home;
static std::vector<char> stacks[kLanes];
static std::function<void(int)> body;
static const unsigned long long* all_lanes(unsigned long long x) {
    const int me = lane_now, set = ops[me]++ & 1;
    vals[set][me] = x;
    lane_now = (me + 1) % kLanes;
    swapcontext(&ctxs[me], &ctxs[lane_now]);
    return vals[set];
}
static void run_lane() {
    const int me = lane_now;
    body(me);
    if (me + 1 < kLanes) { lane_now = me + 1; setcontext(&ctxs[me + 1]); }
    setcontext(&home);
}
static void warp(std::function<void(int)> f) {
    body = f;
    for (int l = 0; l < kLanes; ++l) {
        ops[l] = 0;
        stacks[l].resize(1 << 16);
        getcontext(&ctxs[l]);
        ctxs[l].uc_stack.ss_sp = stacks[l].data(); ctxs[l].uc_stack.ss_size = stacks[l].size(); ctxs[l].uc_link = nullptr;
        makecontext(&ctxs[l], run_lane, 0);
    }
    lane_now = 0;
    swapcontext(&home, &ctxs[0]);
}
template <typename T> unsigned long long bits_of(T x) { unsigned long long u = 0; memcpy(&u, &x, sizeof(T)); return u; }
template <typename T> T of_bits(unsigned long long u) { T x; memcpy(&x, &u, sizeof(T)); return x; }
template <typename T> T __shfl_sync(unsigned, T x, int l) { return of_bits<T>(all_lanes(bits_of(x))[l & 31]); }
template <typename T> T __shfl_xor_sync(unsigned, T x, int o) { const int me = lane_now; return of_bits<T>(all_lanes(bits_of(x))[me ^ o]); }
template <typename T> T __shfl_up_sync(unsigned, T x, int o) { const int me = lane_now; return of_bits<T>(all_lanes(bits_of(x))[me >= o ? me - o : me]); }
inline unsigned __ballot_sync(unsigned, bool x) { const auto* v = all_lanes(x); unsigned m = 0; for (int l = 0; l < kLanes; ++l) m |= (unsigned)(v[l] != 0) << l; return m; }
inline bool __any_sync(unsigned m, bool x) { return __ballot_sync(m, x) != 0; }
inline unsigned __reduce_add_sync(unsigned, unsigned x) { const auto* v = all_lanes(x); unsigned s = 0; for (int l = 0; l < kLanes; ++l) s += (unsigned)v[l]; return s; }
inline int __reduce_max_sync(unsigned, int x) { const auto* v = all_lanes(bits_of(x)); int s = x; for (int l = 0; l < kLanes; ++l) s = max(s, of_bits<int>(v[l])); return s; }
inline float __fdividef(float a, float b) { return a / b; }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
#include "cb_attn_sched32.cuh"
int main() {
    CbAttnParams p = {};
    int narrow_wanted = 0;
    while (scanf("%d %d %d %d %d %d %d", &p.B, &p.T, &p.G, &p.Hkv, &p.D, &p.nc, &narrow_wanted) == 7) {
        std::vector<int> n(p.B), c(p.B);
        for (int b = 0; b < p.B; ++b) if (scanf("%d %d", &n[b], &c[b]) != 2) return 1;
        p.n_nodes = n.data(); p.ctx_len = c.data(); p.P = 16; p.max_pages = 1 << 20;
        p.NPT = CB_MT / p.G; p.npt_inv = 65536u / (unsigned)p.NPT + 1u; p.MT = (p.T + p.NPT - 1) / p.NPT;
        cb_attn_weights(p);
        for (int k = 0; k < p.nc; ++k) {
            long long tot = 0, g0 = 0, g1 = 0, pre = 0;
            int rg0 = 0, b0 = 0, wrong = 0;
            warp([&](int lane) {
                const long long t = cb_sched_total(p, lane), a = cb_range_start(t, p.nc, k), e = cb_range_start(t, p.nc, k + 1);
                int rg = 0, b = 0;
                long long at = 0;
                if (a < e) cb_sched_locate(p, a, lane, &rg, &b, &at);
                long long t2 = -1, a2 = -1, e2 = -1, at2 = 0;
                int rg2 = 0, b2 = 0;
                const bool narrow = cb_sched_of_32(p, k, lane, &t2, &a2, &e2, &rg2, &b2, &at2);
                if (narrow != (narrow_wanted != 0)) wrong = 1;
                if (narrow && (t2 != t || a2 != a || e2 != e)) wrong = 2;
                if (narrow && a < e && (rg2 != rg || b2 != b || at2 != at)) wrong = 3;
                if (lane == 0) { tot = t; g0 = a; g1 = e; rg0 = rg; b0 = b; pre = at; }
            });
            if (wrong) { printf("schedule in 32 bits: %d\n", wrong); return 1; }
            CbWalker wk;
            CbUnit u;
            wk.init(p, g0, g1, rg0, b0, pre);
            while (wk.next_pair(p, &u)) {
                const int pair = u.nrt == kTwoHeads;
                if (pair && (u.t0 != 0 || u.t1 != u.tiles || u.kh + 2 > p.Hkv)) { printf("not a pair\n"); return 1; }
                printf("%d %d %d %d %d %d %d %d %d ", k, u.b, u.kh, u.rg, pair ? 1 : u.nrt, u.tiles, u.t0, u.t1, pair);
            }
        }
        printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def walk_pairs(tmp_path_factory):
    from paper_2511_21699_b200 import build as b
    d = tmp_path_factory.mktemp("pairs")
    (d / "shim.cpp").write_text(_SHIM)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(cuda, "include"), "-I", os.path.join(b.ROOT, "include"), "-I", b.CSRC,
                           str(d / "shim.cpp"), "-o", str(d / "shim")])

    def f(cfg, ctx, n, n_ctas, narrow):
        """n_ctas lists of (share, is it two heads')"""
        text = "%d %d %d %d %d %d %d\n" % (cfg.batch, cfg.max_nodes, cfg.gqa, cfg.n_kv_heads, cfg.head_dim, n_ctas, narrow)
        text += " ".join("%d %d" % x for x in zip(n, ctx))
        r = subprocess.run([str(d / "shim")], input=text, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stdout[-200:]
        shares = [[] for _ in range(n_ctas)]
        for x in np.array(r.stdout.split(), np.int64).reshape(-1, 9):
            shares[x[0]].append((tuple(int(y) for y in x[1:8]), int(x[8])))
        return shares
    return f


def paired(shares):
    """A CTA's shares as it takes them: two neighbouring heads' whole units of one row tile together, from the front."""
    out, k = [], 0
    while k < len(shares):
        b, kh, rg, nrt, tiles, t0, t1 = shares[k]
        two = (k + 1 < len(shares) and nrt == 1 and (t0, t1) == (0, tiles) and shares[k + 1] == (b, kh + 1, rg, 1, tiles, 0, tiles))
        out.append((shares[k], int(two)))
        k += 1 + two
    return out


@pytest.mark.parametrize("batch,hq,hkv,T,d,lo,hi", SHAPES + [(40, 6, 3, 20, 128, 0, 400), (9, 40, 40, 1, 64, 1, 130), (2, 5, 5, 128, 128, 700, 900),
                                                             (28, 64, 8, 110, 128, 377, 377), (32, 64, 8, 110, 64, 0, 500), (33, 16, 16, 7, 64, 3, 60)])
def test_every_pair_and_no_other(walk_pairs, batch, hq, hkv, T, d, lo, hi):
    cfg = _cfg(batch, hq, hkv, T, d)
    rng = np.random.default_rng(batch)
    ctx = rng.permutation(np.round(np.linspace(lo, hi, batch)).astype(np.int64))
    pairs = {0: 0, 1: 0}                                         # in the first row group, in a later one
    for n in (np.full(batch, T), rng.integers(0, T + 1, batch)):
        for n_ctas in (148, 160, 7, 1):
            want = [paired(c) for c in stream_k_shares(cfg, ctx, n, n_ctas)]
            assert walk_pairs(cfg, ctx, n, n_ctas, int(batch <= 32)) == want
            for c in want:
                for (_, _, rg, *_), two in c:
                    pairs[min(rg, 1)] += two
    if hkv > 1:                                                  # a single CTA holds every unit whole
        assert pairs[0] + pairs[1] > 0
    if (hq, hkv, T) == (64, 8, 110):
        assert pairs[1] > 0


def test_schedule_in_32_bits_ends_where_a_sequence_reaches_2_26(walk_pairs):
    cfg = _cfg(2, 128, 128, 128, 128)                            # W = 128 heads x (4 positions a tile + 8)
    for tiles, narrow in ((131069, 1), (131070, 0)):
        ctx = np.array([(tiles - 1) * 128, 5])
        n = np.array([128, 128])
        assert walk_pairs(cfg, ctx, n, 148, narrow) == [paired(c) for c in stream_k_shares(cfg, ctx, n, 148)]
