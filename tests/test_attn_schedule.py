"""Tree attention's split over the persistent CTAs, from the kernel's own header compiled for the host: what every CTA works on against
its restatement in the harness, and launches whose units have all one row tile, or all two, cut where weights of 2 : 1 cut them (the
places where a unit is shared decide the last bit of its rows)."""
import os
import subprocess

import numpy as np
import pytest

import workloads as W
from tests.harness import stream_k_shares

_SHIM = r"""
#include <cstdio>
#include <cstdlib>
#include <algorithm>
#include <vector>
using std::min; using std::max;
// one lane a warp: the header's collectives over a single sequence are not called here
template <typename T> T __shfl_xor_sync(unsigned, T x, int) { return x; }
template <typename T> T __shfl_up_sync(unsigned, T x, int) { return x; }
template <typename T> T __shfl_sync(unsigned, T x, int) { return x; }
inline unsigned __ballot_sync(unsigned, bool x) { return x; }
inline int __reduce_max_sync(unsigned, int x) { return x; }
inline float __fdividef(float a, float b) { return a / b; }
inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
#include "cb_attn.cuh"
int main() {
    CbAttnParams p = {};
    int w1 = 0, w2 = 0;
    while (scanf("%d %d %d %d %d %d %d %d", &p.B, &p.T, &p.G, &p.Hkv, &p.D, &p.nc, &w1, &w2) == 8) {
        std::vector<int> n(p.B), c(p.B);
        for (int b = 0; b < p.B; ++b) if (scanf("%d %d", &n[b], &c[b]) != 2) return 1;
        p.n_nodes = n.data(); p.ctx_len = c.data(); p.P = 16; p.max_pages = 1 << 20;
        p.NPT = CB_MT / p.G; p.npt_inv = 65536u / (unsigned)p.NPT + 1u; p.MT = (p.T + p.NPT - 1) / p.NPT;
        cb_attn_weights(p);
        if (w1) { p.w1 = w1; p.w2 = w2; p.d1 = p.d2 = 0; }
        long long tot = 0;
        for (int b = 0; b < p.B; ++b) tot += cb_seq_shape(p, b).W;
        for (int k = 0; k < p.nc; ++k) {
            const long long g0 = cb_range_start(tot, p.nc, k), g1 = cb_range_start(tot, p.nc, k + 1);
            long long pre = 0;
            int rg0 = 0, b0 = 0;
            bool found = false;                                // cb_sched_locate, one sequence at a time
            for (int rg = 0; rg < cb_max_row_groups(p) && !found; ++rg)
                for (int b = 0; b < p.B && !found; ++b) {
                    const long long w = cb_seq_shape(p, b).w_of(p.Hkv, rg);
                    if (g0 < pre + w) { rg0 = rg; b0 = b; found = true; } else pre += w;
                }
            CbWalker wk;
            CbUnit u;
            wk.init(p, g0, g1, rg0, b0, pre);
            while (wk.next(p, &u)) {
                const int wt = wk.s.wt(u.rg);
                const long long x0 = wk.pre + (long long)u.kh * wk.s.unit(u.rg) + wk.s.dec(u.rg);
                for (int t : {u.t0, u.t1 - 1})                 // whose tile it is, asked the other way round
                    if (cb_cta_of(tot, p.nc, x0 + (long long)t * wt) != k) { printf("wrong owner\n"); return 1; }
                printf("%d %d %d %d %d %d %d %d ", k, u.b, u.kh, u.rg, u.nrt, u.tiles, u.t0, u.t1);
            }
        }
        printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    from paper_2511_21699_b200 import build as b
    d = tmp_path_factory.mktemp("schedule")
    (d / "shim.cpp").write_text(_SHIM)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(cuda, "include"), "-I", os.path.join(b.ROOT, "include"), "-I", b.CSRC,
                           str(d / "shim.cpp"), "-o", str(d / "shim")])

    def f(cfg, ctx, n, n_ctas, weights=(0, 0)):
        text = "%d %d %d %d %d %d %d %d\n" % ((cfg.batch, cfg.max_nodes, cfg.gqa, cfg.n_kv_heads, cfg.head_dim, n_ctas) + weights)
        text += " ".join("%d %d" % x for x in zip(n, ctx))
        r = subprocess.run([str(d / "shim")], input=text, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stdout[-200:]
        shares = [[] for _ in range(n_ctas)]
        for x in np.array(r.stdout.split(), np.int64).reshape(-1, 8):
            shares[x[0]].append(tuple(int(y) for y in x[1:]))
        return shares
    return f


def _cfg(batch, hq, hkv, T, d):
    return W.CbConfig("schedule", batch, 2, 2, 64, 2, T, 8, 0, hq, hkv, d, (0, 1), 100, 1.1, 0.3, (4, 8), 64)


SHAPES = [(64, 40, 40, 32, 128, 2048, 2048), (128, 64, 8, 128, 128, 32768, 32768), (32, 32, 8, 64, 128, 1024, 8192), (39, 40, 40, 9, 128, 220, 220),
          (7, 8, 1, 40, 128, 0, 20000), (1, 16, 2, 20, 64, 300, 300), (13, 32, 8, 61, 64, 777, 5003), (150, 8, 4, 128, 128, 5, 300), (3, 64, 8, 100, 128, 3000, 4000)]


@pytest.mark.parametrize("batch,hq,hkv,T,d,lo,hi", SHAPES)
@pytest.mark.parametrize("trees", ["one_kind", "ragged"])
def test_ranges_of_the_persistent_ctas(walk, batch, hq, hkv, T, d, lo, hi, trees):
    cfg = _cfg(batch, hq, hkv, T, d)
    rng = np.random.default_rng(batch)
    ctx = rng.permutation(np.round(np.linspace(lo, hi, batch)).astype(np.int64))
    npt = 128 // cfg.gqa
    full = T if T <= npt else T // (2 * npt) * 2 * npt                 # trees whose row groups have all two row tiles
    if trees == "one_kind" and full == 0:
        pytest.skip("a tree of this size has one row tile in some group")
    n = np.full(batch, full) if trees == "one_kind" else rng.integers(0, T + 1, batch)
    for n_ctas in (148, 160, 7):
        shares = walk(cfg, ctx, n, n_ctas)
        assert shares == stream_k_shares(cfg, ctx, n, n_ctas)
        assert sum(s[6] - s[5] for c in shares for s in c) == sum(                                    # every tile once
            cfg.n_kv_heads * (1 if T <= npt else -(-(-(-int(k) // npt)) // 2)) * (-(-int(c) // 128) + 1) for k, c in zip(n, ctx) if k > 0)
        if trees == "one_kind":
            assert shares == walk(cfg, ctx, n, n_ctas, (1, 2))
