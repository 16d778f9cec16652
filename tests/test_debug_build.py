"""The checking build of the library (-DCB_DEBUG): the stand-in for a memory checker.  Without a GPU: it builds, exports
the same symbols and asks for a larger workspace (the guard areas).  On a GPU, in a process of its own that loads it in
place of the regular library: the tiny draft-and-verify step gives the oracle's results with a clean status, and a guard
byte overwritten from the host is reported by cb_poll_status."""
import ctypes
import os
import subprocess
import sys

import pytest

from tests.conftest import ROOT


def test_checking_build_exports_and_guards_need_no_gpu():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2511_21699_b200 import _lib
    regular, checking = ctypes.CDLL(os.path.join(ROOT, "paper_2511_21699_b200", "libcacheback.so")), ctypes.CDLL(_lib.SO_DEBUG_PATH)
    for name in _lib.EXPORTS:
        assert hasattr(checking, name), name
    assert regular.cb_debug_build() == 0 and checking.cb_debug_build() == 1
    cfg = _lib.CbConfigC(1, 2, 3, 4096, 4, 16, 4, 5, 32000, 8, 8, 64, 16, 0)
    a, b = ctypes.c_size_t(0), ctypes.c_size_t(0)
    for lib in (regular, checking):
        lib.cb_workspace_bytes.argtypes = [ctypes.POINTER(_lib.CbConfigC), ctypes.POINTER(ctypes.c_size_t)]
    assert regular.cb_workspace_bytes(ctypes.byref(cfg), ctypes.byref(a)) == 0
    assert checking.cb_workspace_bytes(ctypes.byref(cfg), ctypes.byref(b)) == 0
    assert b.value == a.value + 10 * _lib.CB_GUARD_BYTES          # one guard area behind each of the ten regions


_CHILD = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
import __graft_entry__
from paper_2511_21699_b200 import _lib, Cacheback
assert _lib.load().cb_debug_build() == 1
__graft_entry__.smoke()                                  # update, draft, attention, acceptance on the tiny config against the oracle
import workloads as W
cfg = W.get_config("c1_tiny")
cb = Cacheback.from_config(cfg)
st, _ = cb.cb_poll_status()
assert st == 0, st
# a stray write just behind the first workspace region (the table headers: batch * 16 bytes, rounded up to 256), made from the host
base = (cb.workspace.data_ptr() + 255) // 256 * 256 - cb.workspace.data_ptr()
cb.workspace[base + 256 + 7] = 0
st, _ = cb.cb_poll_status()
assert st == _lib.CB_ERR_CANARY, st
cb.workspace[base + 256 + 7] = 0xC5
st, _ = cb.cb_poll_status()
assert st == 0, st
# a page id outside the pool in the block table: recorded, the tile reads as zeros, nothing faults
from workloads import device as wdev
from workloads.tensors import TID
ctx = W.ctx_lens(cfg)
bt, num_pages = W.make_block_table(cfg, ctx)
bt = bt.copy(); bt[0, 3] = num_pages + 1000
bf = torch.bfloat16
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
B, T = cfg.batch, cfg.max_nodes
kp = wdev.normal_tensor((num_pages, cfg.page_size, cfg.n_kv_heads, cfg.head_dim), bf, 0, TID.K_POOL)
vp = wdev.normal_tensor((num_pages, cfg.page_size, cfg.n_kv_heads, cfg.head_dim), bf, 0, TID.V_POOL)
q = wdev.normal_tensor((B, T, cfg.n_q_heads, cfg.head_dim), bf, 0, TID.Q)
kt = wdev.normal_tensor((B, T, cfg.n_kv_heads, cfg.head_dim), bf, 0, TID.K_TREE)
vt = wdev.normal_tensor((B, T, cfg.n_kv_heads, cfg.head_dim), bf, 0, TID.V_TREE)
mask = torch.zeros(B, T, 1, dtype=torch.int32, device="cuda"); mask[:, 0, 0] = 1
out = cb.cb_tree_attn(q, kp, vp, dev(bt), dev(ctx), kt, vt, mask, torch.ones(B, dtype=torch.int32, device="cuda"))
torch.cuda.synchronize()
st, _ = cb.cb_poll_status()
assert st == _lib.CB_ERR_INVALID_ARG, st
assert torch.isfinite(out.float()).all()
# prompts through the block kernel: the oracle's tables, then a planted index word that names an entry the table cannot have
from oracle import cb_oracle
LL, FL, LC, FC, n = 2, 3, 4096, 4, 1500
toks = np.minimum(np.random.default_rng(4).zipf(1.3, (2, 2 * n)) - 1, 900).astype(np.int32)
cb = Cacheback(2, LL, FL, LC, FC, 32, 8, 8, 1000, 8, 8, 64)
tab = [cb_oracle.OracleTable(LL, FL, LC, FC) for _ in range(2)]
z, n1, n2 = (dev(np.full(2, x, np.int32)) for x in (0, n, 2 * n))
for a, b, ha, hb in ((z, n1, 0, n), (n1, n2, n, 2 * n)):
    cb.cb_update_bulk(dev(toks), a, b)
    for s in range(2):
        tab[s].update(toks[s], ha, hb)
        assert all(np.array_equal(x, y) for x, y in zip(cb.cb_table_dump_arrays(s), tab[s].dump_arrays()))
assert cb.cb_poll_status()[0] == 0
M64 = (1 << 64) - 1
h = 0x9E3779B97F4A7C15 ^ LL                             # the key's hash: its tag and its bucket
key = toks[0, :2] * 0 + 950                               # a leader that the tables do not have
for k in key:
    h = ((h ^ int(k)) * 0xFF51AFD7ED558CCD) & M64
    h ^= h >> 32
h ^= h >> 33
h = (h * 0xC4CEB9FE1A85EC53) & M64
h ^= h >> 33
nslots = 4 * LC
base = (cb.workspace.data_ptr() + 255) // 256 * 256 - cb.workspace.data_ptr()
index = cb.workspace[base + 512:base + 512 + 4 * nslots].view(torch.int32)           # behind the headers and their guard area
bucket = index[32 * ((h >> 32) & (nslots // 32 - 1)):][:32]
free = int((bucket == 0).nonzero()[0])
bucket[free] = int(np.uint32(((h & 0xFFFFFFFF) %% 4094 + 1) << 20 | (LC + 7)).view(np.int32))
more = np.concatenate([toks, np.full((2, 80), 950, np.int32)], 1)
cb.cb_update_bulk(dev(more), n2, dev(np.full(2, 2 * n + 80, np.int32)))
assert cb.cb_poll_status()[0] == _lib.CB_ERR_INVALID_ARG
bucket[free] = 0
# a selection of the frozen builder that gives up at its first barrier: the call says so, and nothing behind it goes by what is missing
import ctypes as C
L = _lib.load()
L.cb_debug_frozen_build.argtypes = L.cb_frozen_build.argtypes + [C.c_uint32]
L.cb_debug_frozen_build.restype = C.c_int32
N, LL, FL, LC, FC = 20000, 2, 3, 1 << 15, 4
corpus = np.random.default_rng(3).integers(0, 200, N).astype(np.int32)
fc = _lib.CbFrozenConfigC(LL, FL, LC, FC)
tb, sb = C.c_size_t(0), C.c_size_t(0)
assert L.cb_frozen_bytes(C.byref(fc), C.byref(tb)) == 0 and L.cb_frozen_build_bytes(C.byref(fc), N, C.byref(sb)) == 0
table = torch.empty(tb.value, dtype=torch.uint8, device="cuda")
scratch = torch.full((sb.value,), 0xA5, dtype=torch.uint8, device="cuda")           # ranges that nobody wrote point far outside
assert table.data_ptr() %% 256 == 0 and scratch.data_ptr() %% 256 == 0
d = dev(corpus)
args = (C.byref(fc), d.data_ptr(), N, table.data_ptr(), tb.value, scratch.data_ptr(), sb.value, torch.cuda.current_stream().cuda_stream)
assert L.cb_debug_frozen_build(*args, 0) == 5                                       # CB_ERR_TIMEOUT
# the windows' array: the last third of the region before the leaders' four words each at the scratch's end
S = 1024
while S < 2 * (N - LL - FL + 1):
    S *= 2
up = lambda x: (x + 255) // 256 * 256
wpos = sb.value - up(LC * 16) - up(S * 6) + S * 4
assert bool((scratch[wpos:wpos + S * 2] == 0xA5).all())
assert bool((scratch[sb.value - up(LC * 16) + LC * 4:sb.value - up(LC * 16) + LC * 8] == 0xA5).all())       # no range was given out
bad = dev(np.concatenate([[-1], corpus[1:]]).astype(np.int32))                      # reported even where a negative token was recorded first
assert L.cb_debug_frozen_build(args[0], bad.data_ptr(), *args[2:], 0) == 5
assert L.cb_frozen_build(*args) == 0
nl = C.c_int32(0)
lead, nf, fol = np.zeros((LC, LL), np.int32), np.zeros(LC, np.int32), np.zeros((LC, FC, FL), np.int32)
ip = lambda a: a.ctypes.data_as(C.c_void_p)
assert L.cb_frozen_dump(args[0], table.data_ptr(), tb.value, C.byref(nl), ip(lead), ip(nf), ip(fol)) == 0
oL, onf, oF = cb_oracle.frozen_build(corpus, LL, FL, LC, FC)
n = nl.value
assert n == len(oL) and np.array_equal(lead[:n], oL) and np.array_equal(nf[:n], onf) and np.array_equal(fol[:n], oF)
print("checking build ok")
"""


@pytest.mark.gpu
def test_checking_build_runs_the_tiny_step_and_reports_planted_errors():
    from paper_2511_21699_b200 import _lib
    env = dict(os.environ, CACHEBACK_LIBRARY=_lib.SO_DEBUG_PATH)
    r = subprocess.run([sys.executable, "-c", _CHILD % ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "checking build ok" in r.stdout, (r.stdout[-2000:], r.stderr[-3000:])
