"""GPU parity of tree attention on launches that mix units of one and of two row tiles: every unit that two or more CTAs share and every
unit beside one of the other kind at a CTA's seam, at the weights that the launcher gives their tiles (3 : 2 with head_dim 128, 2 : 1
with 64), over contexts of none to several tiles."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.harness import (Problem, bf16_to_f64, dev, device_attn_inputs, oracle_attn_rows_by_head, stream_k_shares, synthetic_trees,
                           tree_mask_from_parents)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("batch,hq,hkv,T,ctx", [(40, 8, 2, 61, (0, 1, 127, 128, 129, 700)), (150, 8, 4, 128, (5, 300)), (3, 64, 8, 100, (3000, 4000))])
def test_attn_mixed_units(oracle, d, batch, hq, hkv, T, ctx):
    from paper_2511_21699_b200 import Cacheback
    cfg = W.CbConfig("mixed_units", batch, 2, 2, 64, 2, T, 8, 0, hq, hkv, d, (0, max(ctx)), 100, 1.1, 0.3, (4, 8), 64)
    prob = Problem(cfg)
    rng = np.random.default_rng(batch + d)
    prob.ctx = rng.choice(ctx, batch).astype(np.int32)
    prob.bt, prob.num_pages = W.make_block_table(cfg, np.maximum(prob.ctx, 1))
    par, dep, mask, n = synthetic_trees(cfg, full=False)
    n[:] = rng.integers(1, T + 1, batch)
    for b in range(batch):
        par[b], dep[b] = W.random_tree(cfg.seed, b, int(n[b]), cfg.max_depth, T)
        mask[b] = tree_mask_from_parents(par[b], int(n[b]), (T + 31) // 32)
    owners, seams = {}, set()
    for c, shares in enumerate(stream_k_shares(cfg, prob.ctx, n, min(torch.cuda.get_device_properties(0).multi_processor_count, 160))):
        for s in shares:
            owners.setdefault(s[:4], set()).add(c)
        for a, b in zip(shares, shares[1:]):
            if a[3] != b[3]:
                seams |= {a[:4], b[:4]}
    shared = {u for u, cs in owners.items() if len(cs) > 1}
    assert len(shared) >= 10 or len(seams) >= 10
    d_in = device_attn_inputs(cfg, prob)
    cb = Cacheback.from_config(cfg)
    lse = torch.full((batch, hq, T), 7.0, dtype=torch.float32, device="cuda")
    out = cb.cb_tree_attn(d_in["q"], d_in["k_pool"], d_in["v_pool"], d_in["block_table"], d_in["ctx_len"], d_in["k_tree"], d_in["v_tree"],
                          dev(mask.view(np.int32)), dev(n), lse=lse, max_ctx=int(prob.ctx.max()))
    assert cb.cb_poll_status()[0] == 0
    npt = 128 // cfg.gqa
    rows = []
    for b, kh, rg, nrt in sorted(shared | seams):
        lo, hi = rg * 2 * npt, min(rg * 2 * npt + nrt * npt, int(n[b]))
        for i in sorted({lo, hi - 1, int(rng.integers(lo, hi))}):
            rows.append((b, kh * cfg.gqa + int(rng.integers(0, cfg.gqa)), i))
    rows = np.array(rows, np.int64)
    ref, ref_lse = oracle_attn_rows_by_head(oracle, cfg, prob, mask, rows)
    bb, hh, ii = (torch.from_numpy(rows[:, k]).cuda() for k in range(3))
    o, l = bf16_to_f64(out[bb, ii, hh]), lse[bb, hh, ii].cpu().numpy().astype(np.float64)
    # bf16 inputs and probabilities, fp32 sums, bf16 output: 2^-9 a term in P, 2^-8 in the output
    assert np.all(np.abs(o - ref) <= 2e-2 + 1e-2 * np.abs(ref)) and np.all(np.abs(l - ref_lse) <= 2e-3)
    assert np.all(np.linalg.norm(o - ref, axis=1) <= 1e-2 * np.linalg.norm(ref, axis=1))
    gone = np.arange(T)[None] >= n[:, None]
    assert not out.cpu().float().numpy()[gone].any()
