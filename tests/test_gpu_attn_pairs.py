"""GPU parity of tree attention where a CTA takes two heads' whole units at once, a chain each: short units of one row tile, odd and even
numbers of heads, empty trees and contexts between them, ranges that end between the two heads, and units of later row groups."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.harness import (Problem, bf16_to_f64, dev, device_attn_inputs, oracle_attn_rows_by_head, stream_k_shares, synthetic_trees,
                           tree_mask_from_parents)
from tests.test_attn_schedule_pairs import paired

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("batch,hq,hkv,T,ctx", [(60, 10, 10, 33, (0, 1, 127, 128, 129, 500)), (70, 28, 7, 17, (3, 64, 200)), (24, 40, 40, 128, (100, 900)),
                                                (130, 32, 32, 2, (5,))])
def test_attn_two_heads_at_once(oracle, d, batch, hq, hkv, T, ctx):
    from paper_2511_21699_b200 import Cacheback
    cfg = W.CbConfig("pairs", batch, 2, 2, 64, 2, T, 8, 0, hq, hkv, d, (0, max(ctx)), 100, 1.1, 0.3, (4, 8), 64)
    prob = Problem(cfg)
    rng = np.random.default_rng(batch + d)
    prob.ctx = rng.choice(ctx, batch).astype(np.int32)
    prob.bt, prob.num_pages = W.make_block_table(cfg, np.maximum(prob.ctx, 1))
    par, dep, mask, n = synthetic_trees(cfg, full=False)
    n[:] = rng.integers(0, T + 1, batch)
    for b in range(batch):
        par[b], dep[b] = W.random_tree(cfg.seed, b, max(int(n[b]), 1), cfg.max_depth, T)
        mask[b] = tree_mask_from_parents(par[b], int(n[b]), (T + 31) // 32)
    shares = stream_k_shares(cfg, prob.ctx, n, min(torch.cuda.get_device_properties(0).multi_processor_count, 160))
    assert any(a[:1] == b[:1] and a[1] + 1 == b[1] and a[4:] == b[4:] and a[5] == 0 and a[6] == a[4] for c in shares for a, b in zip(c, c[1:]))
    d_in = device_attn_inputs(cfg, prob)
    cb = Cacheback.from_config(cfg)
    lse = torch.full((batch, hq, T), 7.0, dtype=torch.float32, device="cuda")
    out = cb.cb_tree_attn(d_in["q"], d_in["k_pool"], d_in["v_pool"], d_in["block_table"], d_in["ctx_len"], d_in["k_tree"], d_in["v_tree"],
                          dev(mask.view(np.int32)), dev(n), lse=lse, max_ctx=int(prob.ctx.max()))
    assert cb.cb_poll_status()[0] == 0
    # the first and last row of every head, of sequences at both ends of the batch and some between
    rows = np.array([(b, h, i) for b in sorted({0, 1, batch - 2, batch - 1, *rng.integers(0, batch, 6).tolist()}) for h in range(hq)
                     for i in sorted({0, int(n[b]) - 1, int(n[b]) // 2}) if 0 <= i < n[b]], np.int64)
    ref, ref_lse = oracle_attn_rows_by_head(oracle, cfg, prob, mask, rows)
    bb, hh, ii = (torch.from_numpy(rows[:, k]).cuda() for k in range(3))
    o, l = bf16_to_f64(out[bb, ii, hh]), lse[bb, hh, ii].cpu().numpy().astype(np.float64)
    # bf16 inputs and probabilities, fp32 sums, bf16 output: 2^-9 a term in P, 2^-8 in the output
    assert np.all(np.abs(o - ref) <= 2e-2 + 1e-2 * np.abs(ref)) and np.all(np.abs(l - ref_lse) <= 2e-3)
    assert np.all(np.linalg.norm(o - ref, axis=1) <= 1e-2 * np.linalg.norm(ref, axis=1))
    gone = np.arange(T)[None] >= n[:, None]
    assert not out.cpu().float().numpy()[gone].any()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("batch,T,full,ctx", [(28, 110, True, (377,)), (40, 128, False, (0, 127, 129, 300)), (60, 41, False, (5, 200))])
def test_attn_two_heads_at_once_in_later_row_groups(oracle, d, batch, T, full, ctx):
    """64/8 heads: 16 nodes a row tile, so trees of an odd number of them end in a row group of one row tile.  The rows of every such pair."""
    from paper_2511_21699_b200 import Cacheback
    cfg = W.CbConfig("pairs_later", batch, 2, 2, 64, 2, T, 8, 0, 64, 8, d, (0, max(ctx)), 100, 1.1, 0.3, (4, 8), 64)
    prob = Problem(cfg)
    rng = np.random.default_rng(batch + d)
    prob.ctx = rng.choice(ctx, batch).astype(np.int32)
    prob.bt, prob.num_pages = W.make_block_table(cfg, np.maximum(prob.ctx, 1))
    par, dep, mask, n = synthetic_trees(cfg, full=full)
    if not full:
        n[:] = rng.integers(1, T + 1, batch)
        for b in range(batch):
            par[b], dep[b] = W.random_tree(cfg.seed, b, int(n[b]), cfg.max_depth, T)
            mask[b] = tree_mask_from_parents(par[b], int(n[b]), (T + 31) // 32)
    pairs = [s for c in stream_k_shares(cfg, prob.ctx, n, min(torch.cuda.get_device_properties(0).multi_processor_count, 160))
             for s, two in paired(c) if two and s[2] > 0]
    assert len(pairs) >= 10
    d_in = device_attn_inputs(cfg, prob)
    cb = Cacheback.from_config(cfg)
    lse = torch.full((batch, 64, T), 7.0, dtype=torch.float32, device="cuda")
    out = cb.cb_tree_attn(d_in["q"], d_in["k_pool"], d_in["v_pool"], d_in["block_table"], d_in["ctx_len"], d_in["k_tree"], d_in["v_tree"],
                          dev(mask.view(np.int32)), dev(n), lse=lse, max_ctx=int(prob.ctx.max()))
    assert cb.cb_poll_status()[0] == 0
    # of both heads' units: first and last node of the row tile, each with one of the group's eight query heads
    rows = np.array([(b, (kh + k) * 8 + int(rng.integers(0, 8)), i) for b, kh, rg, *_ in pairs for k in (0, 1)
                     for i in sorted({rg * 32, min(rg * 32 + 16, int(n[b])) - 1})], np.int64)
    ref, ref_lse = oracle_attn_rows_by_head(oracle, cfg, prob, mask, rows)
    bb, hh, ii = (torch.from_numpy(rows[:, k]).cuda() for k in range(3))
    o, l = bf16_to_f64(out[bb, ii, hh]), lse[bb, hh, ii].cpu().numpy().astype(np.float64)
    # bf16 inputs and probabilities, fp32 sums, bf16 output: 2^-9 a term in P, 2^-8 in the output
    assert np.all(np.abs(o - ref) <= 2e-2 + 1e-2 * np.abs(ref)) and np.all(np.abs(l - ref_lse) <= 2e-3)
    assert np.all(np.linalg.norm(o - ref, axis=1) <= 1e-2 * np.linalg.norm(ref, axis=1))
    gone = np.arange(T)[None] >= n[:, None]
    assert not out.cpu().float().numpy()[gone].any()
