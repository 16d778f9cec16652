"""GPU parity of tree attention's cluster mode where the bound that the caller gives on the contexts is exact, a tile too high, far too high
or the block table's own width: the first copy's page is asked for on the bound's account before the length is known."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.harness import Problem, bf16_to_f64, dev, device_attn_inputs, oracle_attn_rows_by_head, synthetic_trees

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("hq,hkv,ctx", [(16, 16, [2000]), (8, 4, [1, 4000, 700]), (32, 8, [0, 130]), (4, 1, [3333])])
@pytest.mark.parametrize("bound", ["exact", "next_tile", "far", "none"])
def test_attn_cluster_bound(oracle, d, hq, hkv, ctx, bound):
    from paper_2511_21699_b200 import Cacheback
    B, T = len(ctx), 30
    cfg = W.CbConfig("cluster_guess", B, 2, 2, 64, 2, T, 8, 0, hq, hkv, d, (0, 6000), 100, 1.1, 0.3, (4, 8), 64)
    prob = Problem(cfg)
    prob.ctx = np.array(ctx, np.int32)
    prob.bt, prob.num_pages = W.make_block_table(cfg, np.full(B, 6000, np.int32))
    _, _, mask, n = synthetic_trees(cfg)
    x = device_attn_inputs(cfg, prob)
    cb = Cacheback.from_config(cfg)
    lse = torch.empty(B, hq, T, dtype=torch.float32, device="cuda")
    top = max(ctx)
    args = dict(exact=dict(max_ctx=max(top, 1)), next_tile=dict(max_ctx=top + 128), far=dict(max_ctx=5999), none={})[bound]
    out = cb.cb_tree_attn(x["q"], x["k_pool"], x["v_pool"], x["block_table"], x["ctx_len"], x["k_tree"], x["v_tree"], dev(mask.view(np.int32)), dev(n), lse=lse, **args)
    assert cb.cb_poll_status()[0] == 0
    rows = np.array([(b, h, i) for b in range(B) for h in (0, hq - 1) for i in (0, int(n[b]) - 1)], np.int64)
    ref, ref_lse = oracle_attn_rows_by_head(oracle, cfg, prob, mask, rows)
    bb, hh, ii = (torch.from_numpy(rows[:, k]).cuda() for k in range(3))
    o, l = bf16_to_f64(out[bb, ii, hh]), lse[bb, hh, ii].cpu().numpy().astype(np.float64)
    # bf16 inputs and probabilities, fp32 sums, bf16 output: 2^-9 a term in P, 2^-8 in the output
    assert np.all(np.abs(o - ref) <= 2e-2 + 1e-2 * np.abs(ref)) and np.all(np.abs(l - ref_lse) <= 2e-3)
    assert np.all(np.linalg.norm(o - ref, axis=1) <= 1e-2 * np.linalg.norm(ref, axis=1))
