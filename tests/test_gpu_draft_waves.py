"""Three sequences of update and draft on an SM: with short follower lists the draft kernel's registers leave room for three blocks of 256
threads, so batches of two to three blocks an SM are one wave (a second wave is another chain of look-ups, a quarter of the call)."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.harness import dev

pytestmark = pytest.mark.gpu


def _best_us(batch):
    from paper_2511_21699_b200 import Cacheback
    cfg = W.CbConfig("waves", batch, 2, 4, 1024, 4, 64, 8, 16, 8, 8, 64, (600, 600), 2000, 1.1, 0.3, (4, 8), 64)
    toks, _ = W.make_streams(cfg, np.full(batch, 600, np.int32))
    tokens, new = dev(toks), dev(np.full(batch, 600, np.int32))
    old = new - 4
    cb = Cacheback.from_config(cfg)
    cb.cb_update_bulk(tokens, torch.zeros_like(old), old)
    tree = cb.alloc_tree()
    cb.cb_update_draft_tree(tokens, old, new, tree)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(20):
            cb.cb_update_draft_tree(tokens, old, new, tree)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(20):
        a.record()
        graph.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / 20)
    assert cb.cb_poll_status()[0] == 0
    return best


def test_three_sequences_an_sm():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    two, three = _best_us(2 * sms), _best_us(2 * sms + 8)
    # 1.02 with three blocks an SM, 1.3 with two; the best of 20 runs of 20 calls differs by 1% from one time to the next
    assert three <= 1.15 * two, (two, three)
