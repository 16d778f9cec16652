"""GPU parity of cb_update_bulk's block kernel where the blocks are dealt to few and to very unequal sequences, and where a part has more
than 512 leaders, of which some have one follower, some as many as an entry holds, some more and some are stored already."""
import numpy as np
import pytest
import torch

from tests.harness import dev
from tests.test_gpu_table import _assert_tables_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("LL,FL,LC,FC", [(3, 4, 32768, 4), (1, 8, 32768, 2), (2, 1, 32768, 7), (4, 3, 32768, 1)])
@pytest.mark.parametrize("runs", [[8192], [8192, 64], [8192, 0, 33, 64, 2048, 2047, 8191], [100] * 31 + [8000], [1200] * 100 + [0, 8192, 65], [90] * 147, [70] * 148])
def test_bulk_parts(oracle, LL, FL, LC, FC, runs):
    from paper_2511_21699_b200 import Cacheback
    B, w = len(runs), LL + FL
    rng = np.random.default_rng(B * 10 + LL)
    n1 = np.array([x + w - 1 if x else 0 for x in runs], np.int32)
    n2 = (n1 + np.array([min(x, 700) for x in runs])).astype(np.int32)
    # half of the text is a permutation (leaders of one follower), half is drawn from few tokens (leaders of many)
    toks = np.stack([rng.permutation(int(n2.max()) * 2)[: int(n2.max())] for _ in range(B)]).astype(np.int32) + 50
    few = rng.random(toks.shape) < 0.5
    toks[few] = np.minimum(rng.zipf(1.5, toks.shape) - 1, 40)[few]
    check = sorted({0, 1 % B, B // 2, B - 2 if B > 1 else 0, B - 1})
    cb = Cacheback(B, LL, FL, LC, FC, 32, 8, 8, 32000, 8, 8, 64)
    tabs = {b: oracle.OracleTable(LL, FL, LC, FC) for b in check}
    d, zero = dev(toks), torch.zeros(B, dtype=torch.int32, device="cuda")
    for lo, hi in ((np.zeros(B, np.int32), n1), (n1, n2)):
        cb.cb_update_bulk(d, dev(lo), dev(hi))
        for b in check:
            tabs[b].update(toks[b], int(lo[b]), int(hi[b]))
        _assert_tables_equal(cb, tabs, check)
    st, cnt = cb.cb_poll_status()
    assert st == 0 and cnt["inserts"] == int(np.maximum(n2 - w + 1, 0).sum())
