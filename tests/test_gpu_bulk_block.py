"""GPU parity: cb_update_bulk's runs of up to 8,192 windows, which blocks reduce in shared memory, against the oracle's sequential
update, at the sizes where that can go wrong: the ends of the range (63 / 64 windows, 8,191 / 8,192 / 8,193), one distinct window and
8,192 of them, leaders with more followers than an entry holds, more sequences than blocks, tables that hold leaders already (and
places that deleted ones left), runs that could evict a leader beside runs that cannot, every leader and follower length."""
import numpy as np
import pytest
import torch

from tests.harness import dev
from tests.test_gpu_table import _assert_tables_equal

pytestmark = pytest.mark.gpu


def _tokens(kind, B, n, rng):
    if kind == "one":                                          # a single distinct window
        return np.full((B, n), 7, np.int32)
    if kind == "distinct":                                     # no token twice
        return np.stack([rng.permutation(n * 2)[:n] for _ in range(B)]).astype(np.int32)
    if kind == "pair":                                         # one leader with very many followers
        t = rng.integers(100, 30000, (B, n))
        t[:, ::2] = 5
        return t.astype(np.int32)
    return np.minimum(rng.zipf(1.2, (B, n)) - 1, 30000).astype(np.int32)


CASES = [  # LL, FL, LC, FC, kind of text, windows of the sequences' first run, windows of a second one
    (3, 4, 16384, 4, "zipf", [63, 64, 65, 1000, 8191, 8192, 8193, 0], [70, 8192, 1, 8000, 64, 0, 300, 5000]),
    (2, 3, 16384, 6, "distinct", [8192, 4096, 4097], [64, 100, 8000]),
    (1, 3, 16384, 8, "one", [8192, 64], [8192, 64]),
    (1, 5, 8192, 128, "pair", [4000, 2500, 700], [600, 3000, 64]),
    (1, 1, 8192, 40, "zipf", [5000, 100], [3000, 2000]),
    (4, 8, 16384, 1, "zipf", [6000, 8192], [2000, 300]),
    (2, 8, 512, 3, "zipf", [100, 400, 700, 64], [500, 100, 90, 448]),     # first runs that fit the leader capacity and that do not
    (2, 4, 1024, 4, "zipf", [64 + k % 40 for k in range(200)], [90] * 200),
]


@pytest.mark.parametrize("LL,FL,LC,FC,kind,first,second", CASES)
@pytest.mark.parametrize("scratch", [False, True])
def test_bulk_runs_in_blocks(oracle, LL, FL, LC, FC, kind, first, second, scratch):
    from paper_2511_21699_b200 import Cacheback
    B, w = len(first), LL + FL
    n1 = np.array([x + w - 1 if x else 0 for x in first], np.int32)
    n2 = (n1 + np.array(second)).astype(np.int32)
    rng = np.random.default_rng(LL * 100 + FL)
    toks = _tokens(kind, B, int(n2.max()) + 8, rng)
    cb = Cacheback(B, LL, FL, LC, FC, 32, 8, 8, 32000, 8, 8, 64)
    if scratch:
        cb.cb_bulk_scratch_attach(int(n2.sum()))
    check = list(range(B)) if B <= 8 else [0, 1, 77, 147, 148, 149, 198, 199]
    tabs = {b: oracle.OracleTable(LL, FL, LC, FC) for b in check}
    d, zero = dev(toks), torch.zeros(B, dtype=torch.int32, device="cuda")
    cb.cb_update_bulk(d, zero, dev(n1))
    for b in check:
        tabs[b].update(toks[b], 0, int(n1[b]))
    _assert_tables_equal(cb, tabs, check)
    cb.cb_update_bulk(d, dev(n1), dev(n2))
    for b in check:
        tabs[b].update(toks[b], int(n1[b]), int(n2[b]))
    _assert_tables_equal(cb, tabs, check)
    st, cnt = cb.cb_poll_status()
    assert st == 0 and cnt["inserts"] == int(np.maximum(n2 - w + 1, 0).sum())
    cb.cb_reset()                                               # a table that was in use, empty again
    cb.cb_update_bulk(d, zero, dev(n1))
    tabs = {b: oracle.OracleTable(LL, FL, LC, FC) for b in check}
    for b in check:
        tabs[b].update(toks[b], 0, int(n1[b]))
    _assert_tables_equal(cb, tabs, check)
    assert cb.cb_poll_status()[0] == 0
