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
    if not scratch:                                             # the counters are those of the windows one after the other
        one = Cacheback(B, LL, FL, LC, FC, 32, 8, 8, 32000, 8, 8, 64)
        one.cb_update(d, zero, dev(n1))
        one.cb_update(d, dev(n1), dev(n2))
        ref = one.cb_poll_status()[1]
        assert [cnt[k] for k in ("inserts", "leader_evictions", "follower_evictions")] == [ref[k] for k in ("inserts", "leader_evictions", "follower_evictions")]
    cb.cb_reset()                                               # a table that was in use, empty again
    cb.cb_update_bulk(d, zero, dev(n1))
    tabs = {b: oracle.OracleTable(LL, FL, LC, FC) for b in check}
    for b in check:
        tabs[b].update(toks[b], 0, int(n1[b]))
    _assert_tables_equal(cb, tabs, check)
    assert cb.cb_poll_status()[0] == 0


@pytest.mark.parametrize("few,many,n,LC", [(128, 512, 1500, 1024), (128, 1024, 50, 1024)])
def test_runs_in_order_go_side_by_side(few, many, n, LC):
    """Runs that could evict a leader, or are short, are chains of one warp each: four (eight) times as many sequences take about as long
    where all of them are at work at once.  One block after the other took 3.5 (5.8) times as long, all at once 1.1 (1.4)."""
    from paper_2511_21699_b200 import Cacheback
    took = []
    for B in (few, many):
        cb = Cacheback(B, 2, 4, LC, 4, 32, 8, 8, 32000, 8, 8, 64)
        d = dev(_tokens("zipf", 1, n, np.random.default_rng(3)).repeat(B, 0))
        zero, end = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.full((B,), n, dtype=torch.int32, device="cuda")
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            cb.cb_update_bulk(d, zero, end)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        took.append(min(times))
        assert cb.cb_poll_status()[0] == 0
    assert took[1] < 2.2 * took[0], took


@pytest.mark.parametrize("form", ["rows", "transposed", "strided", "flat"])
def test_one_sequence_whatever_its_stride(oracle, form):
    """A batch of one: the stride of its only row means nothing, and a run longer than a block takes is not lost by it."""
    from paper_2511_21699_b200 import Cacheback
    LL, FL, LC, FC, n = 2, 3, 16384, 4, 10000
    toks = _tokens("zipf", 1, n, np.random.default_rng(9))
    d = dev(toks)
    d = dict(rows=d, transposed=d.reshape(n, 1).clone().t(), strided=torch.as_strided(d, (1, n), (77, 1)), flat=d[0])[form]
    assert d.is_contiguous() and (form == "rows") == (d.stride(0) == n)
    cb = Cacheback(1, LL, FL, LC, FC, 32, 8, 8, 500, 8, 8, 64)
    zero, n1, n2 = (dev(np.array([x], np.int32)) for x in (0, 9000, 9500))
    tab = oracle.OracleTable(LL, FL, LC, FC)
    cb.cb_update_bulk(d, zero, n1)
    tab.update(toks[0], 0, 9000)
    _assert_tables_equal(cb, {0: tab}, [0])
    cb.cb_update_bulk(d, n1, n2)
    tab.update(toks[0], 9000, 9500)
    _assert_tables_equal(cb, {0: tab}, [0])
    assert cb.cb_poll_status()[0] == 0
    if form != "flat":                                          # the call that appends to the row takes its room from the tensor too
        tree = cb.cb_draft_tree(d, n2)
        logits = torch.zeros(1, 32, 500, device="cuda")
        logits[..., 3] = 1.0
        cb.cb_accept_update_draft_tree(tree, logits, d, n2)
        assert cb.cb_poll_status()[0] == 0 and int(n2[0]) > 9500


def test_run_longer_than_its_row_is_reported():
    """n_new beyond the row of several: the windows that no kernel is left to take are reported."""
    from paper_2511_21699_b200 import Cacheback
    cb = Cacheback(3, 2, 3, 16384, 4, 32, 8, 8, 500, 8, 8, 64)
    t = torch.zeros(3, 8000, dtype=torch.int32, device="cuda")
    n = dev(np.array([100, 9000, 100], np.int32))
    cb.cb_update_bulk(t, torch.zeros_like(n), n)
    assert cb.cb_poll_status()[0] == 1                          # CB_ERR_INVALID_ARG
    assert [len(cb.cb_table_dump_arrays(b)[0]) for b in range(3)] == [1, 0, 1]
