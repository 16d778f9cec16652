"""The walk that takes two whole units of one row tile at a time: the same shares as the walk over single units, whatever the ranges cut."""
import numpy as np
import pytest

from tests import test_attn_schedule as single
from tests.harness import stream_k_shares
from tests.test_attn_schedule import SHAPES, _cfg, walk  # noqa: F401  (walk is a fixture)


@pytest.fixture(scope="module")
def walk_pairs(tmp_path_factory):
    loop = single._SHIM.index("while (wk.next(p, &u)) {")
    body = single._SHIM[loop:].replace("while (wk.next(p, &u)) {", """while (wk.next_pair(p, &u)) for (int both = u.nrt == kTwoHeads, hd = 0; hd <= both; ++hd) {
                if (both) { if (hd == 0 && (u.t0 || u.t1 != u.tiles || u.kh + 2 > p.Hkv)) return 2; u.nrt = 1; u.kh += hd; }""", 1)
    old, single._SHIM = single._SHIM, single._SHIM[:loop] + body
    try:
        yield single.walk.__wrapped__(tmp_path_factory) if hasattr(single.walk, "__wrapped__") else single.walk(tmp_path_factory)
    finally:
        single._SHIM = old


@pytest.mark.parametrize("batch,hq,hkv,T,d,lo,hi", SHAPES + [(40, 6, 3, 20, 128, 0, 400), (9, 40, 40, 1, 64, 1, 130), (2, 5, 5, 128, 128, 700, 900)])
def test_pairs_are_the_single_units(walk_pairs, batch, hq, hkv, T, d, lo, hi):
    cfg = _cfg(batch, hq, hkv, T, d)
    rng = np.random.default_rng(batch)
    ctx = rng.permutation(np.round(np.linspace(lo, hi, batch)).astype(np.int64))
    for n in (np.full(batch, T), rng.integers(0, T + 1, batch)):
        for n_ctas in (148, 160, 7, 1):
            assert walk_pairs(cfg, ctx, n, n_ctas) == stream_k_shares(cfg, ctx, n, n_ctas)
