"""GPU parity of cb_frozen_build where its steps change hands, against the oracle's counting: leaders with as many windows as a warp, a
block of either size and the second hash table take (and one more), all of them different, all the same or tied in count; the LC-th
best leader among ties and with a count that one histogram does not hold; every leader length; negative tokens; tables that are used
again."""
import numpy as np
import pytest

from tests.harness import dev

pytestmark = pytest.mark.gpu


def _blocks(counts, FL, spread, rng):
    """A stream of blocks [leader, follower ...]: counts[k] of leader k, in random order, follower tokens from `spread` values."""
    lead = np.repeat(np.arange(len(counts)), counts)
    rng.shuffle(lead)
    fol = 100 + rng.integers(0, spread, (len(lead), FL)) if spread else np.full((len(lead), FL), 100)
    return np.concatenate([lead[:, None], fol], 1).reshape(-1).astype(np.int32)


def _check(oracle, corpus, LL, FL, LC, FC):
    from paper_2511_21699_b200 import FrozenTable
    t = FrozenTable(LL, FL, LC, FC)
    for _ in range(2):                                          # the second build finds the table of the first
        t.cb_frozen_build(dev(corpus))
        L, nf, F = t.cb_frozen_dump()
        oL, onf, oF = oracle.frozen_build(corpus, LL, FL, LC, FC)
        assert np.array_equal(L, oL) and np.array_equal(nf, onf) and np.array_equal(F, oF)


@pytest.mark.parametrize("spread", [0, 2, 40, 1 << 20])          # one follower, ties of few kinds, many kinds, all different
@pytest.mark.parametrize("FL,FC", [(1, 1), (3, 8), (4, 33), (8, 128)])
def test_groups_of_every_size(oracle, spread, FL, FC):
    rng = np.random.default_rng(spread + FL)
    corpus = _blocks([1, 2, 31, 32, 33, 64, 511, 512, 513, 1000, 4095, 4096, 4097, 6000], FL, spread, rng)
    _check(oracle, corpus, 1, FL, 64, FC)
    _check(oracle, corpus, 1, FL, 1 << 17, FC)


@pytest.mark.parametrize("LL", [1, 2, 3, 4])
@pytest.mark.parametrize("LC", [1, 2, 3, 7, 300, 5000])
def test_leaders_at_the_cut(oracle, LL, LC):
    rng = np.random.default_rng(LL * 10 + LC)
    few = rng.integers(0, 3, 30000)                              # counts above 4,095
    flat = rng.integers(0, 70000, 20000)                         # nearly all counts tie; tokens of two digits and more
    big = (np.int64(1) << 31) - 1 - rng.integers(0, 50, 3000)    # tokens of three digits
    _check(oracle, np.concatenate([few, flat, big]).astype(np.int32), LL, 3, LC, 5)


def test_negative_tokens_are_reported_and_their_windows_left_out(oracle):
    from paper_2511_21699_b200 import FrozenTable, CachebackError
    rng = np.random.default_rng(5)
    a, b = rng.integers(0, 50, 3000).astype(np.int32), rng.integers(0, 50, 2000).astype(np.int32)
    t = FrozenTable(2, 3, 512, 4)
    with pytest.raises(CachebackError, match="invalid argument"):
        t.cb_frozen_build(dev(np.concatenate([a, [-1], b]).astype(np.int32)))
    L, nf, F = t.cb_frozen_dump()
    # the same windows without the token: no two-token leader and its follower may span the gap
    pad = np.arange(1 << 20, (1 << 20) + 8, dtype=np.int32)      # windows that touch the padding have leaders or followers of their own
    got = {tuple(l): [tuple(f) for f in F[i][: nf[i]]] for i, l in enumerate(L)}
    oL, onf, oF = oracle.frozen_build(np.concatenate([a, pad, b]).astype(np.int32), 2, 3, 1 << 14, 128)
    want = {tuple(l): [tuple(f) for f in oF[i][: onf[i]] if max(f) < 1 << 20] for i, l in enumerate(oL) if max(l) < 1 << 20}
    for l, fs in got.items():
        assert set(fs) <= set(want[l])
    _check(oracle, a, 2, 3, 512, 4)                              # a clean corpus afterwards
