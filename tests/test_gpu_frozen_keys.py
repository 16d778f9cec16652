"""GPU parity of cb_frozen_build on either side of the line at which its leader table holds the leaders' tokens as one number (they fit 63
bits) or the position of an occurrence: every leader length, at the largest token that fits and the next, over corpora whose LC-th best
leader occurs once, twice and more, with all leaders taken and with leaders of more than 4,096 windows."""
import numpy as np
import pytest

from tests.test_gpu_frozen_groups import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("LL,top", [(1, (1 << 31) - 1), (2, (1 << 31) - 1), (3, (1 << 21) - 1), (3, 1 << 21), (4, (1 << 15) - 1), (4, 1 << 15), (4, (1 << 31) - 1),
                                    (1, 0), (4, 1)])
@pytest.mark.parametrize("LC", [1, 40, 1 << 15])
def test_leaders_as_numbers_and_as_positions(oracle, LL, top, LC):
    rng = np.random.default_rng(LL * 100 + LC)
    few = np.minimum(rng.zipf(1.6, 9000) - 1, top)               # counts of thousands
    low, high = rng.integers(0, min(top, 300) + 1, 3000), top - rng.integers(0, min(top, 300) + 1, 3000)   # both ends of the tokens
    once = rng.integers(0, top + 1, 4000)                        # mostly leaders of one window
    twice = np.tile(rng.integers(0, top + 1, 700), 2)
    _check(oracle, np.concatenate([few, low, high, once, twice]).astype(np.int32), LL, 2, LC, 3)
    _check(oracle, np.concatenate([once, [top]]).astype(np.int32), LL, 3, LC, 2)
