"""GPU parity of cb_frozen_build for leaders of so many distinct windows that the best are looked for by a histogram of their counts: as many
ties at the deciding count as are copied to shared memory and one more, none that occurs twice, counts beyond the histogram's last bin."""
import numpy as np
import pytest

from tests.test_gpu_frozen_groups import _check

pytestmark = pytest.mark.gpu


def _one_leader(followers, rng):
    """Leader 0 followed by the given tokens (from 10 on), in random order."""
    f = rng.permutation(np.asarray(followers))
    return np.stack([np.zeros(len(f), np.int64), f + 10], 1).reshape(-1).astype(np.int32)


@pytest.mark.parametrize("FC", [1, 8, 128])
@pytest.mark.parametrize("kind", ["zipf", "once", "2047 twice", "2048 twice", "2049 twice", "few often", "many often"])
def test_big_leader(oracle, kind, FC):
    rng = np.random.default_rng(len(kind) + FC)
    once = np.arange(100000, 106000)
    if kind == "zipf":
        f = np.minimum(rng.zipf(1.15, 60000), 1 << 20)
    elif kind == "once":
        f = once
    elif kind.endswith("twice"):
        f = np.concatenate([np.repeat(rng.choice(90000, int(kind.split()[0]), replace=False), 2), once])
    elif kind == "few often":                                   # FC of them do not reach the last bin
        f = np.concatenate([np.repeat(np.arange(FC - 1), 1500), np.repeat(np.arange(500, 600), 3), once])
    else:                                                       # more than FC in the last bin, ties among them
        f = np.concatenate([np.repeat(np.arange(FC + 5), 1100 + np.arange(FC + 5) // 3), once])
    _check(oracle, _one_leader(f, rng), 1, 1, 300, FC)
