"""GPU: the drafting kernels' shared memory around the 48 KB that a block gets without asking, static part included: sizes whose dynamic
part alone is below 48 KB (44,288 to 49,140 bytes here), one below and one above; acceptance + update + draft in one launch against the
separate calls."""
import pytest
import torch

from tests.test_gpu_fused_short import test_fused_call_equals_separate_calls_from_short_histories as fused_equals_separate

pytestmark = pytest.mark.gpu

SIZES = [(4, 128, T) for T in range(100, 108)] + [(4, FC, 128) for FC in (77, 78, 82, 85, 86, 87, 88)] + [(1, 103, 105), (1, 128, 105), (1, 128, 106), (8, 128, 128)]


def _bytes(FL, FC, T):
    """Dynamic shared memory of a drafting block: nodes, mask rows, six arrays by leaf, staged followers."""
    leaves = min(T, (T - 1) // FL + 1)
    return 4 * ((3 + (T + 31) // 32) * T + 6 * leaves + leaves * FL * max(1, min(FC, T - 1)))


def test_sizes_lie_where_they_should():
    b = [_bytes(*s) for s in SIZES]
    assert min(b) < 44 * 1024 and max(b) > 64 * 1024 and sum(44256 < x <= 48 * 1024 for x in b) >= 12 and sum(48 * 1024 - 160 < x <= 48 * 1024 for x in b) >= 1


@pytest.mark.parametrize("FL,FC,T", SIZES)
def test_fused_call_around_the_unasked_limit(FL, FC, T):
    fused_equals_separate(1, FL, FC, T, 10, torch.bfloat16 if T % 2 else torch.float32)
