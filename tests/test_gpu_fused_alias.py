"""GPU: acceptance + update + draft in one launch where the next tree goes into the verified tree's own arrays, against the same call with
arrays of its own: most of the grid's CTAs belong to rows that the verified tree does not have, among them rows that the next tree
has, in grids that are resident at once and in larger ones; empty trees, trees of one node and full ones."""
import numpy as np
import pytest
import torch

from tests.harness import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,V,LL,FC,dtype", [(1, 128, 40000, 1, 8, torch.bfloat16), (3, 64, 5000, 2, 4, torch.float32), (96, 128, 20000, 1, 8, torch.bfloat16),
                                               (40, 128, 9000, 1, 40, torch.float32), (200, 33, 3000, 1, 4, torch.float32), (16, 1, 700, 2, 4, torch.float32)])
def test_next_tree_in_the_verified_trees_arrays(B, T, V, LL, FC, dtype):
    from paper_2511_21699_b200 import Cacheback
    FL, depth, N, steps = 3, 9, 600, 30
    rng = np.random.default_rng(B + T)
    text = rng.integers(0, 12, (B, N)).astype(np.int32)
    text[:, 60:] = text[:, :-60]
    text[2::3] = rng.integers(0, V, (len(text[2::3]), N))          # sequences that the drafter has nothing for: trees of one node
    a, b = (Cacheback(B, LL, FL, 1024, FC, T, T // 4, depth, V, 8, 8, 64) for _ in range(2))
    length = rng.integers(1, 200, B).astype(np.int32)
    toks = [dev(np.where(np.arange(N)[None] < length[:, None], text, 0)) for _ in range(2)]
    n = [dev(length) for _ in range(2)]
    tree = []
    for cb, t, l in zip((a, b), toks, n):
        cb.cb_update(t, torch.zeros_like(l), l)
        tree.append(cb.cb_draft_tree(t, l))
        tree[-1]["n_nodes"][::7] = 0                              # emits nothing; the next tree has a root again
    spare = b.alloc_tree()
    x = torch.empty(B, T, V, dtype=dtype, device="cuda")
    g = torch.Generator(device="cuda")
    sizes = set()
    for step in range(steps):
        g.manual_seed(step)
        x.normal_(generator=g)
        # on the path that follows the text, the text's next token is the maximum
        dep = tree[0]["depth"].long().clamp(min=0)
        at = (n[0].long()[:, None] + dep).clamp(max=N - 1)
        nxt = torch.from_numpy(text).cuda().long().gather(1, at)
        if step % 4:                                              # every fourth step all children fail
            x.scatter_(2, nxt[:, :, None], 32.0)
        ra = a.cb_accept_update_draft_tree(tree[0], x, toks[0], n[0])
        rb = b.cb_accept_update_draft_tree(tree[1], x, toks[1], n[1], next_tree=spare)
        tree[1], spare = spare, tree[1]
        for k in ("n_accept", "accept_nodes", "out_tokens", "target_ids"):
            assert torch.equal(ra[k], rb[k]), (step, k)
        for k in ("n_nodes", "tokens", "parent", "depth", "mask"):
            assert torch.equal(tree[0][k], tree[1][k]), (step, k)
        assert torch.equal(n[0], n[1]) and torch.equal(toks[0], toks[1])
        sizes |= set(tree[0]["n_nodes"].tolist())
    assert T == 1 or max(sizes) > 1 + min(sizes)                  # trees grew into rows that the ones before did not have
    assert a.cb_poll_status()[0] == b.cb_poll_status()[0] == 0
