"""GPU: acceptance + append + update + draft in one launch against the four separate calls, from histories shorter than a window on (the
end of the history that the launch keeps in shared memory then starts at the sequence's beginning) up to several windows, through
steps that emit one to many tokens, with trees of one leaf, follower lists below and above a warp's lanes, and a size cap that cuts levels."""
import numpy as np
import pytest
import torch

from tests.harness import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("LL,FL,FC,T,depth", [(1, 1, 2, 5, 3), (2, 4, 4, 64, 8), (3, 5, 8, 128, 10), (1, 3, 128, 96, 24), (4, 8, 40, 33, 16), (2, 3, 33, 1, 4)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_fused_call_equals_separate_calls_from_short_histories(LL, FL, FC, T, depth, dtype):
    from paper_2511_21699_b200 import Cacheback
    B, V, N = 18, 40, 400
    rng = np.random.default_rng(LL * 100 + FL * 10 + FC)
    # text of few tokens with a period in it, so that windows repeat and drafts are accepted
    text = rng.integers(0, 6, (B, N)).astype(np.int32)
    text[:, 40:] = text[:, :-40][:, : N - 40]
    a, b = (Cacheback(B, LL, FL, 256, FC, T, T // 4, depth, V, 8, 8, 64) for _ in range(2))
    length = np.arange(1, B + 1).astype(np.int32)
    toks = [dev(np.where(np.arange(N)[None] < length[:, None], text, 0)) for _ in range(2)]
    n = [dev(length) for _ in range(2)]
    zero = torch.zeros(B, dtype=torch.int32, device="cuda")
    for cb, t, l in zip((a, b), toks, n):
        cb.cb_update(t, zero, l)
    tree = [a.cb_draft_tree(toks[0], n[0]), b.cb_draft_tree(toks[1], n[1])]
    arange = torch.arange(N, device="cuda")[None]
    for step in range(12):
        # the target: the text's continuation for nodes on the path that follows it, another token elsewhere
        par, tok, dep = (tree[0][k].cpu().numpy() for k in ("parent", "tokens", "depth"))
        pos = n[0].cpu().numpy()
        x = rng.standard_normal((B, T, V)).astype(np.float32)
        for s in range(B):
            on = {0}
            for i in range(T):
                if i > 0 and par[s, i] in on and tok[s, i] == text[s, min(pos[s] - 1 + dep[s, i], N - 1)]:
                    on.add(i)
                x[s, i, text[s, min(pos[s] + max(dep[s, i], 0), N - 1)] if i in on else 39] = 16.0
        x = dev(x, dtype)
        ra = a.cb_accept_update_draft_tree(tree[0], x, toks[0], n[0])
        rb = b.cb_accept(tree[1], logits=x)
        m = rb["n_accept"]
        new = n[1] + m + 1
        out = rb["out_tokens"].gather(1, (arange - n[1][:, None]).clamp(0, depth).long())
        toks[1] = torch.where((arange >= n[1][:, None]) & (arange < new[:, None]), out, toks[1]).contiguous()
        b.cb_update(toks[1], n[1], new)
        n[1] = new
        tree[1] = b.cb_draft_tree(toks[1], n[1])
        for k in ("n_accept", "accept_nodes", "out_tokens", "target_ids"):
            assert torch.equal(ra[k], rb[k]), (step, k)
        assert torch.equal(n[0], n[1]) and torch.equal(toks[0], toks[1])
        for k in ("n_nodes", "tokens", "parent", "depth", "mask"):
            assert torch.equal(tree[0][k], tree[1][k]), (step, k)
    for s in range(B):
        assert a.cb_table_dump(s) == b.cb_table_dump(s)
    sa, ca = a.cb_poll_status()
    sb, cb_ = b.cb_poll_status()
    assert sa == sb == 0 and ca["inserts"] == cb_["inserts"] and ca["query_hits"] == cb_["query_hits"]
