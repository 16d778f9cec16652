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


def test_a_depth_beyond_the_tree_and_a_length_below_zero_stay_inside_the_kept_tail():
    """Malformed inputs: a tree whose one accepted node names a depth of 300 (the step emits 301 places, of which the launch keeps 256 on
    chip), and a sequence of negative length (nothing is appended, reported)."""
    from paper_2511_21699_b200 import Cacheback
    V, T, N = 64, 8, 1000
    cb = Cacheback(2, 2, 3, 256, 4, T, 2, 400, V, 8, 8, 64)
    toks = torch.zeros(2, N, dtype=torch.int32, device="cuda")
    toks[:, :500] = torch.arange(500, device="cuda") % 50
    tree = cb.alloc_tree()
    for k, fill in (("tokens", -1), ("parent", -1), ("depth", -1), ("mask", 0)):
        tree[k].fill_(fill)
    tree["n_nodes"].copy_(dev(np.array([2, 1], np.int32)))
    tree["tokens"][:, 0] = 49
    tree["depth"][:, 0] = 0
    tree["tokens"][0, 1], tree["parent"][0, 1], tree["depth"][0, 1] = 7, 0, 300
    logits = torch.zeros(2, T, V, device="cuda")
    logits[..., 7] = 1.0
    n = dev(np.array([500, -5], np.int32))
    nxt = cb.alloc_tree()
    res = cb.cb_accept_update_draft_tree(tree, logits, toks, n, next_tree=nxt)
    assert cb.cb_poll_status()[0] == 1                          # CB_ERR_INVALID_ARG, of the second sequence
    assert res["n_accept"].tolist() == [300, 0] and n.tolist() == [801, -5]
    assert (res["out_tokens"][0, :299] == -1).all() and res["out_tokens"][0, 299:301].tolist() == [7, 7]
    assert (toks[0, 500:756] == -1).all() and not toks[0, 756:].any() and torch.equal(toks[1, :500], torch.arange(500, device="cuda", dtype=torch.int32) % 50)
    assert int(nxt["n_nodes"][1]) == 0
