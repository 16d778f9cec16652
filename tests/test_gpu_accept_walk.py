"""GPU parity of the acceptance walk over the forms of a tree: chains of up to 127 levels (as many rounds of the walk as there can be),
stars, single nodes, trees of every size around a warp's lanes, breaks at every level, malformed parents and depths; through target
ids and through logits, with grids that take their chunk at once (batch 1) and grids that do not."""
import numpy as np
import pytest
import torch

from tests.harness import dev

pytestmark = pytest.mark.gpu


def _trees(kind, B, T, rng):
    par = np.full((B, T), -1, np.int32)
    dep = np.full((B, T), -1, np.int32)
    n = np.full(B, T, np.int32) if kind != "ragged" else rng.integers(0, T + 1, B).astype(np.int32)
    for b in range(B):
        dep[b, :1] = 0
        for i in range(1, n[b]):
            p = {"chain": i - 1, "star": 0}.get(kind, i - 1 if rng.random() < 0.6 else int(rng.integers(0, i)))
            par[b, i], dep[b, i] = p, dep[b, p] + 1
        par[b, n[b]:] = dep[b, n[b]:] = -1
        if n[b] == 0:
            dep[b, 0] = -1
    return par, dep, n


@pytest.mark.parametrize("kind", ["chain", "star", "random", "ragged"])
@pytest.mark.parametrize("T", [1, 2, 31, 32, 33, 64, 65, 96, 127, 128])
def test_walk_over_forms_of_trees(oracle, kind, T):
    from paper_2511_21699_b200 import Cacheback
    rng = np.random.default_rng(T * 7 + len(kind))
    dmax, V, B = max(T - 1, 1), 57, 33
    for batch, dtype in ((1, torch.float32), (B, torch.bfloat16)):
        par, dep, n = _trees(kind, batch, T, rng)
        tok = rng.integers(0, 50, (batch, T)).astype(np.int32)
        tgt = rng.integers(0, 50, (batch, T)).astype(np.int32)
        for b in range(batch):
            for i in range(1, n[b]):                            # most nodes match their parent's target
                if rng.random() < (0.97 if kind == "chain" else 0.8):
                    tok[b, i] = tgt[b, par[b, i]]
        cb = Cacheback(batch, 2, 4, 64, 4, T, 0, dmax, V, 8, 8, 64)
        tree = dict(tokens=dev(tok), parent=dev(par), depth=dev(dep), n_nodes=dev(n))
        x = np.zeros((batch, T, V), np.float32)
        np.put_along_axis(x, tgt[:, :, None], 1.0, 2)
        for res in (cb.cb_accept(tree, target_ids=dev(tgt)), cb.cb_accept(tree, logits=dev(x, dtype))):
            r = {k: v.cpu().numpy() for k, v in res.items()}
            for b in range(batch):
                t = np.where(np.arange(T) < n[b], tgt[b], -1).astype(np.int32)
                m, nodes, out = oracle.accept(tok[b], par[b], dep[b], int(n[b]), t, dmax) if n[b] else (0, np.full(dmax, -1), np.full(dmax + 1, -1))
                assert r["n_accept"][b] == m and np.array_equal(r["accept_nodes"][b], nodes) and np.array_equal(r["out_tokens"][b], out), (kind, T, b)
        assert cb.cb_poll_status()[0] == 0


def test_malformed_trees_are_not_followed():
    """Parents at or behind their node, negative ones, depths outside the range: such nodes (and those below a bad parent) count as
    unverified, the others as ever."""
    from paper_2511_21699_b200 import Cacheback
    T, dmax = 8, 6
    tok = np.array([[1, 2, 3, 4, 5, 6, 7, 8]], np.int32)
    tgt = np.array([[2, 3, 4, 5, 6, 7, 8, 9]], np.int32)         # the chain 0 -> 1 -> 2 -> ... matches throughout
    chain, depth = [-1, 0, 1, 2, 3, 4, 5, 6], [0, 1, 2, 3, 4, 5, 6, 7]
    for at, p, want in ((3, 5, 2), (3, 3, 2), (4, -1, 3), (1, -7, 0), (7, 7, 6)):
        par, dep = np.array([chain], np.int32), np.array([depth], np.int32)
        par[0, at] = p
        cb = Cacheback(1, 2, 4, 64, 4, T, 0, dmax, 57, 8, 8, 64)
        r = cb.cb_accept(dict(tokens=dev(tok), parent=dev(par), depth=dev(dep), n_nodes=dev(np.array([T], np.int32))), target_ids=dev(tgt))
        assert int(r["n_accept"][0]) == want, (at, p)
        assert r["accept_nodes"][0].cpu().tolist() == list(range(1, want + 1)) + [-1] * (dmax - want)
        assert r["out_tokens"][0].cpu().tolist() == list(range(2, want + 3)) + [-1] * (dmax - want)


@pytest.mark.parametrize("batch", [1, 40])                       # a chunk's loads at once, and four at a time
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("V", [1, 3, 4, 7, 8, 9, 1023, 1025, 2047, 2049, 8191, 8193, 16385, 32771])
def test_first_maximum_among_ties(V, dtype, batch):
    """Five values and -inf only, so that the maximum stands many times in a vector of logits, in several of a thread's, a warp's and a
    block's; rows of one value throughout; rows at odd offsets.  The targets are exact."""
    from paper_2511_21699_b200 import Cacheback
    T = 12
    g = torch.Generator().manual_seed(V)
    store = torch.randint(-2, 3, (batch, T, V + 3), generator=g).float()
    store[torch.rand(store.shape, generator=g) < 0.3] = float("-inf")
    store[:, 1], store[:, 2] = -0.0, float("-inf")
    store[:, 3, : V // 2] = -3.0
    x = store.to(dtype).cuda()[:, :, :V]
    cb = Cacheback(batch, 2, 4, 64, 4, T, 0, T, V, 8, 8, 64)
    chain = torch.arange(T, dtype=torch.int32).repeat(batch, 1)
    r = cb.cb_accept(dict(tokens=torch.zeros_like(chain).cuda(), parent=(chain - 1).cuda(), depth=chain.cuda(),
                          n_nodes=torch.full((batch,), T, dtype=torch.int32).cuda()), logits=x)
    assert np.array_equal(r["target_ids"].cpu().numpy(), store[:, :, :V].numpy().argmax(2))
    assert cb.cb_poll_status()[0] == 0
