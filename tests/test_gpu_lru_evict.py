"""GPU parity of one eviction (lru_evict_kernel) against the oracle's one-token-at-a-time LRU trie: fan-outs around the
sizes at which a children table is read by a lane, a warp, the cluster, or more than once, and thresholds at every
kind of place (between stamps, inside one, inside an edge, in a run of edges of one stamp)."""
import random

import pytest

import oracle
import paper_2606_17059_gb300 as g
from gpu_util import same_snapshot
from oracle.lru import LRUTrie
from test_gpu_lru import _access, _insert, _oracle_export

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


def _evict_both(r, o, n):
    k = 0
    while k < n and o.evict() is not None:
        k += 1
    assert g.p2p_lru_evict(r.handle, 0, n) == k
    assert same_snapshot(r.download(0), _oracle_export(o)), n


# Children of the root and of an inner node; tables are up to a quarter live, the root's has 64 slots more.
@pytest.mark.parametrize("fan", [1, 2, 4, 5, 15, 17, 33, 63, 65, 130, 260, 600])
def test_eviction_at_fan_outs(fan):
    rng = random.Random(fan)
    seqs = [[rng.randrange(-(1 << 31), 1 << 31)] + [rng.randrange(3) for _ in range(rng.randint(0, 2))] for _ in range(fan)]
    seqs += [[9, 9] + [rng.randrange(-40, 4 * fan)] + [rng.randrange(3) for _ in range(rng.randint(0, 2))] for _ in range(fan)]
    r, o = g.Router(1), LRUTrie()
    g.p2p_lru_enable(r.handle, 0)
    _insert(r, 0, seqs, 1)
    for s in seqs:
        o.insert(s, 1)
    n = o.n_tokens
    for t, share in ((2, 0.05), (3, 0.1), (4, 0.0), (5, 0.2)):
        # Accesses that end inside edges leave runs of edges of one stamp, the boundary's among them.
        reqs = [list(rng.choice(seqs))[: rng.randint(1, 5)] for _ in range(max(1, fan // 4))]
        assert _access(r, 0, reqs, t).tolist() == [o.access(s, t) for s in reqs]
        _evict_both(r, o, max(1, int(share * n)))
    _evict_both(r, o, 1)
    assert g.p2p_lru_evict(r.handle, 0, 10**9) == o.n_tokens
    assert r.download(0)["label_off"].tolist() == [0]


def test_eviction_along_chains():
    """Edges cut by accesses into long runs, some of one stamp and some of several: every count from one token up."""
    rng = random.Random(5)
    base = [[rng.randrange(3) for _ in range(60)] for _ in range(4)]
    for n in (1, 2, 3, 5, 7, 11, 30, 59, 60, 61, 100):
        r, o = g.Router(1), LRUTrie()
        g.p2p_lru_enable(r.handle, 0)
        _insert(r, 0, base, 1)
        for s in base:
            o.insert(s, 1)
        t = 1
        for k in (55, 40, 40, 22, 7):
            t += rng.choice([0, 1])
            reqs = [s[: k + rng.randint(-3, 3)] for s in base[: rng.randint(1, 4)]]
            assert _access(r, 0, reqs, t).tolist() == [o.access(s, t) for s in reqs]
        _evict_both(r, o, n)
        _evict_both(r, o, n)


@pytest.mark.parametrize("fan,inner,kids", [(4500, 0, 0), (60, 40, 140)])
def test_eviction_of_large_tables(fan, inner, kids):
    """A root larger than the threads keep (8,192 slots), and more than 32 nodes of one level with tables that the
    whole cluster reads; stamps that differ in every byte, in one, and not at all."""
    rng = random.Random(fan)
    seqs = [[rng.randrange(-(1 << 31), 1 << 31), 3][: rng.randint(1, 2)] for _ in range(fan)]
    seqs += [[i, 7, 7, rng.randrange(1 << 20)] for i in range(inner) for _ in range(kids)]
    r, o = g.Router(1), LRUTrie()
    g.p2p_lru_enable(r.handle, 0)
    _insert(r, 0, seqs, 5)
    for s in seqs:
        o.insert(s, 5)
    _evict_both(r, o, 30)
    for t in (6, 300, 70000, (1 << 24) + 9, (1 << 32) - 2):
        reqs = [list(rng.choice(seqs)) for _ in range(40)]
        assert _access(r, 0, reqs, t).tolist() == [o.access(s, t) for s in reqs]
        _evict_both(r, o, 25)


def test_accesses_that_end_around_the_steps_of_a_compare():
    """Edges left, or followed to the end, after every count of tokens around 32, 256, 512 and 1,024."""
    rng = random.Random(11)
    edges = [n + d for n in (32, 256, 512, 544, 768, 1024, 1056) for d in (-1, 0, 1)]
    base = [rng.randrange(1000) for _ in range(1100)]
    r, o = g.Router(1), LRUTrie()
    g.p2p_lru_enable(r.handle, 0)
    seqs = [base, base[:512] + [2000, 1]]
    _insert(r, 0, seqs, 1)
    for s in seqs:
        o.insert(s, 1)
    for t, k in enumerate(edges, 2):
        for reqs in ([base[:k] + [3000]], [base[:k]]):
            assert _access(r, 0, reqs, t).tolist() == [o.access(s, t) for s in reqs]
    assert same_snapshot(r.download(0), _oracle_export(o))
    _evict_both(r, o, 40)
