"""Compaction of a level with more big child tables than the warps' list holds (2,048): the rest are copied by one
thread each, whatever their size."""
import numpy as np
import pytest

import oracle
import paper_2606_17059_gb300 as g
from gpu_util import (assert_same_route, csr_from_lists, route_device, router_from_seqlists, same_snapshot,
                      seqlist_from_lists)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


# Nodes with this many children each: tables of 32, 64 or 128, and 256 slots or more.
@pytest.mark.parametrize("n_nodes,n_children", [(2300, 13), (2300, 40), (2100, 90)])
def test_more_big_tables_on_a_level_than_units(n_nodes, n_children):
    rng = np.random.default_rng(n_children)
    tail = rng.integers(1, 1 << 20, size=(n_nodes, n_children, 4)).tolist()
    seqs = [[1 + i, 7, 1000 * c + i] + tail[i][c] for i in range(n_nodes) for c in range(n_children)]
    r, o = router_from_seqlists([seqlist_from_lists(seqs)]), oracle.build_trees([seqlist_from_lists(seqs)])
    gone = [s for k, s in enumerate(seqs) if k % 5 < 3]  # three in five labels: the tree is compacted
    sl, op = seqlist_from_lists(gone), np.ones(len(gone), np.int32)
    assert r.apply_delta(0, op, sl) == 0
    o[0].apply_ops(op, sl, 0, len(gone))
    assert r.stats(0)["stale_label"] == 0
    assert same_snapshot(r.download(0), o[0].export())
    reqs = [seqs[k][: 3 + k % 5] for k in rng.integers(0, len(seqs), size=4000).tolist()]
    tok, off = csr_from_lists(reqs)
    gm, gp = route_device(r, tok, off, [0], 1)
    om, op_, _ = oracle.route(o, tok, off, [0], 1)
    assert_same_route(gm, gp, om, op_, "after compaction")


# A root of 32,768 slots (units of 256), and of 262,144 (units of 512).
@pytest.mark.parametrize("n", [8000, 40000])
def test_units_of_a_root(n):
    rng = np.random.default_rng(n)
    seqs = np.concatenate([np.arange(n)[:, None] * 7 + 1, rng.integers(1, 1 << 20, size=(n, 20))], axis=1).tolist()
    r, o = router_from_seqlists([seqlist_from_lists(seqs)]), oracle.build_trees([seqlist_from_lists(seqs)])
    gone = [s for k, s in enumerate(seqs) if k % 5 < 3]
    sl, op = seqlist_from_lists(gone), np.ones(len(gone), np.int32)
    assert r.apply_delta(0, op, sl) == 0
    o[0].apply_ops(op, sl, 0, len(gone))
    assert r.stats(0)["stale_label"] == 0
    assert same_snapshot(r.download(0), o[0].export())
