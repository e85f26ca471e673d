"""Deltas whose first pool runs start at one place and differ in length: what one op's run is found to share with an
interned label holds for another op only as far as that op's own run goes.  Against the CPU oracle, through the bulk
rounds and (with one op of three runs in the call) through the delta kernel alone."""
import numpy as np
import pytest

import oracle
import paper_2606_17059_gb300 as g
import workload as wl
from gpu_util import router_from_seqlists, same_snapshot, seqlist_from_lists

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


# The shorter run ends within the label, at its end less one, or after what a lane compares alone (9 and 128 tokens).
@pytest.mark.parametrize("cut", [10, 64, 129, 150, 299])
@pytest.mark.parametrize("order", ["long first", "short first"])
@pytest.mark.parametrize("alone", [False, True], ids=["bulk rounds", "delta kernel"])
def test_runs_of_one_start_and_several_lengths(cut, order, alone):
    rng = np.random.default_rng(cut)
    L, n = 300, 96
    labels = [np.concatenate([[5000 + k], rng.integers(0, 50, L - 1)]) for k in range(n)]
    held = [np.concatenate([x, [7000]]) for x in labels] + [np.concatenate([x, [7001, 3]]) for x in labels]
    pool, ops, sb, so, sl = [], [], [0], [], []

    def add(op, runs):
        ops.append(op)
        for at, ln in runs:
            so.append(at)
            sl.append(ln)
        sb.append(len(so))

    at, size = [], 0
    for k in range(n):  # per label: its tokens, then others in the place of its rest, then the rest itself
        other = labels[k][cut:].copy()
        other[(L - cut) // 2] += 1000
        rest = np.concatenate([labels[k][cut:], [7000]])
        at.append((size, size + L, size + L + (L - cut)))
        pool += [labels[k], other, rest]
        size += L + (L - cut) + len(rest)
    for k in range(n):
        full, other, rest = at[k]
        long_op = [(0, [(full, L)])]
        short_ops = [(0, [(full, cut), (other, L - cut)]),  # leaves the label inside
                     (1, [(full, cut), (other, L - cut)]),  # ... and goes again
                     (1, [(full, cut), (rest, L - cut + 1)]),  # a held sequence in two runs
                     (0, [(full, cut), (other, 1 + (L - cut) // 2)])]
        for op, runs in (long_op + short_ops if order == "long first" else short_ops + long_op):
            add(op, runs)
    if alone:
        add(0, [(0, 1), (1, 1), (2, 1)])
    q = wl.SeqList(np.array(sb, np.int64), np.array(so, np.int64), np.array(sl, np.int32),
                   np.concatenate(pool).astype(np.int32))
    sls = [seqlist_from_lists([x.tolist() for x in held])]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    op = np.array(ops, np.int32)
    assert r.apply_delta(0, op, q) == o[0].apply_ops(op, q)
    assert same_snapshot(r.download(0), o[0].export())


@pytest.mark.parametrize("seed", range(4))
def test_sequences_of_many_runs_share_nothing_by_their_place(seed):
    """Ops of three runs are put together in scratch, where one sequence after another has the same place: what the
    last one matched says nothing of the next.  They differ early or late within a label, below a node of few
    children and of many (which the kernel starts from directly)."""
    rng = np.random.default_rng(seed)
    L, n = 200, 40
    labels = [np.concatenate([[5000 + k], rng.integers(0, 50, L - 1)]) for k in range(n)]
    held, seqs, ops = [], [], []
    for k in range(n):
        held += [np.concatenate([labels[k], [7000 + j, 1, 2]]) for j in range(2 if k % 2 else 70)]
        for j in range(4):
            off = labels[k].copy()
            off[[1, 70, 130, L - 1][j]] += 1000
            seqs += [np.concatenate([labels[k], [9000 + j]]), np.concatenate([off, [7000 + j, 1, 2]])]
            ops += [0, int(rng.integers(2))]
        seqs += [held[-1], np.concatenate([labels[k][: L - 1], [6000, 7000]])]
        ops += [1, 0]
    sb, so, sl, pool = [0], [], [], []
    for s in seqs:
        a, b = sorted(rng.integers(0, len(s) + 1, 2))
        for lo, hi in ((0, a), (a, b), (b, len(s))):
            so.append(len(pool))
            sl.append(hi - lo)
            pool.extend(s[lo:hi])
        sb.append(len(so))
    q = wl.SeqList(np.array(sb, np.int64), np.array(so, np.int64), np.array(sl, np.int32), np.array(pool, np.int32))
    sls = [seqlist_from_lists([x.tolist() for x in held])]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    op = np.array(ops, np.int32)
    assert r.apply_delta(0, op, q) == o[0].apply_ops(op, q)
    assert same_snapshot(r.download(0), o[0].export())
