"""GPU parity of the delta's bulk rounds (delta_bulk.cu: ops that do not meet are applied at once) against the CPU
oracle: deltas made of the ops that do meet, or nearly do.  After every call the canonical export equals the
oracle's byte for byte, the count of absent DELETEs agrees, and a route over the trees matches."""
import random

import numpy as np
import pytest

import oracle
import paper_2606_17059_gb300 as g
import workload as wl
from gpu_util import assert_same_route, csr_from_lists, route_device, router_from_seqlists, same_snapshot, seqlist_from_lists

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


def _runs(seqs, cuts):
    """Sequence list whose sequence i is cut into two pool runs at cuts[i]; equal first runs share one pool copy."""
    pool, at, sb, so, sl = [], {}, [0], [], []
    for s, c in zip(seqs, cuts):
        for part, share in ((s[:c], True), (s[c:], False)):
            key = tuple(part)
            if not (share and key in at):
                at[key] = len(pool)
                pool.extend(part)
            so.append(at[key])
            sl.append(len(part))
        sb.append(len(so))
    return wl.SeqList(np.array(sb, np.int64), np.array(so, np.int64), np.array(sl, np.int32), np.array(pool, np.int32))


def _check(r, trees, calls, reqs):
    for n, (p, ops, sl) in enumerate(calls):
        op = np.array(ops, np.int32)
        assert r.apply_delta(p, op, sl) == trees[p].apply_ops(op, sl), f"call {n}: absent DELETEs"
        assert same_snapshot(r.download(p), trees[p].export()), f"call {n}"
    tok, off = csr_from_lists(reqs)
    P = len(trees)
    gm, gp = route_device(r, tok, off, [0] * P, 0)
    om, op_, _ = oracle.route(trees, tok, off, [0] * P, 0)
    assert_same_route(gm, gp, om, op_, "after the deltas")


# Prompt lengths around what a lane compares alone (8, then 64 tokens), what is interned (128) and a warp's step (256).
@pytest.mark.parametrize("length", [1, 2, 8, 9, 10, 72, 73, 74, 127, 128, 129, 300, 700])
def test_ops_that_meet(length):
    rng = random.Random(length)
    tail = lambda n=None: [rng.randrange(50, 60) for _ in range(n or rng.randint(1, 100))]
    prompts = [[1000 + k] + [rng.randrange(3) for _ in range(length - 1)] for k in range(6)]
    held = [[p + tail() for _ in range(k)] for k, p in enumerate(prompts)]  # 0 .. 5 sequences a prompt
    a = [s for h in held for s in h]
    other = [p + tail() for p in prompts for _ in range(2)]  # (its interned prompts make tree 0's upload split some)
    sls = [seqlist_from_lists(other), seqlist_from_lists(a)]
    r, trees = router_from_seqlists(sls), oracle.build_trees(sls)
    fresh = [9000] + [rng.randrange(3) for _ in range(length)]
    ins, rem = [], []
    ins += [prompts[0] + tail() for _ in range(40)]           # many sequences of a prompt the tree does not hold
    ins += [fresh + tail() for _ in range(3)] + [fresh]       # ... and one that is its prompt itself
    ins += [prompts[5][: max(1, length // 2)], prompts[5][: max(1, length - 1)] + [77]]  # ends and leaves inside an edge
    ins += [prompts[4] + [50 + k] for k in range(10)]          # tables that have to grow
    ins += [held[3][0], held[3][0], held[3][0] + [1]]          # counts, and a leaf that gets a child
    rem += held[2] + held[3][1:] + held[4][:3] + held[5]       # folds, and prompts that vanish
    rem += [prompts[1] + [1, 2], [4242], held[1][0][:-1]]      # not stored
    ops = [(0, s) for s in ins] + [(1, s) for s in rem]
    again = [(1, ins[0]), (0, ins[0]), (1, ins[0]), (1, ins[0]), (0, held[2][0]), (1, held[2][0]), (1, ins[41])]
    rng.shuffle(ops)
    ops += again
    cuts = [min(len(s), rng.choice([length, length, 0, len(s), 5])) for _, s in ops]
    seqs = [s for _, s in ops]
    calls = [(1, [o for o, _ in ops], _runs(seqs, cuts))]
    # Taken back one by one from the other end: every DELETE has a stored sequence or is a counted no-op.
    back = [(1 - o, s) for o, s in reversed(ops)]
    calls.append((1, [o for o, _ in back], seqlist_from_lists([s for _, s in back])))
    reqs = [s + [3] for s in seqs[::3]] + prompts + [s[:-1] for s in a]
    _check(r, trees, calls, reqs)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 257, 1000])
def test_batch_sizes_and_runs(n):
    """Deltas of n ops over three trees (sizes around a warp and a CTA), of one, two and three pool runs (the last
    are delta_kernel's alone), in one call over all trees from device memory."""
    import torch
    rng = random.Random(n)
    V = 4
    stored = [[[rng.randrange(V) for _ in range(rng.randint(1, 20))] for _ in range(60)] for _ in range(3)]
    sls = [seqlist_from_lists(s) for s in stored]
    for runs in (1, 2, 3):
        r, trees = router_from_seqlists(sls), oracle.build_trees(sls)
        ops, seqs, pb = [], [], [0]
        for p in range(3):
            for _ in range(n if p != 1 else n // 2):
                if rng.random() < 0.5:
                    ops.append(1)
                    seqs.append(list(rng.choice(stored[p])))
                else:
                    ops.append(0)
                    seqs.append(rng.choice(stored[p])[: rng.randint(0, 20)] + [rng.randrange(V) for _ in range(rng.randint(0, 20))])
            pb.append(len(ops))
        sb, so, sl, pool = [0], [], [], []
        for s in seqs:
            marks = sorted(rng.randint(0, len(s)) for _ in range(runs - 1))
            for lo, hi in zip([0] + marks, marks + [len(s)]):
                so.append(len(pool))
                sl.append(hi - lo)
                pool.extend(s[lo:hi])
            sb.append(len(so))
        host = wl.SeqList(np.array(sb, np.int64), np.array(so, np.int64), np.array(sl, np.int32), np.array(pool or [0], np.int32))
        op = np.array(ops, np.int32)
        dev = wl.SeqList(*(torch.from_numpy(x).cuda() for x in (host.seg_begin, host.seg_off, host.seg_len, host.pool)))
        got = r.apply_delta(-1, torch.from_numpy(op).cuda(), dev, torch.from_numpy(np.array(pb, np.int64)).cuda(), on_device=True)
        assert got == sum(trees[p].apply_ops(op, host, pb[p], pb[p + 1]) for p in range(3))
        for p in range(3):
            assert same_snapshot(r.download(p), trees[p].export()), (runs, p)


def test_a_root_table_that_has_to_grow():
    """Thousands of new first tokens at once: the root's table only grows between launches, and the rounds run again
    after it has."""
    rng = random.Random(3)
    sls = [seqlist_from_lists([[5, 6, 7]])]
    r, trees = router_from_seqlists(sls), oracle.build_trees(sls)
    seqs = [[rng.randrange(1 << 20)] + [rng.randrange(9) for _ in range(rng.randint(0, 90))] for _ in range(5000)]
    sl = seqlist_from_lists(seqs)
    _check(r, trees, [(0, [0] * 5000, sl), (0, [1] * 5000, sl)], seqs[:300])


@pytest.mark.parametrize("seed", range(12))
def test_room_running_out(seed):
    """INSERTs that run out of node, slot and label room again and again while other warps still find some: every
    reservation keeps its own room."""
    rng = random.Random(seed)
    sls = [seqlist_from_lists([[1, 2, 3]]) for _ in range(4)]
    r, trees = router_from_seqlists(sls), oracle.build_trees(sls)
    for p in range(4):
        seqs = [[rng.randrange(60) for _ in range(rng.randint(1, 90))] for _ in range(2500)]
        _check(r, trees, [(p, [0] * 2500, seqlist_from_lists(seqs))], seqs[:50])


@pytest.mark.parametrize("n_fill", [0, 6000])
def test_edges_left_around_the_lane_spans(n_fill):
    """INSERTs that leave an edge, and DELETEs and repeats that follow it, after every count of tokens around those that
    a lane compares alone (9, then 8 per op of its warp, 128 at most), in one pool run and in two; with and without
    enough other ops that a warp has two."""
    rng = random.Random(n_fill)
    lens = [1, 8, 9, 10, 16, 17, 18, 24, 25, 26, 33, 127, 128, 136, 137, 138, 300]
    base = [[i] + [rng.randrange(1000) for _ in range(320)] for i in range(len(lens))]
    r, o = router_from_seqlists([seqlist_from_lists(base)]), oracle.build_trees([seqlist_from_lists(base)])
    for cuts in (0, 1):
        ops, seqs = [], []
        for i, k in enumerate(lens):
            seqs += [base[i][:k] + [1000 + cuts, 5], base[i][:k] + [1000 + cuts], base[i], base[i][:k]]
            ops += [0, 1, 0, 1]
        fill = [[5000 + cuts * n_fill + j, 1] for j in range(n_fill)]
        ops, seqs = np.array(ops + [0] * n_fill, np.int32), seqs + fill
        sl = _runs(seqs, [min(len(s), 1 + 7 * (i % 30)) if cuts else len(s) for i, s in enumerate(seqs)])
        r.apply_delta(0, ops, sl)
        o[0].apply_ops(ops, sl, 0, len(ops))
        assert same_snapshot(r.download(0), o[0].export()), cuts


def test_a_round_that_asks_for_more_than_an_arena_can_hold():
    """Many INSERTs of one long new prompt: counted for each of them they ask for 1.15 G tokens, past the arenas' reach,
    though together they take it once."""
    n, L = 1100, 1 << 20
    rng = np.random.default_rng(3)
    pool = np.concatenate([rng.integers(0, 1000, size=L), np.arange(n)]).astype(np.int32)
    sb = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
    so = np.stack([np.zeros(n), L + np.arange(n)], axis=1).astype(np.int64).reshape(-1)
    sl = np.tile([L, 1], n).astype(np.int32)
    seqs = wl.SeqList(sb, so, sl, pool)
    r = router_from_seqlists([seqlist_from_lists([[5]])])
    r.apply_delta(0, np.zeros(n, np.int32), seqs)
    st = r.download(0)
    lens = np.sort(np.asarray(st["label_len"]))
    assert len(lens) == n + 3 and lens[-1] == L and (lens[1:-1] == 1).all() and int(np.sum(st["term_count"])) == n + 1
    tok, off = csr_from_lists([pool[:L].tolist() + [3], pool[: L // 2].tolist() + [-1], [5]])
    gm, _ = route_device(r, tok, off, [0], 1)
    assert gm.ravel().tolist() == [L + 1, L // 2, 1]


@pytest.mark.parametrize("P,per,one", [(1, 1, 0), (1, 12, 0), (1, 13, 0), (5, 12, 3), (5, 2, 13), (5, 0, 1), (5, 0, 40),
                                       (310, 3, 2), (310, 6, 0)])
def test_deltas_of_a_few_ops(P, per, one):
    """Up to 12 ops a tree the delta kernel takes a delta alone (fewer in all on many trees), from host and from device
    memory; `one` more go to the last tree."""
    import torch
    rng = random.Random(P * 100 + per)
    stored = [[[rng.randrange(4) for _ in range(rng.randint(1, 20))] for _ in range(12)] for _ in range(P)]
    sls = [seqlist_from_lists(s) for s in stored]
    r, trees = router_from_seqlists(sls), oracle.build_trees(sls)
    ops, seqs, pb = [], [], [0]
    for p in range(P):
        for _ in range(per + (one if p == P - 1 else 0)):
            ops.append(rng.randrange(2))
            seqs.append(rng.choice(stored[p])[: rng.randint(0, 20)] + [rng.randrange(4)])
        pb.append(len(ops))
    sl, op, pb = seqlist_from_lists(seqs), np.array(ops, np.int32), np.array(pb, np.int64)
    dev = wl.SeqList(*(torch.from_numpy(x).cuda() for x in (sl.seg_begin, sl.seg_off, sl.seg_len, sl.pool)))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    few = max(np.diff(pb)) <= 12 and (P <= 2 * sms or len(ops) <= 8 * sms)
    for turn in range(2):
        r.kernel_clock(True)
        got = r.apply_delta(-1, op, sl, pb) if turn else r.apply_delta(-1, torch.from_numpy(op).cuda(), dev, torch.from_numpy(pb).cuda(), on_device=True)
        assert got == sum(t.apply_ops(op, sl, int(pb[p]), int(pb[p + 1])) for p, t in enumerate(trees))
        assert ("bulk_resolve_kernel" in r.kernel_times()) != few
    for p in range(0, P, max(1, P // 7)):
        assert same_snapshot(r.download(p), trees[p].export()), p
    assert same_snapshot(r.download(P - 1), trees[P - 1].export())


@pytest.mark.parametrize("n", [5, 32, 60])
def test_a_tree_with_room_is_not_grown(n):
    """INSERTs of one new prompt, which together take it once: the arenas that hold them (and a next call like it) stay
    as they are, though n prompts would not fit."""
    r, trees = router_from_seqlists([seqlist_from_lists([[1, 2, 3]])]), oracle.build_trees([seqlist_from_lists([[1, 2, 3]])])
    before = r.stats(0)
    prompt = list(range(1000, 1000 + before["cap_label"] // 4))
    sl, op = _runs([prompt + [k] for k in range(n)], [len(prompt)] * n), np.zeros(n, np.int32)
    assert r.apply_delta(0, op, sl) == trees[0].apply_ops(op, sl)
    assert same_snapshot(r.download(0), trees[0].export())
    after = r.stats(0)
    assert all(after[k] == before[k] for k in ("cap_node", "cap_child", "cap_label")), (before, after)


@pytest.mark.parametrize("held,new", [(0, 1), (0, 3), (2, 1), (2, 30), (8, 1), (8, 9), (30, 3), (60, 70), (130, 1), (200, 900), (1000, 1100)])
def test_tables_that_grow_within_a_round(held, new):
    """Nodes with `held` children that get `new` leaves in one call (and one with a single one, and a few that are left
    alone): tables of every size class move, by a lane, by a warp with a bit mask, and by compare-and-swap."""
    rng = random.Random(held * 31 + new)
    kids = [rng.sample(range(-(1 << 31), 1 << 31), held + new) for _ in range(6)]
    base = [[i, 7, c, 1] for i in range(6) for c in kids[i][:held]] + [[i, 7] for i in range(6)]
    add = [[i, 7, c, 1] for i in range(4) for c in kids[i][held:]] + [[4, 7, kids[4][held], 1]]
    rng.shuffle(add)
    r, o = router_from_seqlists([seqlist_from_lists(base)] * 2), oracle.build_trees([seqlist_from_lists(base)] * 2)
    sl, op = seqlist_from_lists(add + add), np.zeros(2 * len(add), np.int32)
    pb = np.array([0, len(add), 2 * len(add)], np.int64)
    assert r.apply_delta(-1, op, sl, pb) == 0
    reqs = [s[: rng.randint(2, 4)] for s in rng.sample(base + add, min(300, len(base + add)))]
    tok, off = csr_from_lists(reqs)
    for p in range(2):
        o[p].apply_ops(op, sl, int(pb[p]), int(pb[p + 1]))
        assert same_snapshot(r.download(p), o[p].export()), p
    gm, gp = route_device(r, tok, off, [0, 0], 1)
    om, op_, _ = oracle.route(o, tok, off, [0, 0], 1)
    assert_same_route(gm, gp, om, op_, "grown tables")
