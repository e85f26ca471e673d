"""A snapshot uploaded to the device (tables filled and own labels moved there): label lengths around the eight lanes'
steps, shared runs, labels split at a shared head, trees whose labels are nearly all shared, nodes in any order, pinned
and pageable arrays; the export and the routes against the CPU oracle."""
import numpy as np
import pytest

import oracle
import paper_2606_17059_gb300 as g
from gpu_util import assert_same_route, csr_from_lists, route_device, same_snapshot, seqlist_from_lists

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


def _flat(seqs):
    snap = g.p2p_snapshot_build(seqlist_from_lists(seqs))
    flat = {k: np.array(v) for k, v in g.p2p_snapshot_view(snap).items()}
    g.p2p_snapshot_free(snap)
    return flat


def _reversed(flat):
    """The same tree with its nodes (but the root) in reverse order: every child before its parent."""
    n = len(flat["label_off"])
    new = np.concatenate([[0], np.arange(n - 1, 0, -1)]).astype(np.int32)  # old -> new, its own inverse
    out = dict(flat)
    for k in ("label_off", "label_len", "child_begin", "child_count", "term_count"):
        out[k] = np.ascontiguousarray(flat[k][new])
    out["child_idx"] = new[flat["child_idx"]]
    return out


def _cases():
    rng = np.random.default_rng(3)
    run = lambda n: rng.integers(0, 30000, size=n).tolist()
    shared = [run(n) for n in (127, 128, 129, 400, 5000)]
    yield [[]]
    yield [[], [[]], [[5]], [[5], [5, 6]]]
    yield [[[i] + run(n) for i, n in enumerate(range(0, 140))], [run(n) for n in (63, 64, 65, 66, 127, 128, 129, 1000)]]
    yield [[s + run(k) for s in shared for k in (1, 5, 130)], [shared[4][:k] + run(k // 3) for k in (128, 200, 4999)],
           [s + run(2) for s in shared], [s for s in shared]]
    # Nearly all labels are shared runs: more snapshot labels than the spare holds.
    long = [[i] + run(4000) for i in range(60)]
    yield [long, long + [[100 + i, 3] for i in range(50)], [s[:3000] for s in long] + [[7, 7, 7]]]
    yield [[run(rng.integers(1, 90)) for _ in range(5000)]]


@pytest.mark.parametrize("trees", list(_cases()))
@pytest.mark.parametrize("form", ["preorder", "reversed", "pinned"])
def test_upload(trees, form):
    import torch
    r, ots = g.Router(max(len(trees), 1)), []
    flats = [_flat(t) for t in trees]
    for turn in range(2):  # (the second time, the runs are there)
        for p, f in enumerate(flats):
            f = _reversed(f) if form == "reversed" else dict(f)
            if form == "pinned":
                keep = {k: torch.from_numpy(np.ascontiguousarray(v, np.int32)).pin_memory() for k, v in f.items()}
                f = {k: v.numpy() for k, v in keep.items()}
            r.upload(p, f)
            if form == "pinned":
                for v in keep.values():  # (the caller's again once the call has returned)
                    v.fill_(-1)
        for p, f in enumerate(flats):
            assert same_snapshot(r.download(p), f), (turn, p)
    o = oracle.build_trees([seqlist_from_lists(t) for t in trees])
    rng = np.random.default_rng(4)
    reqs = [s[: rng.integers(0, len(s) + 1)] + [9] for t in trees for s in t][:3000] or [[1]]
    tok, off = csr_from_lists(reqs)
    gm, gp = route_device(r, tok, off, [0] * len(o), 1)
    om, op, _ = oracle.route(o, tok, off, [0] * len(o), 1)
    assert_same_route(gm, gp, om, op, form)


@pytest.mark.parametrize("kids", [1, 510, 511, 512])
def test_both_sides_of_the_line_between_host_and_device(kids):
    """Trees of up to 512 nodes are put together on the host, with own, shared and split labels on both sides."""
    rng = np.random.default_rng(kids)
    long = rng.integers(0, 30000, size=300).tolist()
    r = g.Router(2)
    r.upload(1, _flat([long + [1], long + [2]]))
    seqs = [[40000 + i] + rng.integers(0, 9, size=rng.integers(0, 140)).tolist() for i in range(kids - 1)] + [long + [3, 3]]
    flat = _flat(seqs)  # (the last one's label is split where the shared run ends: a node more)
    r.kernel_clock(True)
    r.upload(0, flat)
    assert ("upload_kernel" in r.kernel_times()) == (kids + 2 > 512)
    assert same_snapshot(r.download(0), flat)
    o = oracle.build_trees([seqlist_from_lists(seqs), seqlist_from_lists([long + [1], long + [2]])])
    tok, off = csr_from_lists([s[: len(s) // 2 + 1] + [9] for s in seqs])
    gm, gp = route_device(r, tok, off, [0, 0], 1)
    om, op, _ = oracle.route(o, tok, off, [0, 0], 1)
    assert_same_route(gm, gp, om, op, "line")
