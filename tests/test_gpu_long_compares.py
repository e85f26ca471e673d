"""Requests of a staging window and more that leave long labels after every count of tokens around the steps of the
compares (32, 128, 256, 512, 768 and 1,024 tokens), as leaders and as followers, against the CPU oracle; and common
prefixes of groups that end around those steps."""
import random

import numpy as np
import pytest

import oracle
import paper_2606_17059_gb300 as g
from gpu_util import assert_same_route, csr_from_lists, router_from_seqlists, seqlist_from_lists

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g.build()


EDGES = [n + d for n in (32, 64, 128, 256, 512, 768, 1024, 1280, 1536, 2048, 3072, 4096) for d in (-1, 0, 1)]


@pytest.mark.parametrize("grouped", [False, True])
def test_long_labels_left_around_the_steps(grouped):
    import torch
    rng = np.random.default_rng(7)
    run = lambda n: rng.integers(0, 30000, size=n).tolist()
    base, alts = run(9000), [(90 + 13 * j, run(5000)) for j in range(3)]
    trees = [[base], [base[:7000]] + [base[:c] + a for c, a in alts], [base[:c] + a for c, a in alts[:2]]]
    reqs = [base]  # the leader of the group
    for k in EDGES:
        reqs.append(base[:k] + [-5] + run(8400 - k))
        for c, a in alts:
            reqs.append(base[:c] + a[:k] + [-6] + run(8400 - k))
    if grouped:  # past min(2,432, 300 (P - 1)) requests
        reqs += [base[: 8300 + i] for i in range(650 - len(reqs))]
    else:
        random.Random(1).shuffle(reqs)
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    tok, off = csr_from_lists(reqs)
    om, op, _ = oracle.route(o, tok, off, [3, 1, 0], 2)
    t, f = torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()
    m, p = r.route(t, f, [3, 1, 0], 2)
    r.sync()
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "long labels")
    ex = np.array([0, 1, 0], np.uint8)
    m, p, n = r.route_decide(t, f, [3, 1, 0], 2, ex)
    dp, dn = oracle.decide(om, [3, 1, 0], 2, ex)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(p.cpu().numpy(), dp) and np.array_equal(n.cpu().numpy(), dn)


def test_common_prefixes_around_the_steps():
    """Short requests: groups whose members share every count of tokens around the steps with their leader, or end there."""
    import torch
    rng = np.random.default_rng(8)
    run = lambda n: rng.integers(0, 30000, size=n).tolist()
    base = run(1600)
    edges = [k for k in EDGES if 64 <= k < 1500]
    reqs = [base] + [base[:k] + [-7] + run(5) for k in edges] + [base[:k] for k in edges]
    reqs += [base[: 64 + i] for i in range(400)]
    trees = [[base], [base[:k] + [-7] for k in edges[::2]]]
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    tok, off = csr_from_lists(reqs)
    om, op, _ = oracle.route(o, tok, off, [0, 0], 1)
    t, f = torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()
    m, p = r.route(t, f, [0, 0], 1)
    r.sync()
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "common prefixes")
    # Grouped beside a delta (that leaves the trees as they were).
    g.p2p_route_prepare(r.handle, t, t.numel(), f, len(reqs))
    sl = seqlist_from_lists([[7, 7, 7], [7, 7, 7]])
    r.apply_delta(0, np.array([0, 1], np.int32), sl)
    m, p = r.route(t, f, [0, 0], 1)
    r.sync()
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "grouped beside a delta")
