"""The followers' pass of short requests (a lane per follower): rows of every remainder of its tiles of 16 trees and of
its 16-byte stores, groups around a warp's 32 lanes, lookups that queue, walks over several edges, and edges longer
than a lane compares itself (80 tokens), against the CPU oracle."""
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


def _case(rng, P, group_sizes, far):
    """Groups share a prompt of 70 to 90 tokens; behind it the trees hold a few suffixes of the group (whole, cut, or
    split into edges), up to `far` tokens of them on one edge."""
    trees, reqs = [[] for _ in range(P)], []
    for n in group_sizes:
        prompt = [rng.randrange(500) for _ in range(rng.choice([70, 80, 90]))]
        tails = [[rng.randrange(500) for _ in range(rng.choice([1, 3, 79, 80, 81, 82, far]))] for _ in range(6)]
        for t in trees:
            if rng.random() < 0.8:
                for s in rng.sample(tails, rng.randint(0, 4)):
                    cut = rng.choice([0, 1, len(s) // 2, len(s), len(s)])
                    t.append(prompt[: rng.choice([len(prompt), len(prompt), 66])] + s[:cut])
                    if cut == len(s) and rng.random() < 0.5:
                        t.append(prompt + s[: max(1, len(s) // 3)] + [rng.randrange(500)])
        for _ in range(n):
            s = rng.choice(tails)
            reqs.append(prompt + rng.choice([s, s[: len(s) // 2], s + [rng.randrange(500)], [rng.randrange(500)], []]))
    rng.shuffle(reqs)
    return trees, reqs


@pytest.mark.parametrize("P,far", [(2, 200), (3, 90), (4, 500), (15, 83), (16, 200), (17, 161), (33, 82), (64, 300), (97, 100)])
def test_followers(P, far):
    import torch
    rng = random.Random(P * 31 + far)
    line = min(4864, 300 * (P - 1))  # batches above it are grouped on 152 SMs
    sizes = [1, 2, 31, 32, 33, 34, 64, 65, 300]
    while sum(sizes) <= line:
        sizes.append(rng.choice([2, 33, 200, 700]))
    trees, reqs = _case(rng, P, sizes, far)
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    tok, off = csr_from_lists(reqs)
    load = [rng.randrange(60) for _ in range(P)]
    om, op, _ = oracle.route(o, tok, off, load, 2)
    t, f = torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()
    m, p = r.route(t, f, load, 2)
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "route")
    ex = np.array([rng.random() < 0.4 for _ in range(P)], np.uint8)
    m, p, n = r.route_decide(t, f, load, 2, ex)
    dp, dn = oracle.decide(om, load, 2, ex)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(p.cpu().numpy(), dp) and np.array_equal(n.cpu().numpy(), dn)
    # A match matrix that is not on a 16-byte boundary.
    buf = torch.full((len(reqs) * P + 1,), -7, dtype=torch.int32, device="cuda")
    peer = torch.empty(len(reqs), dtype=torch.int32, device="cuda")
    out = buf[1:].view(len(reqs), P)
    r.route(t, f, load, 2, out_match=out, out_peer=peer)
    r.sync()
    assert_same_route(out.cpu().numpy(), peer.cpu().numpy(), om, op, "off a 16-byte boundary")
    assert int(buf[0]) == -7
