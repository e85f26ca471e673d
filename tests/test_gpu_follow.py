"""The followers' pass of short requests, in ordinary batches (a lane per tree) and in large ones (a lane per follower):
rows of every remainder of its tiles of 16 trees and of its 16-byte stores, groups around a warp's 32 lanes, lookups
that queue, walks over several edges, edges longer than a lane compares itself (8 tokens), and followers whose token is
there in few, many and all trees, against the CPU oracle."""
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


def _case(rng, P, group_sizes, far, held=0.8):
    """Groups share a prompt of 70 to 90 tokens; behind it a share `held` of the trees hold a few suffixes of the group
    (whole, cut, or split into edges), up to `far` tokens of them on one edge."""
    trees, reqs = [[] for _ in range(P)], []
    for n in group_sizes:
        prompt = [rng.randrange(500) for _ in range(rng.choice([70, 80, 90]))]
        tails = [[rng.randrange(500) for _ in range(rng.choice([1, 3, 79, 80, 81, 82, far]))] for _ in range(6)]
        for t in trees:
            if rng.random() < held:
                for s in rng.sample(tails, rng.randint(0, 4) if held < 1 else 6):
                    cut = rng.choice([0, 1, len(s) // 2, len(s), len(s)])
                    t.append(prompt[: rng.choice([len(prompt), len(prompt), 66])] + s[:cut])
                    if cut == len(s) and rng.random() < 0.5:
                        t.append(prompt + s[: max(1, len(s) // 3)] + [rng.randrange(500)])
        for _ in range(n):
            s = rng.choice(tails)
            reqs.append(prompt + rng.choice([s, s[: len(s) // 2], s + [rng.randrange(500)], [rng.randrange(500)], []]))
    rng.shuffle(reqs)
    return trees, reqs


def _check(P, trees, tok, off, rng):
    import torch
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
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
    buf = torch.full((om.shape[0] * P + 1,), -7, dtype=torch.int32, device="cuda")
    peer = torch.empty(om.shape[0], dtype=torch.int32, device="cuda")
    out = buf[1:].view(om.shape[0], P)
    r.route(t, f, load, 2, out_match=out, out_peer=peer)
    r.sync()
    assert_same_route(out.cpu().numpy(), peer.cpu().numpy(), om, op, "off a 16-byte boundary")
    assert int(buf[0]) == -7


# From half a wave of lanes (up to 16 trees) or three quarters on, the followers are taken a lane each.
@pytest.mark.parametrize("P,far,held", [(2, 200, 0.8), (3, 90, 1), (15, 83, 0.2), (16, 200, 0.8), (16, 120, 1), (17, 161, 0.1),
                                        (33, 400, 1), (33, 82, 0.3), (64, 300, 0.05), (97, 100, 0.4)])
def test_followers_of_large_batches(P, far, held):
    import torch
    rng = random.Random(P * 37 + far)
    trees, reqs = _case(rng, P, [1, 2, 31, 32, 33, 34, 64, 65, 300, 700, 1500], far, held)
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 3 * 256
    line = wave // 2 if P <= 16 else wave * 3 // 4
    tok, off = csr_from_lists(reqs)
    times = line // len(reqs) + 1  # the batch again and again, each time with other tokens at its requests' ends
    lens = np.diff(off)
    off = np.concatenate([[0], np.cumsum(np.tile(lens, times))]).astype(np.int64)
    tok = np.tile(tok, times)
    last = off[1:][lens[np.arange(len(off) - 1) % len(lens)] > 0] - 1
    change = np.random.default_rng(P).random(len(last)) < 0.5
    tok[last[change]] = np.random.default_rng(far).integers(0, 500, int(change.sum()))
    assert len(off) - 1 >= line
    _check(P, trees, tok, off, rng)


@pytest.mark.parametrize("P,far", [(2, 200), (3, 90), (4, 500), (15, 83), (16, 200), (17, 161), (33, 82), (64, 300), (97, 100)])
def test_followers(P, far):
    import torch
    rng = random.Random(P * 31 + far)
    line = min(torch.cuda.get_device_properties(0).multi_processor_count * 32, 300 * (P - 1))  # batches above it are grouped
    sizes = [1, 2, 31, 32, 33, 34, 64, 65, 300]
    while sum(sizes) <= line:
        sizes.append(rng.choice([2, 33, 200, 700]))
    trees, reqs = _case(rng, P, sizes, far)
    tok, off = csr_from_lists(reqs)
    _check(P, trees, tok, off, rng)
