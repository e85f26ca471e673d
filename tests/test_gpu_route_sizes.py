"""Batches on both sides of the line between ungrouped and grouped routing, and of the grouped path's own lines (the
hash kernel's requests per warp, the two follower lists, long requests), against the CPU oracle."""
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


def _case(rng, P, B, stem_len, tail):
    """Trees holding stems with several tails; requests that share a stem's first 63, 64, 65 or more tokens, short
    ones, empty ones and duplicates."""
    V = 400
    stems = [[rng.randrange(V) for _ in range(stem_len)] for _ in range(5)]
    trees = []
    for _ in range(P):
        t = []
        for s in stems:
            if rng.random() < 0.6:
                cut = rng.choice([63, 64, 65, stem_len // 2, stem_len])
                t += [s[:cut] + [rng.randrange(V) for _ in range(rng.randint(0, tail))] for _ in range(rng.randint(1, 3))]
        trees.append(t)
    reqs = []
    while len(reqs) < B:
        k = rng.random()
        s = rng.choice(stems)
        if k < 0.75:
            reqs.append(s[: rng.choice([63, 64, 65, 66, stem_len // 2, stem_len])] + [rng.randrange(V) for _ in range(rng.randint(0, tail))])
        elif k < 0.85 and reqs:
            reqs.append(rng.choice(reqs))
        elif k < 0.95:
            reqs.append([rng.randrange(V) for _ in range(rng.randint(0, 3 * tail))])
        else:
            reqs.append([])
    return trees, reqs


def _line(P, long):
    """The most requests that are routed without grouping on P trees."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return min(sms * (4 if P <= 8 else 2 if P <= 32 else 1) if long else sms * 32, 300 * (P - 1))


def _requests(P, B, long):
    """B requests, or (a text) that many more than the line."""
    return B if isinstance(B, int) else _line(P, long) + int(B)


# Batches around the line, around the CTA sizes of the ungrouped pass (a warp, two and eight a SM) and well off both.
@pytest.mark.parametrize("P,B", [(1, 1), (1, 40), (2, 299), (2, "+0"), (2, "+1"), (2, 309), (4, "+0"), (4, "+1"), (20, "+0"), (20, "+1"),
                                 (3, 33), (33, 7), (45, 5300), (20, 152), (20, 153), (20, 1217)])
def test_both_sides_of_the_grouping_line(P, B):
    import torch
    B = _requests(P, B, False)
    rng = random.Random(P * 10007 + B)
    trees, reqs = _case(rng, P, B, 200, 12)
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    tok, off = csr_from_lists(reqs)
    load = [rng.randrange(5) for _ in range(P)]
    om, op, _ = oracle.route(o, tok, off, load, 2)
    t, f = torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()
    n0 = r.launch_count()
    m, p = r.route(t, f, load, 2)
    assert (r.launch_count() - n0 == 1) == (B <= _line(P, False))
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "route")
    ex = np.array([rng.random() < 0.4 for _ in range(P)], np.uint8)
    m, p, n = r.route_decide(t, f, load, 2, ex)
    dp, dn = oracle.decide(om, load, 2, ex)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(p.cpu().numpy(), dp) and np.array_equal(n.cpu().numpy(), dn)
    # Announced ahead, with a delta in between (a small batch has nothing to prepare).
    g.p2p_route_prepare(r.handle, t, t.numel(), f, B)
    sl = seqlist_from_lists([[7, 7, 7]])
    r.apply_delta(0, np.zeros(1, np.int32), sl)
    r.apply_delta(0, np.ones(1, np.int32), sl)
    m, p = r.route(t, f, load, 2)
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "after prepare")
    # A request with bad offsets matches nothing, has no peer and is reported.
    bad = off.copy()
    bad[-1] = len(tok) + 5
    m, p = r.route(t, torch.from_numpy(bad).cuda(), load, 2)
    with pytest.raises(g.P2PError):
        r.sync()
    assert_same_route(m.cpu().numpy()[:-1], p.cpu().numpy()[:-1], om[:-1], op[:-1], "beside a bad request")
    assert not m.cpu().numpy()[-1].any() and int(p[-1]) == -1


@pytest.mark.parametrize("P,B", [(2, 3), (3, "+0"), (3, "+1"), (9, "+0"), (9, "+1"), (9, 2390), (33, "+0"), (33, "+1")])
def test_long_requests_on_both_sides(P, B):
    import torch
    B = _requests(P, B, True)
    rng = random.Random(P + B)
    trees, reqs = _case(rng, P, 40, 9000, 30)
    full = [q + [rng.randrange(9) for _ in range(max(0, 4200 - len(q)))] for q in reqs]
    reqs = [full[rng.randrange(40)][: rng.choice([4500, 9050])] + [rng.randrange(9)] for _ in range(B)]
    sls = [seqlist_from_lists(t) for t in trees]
    r, o = router_from_seqlists(sls), oracle.build_trees(sls)
    tok, off = csr_from_lists(reqs)
    om, op, _ = oracle.route(o, tok, off, [0] * P, 1)
    t, f = torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()
    n0 = r.launch_count()
    m, p = r.route(t, f, [0] * P, 1)
    r.sync()
    assert (r.launch_count() - n0 == 1) == (B <= _line(P, True))
    assert_same_route(m.cpu().numpy(), p.cpu().numpy(), om, op, "long")
    ex = np.zeros(P, np.uint8)
    ex[0] = 1
    m, p, n = r.route_decide(t, f, [0] * P, 1, ex)
    dp, dn = oracle.decide(om, [0] * P, 1, ex)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(p.cpu().numpy(), dp) and np.array_equal(n.cpu().numpy(), dn)
