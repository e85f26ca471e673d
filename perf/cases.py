"""The work that is measured: what a router process has this engine do, through its public calls.

A case names a workload preset of the generator (``base``, 0 to 4: see ``workload/wl.h``) for the kind of prompts
and the tree contents, its own numbers of trees, sequences and requests, and a ``kind`` of pass:

  route     a batch of requests on the device is matched against every tree and routed (``decide``: with peers
            taken out and the next-best target, in the same pass)
  host      the same for a batch in pinned host memory, copies included
  decide    the decision made again from a match matrix after peers pushed back, and the expected hit rates
  refresh   one peer's small anti-entropy delta arrives in host memory, is applied, and a few requests are routed
  step      every replica takes its delta from device memory, then a batch is routed (announced ahead)
  learn     a routed batch goes into the trees it was sent to; the peers' later evictions take it out again
  cache     the own cache trie serves a batch, takes it in and evicts as many tokens as it is short of
  snapshot  one peer's full snapshot arrives in host memory and replaces its replica, then a few requests are routed

Passes that change trees come back to where they began after every pass or every second one (``cache`` settles),
as a router's trees do in steady service, so that a pass can be repeated.
"""
from __future__ import annotations

import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2606_17059_gb300 as g
import workload as wl

_THREADS = min(16, os.cpu_count() or 1)
_PROBE = 1025  # requests routed after a change of the trees, whose results show it


def listed():
    return [
        # A handful of requests arriving together at a small cluster: launches and latency.
        dict(name="route, 33 requests", kind="route", base=0, P=4, n_seq=1000, B=33, decide=False),
        # An ordinary batch of few-shot prompts, 16 peers (the generator's second preset as it is).
        dict(name="route, 65,536 requests", kind="route", base=1, P=16, n_seq=20000, B=65536, decide=False),
        # Stale replicas of 64 peers, some of them suspected or pushing back, an odd batch.
        dict(name="route, peers excluded", kind="route", base=2, P=64, n_seq=20000, B=200003, decide=True),
        # Long-context prompts of 4,096 to 32,768 tokens that leave the cached prefixes half-way.
        dict(name="route, long context", kind="route", base=3, P=32, n_seq=5000, B=8191, decide=False),
        # Requests in host memory, as a front end without device buffers hands them over.
        dict(name="route from the host", kind="host", base=1, P=16, n_seq=20000, B=270001),
        # Push-back after a large batch was matched: the decision alone, over the whole match matrix.
        dict(name="decide, 1,048,576 rows", kind="decide", base=4, P=256, n_seq=0, B=1048576),
        # One peer's delta of a few hundred changes since its last message.
        dict(name="refresh one replica", kind="refresh", base=1, P=16, n_seq=20000, B=_PROBE, ops=300),
        # The scale step on 256 replicas: 5% + 5% of every replica's sequences change, then the batch.
        dict(name="step, 256 replicas", kind="step", base=4, P=256, n_seq=40000, B=262144),
        # After the requests were sent and acknowledged: the sender's estimates learn them.
        dict(name="learn 16,384 requests", kind="learn", base=1, P=16, n_seq=20000, B=16384),
        # The node's own cache at capacity.
        dict(name="cache, 4,096 requests", kind="cache", base=1, P=2, n_seq=20000, B=4096),
        # A peer's full broadcast (after it restarted, or its deltas were lost).
        dict(name="snapshot of one peer", kind="snapshot", base=1, P=16, n_seq=20000, B=4 * _PROBE),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, any tree count from 1 to 256 and any batch up to the listed ones' sizes."""
    kind = rng.choice(["route", "route", "route", "host", "decide", "refresh", "step", "learn", "cache", "snapshot"])
    c = dict(kind=kind, base=rng.choice([0, 1, 2, 3] if kind == "route" else [0, 1, 2]))
    c["P"] = _log(rng, 1, 256) if kind != "cache" else rng.randint(1, 4)
    c["n_seq"] = _log(rng, 200, 20000)
    if c["P"] * c["n_seq"] > 640000:  # (the trees are built on the host)
        c["n_seq"] = 640000 // c["P"]
    if kind == "route":
        c["B"] = _log(rng, 1, 8191 if c["base"] == 3 else 200003)
        c["decide"] = rng.random() < 0.4
        if c["base"] == 3:
            c["n_seq"] = max(100, c["n_seq"] // 8)
    elif kind == "host":
        c["B"] = _log(rng, 1, 200003)
    elif kind == "decide":
        c["base"], c["n_seq"] = 4, 0
        c["B"] = _log(rng, 1, (1 << 28) // max(c["P"], 16))
    elif kind == "refresh":
        c["B"], c["ops"] = _PROBE, _log(rng, 2, 2000)
    elif kind == "step":
        c["base"], c["B"] = rng.choice([1, 4]), _log(rng, 64, 65536)
    elif kind == "learn":
        c["B"] = _log(rng, 16, 16384)
    elif kind == "cache":
        c["B"] = _log(rng, 16, 4096)
    else:
        c["B"] = 4 * _PROBE
    return c


def _params(case):
    prm = wl.preset(case["base"])
    prm.update(P=case["P"], B=max(case["B"], 1))
    if case["n_seq"]:
        # Fewer sequences a tree than the preset's hold proportionally fewer prompts, so that every cached prompt
        # keeps several suffixes (at least 32 prompts).
        prm["n_prefix"] = max(min(32, prm["n_prefix"]), prm["n_prefix"] * case["n_seq"] // prm["n_seq"])
        prm["n_seq"] = case["n_seq"]
    return prm


def _build(W):
    """A router whose P trees hold the workload's sequences (snapshots built on host threads)."""
    r = g.Router(W.P)

    def snapshot(p):
        return g.p2p_snapshot_build(W.tree(p))

    with ThreadPoolExecutor(max_workers=_THREADS) as ex:
        for p, snap in enumerate(ex.map(snapshot, range(W.P))):
            r.upload(p, g.p2p_snapshot_view(snap))
            g.p2p_snapshot_free(snap)
    r.sync()
    return r


def _requests(W, b0, b1):
    tok, off = W.requests(b0, b1, n_threads=_THREADS)
    return torch.from_numpy(tok).cuda(), torch.from_numpy(off).cuda()


def _on_device(s):
    return wl.SeqList(*(torch.from_numpy(np.ascontiguousarray(a)).cuda()
                        for a in (s.seg_begin, s.seg_off, s.seg_len, s.pool)))


def prepare(case, seed):
    kind, B, P = case["kind"], case["B"], case["P"]
    rs = np.random.RandomState(seed % (1 << 32))
    st = dict(kind=kind, B=B, turn=0)
    if kind == "decide":
        # A match matrix as routes write it: most trees hold nothing of a request, some its whole prompt.
        gen = torch.Generator(device="cuda").manual_seed(seed)
        prompt = torch.randint(128, 4097, (B, 1), generator=gen, device="cuda", dtype=torch.int32)
        kept = torch.randint(0, 4, (B, P), generator=gen, device="cuda", dtype=torch.int8)
        match = torch.where(kept == 0, prompt, torch.where(kept == 1, prompt % 5, torch.zeros_like(prompt)))
        st["match"] = match.to(torch.int32).contiguous()
        st["offsets"] = torch.cat([torch.zeros(1, device="cuda", dtype=torch.int64),
                                   torch.cumsum(prompt[:, 0].to(torch.int64) + 80, 0)])
        st["load"] = rs.randint(0, 256, P).astype(np.int32)
        st["alpha"] = 2
        st["excluded"] = (rs.rand(P) < 0.05).astype(np.uint8)
        st["router"] = g.Router(P)
        st["hit"] = torch.empty(B, dtype=torch.float32, device="cuda")
        return st
    W = wl.Workload(params=_params(case), seed=seed)
    st["router"] = r = _build(W)
    st["load"], st["alpha"] = W.load(), W.alpha
    if kind == "host":
        n = int(wl._load().wl_requests_size(W._h, 0, B, _THREADS))
        st["tokens"] = torch.empty(max(n, 1), dtype=torch.int32, pin_memory=True)
        _, off = W.requests(0, B, n_threads=_THREADS, out_tokens=st["tokens"].numpy())
        st["offsets"] = torch.from_numpy(off).pin_memory()
        st["match"] = torch.empty((B, P), dtype=torch.int32, pin_memory=True)
        st["peer"] = torch.empty(B, dtype=torch.int32, pin_memory=True)
        return st
    if kind == "cache":
        # Four batches in turn, so that a batch comes back when the cache has lost part of it; the cache evicts
        # about half of what a batch brings in when none of it is cached.
        st["batches"] = [_requests(W, k * B, (k + 1) * B) for k in range(4)]
        st["evict"] = int(B * ((W.params["suf_lo"] + W.params["suf_hi"]) / 2 +
                               W.params["fresh_frac"] * (W.params["pre_lo"] + W.params["pre_hi"]) / 2) / 2)
        st["match"] = torch.empty(B, dtype=torch.int32, device="cuda")
        g.p2p_lru_enable(r.handle, 0)
        return st
    st["tokens"], st["offsets"] = _requests(W, 0, B)
    if kind == "route":
        st["excluded"] = (rs.rand(P) < 0.1).astype(np.uint8) if case["decide"] else None
        st["decide"] = case["decide"]
    elif kind in ("refresh", "step"):
        # A delta and the one that takes it back (its sequences are all different, so their order is free).
        peer = int(rs.randint(P)) if kind == "refresh" else None
        n_live = case["n_seq"]
        f = min(0.4, case["ops"] / 2 / n_live) if kind == "refresh" else 0.05
        p0, p1 = (peer, peer + 1) if kind == "refresh" else (0, P)
        W.delta_make(0, f, f, p0, p1, n_threads=_THREADS)
        d = W.delta(p0, p1, n_threads=_THREADS)
        st["peer"] = peer
        if kind == "refresh":
            st["deltas"] = [(d.op, d.seqs), (1 - d.op, d.seqs)]
        else:
            seqs = _on_device(d.seqs)
            st["deltas"] = [(torch.from_numpy(op).cuda(), seqs) for op in (d.op, 1 - d.op)]
            st["ranges"] = torch.from_numpy(d.peer_begin).cuda()
    elif kind == "learn":
        # The DELETEs by which the peers later evict the same sequences: each request once, by the tree it went to.
        _, peer = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
        r.sync()
        order = torch.argsort(peer, stable=True)
        off = st["offsets"]
        st["evicted"] = wl.SeqList(torch.arange(B + 1, device="cuda"), off[:-1][order].contiguous(),
                                   (off[1:] - off[:-1])[order].to(torch.int32).contiguous(), st["tokens"])
        st["ranges"] = torch.searchsorted(peer[order].contiguous(), torch.arange(P + 1, device="cuda", dtype=torch.int32))
        st["delete"] = torch.ones(B, dtype=torch.int32, device="cuda")
        st["probe"] = off[: min(B, _PROBE) + 1].contiguous()
    elif kind == "snapshot":
        # The peer's broadcasts before and after a tenth of its sequences changed.
        peer = int(rs.randint(P))
        flats = []
        for k in range(2):
            snap = g.p2p_snapshot_build(W.tree(peer))
            flats.append(g.p2p_snapshot_view(snap))
            g.p2p_snapshot_free(snap)
            W.delta_make(k, 0.1, 0.1, peer, peer + 1)
        st["peer"], st["flats"] = peer, flats[::-1]
    return st


def run(st):
    kind, r = st["kind"], st["router"]
    k = st["turn"]
    st["turn"] = k + 1
    if kind == "decide":
        peer, nxt = r.decide(st["match"], st["load"], st["alpha"], st["excluded"])
        g.p2p_hit_rate(r.handle, st["match"], st["offsets"], st["B"], peer, st["hit"])
        return {"peer": peer, "next": nxt, "hit": st["hit"]}
    if kind == "host":
        m, p = r.route_host(st["tokens"].numpy(), st["offsets"].numpy(), st["load"], st["alpha"], st["match"].numpy(),
                            st["peer"].numpy())
        return {"match": m, "peer": p}
    if kind == "route":
        if st["decide"]:
            m, p, n = r.route_decide(st["tokens"], st["offsets"], st["load"], st["alpha"], st["excluded"])
            return {"match": m, "peer": p, "next": n}
        m, p = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
        return {"match": m, "peer": p}
    if kind == "refresh":
        op, seqs = st["deltas"][k % 2]
        absent = r.apply_delta(st["peer"], op, seqs)
        m, p = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
        return {"absent": absent, "match": m, "peer": p}
    if kind == "step":
        op, seqs = st["deltas"][k % 2]
        g.p2p_route_prepare(r.handle, st["tokens"], st["tokens"].numel(), st["offsets"], st["B"])
        absent = r.apply_delta(-1, op, seqs, st["ranges"], on_device=True)
        m, p = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
        return {"absent": absent, "match": m, "peer": p}
    if kind == "learn":
        m, p = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
        n = r.update_estimates(st["tokens"], st["offsets"], p)
        m2, p2 = r.route(st["tokens"], st["probe"], st["load"], st["alpha"])
        absent = r.apply_delta(-1, st["delete"], st["evicted"], st["ranges"], on_device=True)
        return {"match": m, "peer": p, "inserted": n, "match_after": m2, "peer_after": p2, "absent": absent}
    if kind == "cache":
        tok, off = st["batches"][k % 4]
        g.p2p_lru_insert(r.handle, 0, tok, tok.numel(), off, st["B"], 2 * k + 1)
        n = g.p2p_lru_evict(r.handle, 0, st["evict"])
        tok, off = st["batches"][(k + 1) % 4]
        g.p2p_lru_access(r.handle, 0, tok, tok.numel(), off, st["B"], 2 * k + 2, st["match"])
        return {"evicted": n, "match": st["match"]}
    r.upload(st["peer"], st["flats"][k % 2])
    m, p = r.route(st["tokens"], st["offsets"], st["load"], st["alpha"])
    return {"match": m, "peer": p}


def work(case):
    """Bytes a pass cannot do without, with the mean lengths of the workload: each input read and each output
    written once.  What a walk reads of the trees depends on the requests and is left out."""
    kind, B, P = case["kind"], case["B"], case["P"]
    prm = _params(case)
    suffix = (prm["suf_lo"] + prm["suf_hi"]) / 2
    prefix = (prm["pre_lo"] + prm["pre_hi"]) / 2
    length = prefix * (0.55 if prm["diverge"] else 1.0) + (prm["req_suf_lo"] + prm["req_suf_hi"]) / 2
    route = B * (4 * length + 8) + 4 * B * P + 4 * B
    if kind == "decide":
        nbytes = B * (4 * P + 4 + 4 + 8 + 4)
    elif kind in ("route", "host"):
        nbytes = route + (4 * B if case.get("decide") else 0)
    elif kind in ("refresh", "step"):
        ops = case["ops"] if kind == "refresh" else 0.1 * case["n_seq"] * P
        nbytes = route + ops * (4 + 8 + 2 * 12 + 4 * suffix + 4 * suffix / 2) + 4 * prefix * prm["n_prefix"]
    elif kind == "learn":
        nbytes = route + B * (4 + 16 + 4 * suffix)  # a request's tokens count once; its new tokens are written
    elif kind == "cache":
        new = B * (suffix + prm["fresh_frac"] * prefix) / 2
        nbytes = 2 * B * (4 * length + 8) + 4 * B + 8 * new
    else:
        nodes = 2 * case["n_seq"]
        labels = 4 * (case["n_seq"] * suffix + prefix * prm["n_prefix"] * prm["assign_prob"])
        nbytes = route + 2 * (nodes * 28 + labels)
    return {"bytes": float(nbytes), "flops": 0.0}


def tolerance(case):
    # Token counts and tree indices; the hit rate is one correctly rounded division of two whole numbers below 2^24.
    return "exact"


def exact(case, seed):
    """The decision in plain torch (64-bit scores), the hit rate in 64 bits; a route by comparing every request with
    every stored sequence where that is short."""
    st = None
    if case["kind"] == "decide":
        st = prepare(case, seed)
        load = torch.from_numpy(st["load"]).cuda().to(torch.int64)
        ex = torch.from_numpy(st["excluded"]).cuda().bool()
        P, B = case["P"], case["B"]
        idx = torch.arange(P, device="cuda")
        peer = torch.full((B,), -1, dtype=torch.int32, device="cuda")
        nxt = peer.clone()
        hit = torch.zeros(B, dtype=torch.float64, device="cuda")
        length = st["offsets"][1:] - st["offsets"][:-1]
        for a in range(0, B, 65536):
            m = st["match"][a: a + 65536].to(torch.int64)
            key = ((m - st["alpha"] * load + (1 << 30)) * 65536 + (65535 - load)) * 65536 + (65535 - idx)
            key = torch.where(ex, torch.full_like(key, -1), key)
            best, arg = torch.topk(key, min(2, P), dim=1)
            arg = torch.where(best >= 0, arg, torch.full_like(arg, -1)).to(torch.int32)
            peer[a: a + 65536] = arg[:, 0]
            if P > 1:
                nxt[a: a + 65536] = arg[:, 1]
            got = m.gather(1, arg[:, :1].clamp(min=0).to(torch.int64))[:, 0].double() / length[a: a + 65536].double()
            hit[a: a + 65536] = torch.where(arg[:, 0] >= 0, got, torch.zeros_like(got))
        return {"peer": peer, "next": nxt, "hit": hit}
    if case["kind"] != "route" or case["decide"] or case["base"] == 3 or case["B"] * case["P"] * case["n_seq"] > 400000:
        return None
    W = wl.Workload(params=_params(case), seed=seed)
    tok, off = W.requests(0, case["B"])
    load = W.load().astype(np.int64)
    match = np.zeros((case["B"], W.P), np.int64)
    for p in range(W.P):
        for s in (W.tree(p).seq(i) for i in range(case["n_seq"])):
            for b in range(case["B"]):
                q = tok[off[b]: off[b + 1]]
                n = min(len(q), len(s))
                if n and q[0] == s[0]:
                    differ = np.flatnonzero(q[:n] != s[:n])
                    match[b, p] = max(match[b, p], differ[0] if len(differ) else n)
    score = match - W.alpha * load
    peer = np.array([min(range(W.P), key=lambda p: (-score[b, p], load[p], p)) for b in range(case["B"])], np.int64)
    return {"match": match, "peer": peer}
