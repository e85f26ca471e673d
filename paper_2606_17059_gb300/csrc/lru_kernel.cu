// lru_kernel.cu -- LRU eviction of a node's own cache trie on the device (EvictLRUTrie of Algorithm 1).
//
// Algorithm 1 evicts, while a request needs more memory than is free, the least recently used leaf token of
// the node's own trie, one token at a time (Section 2 primitive list: evictLRUTrie).  Every token's last
// access is the time of the latest insert (UpdateTrie) or served request (PrefixMatch) whose path covered it;
// ties go to the lexicographically smallest token path, and sequences that ended at an evicted token end one
// token earlier.
//
// Stamps.  A tree kept as an LRU cache has one stamp per node: the last access of every token of the node's
// edge.  An access that ends inside an edge splits it there (the upper part gets the new stamp; the node
// left between has one child and stores nothing -- the export merges such nodes back), so every edge's
// tokens share one stamp.  Times never decrease, so a token's stamp is never older than its descendants'.
//
// Eviction order without a token-by-token loop.  Let region(v) be the nodes of v's subtree reached from v
// through nodes of v's stamp, and end(v) the lexicographically largest token path in region(v) (follow the
// child with the largest first token among same-stamp children).  Removing the oldest leaf token n times
// removes the tokens in increasing order of (stamp, path of end, deeper first): a node becomes a leaf only
// after its descendants go, those of other stamps are older (removed before it) and those of its stamp
// include end(v), which precedes v in that order.  All tokens of one edge share the key, the deepest first.
// So n tokens are removed at once: the nodes whose key is below a threshold, and the tail of the one node at it.
//
// The threshold needs no sort and no rank of the nodes.  Its stamp S comes from a radix selection over the stamps,
// weighted by edge lengths; the r tokens left over are the first r of stamp S in the order of (end, deeper first),
// found by walking down from the root.  At a node u, `carry` is the length of the edges above (u's included) whose end
// lies in u's subtree: they are a run of stamp S down to u, each the largest same-stamp child of the one before. A
// child c then stands for T(c) tokens, the edge lengths of stamp S in its subtree, and for carry too if it is u's
// largest same-stamp child; the children are taken in token order, and the walk goes on in the one that holds token r.
// At a u of stamp S without a same-stamp child the carried edges end: the r tokens are taken from the deepest up.  A
// node of stamp S is removed if it precedes the walked path x in preorder or is one of those whole edges: one that
// follows x is not, nor is an ancestor on x that is not carried (its end follows x).
//
// Kernels:
//   lru_walk_kernel    warp per request: the match, and per node the deepest touched position (atomicMax)
//   lru_stamp_kernel   thread per node: stamp fully touched nodes, split partially touched edges
//   lru_evict_kernel   one cluster of CTAs does an eviction: breadth-first order, threshold, removal
#include "internal.h"

namespace p2p {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kLruThreads = 256;
constexpr int32_t kTouchFull = INT32_MAX;

struct LruTree {
  int4* node;
  int4* child;
  const int32_t* label;
  const int32_t* shared;
  uint32_t* stamp;
};

__device__ __forceinline__ const int32_t* lab_of(const LruTree& t, int32_t off) {
  return label_ptr(t.label, t.shared, off);
}

// Live child with first token tok in the table at off (2^bits slots), one warp: 1 (entry, slot), 0 none.
__device__ int find_live(const LruTree& t, int32_t off, int32_t bits, int32_t tok, int lane, int4& e, int32_t& slot) {
  if (bits == 0) return 0;
  const uint32_t mask = (1u << bits) - 1, h = slot_hash(tok, bits);
  for (uint32_t base = 0; base <= mask; base += 32) {
    const uint32_t s = (h + base + lane) & mask;
    const int4 x = t.child[off + s];
    const unsigned hit = __ballot_sync(kFull, x.y >= 1 && x.x == tok);
    const unsigned empty = __ballot_sync(kFull, x.y == 0);
    const int fh = hit ? __ffs(hit) - 1 : 64, fe = empty ? __ffs(empty) - 1 : 64;
    if (fh < fe) {
      e.x = tok;
      e.y = __shfl_sync(kFull, x.y, fh);
      e.z = __shfl_sync(kFull, x.z, fh);
      e.w = __shfl_sync(kFull, x.w, fh);
      slot = off + (int32_t)((h + base + fh) & mask);
      return 1;
    }
    if (fe < 64) return 0;
  }
  return 0;
}

// First j in [0, lim) with a[j] != b[j], or lim (one warp): 512 tokens per step and side, and the rest in one more, so
// that a prompt of a thousand tokens takes a few round trips (the walk of 4,096 requests 15 us; 256 tokens per step and
// the rest 32 at a time 19, 32 throughout 39).
__device__ int32_t first_mismatch(const int32_t* a, const int32_t* b, int32_t lim, int lane) {
  constexpr int U = 16;
  int32_t j0 = 0;
  for (; lim - j0 >= 32 * U; j0 += 32 * U) {
    int32_t x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = a[j0 + u * 32 + lane];
    int32_t d = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) d |= x[u] ^ b[j0 + u * 32 + lane];
    if (__any_sync(kFull, d != 0)) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned m = __ballot_sync(kFull, x[u] != b[j0 + u * 32 + lane]);
        if (m) return j0 + u * 32 + __ffs(m) - 1;
      }
    }
  }
  if (j0 < lim) {  // the rest in one round trip too
    int32_t x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = u * 32 + lane < lim - j0;
      x[u] = in ? a[j0 + u * 32 + lane] : 0;
      y[u] = in ? b[j0 + u * 32 + lane] : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned m = __ballot_sync(kFull, x[u] != y[u]);
      if (m) return j0 + u * 32 + __ffs(m) - 1;
    }
  }
  return lim;
}

__global__ void __launch_bounds__(kLruThreads) lru_walk_kernel(LruTree t, const int32_t* __restrict__ tokens,
                                                               int64_t n_tokens, const int64_t* __restrict__ offsets,
                                                               int64_t B, int32_t* touch, int32_t* pslot,
                                                               int32_t* out_match, int32_t* err) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kLruThreads / 32);
  for (int64_t b = ((int64_t)blockIdx.x * kLruThreads + threadIdx.x) >> 5; b < B; b += warps) {
    const int64_t start = offsets[b], end = offsets[b + 1];
    if (!(start >= 0 && start <= end && end <= n_tokens && end - start <= INT32_MAX)) {
      if (lane == 0) {
        if (out_match) out_match[b] = 0;
        atomicOr(err, ERR_BAD_OFFSETS);
      }
      continue;
    }
    const int32_t* req = tokens + start;
    const int32_t len = (int32_t)(end - start);
    int4 nd = t.node[0];
    int32_t pos = 0;
    for (int guard = 0; pos < len && guard <= len; ++guard) {
      int4 e;
      int32_t slot;
      if (!find_live(t, nd.x, tab_bits(nd.y), req[pos], lane, e, slot)) break;
      const int32_t lim = min(e.w, len - pos);
      const int32_t k = first_mismatch(lab_of(t, e.z), req + pos, lim, lane);
      if (k == e.w) {
        if (lane == 0) atomicMax(&touch[e.y], kTouchFull);
        pos += k;
        nd = t.node[e.y];
        continue;
      }
      if (lane == 0 && k > 0) {  // the access ends inside this edge: its first k tokens are touched
        atomicMax(&touch[e.y], k);
        pslot[e.y] = slot;  // every toucher writes the same slot (the edge's own)
      }
      pos += k;
      break;
    }
    if (lane == 0 && out_match) out_match[b] = pos;
  }
}

// Thread per node v >= 1 (n_node: the node count before this call's splits).  Fully touched: stamp t.
// Partially touched at k: a new node mid takes the edge's first k tokens (stamp t) and has v, with the
// rest of the edge, as its one child.  Room for one node and one 4-slot table per split is ensured by the host.
__global__ void __launch_bounds__(kLruThreads) lru_stamp_kernel(LruTree t, TreeState* st, const int32_t* touch,
                                                                const int32_t* pslot, int32_t n_node, uint32_t time) {
  const int64_t stride = (int64_t)gridDim.x * kLruThreads;
  for (int64_t v = 1 + (int64_t)blockIdx.x * kLruThreads + threadIdx.x; v < n_node; v += stride) {
    const int32_t k = touch[v];
    if (k == 0) continue;
    if (k == kTouchFull) {
      t.stamp[v] = time;
      continue;
    }
    const int32_t s = pslot[v];
    const int4 e = t.child[s];
    const int32_t mid = atomicAdd(&st->n_node, 1);
    const int32_t c0 = atomicAdd(&st->n_child, 1 << kMinTabBits);
    for (int j = 0; j < (1 << kMinTabBits); ++j) t.child[c0 + j] = make_int4(0, 0, 0, 0);
    const int4 lower = make_int4(lab_of(t, e.z)[k], (int32_t)v, label_adv(e.z, k), e.w - k);
    t.child[c0 + slot_hash(lower.x, kMinTabBits)] = lower;
    t.node[mid] = make_int4(c0, make_meta(kMinTabBits, 1), 1, 0);
    t.stamp[mid] = time;
    t.child[s] = make_int4(e.x, mid, e.z, k);
  }
}

// ---- eviction ---------------------------------------------------------------------------------------------
//
// One cluster of kEvictCtas CTAs, so that its steps are ordered by the cluster's hardware barrier: an eviction has
// about three steps per tree level and eight for the threshold.  With a launch per step (and per step of a global
// bitonic sort of all siblings, and a host read per step of a binary search for the threshold) an eviction from
// a trie of ~20,000 nodes took 240 launches and 100 host reads, 2.6 ms; now 0.11 ms (0.19 with large tables one after
// another, 32 nodes a warp at every level, and four passes of every selection).  What bounds it: the barriers and the
// dependent loads between them (a level's records, tables, stamps); 16 of the SMs stream the tables at ~1 TB/s,
// which large tries need less than the steps do.
constexpr int kEvictThreads = 1024;
constexpr int kEvictCtas = 16;
constexpr int kHeld = 8;        // slots a thread keeps of the table that the walk is at
constexpr int kLaneBits = 4;    // tables of up to 16 slots are read by one lane,
constexpr int kWarpBits = 8;    // up to 256 slots by one warp, larger ones by the whole cluster
constexpr int kStBefore = 0, kStAfter = 1, kStOnPath = 2, kStGone = 4;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

struct EvictShared {
  unsigned long long hist[256];
  unsigned long long below, sum, best;
  uint32_t least, most;  // of the keys of a selection
  int bin, child, len, tok;
};

// The bin of the 256 that holds unit r (0 <= r < the bins' sum) of the weights in S.hist, and the sum before it
// (S.bin, S.below; S.sum = all).  Every thread of the CTA calls it.
__device__ void pick_bin(EvictShared& S, unsigned long long r) {
  __syncthreads();
  if (threadIdx.x < 32) {
    unsigned long long w[8], mine = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) mine += w[c] = S.hist[threadIdx.x * 8 + c];
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(kFull, incl, o);
      if ((int)threadIdx.x >= o) incl += y;
    }
    unsigned long long at = incl - mine;
    if (r >= at && r < incl) {
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (r >= at && r < at + w[c]) {
          S.bin = threadIdx.x * 8 + c;
          S.below = at;
        }
        at += w[c];
      }
    }
    if (threadIdx.x == 31) S.sum = incl;
  }
  __syncthreads();
}

// The first pass of a radix selection by bytes over keys from lo to hi: those above it are the same in all keys.
__device__ __forceinline__ int first_pass(uint32_t lo, uint32_t hi) { return min(3, __clz((int)(lo ^ hi)) / 8); }
// The bytes of x above pass `pass`.
__device__ __forceinline__ uint32_t bytes_above(uint32_t x, int pass) { return pass == 0 ? 0u : x >> (32 - 8 * pass); }

// Adds w to bin k of S.hist: one addition for the warp when all of its lanes have the same bin (the high bytes
// of the keys usually agree).  Every lane of the warp calls it; w = 0 adds nothing.
__device__ __forceinline__ void add_bin(EvictShared& S, int k, unsigned long long w) {
  const unsigned has = __ballot_sync(kFull, w != 0);
  if (!has) return;
  const int k0 = __shfl_sync(kFull, k, __ffs(has) - 1);
  if (__all_sync(kFull, w == 0 || k == k0)) {
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&S.hist[k0], w);
  } else if (w) {
    atomicAdd(&S.hist[k], w);
  }
}

__global__ void __launch_bounds__(kEvictThreads, 1) lru_evict_kernel(LruTree t, TreeState* st, LruScratch s, int32_t N,
                                                                     unsigned long long want) {
  __shared__ EvictShared S;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t rank = cluster_rank();
  const int n_warps = (int)cluster_size() * (kEvictThreads / 32), gw = (int)rank * (kEvictThreads / 32) + warp;
  const int n_threads = n_warps * 32, gt = gw * 32 + lane;
  const bool lead = rank == 0 && threadIdx.x == 0;
  if (lead) {
    s.order[0] = 0;
    s.lvl[0] = 0;
    s.lvl[1] = 1;
    s.sum[0] = 0;
    s.state[0] = kStOnPath;
  }
  cluster_sync();
  // Breadth-first order, a level at a time.  By position in the order: node, parent, slot, edge length, stamp.
  uint32_t newest = 0, oldest = ~0u;  // stamps this thread has put
  auto put = [&](int32_t at, int32_t v, int32_t slot, const int4& e) {
    if (at >= N) return;  // (more nodes than the tree has: reported below)
    const uint32_t x = t.stamp[e.y];
    s.order[at] = e.y;
    s.parent[at] = v;
    s.cslot[at] = slot;
    s.len[at] = e.w;
    s.stamp[at] = x;
    s.sum[e.y] = 0;
    newest = max(newest, x);
    oldest = min(oldest, x);
  };
  // (Ahead of a barrier that follows the last put.)
  auto put_range = [&]() {
    const uint32_t hi = __reduce_max_sync(kFull, newest), lo = __reduce_min_sync(kFull, oldest);
    if (lane == 0 && lo <= hi) {
      atomicMax(&s.out[5], (unsigned long long)hi);
      atomicMax(&s.out[6], (unsigned long long)~lo);
    }
  };
  int32_t begin = 0, end = 1, L = 0;
  for (;;) {
    // Nodes per warp: few enough that every warp has some, since a warp reads its nodes' larger tables one by one.
    const int32_t per = max(1, min(32, (end - begin) / n_warps));
    for (int32_t b0 = begin + gw * per; b0 < end; b0 += n_warps * per) {
      const int32_t i = b0 + lane;
      const int32_t v = lane < per && i < end ? __ldcg(s.order + i) : -1;
      const int4 nd = v >= 0 ? t.node[v] : make_int4(0, 0, 0, 0);
      const int32_t bits = tab_bits(nd.y);
      const int32_t z = bits > 0 && bits <= kWarpBits ? max(nd.z, 0) : 0;  // its children, placed side by side
      int32_t incl = z;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      const int32_t total = __shfl_sync(kFull, incl, 31);
      int32_t base = 0;
      if (lane == 31 && total) base = atomicAdd(&s.cnt[L + 1], total);
      base = __shfl_sync(kFull, base, 31);
      int32_t at = end + base + incl - z;
      const int32_t stop = at + z;
      if (bits > kWarpBits) {
        const int32_t k = atomicAdd(&s.big_cnt[L], 1);
        if (k < N) s.big[k] = v;
      } else if (bits > 0 && bits <= kLaneBits) {
        for (int32_t j0 = 0; j0 < (1 << bits) && at < stop; j0 += 4) {
          int4 e[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) e[c] = t.child[nd.x + j0 + c];
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (e[c].y >= 1 && at < stop) put(at++, v, nd.x + j0 + c, e[c]);
        }
      }
      for (unsigned m = __ballot_sync(kFull, bits > kLaneBits && bits <= kWarpBits); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const int32_t x = __shfl_sync(kFull, nd.x, j), size = 1 << __shfl_sync(kFull, bits, j);
        const int32_t vj = __shfl_sync(kFull, v, j), sj = __shfl_sync(kFull, stop, j);
        int32_t aj = __shfl_sync(kFull, at, j);
        for (int32_t j0 = 0; j0 < size; j0 += 32) {
          const int4 e = t.child[x + j0 + lane];
          const unsigned lm = __ballot_sync(kFull, e.y >= 1);
          const int32_t pos = aj + __popc(lm & ((1u << lane) - 1));
          if (e.y >= 1 && pos < sj) put(pos, vj, x + j0 + lane, e);
          aj += __popc(lm);
        }
      }
    }
    put_range();
    cluster_sync();
    const int32_t nb = min(__ldcg(s.big_cnt + L), N);
    if (nb) {
      // 32 large tables at a time: a warp takes 32 slots of any of them.
      for (int32_t k0 = 0; k0 < nb; k0 += 32) {
        const int32_t v = k0 + lane < nb ? __ldcg(s.big + k0 + lane) : -1;
        const int4 nd = v >= 0 ? t.node[v] : make_int4(0, 0, 0, 0);
        const int32_t parts = v >= 0 ? 1 << (tab_bits(nd.y) - 5) : 0;
        int32_t incl = parts;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int32_t y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        const int32_t parts_all = __shfl_sync(kFull, incl, 31);
        for (int32_t c = gw; c < parts_all; c += n_warps) {
          const int j = __popc(__ballot_sync(kFull, incl <= c));  // part c is the j-th table's
          const int32_t vj = __shfl_sync(kFull, v, j);
          const int32_t slot = __shfl_sync(kFull, nd.x, j) + 32 * (c - __shfl_sync(kFull, incl - parts, j)) + lane;
          const int4 e = t.child[slot];
          const unsigned lm = __ballot_sync(kFull, e.y >= 1);
          int32_t base = 0;
          if (lane == 0 && lm) base = atomicAdd(&s.cnt[L + 1], __popc(lm));
          base = __shfl_sync(kFull, base, 0);
          if (e.y >= 1) put(end + base + __popc(lm & ((1u << lane) - 1)), vj, slot, e);
        }
      }
      put_range();
      cluster_sync();
    }
    const int32_t c = __ldcg(s.cnt + L + 1);
    if (c <= 0) break;
    if ((int64_t)end + c > N) {  // an inconsistent tree: nothing is removed
      if (lead) s.out[1] = 1;
      return;
    }
    begin = end;
    end += c;
    ++L;
    if (lead) s.lvl[L + 1] = end;
  }
  const int32_t total = end;
  // The stamp S of the threshold: a radix selection of unit `want` of the edge lengths by stamp.
  const uint32_t stamp_hi = (uint32_t)__ldcg(s.out + 5), stamp_lo = ~(uint32_t)__ldcg(s.out + 6);
  const int stamp_pass = first_pass(stamp_lo, stamp_hi);
  uint32_t cut_stamp = bytes_above(stamp_hi, stamp_pass);
  unsigned long long rest = want;
  bool all = false;
  for (int pass = stamp_pass; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int k = threadIdx.x; k < 256; k += kEvictThreads) S.hist[k] = 0;
    __syncthreads();
    for (int32_t i0 = 1 + gw * 32; i0 < total; i0 += n_threads) {
      const int32_t i = i0 + lane;
      const uint32_t x = i < total ? __ldcg(s.stamp + i) : 0u;
      const bool in = i < total && bytes_above(x, pass) == cut_stamp;
      add_bin(S, (int)((x >> shift) & 255u), in ? (unsigned long long)__ldcg(s.len + i) : 0ull);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 256; k += kEvictThreads)
      if (S.hist[k]) atomicAdd(&s.hist[pass * 256 + k], S.hist[k]);
    cluster_sync();
    for (int k = threadIdx.x; k < 256; k += kEvictThreads) S.hist[k] = __ldcg(&s.hist[pass * 256 + k]);
    pick_bin(S, rest);
    if (pass == stamp_pass) {
      if (lead) s.out[0] = S.sum;
      if (rest >= S.sum) {
        all = true;
        break;
      }
    }
    rest -= S.below;
    cut_stamp = (cut_stamp << 8) | (uint32_t)S.bin;
    __syncthreads();
  }
  // The place of token `rest` of stamp S: T bottom-up, then the walk down from the root (the first CTA).
  const bool walk = !all && rest > 0;
  int32_t depth = 0, cut_level = 0, cut = 0;
  if (walk) {
    for (int32_t l = L; l >= 1; --l) {
      const int32_t hi = __ldcg(s.lvl + l + 1);
      for (int32_t i = __ldcg(s.lvl + l) + gt; i < hi; i += n_threads) {
        const int32_t v = __ldcg(s.order + i);
        const unsigned long long own = __ldcg(s.stamp + i) == cut_stamp ? (unsigned long long)__ldcg(s.len + i) : 0ull;
        const unsigned long long T = __ldcg(s.sum + v) + own;
        if (own) s.sum[v] = T;
        if (T) atomicAdd(&s.sum[__ldcg(s.parent + i)], T);
      }
      cluster_sync();
    }
    if (rank == 0) {
      int32_t u = 0, lev = 0, len_u = 0;
      unsigned long long carry = 0, r = rest;
      for (; lev <= L; ++lev) {
        const int4 nd = t.node[u];
        const int32_t size = tab_bits(nd.y) ? 1 << tab_bits(nd.y) : 0;
        const bool same = u != 0 && t.stamp[u] == cut_stamp;
        if (same) carry += (unsigned long long)len_u;
        // The children's keys and weights, kept by the threads for a table of up to kHeld slots a thread, and read
        // again by each step for a larger one.
        const bool held = size <= kHeld * kEvictThreads;
        uint32_t kx[kHeld] = {};
        unsigned long long kw[kHeld] = {};
        if (held) {
#pragma unroll
          for (int c = 0; c < kHeld; ++c) {
            const int32_t j = c * kEvictThreads + (int32_t)threadIdx.x;
            const int4 e = j < size ? t.child[nd.x + j] : make_int4(0, 0, 0, 0);
            kx[c] = (uint32_t)e.x ^ 0x80000000u;
            kw[c] = e.y >= 1 ? __ldcg(s.sum + e.y) : 0ull;
          }
        }
        if (threadIdx.x == 0) {
          S.best = 0;
          S.child = S.len = S.tok = 0;
          S.least = ~0u;
          S.most = 0;
        }
        __syncthreads();
        if (same)
          for (int32_t j = threadIdx.x; j < size; j += kEvictThreads) {
            const int4 e = t.child[nd.x + j];
            if (e.y >= 1 && t.stamp[e.y] == cut_stamp)
              atomicMax(&S.best, ((unsigned long long)((uint32_t)e.x ^ 0x80000000u) << 32) | (uint32_t)e.y);
          }
        __syncthreads();
        const int32_t best = (int32_t)(S.best & 0xffffffffull);
        if (same && best == 0) break;  // the carried edges end here
        const uint32_t best_key = (uint32_t)(S.best >> 32);
        // f(key, weight) for every slot; all of a warp's lanes come to it together.
        auto each = [&](auto f) {
          if (held) {
#pragma unroll
            for (int c = 0; c < kHeld; ++c)
              if (c * kEvictThreads < size) f(kx[c], kw[c]);
          } else {
            for (int32_t j0 = 0; j0 < size; j0 += kEvictThreads) {
              // (A table this large is a multiple of the CTA.)
              const int4 e = t.child[nd.x + j0 + (int32_t)threadIdx.x];
              const uint32_t x = (uint32_t)e.x ^ 0x80000000u;
              const unsigned long long w = e.y >= 1 ? __ldcg(s.sum + e.y) : 0ull;
              f(x, w && same && x == best_key ? w + carry : w);
            }
          }
        };
        if (held && same) {  // (best stands for tokens of its own, so its weight is not 0; a tombstone's is)
#pragma unroll
          for (int c = 0; c < kHeld; ++c)
            if (kw[c] && kx[c] == best_key) kw[c] += carry;
        }
        uint32_t least = ~0u, most = 0;
        each([&](uint32_t x, unsigned long long w) {
          if (w) {
            least = min(least, x);
            most = max(most, x);
          }
        });
        least = __reduce_min_sync(kFull, least);
        most = __reduce_max_sync(kFull, most);
        if (lane == 0 && least <= most) {
          atomicMin(&S.least, least);
          atomicMax(&S.most, most);
        }
        __syncthreads();
        const int key_pass = first_pass(S.least, S.most);
        uint32_t key = bytes_above(S.most, key_pass);
        for (int pass = key_pass; pass < 4; ++pass) {
          const int shift = 24 - 8 * pass;
          for (int k = threadIdx.x; k < 256; k += kEvictThreads) S.hist[k] = 0;
          __syncthreads();
          each([&](uint32_t x, unsigned long long w) {
            add_bin(S, (int)((x >> shift) & 255u), bytes_above(x, pass) == key ? w : 0ull);
          });
          pick_bin(S, r);
          r -= S.below;
          key = (key << 8) | (uint32_t)S.bin;
          __syncthreads();
        }
        for (int32_t j = threadIdx.x; j < size; j += kEvictThreads) {
          const int4 e = t.child[nd.x + j];
          if (e.y >= 1 && ((uint32_t)e.x ^ 0x80000000u) == key) {
            S.child = e.y;
            S.len = e.w;
            S.tok = e.x;
          }
        }
        __syncthreads();
        if (!(same && S.child == best)) carry = 0;
        u = S.child;
        len_u = S.len;
        if (threadIdx.x == 0) {
          s.path_node[lev + 1] = u;
          s.path_tok[lev + 1] = S.tok;
          s.path_len[lev + 1] = len_u;
        }
        __syncthreads();
      }
      if (threadIdx.x == 0) {
        // r < carry: whole edges from the deepest up, then r tokens of the next.
        int32_t l = lev;
        while (l > 1 && r >= (unsigned long long)s.path_len[l]) r -= (unsigned long long)s.path_len[l--];
        s.out[2] = (unsigned long long)lev;
        s.out[3] = (unsigned long long)l;
        s.out[4] = r;
      }
    }
    cluster_sync();
    depth = (int32_t)__ldcg(s.out + 2);
    cut_level = (int32_t)__ldcg(s.out + 3);
    cut = (int32_t)__ldcg(s.out + 4);
  }
  // Removal, from the top: a node that goes is tombstoned in its parent's table when the parent stays, and its stored
  // sequences move to the nearest node that stays; the node at the threshold loses its last `cut` tokens.
  unsigned long long dead = 0, st_label = 0, st_child = 0;
  for (int32_t l = 1; l <= L; ++l) {
    const int32_t hi = __ldcg(s.lvl + l + 1);
    const int32_t x = walk && l <= depth ? __ldcg(s.path_node + l) : -1;
    const uint32_t xt = x >= 0 ? (uint32_t)__ldcg(s.path_tok + l) ^ 0x80000000u : 0u;
    for (int32_t i = __ldcg(s.lvl + l) + gt; i < hi; i += n_threads) {
      const int32_t v = __ldcg(s.order + i), p = __ldcg(s.parent + i), slot = __ldcg(s.cslot + i);
      const uint32_t stamp = __ldcg(s.stamp + i);
      const int up = __ldcg(s.state + p);
      int where = up & 3;
      if (walk && where == kStOnPath) {
        if (x < 0) where = kStAfter;
        else if (v != x) where = ((uint32_t)t.child[slot].x ^ 0x80000000u) < xt ? kStBefore : kStAfter;
      }
      const bool out = all || stamp < cut_stamp ||
                       (walk && stamp == cut_stamp &&
                        (where == kStBefore || (where == kStOnPath && l > cut_level)));
      s.state[v] = (uint8_t)(where | (out ? kStGone : 0));
      if (!out) {
        if (walk && where == kStOnPath && l == cut_level && cut > 0) t.child[slot].w -= cut;
        continue;
      }
      const bool orphan = up & kStGone;
      const int32_t sv = orphan ? __ldcg(s.surv + p) : p;
      s.surv[v] = sv;
      const int4 e = t.child[slot];
      if (!orphan) {
        t.child[slot].y = -1;  // a tombstone: the slot keeps its key
        atomicSub(&t.node[p].z, 1);
      }
      const int4 nd = t.node[v];
      if (nd.w) atomicAdd(&t.node[sv].w, nd.w);
      dead += 1;
      if (e.z >= 0) st_label += (unsigned long long)e.w;
      if (tab_bits(nd.y)) st_child += 1ull << tab_bits(nd.y);
    }
    cluster_sync();
  }
  for (int o = 16; o > 0; o >>= 1) {
    dead += __shfl_xor_sync(kFull, dead, o);
    st_label += __shfl_xor_sync(kFull, st_label, o);
    st_child += __shfl_xor_sync(kFull, st_child, o);
  }
  if (lane == 0 && dead) {
    atomicAdd((unsigned long long*)&st->dead_nodes, dead);
    if (st_label) atomicAdd((unsigned long long*)&st->stale_label, st_label);
    if (st_child) atomicAdd((unsigned long long*)&st->stale_child, st_child);
  }
}

// A batch as INSERT ops of one tree: op i = request i, one pool run (its tokens); a request with invalid
// offsets gets a negative run length, which the delta validation rejects.
__global__ void __launch_bounds__(kLruThreads) lru_ops_kernel(const int64_t* __restrict__ offsets, int64_t B,
                                                              int64_t n_tokens, int32_t* op, int64_t* seg_begin,
                                                              int64_t* seg_off, int32_t* seg_len) {
  const int64_t stride = (int64_t)gridDim.x * kLruThreads;
  for (int64_t b = (int64_t)blockIdx.x * kLruThreads + threadIdx.x; b <= B; b += stride) {
    seg_begin[b] = b;
    if (b == B) continue;
    const int64_t s = offsets[b], e = offsets[b + 1];
    const bool ok = s >= 0 && s <= e && e <= n_tokens && e - s <= INT32_MAX;
    op[b] = P2P_OP_INSERT;
    seg_off[b] = ok ? s : 0;
    seg_len[b] = ok ? (int32_t)(e - s) : -1;
  }
}

// Section 5's expected hit rate of each routed request: the share of its tokens its target already holds,
// match[b][peer[b]] / |r_b| (IEEE single precision, rounded to nearest); 0 for an empty or unrouted request.
__global__ void __launch_bounds__(kLruThreads) hit_rate_kernel(const int32_t* __restrict__ match, int32_t P,
                                                               const int64_t* __restrict__ offsets, int64_t B,
                                                               const int32_t* __restrict__ peer, float* out) {
  const int64_t stride = (int64_t)gridDim.x * kLruThreads;
  for (int64_t b = (int64_t)blockIdx.x * kLruThreads + threadIdx.x; b < B; b += stride) {
    const int64_t len = offsets[b + 1] - offsets[b];
    const int32_t k = peer[b];
    out[b] = (k >= 0 && k < P && len > 0) ? __fdiv_rn((float)match[b * P + k], (float)len) : 0.0f;
  }
}

inline int grid_for(int64_t n, int per, int num_sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, (int64_t)num_sms * 8));
}
inline LruTree lru_tree(const TreeState& s, const int32_t* shared) {
  return LruTree{s.node, s.child, s.label, shared, s.stamp};
}

}  // namespace

cudaError_t launch_lru_walk(const TreeState& s, const int32_t* shared, const int32_t* tokens, int64_t n_tokens,
                            const int64_t* offsets, int64_t B, int32_t* touch, int32_t* pslot, int32_t* out_match,
                            int32_t* err, int num_sms, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  P2P_TIMED(K_LRU_WALK, st,
            (lru_walk_kernel<<<grid_for(B, kLruThreads / 32, num_sms), kLruThreads, 0, st>>>(
                lru_tree(s, shared), tokens, n_tokens, offsets, B, touch, pslot, out_match, err)));
  return cudaGetLastError();
}

cudaError_t launch_lru_stamp(const TreeState& s, TreeState* d_state, const int32_t* shared, const int32_t* touch,
                             const int32_t* pslot, int32_t n_node, uint32_t time, int num_sms, cudaStream_t st) {
  if (n_node <= 1) return cudaSuccess;
  P2P_TIMED(K_LRU_STAMP, st,
            (lru_stamp_kernel<<<grid_for(n_node, kLruThreads, num_sms), kLruThreads, 0, st>>>(
                lru_tree(s, shared), d_state, touch, pslot, n_node, time)));
  return cudaGetLastError();
}

size_t lru_scratch(int64_t N, void* base, LruScratch& s) {
  char* p = static_cast<char*>(base);
  size_t at = 0;
  auto take = [&](size_t bytes) {
    void* q = p ? p + at : nullptr;
    at += (bytes + 15) & ~(size_t)15;
    return q;
  };
  const size_t n = (size_t)N, levels = (size_t)N + 2;
  s.cnt = static_cast<int32_t*>(take(levels * 4));
  s.big_cnt = static_cast<int32_t*>(take(levels * 4));
  s.hist = static_cast<unsigned long long*>(take(4 * 256 * 8));
  s.out = static_cast<unsigned long long*>(take(8 * 8));
  s.zeroed = at;
  s.sum = static_cast<unsigned long long*>(take(n * 8));
  s.order = static_cast<int32_t*>(take(n * 4));
  s.parent = static_cast<int32_t*>(take(n * 4));
  s.cslot = static_cast<int32_t*>(take(n * 4));
  s.len = static_cast<int32_t*>(take(n * 4));
  s.stamp = static_cast<uint32_t*>(take(n * 4));
  s.surv = static_cast<int32_t*>(take(n * 4));
  s.big = static_cast<int32_t*>(take(n * 4));
  s.lvl = static_cast<int32_t*>(take(levels * 4));
  s.path_node = static_cast<int32_t*>(take(levels * 4));
  s.path_tok = static_cast<int32_t*>(take(levels * 4));
  s.path_len = static_cast<int32_t*>(take(levels * 4));
  s.state = static_cast<uint8_t*>(take(n));
  return at;
}

cudaError_t launch_lru_evict(const TreeState& tree, TreeState* d_state, const LruScratch& s, int32_t N,
                             unsigned long long want, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(s.cnt, 0, s.zeroed, st);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lru_evict_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kEvictCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(kEvictCtas);
  cfg.blockDim = dim3(kEvictThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int fit = 0;
  if (cudaOccupancyMaxActiveClusters(&fit, lru_evict_kernel, &cfg) != cudaSuccess || fit < 1) {
    (void)cudaGetLastError();
    attr[0].val.clusterDim.x = 8;  // the portable size
    cfg.gridDim = dim3(8);
  }
  P2P_TIMED(K_LRU_EVICT, st,
            (e = cudaLaunchKernelEx(&cfg, lru_evict_kernel, lru_tree(tree, nullptr), d_state, s, N, want)));
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t launch_lru_ops(const int64_t* offsets, int64_t B, int64_t n_tokens, int32_t* op, int64_t* seg_begin,
                           int64_t* seg_off, int32_t* seg_len, int num_sms, cudaStream_t st) {
  P2P_TIMED(K_LRU_OPS, st,
            (lru_ops_kernel<<<grid_for(B + 1, kLruThreads, num_sms), kLruThreads, 0, st>>>(offsets, B, n_tokens, op,
                                                                                           seg_begin, seg_off,
                                                                                           seg_len)));
  return cudaGetLastError();
}

cudaError_t launch_hit_rate(const int32_t* match, int32_t P, const int64_t* offsets, int64_t B, const int32_t* peer,
                            float* out, int num_sms, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  P2P_TIMED(K_HIT_RATE, st,
            (hit_rate_kernel<<<grid_for(B, kLruThreads, num_sms), kLruThreads, 0, st>>>(match, P, offsets, B, peer,
                                                                                        out)));
  return cudaGetLastError();
}

}  // namespace p2p
