// delta_bulk.cu -- the ops of a delta that do not meet, applied all at once over the whole GPU.
//
// delta_kernel gives a tree to one CTA and an op to one warp, which walks the tree, then changes it: an op is a
// chain of a dozen dependent loads (10-28 us), and a tree has 16 such chains in flight.  A delta that goes mostly
// to one tree (a routed batch, the own cache) leaves the rest of the GPU idle, and 256 trees keep 4,096 chains
// going where the SMs could hold over 100,000.  But ops on different sequences commute, and nearly all of them
// touch nothing in common: so here every op is walked by one lane of a grid-wide launch that changes nothing, says
// which table slot and which nodes it would touch, and is then applied in a later launch if nothing else wants
// them first.  What is left after kBulkRounds such rounds goes to delta_kernel.
//
// A round, three launches:
//   bulk_resolve_kernel  a lane per op: the read-only walk.  It ends in a place: a node u and a token (a slot of u's
//                        table, whether taken or free).  The op enters the places it needs for itself in a key table
//                        (the smallest op index wins each), its own place first, and the node it depends on in a
//                        node table:
//                          leaf     INSERT of a new leaf edge under u            (u, tok), shares u; if u is a leaf
//                                                                                itself, u's own place too
//                          split    INSERT that leaves the edge (u, tok) inside  (u, tok), shares u
//                          count    INSERT or DELETE that only changes a node's sequence count
//                                                                                its place, shares the node (a DELETE
//                                                                                that leaves it without one: alone)
//                          remove   DELETE of the leaf v under u                 (u, tok), shares u
//                          fold     the same where u then has one child y left and stores nothing: u takes y in
//                                                                                (u, tok), u's own place, u alone;
//                                                                                y's place if it is a leaf, else y
//                                                                                alone
//                          absent   DELETE of a sequence that is not stored      (u, tok)
//                        An op of any other form (a DELETE that takes in a node's only child, say) holds its place and
//                        is left over.
//   bulk_grow_kernel     the tables of nodes that would pass 1/2 claimed with the round's leaves under them.
//   bulk_apply_kernel    an op that won its places, and whose node nobody shares if it needs it alone (and no op of
//                        smaller index needs it alone too), is applied: room for the warp's ops with one reservation
//                        per tree and arena, labels copied by the whole warp, slots, records and counts by the op's
//                        lane.  The others go to the next round's list, and with them those that found no room: the
//                        host then grows their tree, by what the round's ops that could go came to.
// Of the removals under a node with z children that stores nothing only the first z - 2 to arrive go in one round, so
// no node is left with fewer than 2 children unless it is folded.  A leaf's record and what hangs from it are
// changed only by ops that hold its place.  Ops on one sequence always name the same place first, the one with the
// smallest index wins it and the others wait: they apply in op order.  A place that an op could not enter (no room in
// the key table) cannot be entered by the others that name it either, so none of them overtakes it.
//
// What bounds it: each lane's chain of dependent loads (a probe, a compare and a record per tree level), with
// 32 chains a warp in flight.  Long compares are made by the warp, once per launch for an interned label and a
// pool run (the table delta_kernel uses): the lane that enters a pair first compares it, the others go on with
// other edges and look again.
//
// Measured, the delta of a call (delta_kernel alone -> these rounds and delta_kernel behind them): 16,384 routed
// requests into 16 trees, most into one, 8.2 -> 0.18 ms; 4,096 requests into one cache trie 2.46 -> 0.12 ms; 300 ops
// into one tree 189 -> 77 us; 1,024,000 ops on 256 trees of 40,000 sequences 3.58 -> 1.37 ms.
#include "internal.h"

namespace p2p {

// What an op would do, as found by the walk.  u, tok: its place, which was slot `slot` of u's table at table offset
// `tab` then; key: its entry.  Then by kind: k where a split cuts the edge, the leaf a removal takes, the node of a
// count (arg) and its entry (ent); a leaf's entry of u (ent).  The second half only for a fold (v = arg; g, gpos: u's
// own place) and a leaf under a leaf (key2).
struct __align__(32) BulkOp {
  int32_t what;  // B_* | BF_* flags | tree << kTreeShift
  int32_t u, tok, slot;
  int32_t key, arg, ent, pos;
  int32_t key2, key3, ent_u, ent_y;
  int32_t g, gpos, pad0, pad1;
};

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBulkThreads = 256;
constexpr int kBulkWarps = kBulkThreads / 32;
constexpr int kBulkCtasPerSm = 4;   // at most 64 registers a thread (80 and 3 CTAs: the resolve launches of a step of
                                    // 1,024,000 ops 0.90 ms instead of 0.81)
// Label tokens after the first eight that a lane compares alone: a warp of few ops has its lanes compare them together
// instead (one round trip an op, where the lane takes one per eight tokens).  16,384 routed requests, four ops a warp:
// the first resolve launch 8% shorter; a warp of 16 ops or more keeps its 128.
constexpr int kLaneSpan = 128, kLaneSpanPerOp = 8;
constexpr int kLaneBits = 5;        // tables up to 32 slots are moved by one lane,
constexpr int kMaskBits = 9;        // up to 512 by one warp with a bit mask of the slots it has filled
constexpr int kMaskWords = 1 << (kMaskBits - 5);
constexpr int kMaxProbes = 64;      // of the key and node tables
constexpr int kMemoProbes = 4;
constexpr int kMemoWaits = 256;     // looks at a pair another warp compares before the lane's warp compares it too
constexpr int kFoldBits = 6;        // tables a lane searches for the one other child

enum { B_NONE = 0, B_LEAF, B_SPLIT, B_COUNT, B_REMOVE, B_FOLD, B_ABSENT, B_LEFT };
enum { BF_ALONE = 16, BF_REVIVE = 32, BF_MORE = 64, BF_LATER = 128 };  // BF_MORE: the record's second half holds
constexpr int kTreeShift = 8;  // (a tree index has 16 bits)

// Enters (tree, u, tok) of this round for op idx; the table's index, or -1 if it has no room near the key's home.  An
// entry is 32 bits of the place's hash over the complement of the smallest op index.  Two places that share those
// bits and the neighbourhood only wait for one another.
__device__ int32_t enter_key(const BulkTables& T, int32_t tree, int32_t u, int32_t tok, int round, uint32_t idx) {
  const unsigned long long h = mix64((((unsigned long long)(uint32_t)u << 32) | (uint32_t)tok) ^
                                     mix64(((unsigned long long)(uint32_t)tree << 8) | (unsigned)(round + 1)));
  const uint32_t mark = (uint32_t)(h >> 32) | 1u;  // 0 marks an empty entry
  const unsigned long long mine = ((unsigned long long)mark << 32) | (uint32_t)~idx;
  uint32_t s = (uint32_t)h & T.key_mask;
  for (int it = 0; it < kMaxProbes; ++it, s = (s + 1) & T.key_mask) {
    const unsigned long long prev = atomicCAS(&T.keys[s], 0ull, mine);
    if (prev == 0ull) return (int32_t)s;
    if ((uint32_t)(prev >> 32) == mark) {
      if (prev < mine) atomicMax(&T.keys[s], mine);
      return (int32_t)s;
    }
  }
  return -1;
}

// The entry of (tree, node) of this round; -1 if the table has no room for it near its home.
__device__ int32_t enter_node(const BulkTables& T, int32_t tree, int32_t node, int round) {
  const unsigned long long key = 1ull | ((unsigned long long)round << 1) | ((unsigned long long)(uint32_t)node << 8) |
                                 ((unsigned long long)(uint32_t)tree << 40);
  uint32_t s = (uint32_t)(mix64(key) >> 17) & T.node_mask;
  for (int it = 0; it < kMaxProbes; ++it, s = (s + 1) & T.node_mask) {
    const unsigned long long prev = atomicCAS(&T.nodes[s].key, 0ull, key);
    if (prev == 0ull || prev == key) return (int32_t)s;
  }
  return -1;
}

// An op's sequence: token j is a[j] below na, bo[j] from there (bo = the second pool run less na).
struct LaneSeq {
  const int32_t* a;
  const int32_t* bo;
  int32_t na, n;
  __device__ __forceinline__ int32_t at(int32_t j) const { return __ldg((j < na ? a : bo) + j); }
};
__device__ __forceinline__ LaneSeq lane_seq(const BulkArgs& A, int64_t i) {
  const int64_t g0 = A.seg_begin[i], g1 = A.seg_begin[i + 1];
  LaneSeq q;
  q.na = g1 > g0 ? A.seg_len[g0] : 0;
  q.a = A.pool + (g1 > g0 ? A.seg_off[g0] : 0);
  q.bo = q.a;
  q.n = q.na;
  if (g1 - g0 == 2) {
    q.bo = A.pool + A.seg_off[g0 + 1] - q.na;
    q.n = q.na + A.seg_len[g0 + 1];
  }
  return q;
}

// The tree (index into states) of op i, where the ops of lower lanes come before it: a search for the warp's first op,
// and from there a step per tree passed.  The whole warp calls it.
__device__ __forceinline__ int32_t tree_of(const BulkArgs& A, int64_t i) {
  if (!A.peer_begin) return 0;
  const int64_t i0 = __shfl_sync(kFull, i, 0);
  int32_t lo = 0, hi = A.n_trees;  // peer_begin[lo] <= i0 < peer_begin[hi]
  while (hi - lo > 1) {
    const int32_t mid = lo + (hi - lo) / 2;
    if (__ldg(A.peer_begin + mid) <= i0) lo = mid; else hi = mid;
  }
  while (lo + 1 < A.n_trees && __ldg(A.peer_begin + lo + 1) <= i) ++lo;
  return lo;
}

// One lane: the slot of tok in the table of 2^bits slots at off.  Returns 1 (live; e = the entry), 2 (tombstone) or
// 0 (absent); slot = where it is (absent: the first empty slot, or -1).  Two slots per step; kLive: each read as two
// 64-bit words whose first holds key and state, since other lanes claim other keys' slots meanwhile.
template <bool kLive>
__device__ int probe_lane(const int4* child, int32_t off, int32_t bits, int32_t tok, int32_t& slot, int4& e) {
  slot = -1;
  if (bits == 0) return 0;
  const uint32_t mask = (1u << bits) - 1, h = slot_hash(tok, bits);
  for (uint32_t i = 0; i <= mask; i += 2) {
    const uint32_t s0 = (h + i) & mask, s1 = (h + i + 1) & mask;
    int4 x, y;
    if constexpr (kLive) {
      const longlong2 u = __ldcg(reinterpret_cast<const longlong2*>(child + off + s0));
      const longlong2 v = __ldcg(reinterpret_cast<const longlong2*>(child + off + s1));
      x = make_int4((int32_t)u.x, (int32_t)((unsigned long long)u.x >> 32), (int32_t)u.y,
                    (int32_t)((unsigned long long)u.y >> 32));
      y = make_int4((int32_t)v.x, (int32_t)((unsigned long long)v.x >> 32), (int32_t)v.y,
                    (int32_t)((unsigned long long)v.y >> 32));
    } else {
      load_slots(child + off + s0, x, y);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int4 w = c ? y : x;
      if (w.y == 0) {
        slot = off + (int32_t)(c ? s1 : s0);
        return 0;
      }
      if (w.x == tok && (w.y >= 1 || w.y == -1)) {
        slot = off + (int32_t)(c ? s1 : s0);
        e = w;
        return w.y >= 1 ? 1 : 2;
      }
    }
  }
  return 0;
}

// A token of a label or a pool run that a lane reads on from: the whole 256 bytes come to L2 with the first one, where
// a lane's next steps find them.
__device__ __forceinline__ int32_t ld_ahead(const int32_t* p) {
  int32_t x;
  asm("ld.global.nc.L2::256B.b32 %0, [%1];" : "=r"(x) : "l"(p));
  return x;
}

// One lane: first j in [from, to) with lab[j] != q[pos + j], or to; lab[0 .. from) is known to agree.  Eight pairs in
// flight and no test per token: the last step ends at `to` and looks at tokens before it again instead of stopping
// short, so that lanes with ends of their own stay together (with a tested tail per lane the resolve launch had
// three times the instructions in this loop).  Only labels under eight tokens and steps across the two pool runs take
// a token at a time.
__device__ __forceinline__ int32_t diff_lane(const int32_t* lab, const LaneSeq& q, int32_t pos, int32_t from,
                                             int32_t to) {
  for (int32_t j0 = from; j0 < to; j0 += 8) {
    const int32_t s0 = min(j0, to - 8), p0 = pos + s0;
    if (s0 < 0 || (p0 < q.na && q.na - p0 < 8)) {
      const int32_t e = min(to, j0 + 8);
      for (int32_t j = j0; j < e; ++j)
        if (__ldg(lab + j) != q.at(pos + j)) return j;
      continue;
    }
    const int32_t* y = (p0 < q.na ? q.a : q.bo) + p0;
    int32_t x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = ld_ahead(lab + s0 + u);
    unsigned d = 0;  // bit u: token u differs
#pragma unroll
    for (int u = 0; u < 8; ++u) d |= (x[u] != ld_ahead(y + u) ? 1u : 0u) << u;
    if (d) return s0 + __ffs(d) - 1;
  }
  return to;
}

// One warp: first j in [from, to) with a[j] != b[j], or to; 256 tokens per step and side.
__device__ int32_t diff_warp(const int32_t* a, const int32_t* b, int32_t from, int32_t to, int lane) {
  constexpr int U = 8;
  int32_t j0 = from;
  for (; to - j0 >= 32 * U; j0 += 32 * U) {
    int32_t x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = __ldg(a + j0 + u * 32 + lane);
    int32_t d = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) d |= x[u] ^ __ldg(b + j0 + u * 32 + lane);
    if (__any_sync(kFull, d != 0)) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned m = __ballot_sync(kFull, x[u] != __ldg(b + j0 + u * 32 + lane));
        if (m) return j0 + u * 32 + (__ffs(m) - 1);
      }
    }
  }
  for (; j0 < to; j0 += 128) {
    int32_t x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool in = u * 32 + lane < to - j0;
      x[u] = in ? __ldg(a + j0 + u * 32 + lane) : 0;
      y[u] = in ? __ldg(b + j0 + u * 32 + lane) : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned m = __ballot_sync(kFull, x[u] != y[u]);
      if (m) return j0 + u * 32 + (__ffs(m) - 1);
    }
  }
  return to;
}

__device__ __forceinline__ int64_t list_size(const BulkArgs& A, int round) {
  return round == 0 ? A.n : A.counts[round];
}

__global__ void __launch_bounds__(kBulkThreads, kBulkCtasPerSm) bulk_resolve_kernel(BulkArgs A, int round) {
  const int lane = threadIdx.x & 31;
  const int64_t total = list_size(A, round);
  const int64_t warps = (int64_t)gridDim.x * kBulkWarps;
  // Ops per warp: few enough that every warp has some, since a warp's long compares follow one another, and rounded up,
  // since a few warps with a second turn double the launch (16,384 ops: 3.4 a warp, the resolve launches 34 -> 30 us).
  const int32_t per = (int32_t)max((int64_t)1, min((int64_t)32, (total + warps - 1) / warps));
  const int32_t lane_span = min(kLaneSpan, kLaneSpanPerOp * per);
  const int32_t* list = A.lists + (round & 1) * A.n;
  for (int64_t t = (int64_t)blockIdx.x * kBulkThreads + threadIdx.x; t < A.n_trees;
       t += (int64_t)gridDim.x * kBulkThreads) {
    const TreeState& s = A.states[t];  // the arenas' use ahead of this round's reservations
    A.base[3 * t] = s.n_node;
    A.base[3 * t + 1] = s.n_child;
    A.base[3 * t + 2] = s.n_label;
  }
  for (int64_t b0 = (((int64_t)blockIdx.x * kBulkThreads + threadIdx.x) >> 5) * per; b0 < total; b0 += warps * per) {
    int64_t i = b0 + lane;
    bool valid = lane < per && i < total;
    int32_t tree = round == 0 ? tree_of(A, min(i, total - 1)) : 0;
    if (valid && round > 0) i = list[i];
    valid = valid && !A.done[i];
    LaneSeq q{nullptr, nullptr, 0, 0};
    int32_t opc = 0;
    const int4* node = nullptr;
    const int4* child = nullptr;
    const int32_t* label = nullptr;
    if (valid) {
      q = lane_seq(A, i);
      opc = A.op[i];
      if (round > 0) tree = A.ops[i].what >> kTreeShift;
      const TreeState& s = A.states[tree];
      node = s.node;
      child = s.child;
      label = s.label;
    }
    valid = valid && q.n > 0;  // (an empty sequence is the root's own count: left to delta_kernel)
    // The walk: at node u (record nd, reached at pos), its parent g (reached at gpos, gz children, gw sequences)
    // and that one's parent gg.
    int32_t u = 0, pos = 0, g = -1, gpos = 0, gz = 0, gw = 0, gg = -1, ggpos = 0, k = 0, waits = 0;
    int32_t slot = -1;  // where the last probe ended
    int what = B_NONE, flags = 0;
    int4 nd = make_int4(0, 0, 0, 0), ce = nd, nn = nd;
    bool act = valid, held = false;  // held: at the edge ce, waiting for a pair that another warp compares
    int32_t lim = 0, first = 0;
    if (act) nd = __ldg(node);
    while (__any_sync(kFull, act)) {
      bool need = false;
      int32_t memo_at = -1;  // the pair's entry, when this lane is the one to compare it
      const int32_t* lab = nullptr;
      if (act && !held) {
        const int st = probe_lane<false>(child, nd.x, tab_bits(nd.y), q.at(pos), slot, ce);
        if (st != 1) {
          what = opc == P2P_OP_INSERT ? B_LEAF : B_ABSENT;
          flags = st == 2 ? BF_REVIVE : 0;
          act = false;
        } else if (ce.w <= 0 || ce.y <= 0) {  // (not in a valid tree: delta_kernel reports it)
          what = B_LEFT;
          act = false;
        } else {
          nn = __ldg(node + ce.y);
          lim = min(ce.w, q.n - pos);
          lab = label_ptr(label, A.shared, ce.z);
          first = min(lim, 9);
          k = diff_lane(lab, q, pos, 1, first);
          if (k == first && first < lim) {
            if (lim - first <= lane_span) {
              k = diff_lane(lab, q, pos, first, lim);
            } else {
              need = true;
              waits = 0;
            }
          }
        }
      } else if (act) {
        lab = label_ptr(label, A.shared, ce.z);
        need = true;
        held = false;
      }
      // A pair of an interned label and a pool run: how much of it is known to be equal, as far as this op's first run
      // goes (another op's may start at the same place and be longer).  One lane of the warp at a time
      // takes on a pair that nobody has compared yet, so that a launch's first compares spread over all warps (a
      // warp that took on each of its lanes' pairs had 20 of them to do, one after another, with the others waiting).
      int32_t free_at = -1;
      unsigned long long key = 0;
      if (need && ce.z < 0 && A.memo_keys && q.na - pos >= first) {
        const int64_t so = q.a + pos - A.pool;
        if (so <= 0xffffffffll) {
          key = (1ull << 63) | ((unsigned long long)(uint32_t)~ce.z << 32) | (unsigned long long)so;
          uint32_t s = (uint32_t)((key * 0x9E3779B97F4A7C15ull) >> 32) & A.memo_mask;
          for (int it = 0; it < kMemoProbes; ++it, s = (s + 1) & A.memo_mask) {
            const unsigned long long have = __ldcg(A.memo_keys + s);
            if (have == 0ull) {
              free_at = (int32_t)s;
              break;
            }
            if (have == key) {
              const int32_t known = min(__ldcg(A.memo_vals + s), q.na - pos);
              if (known == 0 && ++waits < kMemoWaits) {
                held = true;
              } else if (known >= lim) {
                k = lim;
                need = false;
              } else {
                first = max(first, known);
                memo_at = (int32_t)s;
              }
              break;
            }
          }
        }
      }
      const unsigned fm = __ballot_sync(kFull, free_at >= 0);
      if (free_at >= 0) {
        if (lane == __ffs(fm) - 1 && atomicCAS(A.memo_keys + free_at, 0ull, key) == 0ull) memo_at = free_at;
        else if (++waits < kMemoWaits) held = true;
      }
      if (held) need = false;
      if (!__any_sync(kFull, act && !held)) __nanosleep(200);  // (bounded by kMemoWaits looks)
      for (unsigned m = __ballot_sync(kFull, need); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const int32_t* l = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)lab, j);
        const int32_t* qa = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)(q.a + pos), j);
        const int32_t* qb = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)(q.bo + pos), j);
        const int32_t f = __shfl_sync(kFull, first, j), t = __shfl_sync(kFull, lim, j);
        const int32_t cut = max(f, min(t, __shfl_sync(kFull, q.na - pos, j)));  // below cut: the first pool run
        int32_t kk = diff_warp(l, qa, f, cut, lane);
        if (kk == cut && cut < t) kk = diff_warp(l, qb, cut, t, lane);
        if (lane == j) {
          k = kk;
          if (memo_at >= 0) atomicMax(A.memo_vals + memo_at, min(kk, q.na - pos));
        }
      }
      if (act && !held) {
        if (k == ce.w) {
          gg = g;
          ggpos = gpos;
          g = u;
          gpos = pos;
          gz = nd.z;
          gw = nd.w;
          u = ce.y;
          nd = nn;
          pos += k;
          if (pos == q.n) {  // the sequence ends at node u
            act = false;
            if (opc == P2P_OP_INSERT) what = B_COUNT;
            else if (nd.w == 0) what = B_ABSENT;
            else if (nd.w > 1 || nd.z >= 2) what = B_COUNT, flags = nd.w == 1 ? BF_ALONE : 0;
            else if (nd.z == 1) what = B_LEFT;
            else if (g == 0 || gw > 0 || gz >= 3) what = B_REMOVE;
            else what = gz == 2 ? B_FOLD : B_LEFT;
          }
        } else {
          what = opc == P2P_OP_INSERT ? B_SPLIT : B_ABSENT;
          act = false;
        }
      }
    }
    bool grow = false;
    int4 mine_grow = make_int4(0, 0, 0, 0);
    if (valid) {
      // The op's place and nodes.  An op that ended at a node has its place in the parent's table (the last slot found
      // led to it).
      const bool at_node = pos == q.n;
      const int32_t pu = at_node ? g : u, ppos = at_node ? gpos : pos;
      const int32_t tok = q.at(ppos);
      const uint32_t idx = (uint32_t)i;
      int32_t arg = k, ent = -1;
      const int32_t key = enter_key(A.tab, tree, pu, tok, round, idx);
      if (key < 0) what = B_LEFT;
      int4* out = reinterpret_cast<int4*>(A.ops + i);
      if (what == B_LEAF || what == B_SPLIT || what == B_REMOVE) {
        ent = enter_node(A.tab, tree, pu, round);
        if (ent < 0) {
          what = B_LEFT;
        } else {
          BulkNode* e = A.tab.nodes + ent;
          atomicAdd(&e->shared, 1u);
          if (what == B_LEAF && !(flags & BF_REVIVE)) {
            const uint32_t rank = atomicAdd(&e->leaves, 1u);
            // The leaf that takes a node's table past its half puts it on the list of those to grow.  (The root's table
            // grows between launches only; a leaf past its half waits for that.)
            const int32_t bits = tab_bits(nd.y);
            const int64_t used = (int64_t)tab_used(nd.y) + rank;
            if (tab_full(bits, used + 1)) {
              if (pu == 0) flags |= BF_LATER;
              else grow = rank == 0 || !tab_full(bits, used);
            }
          }
          if (what == B_REMOVE && g != 0 && gw == 0 && (int64_t)atomicAdd(&e->removals, 1u) > (int64_t)gz - 3)
            flags |= BF_LATER;
        }
        if (what == B_REMOVE) arg = u;
        if (what == B_LEAF && pu != 0 && nd.z == 0) {
          const int32_t key2 = enter_key(A.tab, tree, g, q.at(gpos), round, idx);
          if (key2 < 0) what = B_LEFT;
          flags |= BF_MORE;
          out[2] = make_int4(key2, -1, -1, -1);
        }
      } else if (what == B_COUNT) {
        arg = u;
        ent = enter_node(A.tab, tree, u, round);
        if (ent < 0) what = B_LEFT;
        else if (flags & BF_ALONE) atomicMax(&A.tab.nodes[ent].alone, ~idx);
        else atomicAdd(&A.tab.nodes[ent].shared, 1u);
      } else if (what == B_FOLD) {
        arg = u;
        const int4 rec = __ldg(node + pu);
        const int32_t bits = tab_bits(rec.y);
        int4 y = make_int4(0, -1, 0, 0);  // the one other child
        if (bits <= kFoldBits)
          for (int32_t s = 0; s < (1 << bits); ++s) {
            const int4 e = __ldg(child + rec.x + s);
            if (e.y >= 1 && e.y != u) y = e;
          }
        int32_t key2 = -1, key3 = -1, ent_u = -1, ent_y = -1;
        if (y.y >= 1 && gg >= 0) {
          key2 = enter_key(A.tab, tree, gg, q.at(ggpos), round, idx);
          ent_u = enter_node(A.tab, tree, pu, round);
          if (ent_u >= 0) atomicMax(&A.tab.nodes[ent_u].alone, ~idx);
          if (__ldg(node + y.y).z == 0) {
            key3 = enter_key(A.tab, tree, pu, y.x, round, idx);
          } else if ((ent_y = enter_node(A.tab, tree, y.y, round)) >= 0) {
            atomicMax(&A.tab.nodes[ent_y].alone, ~idx);
          }
        }
        if (key2 < 0 || ent_u < 0 || (key3 < 0 && ent_y < 0)) what = B_LEFT;
        flags |= BF_MORE;
        out[2] = make_int4(key2, key3, ent_u, ent_y);
        out[3] = make_int4(gg, ggpos, 0, 0);
      }
      out[0] = make_int4(what | flags | tree << kTreeShift, pu, tok, slot);
      out[1] = make_int4(key, arg, ent, ppos);
      if (grow) mine_grow = make_int4(tree, pu, ent, 0);
    } else if (lane < per && i < A.n && b0 + lane < total && !A.done[i]) {
      A.ops[i].what = B_LEFT;  // an empty sequence
    }
    const unsigned gm = __ballot_sync(kFull, grow);
    if (gm) {
      int32_t at = 0;
      if (lane == 0) at = atomicAdd(&A.counts[kBulkRounds + 1 + round], __popc(gm));
      at = __shfl_sync(kFull, at, 0);
      if (grow) A.grow[at + __popc(gm & ((1u << lane) - 1))] = mine_grow;
    }
  }
}

__device__ __forceinline__ void add64(int64_t* p, int64_t v) {
  if (v) atomicAdd((unsigned long long*)p, (unsigned long long)v);
}

// Moves the table of 2^bits slots at off to the fresh one of 2^nb <= 32 slots at dst, one lane: four slots at a time,
// placed by the bit mask of the slots it has filled.
__device__ void move_table_lane(int4* child, int32_t off, int32_t bits, int32_t dst, int32_t nb) {
  const uint32_t mask = (1u << nb) - 1;
  uint32_t used = 0;
  for (int32_t t0 = 0; bits && t0 < (1 << bits); t0 += 4) {
    int4 e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) e[c] = __ldcg(child + off + t0 + c);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (e[c].y < 1) continue;
      uint32_t sl = slot_hash(e[c].x, nb);
      while ((used >> sl) & 1u) sl = (sl + 1) & mask;
      used |= 1u << sl;
      child[dst + sl] = e[c];
    }
  }
  for (uint32_t t = 0; t <= mask; ++t)
    if (!((used >> t) & 1u)) child[dst + t] = make_int4(0, 0, 0, 0);
}

// The same for up to 2^kMaskBits slots, one warp, with a bit mask in shared memory.
__device__ void move_table_mask(int4* child, int32_t off, int32_t bits, int32_t dst, int32_t nb, uint32_t* used,
                                int lane) {
  const uint32_t mask = (1u << nb) - 1;
  if (lane < kMaskWords) used[lane] = 0;
  __syncwarp();
  for (int32_t t0 = 0; bits && t0 < (1 << bits); t0 += 128) {
    int4 e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int32_t t = t0 + c * 32 + lane;
      e[c] = t < (1 << bits) ? __ldcg(child + off + t) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (e[c].y < 1) continue;
      uint32_t sl = slot_hash(e[c].x, nb);
      while (atomicOr(&used[sl >> 5], 1u << (sl & 31)) >> (sl & 31) & 1u) sl = (sl + 1) & mask;  // (at most 1/2 taken)
      child[dst + sl] = e[c];
    }
  }
  __syncwarp();
  for (int32_t t = lane; t < (1 << nb); t += 32)
    if (!((used[t >> 5] >> (t & 31)) & 1u)) child[dst + t] = make_int4(0, 0, 0, 0);
  __syncwarp();
}

// The same for any size, one warp.
__device__ void move_table_warp(int4* child, int32_t off, int32_t bits, int32_t dst, int32_t nb, int lane) {
  const uint32_t mask = (1u << nb) - 1;
  for (int32_t t = lane; t < (1 << nb); t += 32) child[dst + t] = make_int4(0, 0, 0, 0);
  __syncwarp();
  for (int32_t t0 = 0; bits && t0 < (1 << bits); t0 += 128) {
    int4 e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int32_t t = t0 + c * 32 + lane;
      e[c] = t < (1 << bits) ? __ldcg(child + off + t) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (e[c].y < 1) continue;
      const unsigned long long kv = (unsigned long long)(uint32_t)e[c].x | ((unsigned long long)(uint32_t)e[c].y << 32);
      uint32_t sl = slot_hash(e[c].x, nb);
      for (uint32_t it = 0; it <= mask; ++it, sl = (sl + 1) & mask)
        if (atomicCAS((unsigned long long*)&child[dst + sl], 0ull, kv) == 0ull) {
          child[dst + sl].z = e[c].z;
          child[dst + sl].w = e[c].w;
          break;
        }
    }
  }
  __syncwarp();
}

// A lane per listed node: the round's leaves take its table past 1/2 claimed, so it moves to one of at most 1/4 live
// load (as delta_kernel grows tables), small ones by the lane and larger ones by the warp.  A table that cannot grow
// (no room in the arena) marks the node's entry, and its leaves wait.  (With every node that gets a leaf listed, and
// tables of 64 slots and more zeroed and filled by compare-and-swap, a step of 1,024,000 ops took 130 us of these
// launches; now 47.)
__global__ void __launch_bounds__(kBulkThreads) bulk_grow_kernel(BulkArgs A, int round) {
  __shared__ uint32_t s_used[kBulkWarps][kMaskWords];
  const int lane = threadIdx.x & 31;
  const int32_t total = A.counts[kBulkRounds + 1 + round];
  const int32_t warps = (int32_t)gridDim.x * kBulkWarps;
  // Nodes per warp: few, since a warp moves its larger tables one after another, but not one, since each warp reserves
  // its room in a tree's arena.
  const int32_t per = max(4, min(32, (total + warps - 1) / warps));
  for (int64_t b0 = (int64_t)((int32_t)blockIdx.x * kBulkWarps + (int32_t)(threadIdx.x >> 5)) * per; b0 < total;
       b0 += (int64_t)warps * per) {
    const bool valid = lane < per && b0 + lane < total;
    const int4 gr = valid ? A.grow[b0 + lane] : make_int4(-1, 0, 0, 0);
    const int32_t tree = gr.x, u = gr.y;
    int32_t nb = 0, c0 = 0;
    int4 rec = make_int4(0, 0, 0, 0);
    TreeState* s = A.states + max(tree, 0);
    if (valid) {
      const int64_t leaves = A.tab.nodes[gr.z].leaves;
      rec = s->node[u];
      const int32_t bits = tab_bits(rec.y);
      if (tab_full(bits, (int64_t)tab_used(rec.y) + leaves)) {
        nb = bits ? bits + 1 : kMinTabBits;
        while (nb < kMaxTabBits && ((int64_t)rec.z + leaves) * 4 > ((int64_t)1 << nb)) ++nb;
      }
    }
    const int32_t bits = tab_bits(rec.y);
    // Slots, once per tree and warp.
    for (unsigned m = __ballot_sync(kFull, nb > 0); m;) {
      const int32_t t = __shfl_sync(kFull, tree, __ffs(m) - 1);
      const bool mine = nb > 0 && tree == t;
      const unsigned mm = __ballot_sync(kFull, mine);
      m &= ~mm;
      int64_t sum = mine ? (int64_t)1 << nb : 0, old = mine && bits ? (int64_t)1 << bits : 0;
      const int64_t own = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, sum, o);
        if (lane >= o) sum += y;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) old += __shfl_xor_sync(kFull, old, o);
      const int64_t all = __shfl_sync(kFull, sum, 31);
      TreeState* ts = A.states + t;
      int32_t at = -1;
      if (lane == 0) {
        int32_t have = *(volatile int32_t*)&ts->n_child;
        for (int it = 0; it < (1 << 20) && (int64_t)have + all <= ts->cap_child; ++it) {
          const int32_t prev = atomicCAS(&ts->n_child, have, (int32_t)(have + all));
          if (prev == have) {
            at = have;
            break;
          }
          have = prev;
        }
        if (at >= 0) {
          atomicAdd(&A.base[3 * t + 1], (int32_t)all);
          add64(&ts->stale_child, old);
        }
      }
      at = __shfl_sync(kFull, at, 0);
      if (mine) {
        if (at < 0) {
          A.tab.nodes[gr.z].stuck = 1;
          nb = 0;
        } else {
          c0 = (int32_t)(at + sum - own);
        }
      }
    }
    int4* child = s->child;
    if (nb > 0 && nb <= kLaneBits) move_table_lane(child, rec.x, bits, c0, nb);
    for (unsigned m = __ballot_sync(kFull, nb > kLaneBits); m; m &= m - 1) {
      const int j = __ffs(m) - 1;
      int4* cj = (int4*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)child, j);
      const int32_t off = __shfl_sync(kFull, rec.x, j), bj = __shfl_sync(kFull, bits, j);
      const int32_t dst = __shfl_sync(kFull, c0, j), nj = __shfl_sync(kFull, nb, j);
      if (nj <= kMaskBits) move_table_mask(cj, off, bj, dst, nj, s_used[threadIdx.x >> 5], lane);
      else move_table_warp(cj, off, bj, dst, nj, lane);
    }
    if (nb > 0) s->node[u] = make_int4(c0, make_meta(nb, rec.z), rec.z, rec.w);
  }
}

// Copies, for every lane with n > 0, n tokens to dst: [0, na) from a, the rest from bo (bo[j] for j >= na); the
// whole warp copies.  Long runs (whole prompts) go one after another, 512 tokens per step, the others four at a time,
// 128 tokens of each per step: 16 loads a lane in flight both ways.  (Four at a time throughout, 64 tokens of each,
// every prompt among them took 35 round trips: the apply launch of 1,024,000 ops
// 0.42 -> 0.32 ms.)
constexpr int kCopies = 4, kCopySteps = 4;
constexpr int32_t kLongCopy = 256;
__device__ void copy_runs(int32_t* dst, const int32_t* a, const int32_t* bo, int32_t na, int32_t n, int lane) {
  for (unsigned m = __ballot_sync(kFull, n > kLongCopy); m; m &= m - 1) {
    const int j = __ffs(m) - 1;
    int32_t* d = (int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)dst, j);
    const int32_t* pa = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)a, j);
    const int32_t* pb = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)bo, j);
    const int32_t ca = __shfl_sync(kFull, na, j), cn = __shfl_sync(kFull, n, j);
    for (int32_t t0 = 0; t0 < cn; t0 += 32 * kCopies * kCopySteps) {
      int32_t x[kCopies * kCopySteps];
#pragma unroll
      for (int s = 0; s < kCopies * kCopySteps; ++s) {
        const int32_t t = t0 + s * 32 + lane;
        x[s] = t < cn ? ((t < ca ? pa : pb)[t]) : 0;
      }
#pragma unroll
      for (int s = 0; s < kCopies * kCopySteps; ++s) {
        const int32_t t = t0 + s * 32 + lane;
        if (t < cn) d[t] = x[s];
      }
    }
  }
  unsigned m = __ballot_sync(kFull, n > 0 && n <= kLongCopy);
  while (m) {
    int32_t* d[kCopies];
    const int32_t *pa[kCopies], *pb[kCopies];
    int32_t ca[kCopies], cn[kCopies], most = 0;
#pragma unroll
    for (int c = 0; c < kCopies; ++c) {
      const int j = m ? __ffs(m) - 1 : 0;
      d[c] = (int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)dst, j);
      pa[c] = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)a, j);
      pb[c] = (const int32_t*)__shfl_sync(kFull, (unsigned long long)(uintptr_t)bo, j);
      ca[c] = __shfl_sync(kFull, na, j);
      cn[c] = m ? __shfl_sync(kFull, n, j) : 0;
      m &= m - 1;
      most = max(most, cn[c]);
    }
    for (int32_t t0 = 0; t0 < most; t0 += 32 * kCopySteps) {
      int32_t x[kCopies][kCopySteps];
#pragma unroll
      for (int c = 0; c < kCopies; ++c)
#pragma unroll
        for (int s = 0; s < kCopySteps; ++s) {
          const int32_t t = t0 + s * 32 + lane;
          x[c][s] = t < cn[c] ? ((t < ca[c] ? pa[c] : pb[c])[t]) : 0;
        }
#pragma unroll
      for (int c = 0; c < kCopies; ++c)
#pragma unroll
        for (int s = 0; s < kCopySteps; ++s) {
          const int32_t t = t0 + s * 32 + lane;
          if (t < cn[c]) d[c][t] = x[c][s];
        }
    }
  }
}

__device__ __forceinline__ bool adjacent(const int4& a, const int4& b) {  // label b starts where label a ends
  if (a.z >= 0 && b.z >= 0) return (int64_t)a.z + a.w == b.z;
  if (a.z < 0 && b.z < 0) return (int64_t)~a.z + a.w == (int64_t)~b.z;
  return false;
}

__device__ __forceinline__ bool won(const BulkArgs& A, int32_t key, uint32_t idx) {
  return (uint32_t)__ldcg(A.tab.keys + key) == ~idx;
}
__device__ __forceinline__ bool alone(const BulkArgs& A, int32_t ent, uint32_t idx) {
  const BulkNode& e = A.tab.nodes[ent];
  return e.shared == 0 && e.alone == ~idx;
}

__global__ void __launch_bounds__(kBulkThreads, kBulkCtasPerSm) bulk_apply_kernel(BulkArgs A, int round) {
  const int lane = threadIdx.x & 31;
  const int64_t total = list_size(A, round);
  const int64_t warps = (int64_t)gridDim.x * kBulkWarps;
  const int32_t per = (int32_t)max((int64_t)1, min((int64_t)32, (total + warps - 1) / warps));
  const int32_t* list = A.lists + (round & 1) * A.n;
  int32_t* next = A.lists + ((round + 1) & 1) * A.n;
  for (int64_t b0 = (((int64_t)blockIdx.x * kBulkThreads + threadIdx.x) >> 5) * per; b0 < total; b0 += warps * per) {
    int64_t i = b0 + lane;
    bool valid = lane < per && i < total;
    if (valid && round > 0) i = list[i];
    valid = valid && !A.done[i];
    int what = B_NONE, flags = 0, opc = 0;
    int32_t tree = -1, u = 0, tok = 0, slot = -1, arg = 0, pos = 0;
    bool go = false;
    LaneSeq q{nullptr, nullptr, 0, 0};
    const uint32_t idx = (uint32_t)i;
    const int4* in = reinterpret_cast<const int4*>(A.ops + i);
    TreeState* s = A.states;
    int4 *node = nullptr, *child = nullptr;
    const int32_t* label = nullptr;
    int4 rec = make_int4(0, 0, 0, 0), e = rec;
    if (valid) {
      const int4 x = in[0], y = in[1];
      what = x.x & 15;
      flags = x.x & 0xf0;
      tree = x.x >> kTreeShift;
      u = x.y;
      tok = x.z;
      slot = x.w;
      arg = y.y;
      pos = y.w;
      opc = A.op[i];
      s += tree;
      node = s->node;
      child = s->child;
      label = s->label;
      go = what != B_LEFT && !(flags & BF_LATER) && won(A, y.x, idx);
      if (go && what == B_LEAF && !(flags & BF_REVIVE)) go = !A.tab.nodes[y.z].stuck;
      if (go && what == B_COUNT && (flags & BF_ALONE)) go = alone(A, y.z, idx);
      if (go && (flags & BF_MORE)) {
        const int4 z = in[2];
        go = won(A, z.x, idx);
        if (go && what == B_FOLD)
          go = alone(A, z.z, idx) && (z.y >= 0 ? won(A, z.y, idx) : alone(A, z.w, idx));
      }
      if (what == B_LEFT)  // (not an empty sequence)
        valid = A.seg_begin[i + 1] > A.seg_begin[i] && lane_seq(A, i).n > 0;
      if (go && (what == B_LEAF || what == B_SPLIT || what == B_FOLD)) q = lane_seq(A, i);
      // The place, as the walk found it or, where the table has moved since, looked up again.
      if (go && what <= B_FOLD && what != B_COUNT) {
        rec.x = __ldcg(&node[u].x);
        rec.y = __ldcg(&node[u].y);
        const int32_t bits = tab_bits(rec.y);
        const bool there = slot >= rec.x && slot < rec.x + (bits ? 1 << bits : 0);
        if (!there || (what != B_LEAF && what != B_FOLD) || (flags & BF_REVIVE)) {
          if (there && !(flags & BF_REVIVE)) {
            const longlong2 w = __ldcg(reinterpret_cast<const longlong2*>(child + slot));
            e = make_int4((int32_t)w.x, (int32_t)((unsigned long long)w.x >> 32), (int32_t)w.y,
                          (int32_t)((unsigned long long)w.y >> 32));
            go = e.x == tok && e.y >= 1;  // (always: nothing else may touch this op's slot)
          } else {
            const int st = probe_lane<true>(child, rec.x, bits, tok, slot, e);
            const int expect = what == B_LEAF ? (flags & BF_REVIVE ? 2 : 0) : 1;
            go = st == expect && slot >= 0;
          }
        }
      }
    }
    // A fold: u's own slot, and the child it takes in.
    int4 pe = make_int4(0, 0, 0, 0), ye = pe;
    int32_t pslot = -1;
    int32_t want_n = 0, want_c = 0, want_l = 0;
    if (go && what == B_FOLD) {
      const int4 gp = in[3];
      const int32_t gx = __ldcg(&node[gp.x].x), gy = __ldcg(&node[gp.x].y);
      int32_t ys = -1;
      slot = -1;
      for (int32_t t = 0; t < (1 << tab_bits(rec.y)); ++t) {
        const int4 o = __ldcg(child + rec.x + t);
        if (o.y >= 1 && o.y != arg) ys = t, ye = o;
        if (o.y == arg) slot = rec.x + t, e = o;
      }
      go = ys >= 0 && slot >= 0 && probe_lane<true>(child, gx, tab_bits(gy), q.at(gp.y), pslot, pe) == 1;
      if (go && !adjacent(pe, ye)) want_l = pe.w + ye.w;
    }
    if (go && what == B_LEAF) want_n = 1, want_l = q.n - pos;
    if (go && what == B_SPLIT) {
      want_l = q.n - pos - arg;
      want_n = want_l > 0 ? 2 : 1;
      want_c = 1 << kMinTabBits;
    }
    // Room, once per tree and warp.  Tickets count on past an arena's end, so none has to be taken back and no two get
    // the same room; an op past the end waits until the host has grown the tree, by what the tickets came to.
    int32_t n0 = 0, c0 = 0, l0 = 0;
    for (unsigned m = __ballot_sync(kFull, want_n | want_c | want_l); m;) {
      const int32_t t = __shfl_sync(kFull, tree, __ffs(m) - 1);
      const bool mine = (want_n | want_c | want_l) && tree == t;
      m &= ~__ballot_sync(kFull, mine);
      int32_t sn = mine ? want_n : 0, sc = mine ? want_c : 0;
      int64_t sl = mine ? want_l : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t an = __shfl_up_sync(kFull, sn, o), ac = __shfl_up_sync(kFull, sc, o);
        const int64_t al = __shfl_up_sync(kFull, sl, o);
        if (lane >= o) sn += an, sc += ac, sl += al;
      }
      const int32_t tn = __shfl_sync(kFull, sn, 31), tc = __shfl_sync(kFull, sc, 31);
      const int64_t tl = __shfl_sync(kFull, sl, 31);
      TreeState* ts = A.states + t;
      const int64_t k = lane == 0 ? tn : lane == 1 ? tc : lane == 2 ? tl : 0;
      int64_t at = 0, cap = 0;
      if (k) {
        at = A.base[3 * t + lane] + (int64_t)atomicAdd(&A.taken[((int64_t)round * A.n_trees + t) * 3 + lane],
                                                       (unsigned long long)k);
        cap = lane == 0 ? ts->cap_node : lane == 1 ? ts->cap_child : ts->cap_label;
      }
      const bool ok = __all_sync(kFull, at + k <= cap);
      if (k && at + k <= cap) {
        atomicMax(lane == 0 ? &ts->n_node : lane == 1 ? &ts->n_child : &ts->n_label, (int32_t)(at + k));
        if (!ok) add64(lane == 0 ? &ts->dead_nodes : lane == 1 ? &ts->stale_child : &ts->stale_label, k);
      } else if (k) {
        atomicOr(&ts->status, DELTA_NEED_SPACE | DELTA_NEED_BULK);
        atomicMax(lane == 0 ? &ts->need_node : lane == 1 ? &ts->need_child : &ts->need_label,
                  (int32_t)min(at + k - cap, (int64_t)INT32_MAX));
      }
      const int32_t bn = __shfl_sync(kFull, (int32_t)at, 0), bc = __shfl_sync(kFull, (int32_t)at, 1),
                    bl = __shfl_sync(kFull, (int32_t)at, 2);
      if (mine) {
        go = ok;
        n0 = bn + sn - want_n;
        c0 = bc + sc - want_c;
        l0 = (int32_t)(bl + sl - want_l);
      }
    }
    // The new labels: a leaf's tokens, or a fold's two labels joined.
    {
      const int32_t n = go ? want_l : 0;
      const int32_t *a = q.a, *bo = q.bo;
      int32_t na = 0;
      if (n > 0) {
        if (what == B_FOLD) {
          a = label_ptr(label, A.shared, pe.z);
          bo = label_ptr(label, A.shared, ye.z) - pe.w;
          na = pe.w;
        } else {
          const int32_t at = q.n - n;
          a = q.a + at;
          bo = q.bo + at;
          na = max(q.na - at, 0);
        }
      }
      copy_runs(n > 0 ? s->label + l0 : nullptr, a, bo, na, n, lane);
    }
    int32_t absent = 0, dead = 0, st_child = 0;
    int64_t st_label = 0;
    if (go) {
      switch (what) {
        case B_LEAF: {
          node[n0] = make_int4(0, 0, 0, 1);
          const unsigned long long kv = (unsigned long long)(uint32_t)tok | ((unsigned long long)(uint32_t)n0 << 32);
          if (flags & BF_REVIVE) {
            child[slot].z = l0;
            child[slot].w = want_l;
            child[slot].y = n0;
          } else {
            // The probe's first empty slot, or the next: other leaves of this table claim theirs meanwhile.  The
            // table has room for all of them (bulk_grow_kernel), so this ends within its size.
            const int32_t bits = tab_bits(rec.y);
            const uint32_t mask = (1u << bits) - 1;
            uint32_t sl = (uint32_t)(slot - rec.x);
            for (uint32_t it = 0; it <= mask; ++it, sl = (sl + 1) & mask)
              if (atomicCAS((unsigned long long*)&child[rec.x + sl], 0ull, kv) == 0ull) {
                child[rec.x + sl].z = l0;
                child[rec.x + sl].w = want_l;
                break;
              }
            atomicAdd(&node[u].y, 1 << 5);
          }
          atomicAdd(&node[u].z, 1);
          if (u == 0) {
            const uint32_t h = root_filter_bit(tok);
            atomicOr(s->rfilter + (h >> 5), 1u << (h & 31));
          }
          break;
        }
        case B_SPLIT: {
          const bool tail = want_l > 0;
          const int32_t mid = n0, leaf = n0 + 1;
          const int4 lower = make_int4(label_ptr(label, A.shared, e.z)[arg], e.y, label_adv(e.z, arg), e.w - arg);
          const uint32_t mask = (1u << kMinTabBits) - 1, s0 = slot_hash(lower.x, kMinTabBits);
          uint32_t s1 = s0;
          int4 le = make_int4(0, 0, 0, 0);
          if (tail) {
            le = make_int4(q.at(pos + arg), leaf, l0, want_l);
            s1 = slot_hash(le.x, kMinTabBits);
            if (s1 == s0) s1 = (s1 + 1) & mask;
            node[leaf] = make_int4(0, 0, 0, 1);
          }
          for (uint32_t t = 0; t <= mask; ++t)
            child[c0 + t] = t == s0 ? lower : (tail && t == s1) ? le : make_int4(0, 0, 0, 0);
          node[mid] = make_int4(c0, make_meta(kMinTabBits, tail ? 2 : 1), tail ? 2 : 1, tail ? 0 : 1);
          child[slot] = make_int4(tok, mid, e.z, arg);  // the slot keeps its key; the label starts where it did
          break;
        }
        case B_COUNT:
          atomicAdd(&node[arg].w, opc == P2P_OP_INSERT ? 1 : -1);
          break;
        case B_REMOVE:
        case B_FOLD: {
          const int32_t vb = tab_bits(__ldcg(&node[arg].y));
          child[slot].y = -1;  // a tombstone: the slot keeps its key
          st_label = e.w;
          dead = 1;
          st_child = vb ? 1 << vb : 0;
          if (what == B_REMOVE) {
            atomicAdd(&node[u].z, -1);
          } else {
            // u takes its last child in: the joined label, the child's record.
            child[pslot].z = want_l > 0 ? l0 : pe.z;
            child[pslot].w = pe.w + ye.w;
            node[u] = node[ye.y];
            st_label += want_l;
            dead += 1;
            st_child += tab_bits(rec.y) ? 1 << tab_bits(rec.y) : 0;
          }
          break;
        }
        default:
          absent = 1;
      }
      A.done[i] = 1;
    }
    // The trees' counts, once per tree and warp.
    for (unsigned m = __ballot_sync(kFull, go && (absent || dead)); m;) {
      const int j = __ffs(m) - 1;
      const int32_t t = __shfl_sync(kFull, tree, j);
      const bool mine = go && (absent || dead) && tree == t;
      m &= ~__ballot_sync(kFull, mine);
      int64_t v[4] = {mine ? absent : 0, mine ? dead : 0, mine ? st_child : 0, mine ? st_label : 0};
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(kFull, v[c], o);
      TreeState* ts = A.states + t;
      if (lane == 0) add64(&ts->n_absent, v[0]);
      if (lane == 1) add64(&ts->dead_nodes, v[1]);
      if (lane == 2) add64(&ts->stale_child, v[2]);
      if (lane == 3) add64(&ts->stale_label, v[3]);
    }
    // The rest goes to the next round.
    const bool again = valid && !go;
    const unsigned am = __ballot_sync(kFull, again);
    int32_t at = 0;
    if (lane == 0 && am) at = atomicAdd(&A.counts[round + 1], __popc(am));
    at = __shfl_sync(kFull, at, 0);
    if (again) next[at + __popc(am & ((1u << lane) - 1))] = (int32_t)i;
  }
}

}  // namespace

cudaError_t launch_bulk(const BulkArgs& A, int num_sms, cudaStream_t st, int* launched) {
  *launched = 0;
  if (A.n <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(A.tab.keys, 0, A.n_zero, st);
  if (e != cudaSuccess) return e;
  // A warp per op up to a full wave of resident CTAs (the kernels then take more ops per warp).
  const int grid = (int)std::min<int64_t>((A.n + kBulkWarps - 1) / kBulkWarps, (int64_t)num_sms * kBulkCtasPerSm);
  const int grid_g = (int)std::min<int64_t>((A.n + kBulkThreads - 1) / kBulkThreads, (int64_t)num_sms * 4);
  for (int round = 0; round < kBulkRounds; ++round) {
    P2P_TIMED(K_BULK_RESOLVE, st, (bulk_resolve_kernel<<<grid, kBulkThreads, 0, st>>>(A, round)));
    P2P_TIMED(K_BULK_GROW, st, (bulk_grow_kernel<<<grid_g, kBulkThreads, 0, st>>>(A, round)));
    P2P_TIMED(K_BULK_APPLY, st, (bulk_apply_kernel<<<grid, kBulkThreads, 0, st>>>(A, round)));
    *launched += 3;
  }
  return cudaGetLastError();
}

size_t bulk_scratch(int64_t n, int32_t n_trees, void* base, BulkArgs& A) {
  // Entries: a place per op and a few more for folds, a node per op at most, over all rounds.
  int64_t keys = 1024, nodes = 1024;
  while (keys < 2 * n) keys <<= 1;
  while (nodes < n + n / 4) nodes <<= 1;
  char* p = static_cast<char*>(base);
  size_t at = 0;
  auto take = [&](size_t bytes) {
    void* q = p ? p + at : nullptr;
    at += (bytes + 255) & ~(size_t)255;
    return q;
  };
  A.tab.keys = static_cast<unsigned long long*>(take((size_t)keys * sizeof(unsigned long long)));
  A.tab.key_mask = (uint32_t)(keys - 1);
  A.tab.nodes = static_cast<BulkNode*>(take((size_t)nodes * sizeof(BulkNode)));
  A.tab.node_mask = (uint32_t)(nodes - 1);
  A.taken = static_cast<unsigned long long*>(take((size_t)kBulkRounds * n_trees * 3 * sizeof(unsigned long long)));
  A.counts = static_cast<int32_t*>(take((2 * kBulkRounds + 1) * sizeof(int32_t)));
  A.n_zero = at;  // cleared by the launch up to here
  A.base = static_cast<int32_t*>(take((size_t)n_trees * 3 * sizeof(int32_t)));
  A.ops = static_cast<BulkOp*>(take((size_t)n * sizeof(BulkOp)));
  A.lists = static_cast<int32_t*>(take((size_t)n * 2 * sizeof(int32_t)));
  A.grow = static_cast<int4*>(take((size_t)n * sizeof(int4)));
  return at;
}

}  // namespace p2p
