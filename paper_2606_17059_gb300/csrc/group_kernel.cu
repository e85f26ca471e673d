// group_kernel.cu -- shared-prefix groups of a request batch, ahead of the route kernel.
//
// Requests of one batch often share long prefixes (a few-shot or system prompt in front of each query).
// Their walks in a tree coincide along the shared part, so a batch is routed in two passes: group leaders
// walk every tree as usual, and every other request of a group (a follower) starts from its leader's result.
// For a follower f of leader l with c = LCP(r_f, r_l) (exact, computed here):
//   - if match(r_l, T) < c, then match(r_f, T) = match(r_l, T): both walks stop at the same token;
//   - otherwise match(r_f, T) >= c, and the follower's walk need not compare its first c tokens.
// Both facts hold for the PrefixMatch of Algorithm 1 because a walk depends only on the request tokens it
// has consumed.  Results are therefore identical to independent walks; grouping changes only the work.
//
// Grouping: a request of at least kGroupHead tokens is keyed by a 64-bit hash of its first kGroupHead tokens
// and inserted into an open-addressing table; the smallest request index with that key leads the group.
// A follower whose exact common prefix with its leader is shorter than kGroupHead (a hash collision) routes
// as a leader instead.  The leader choice is deterministic (smallest index); the order of the two request
// lists is not, and only affects scheduling.  In a large batch each group's followers take a contiguous range of the
// follower list (group_ranges_kernel, group_place_kernel): the warps that route them at the same time then read the
// leader's match row, its checkpoints and the tables at the checkpoint nodes once, from cache.
#include "internal.h"

namespace p2p {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kGroupThreads = 256;

__device__ __forceinline__ bool request_range(const int64_t* offsets, int64_t b, int64_t tok_base, int64_t n_tokens,
                                              int64_t& start, int64_t& len) {
  start = offsets[b] - tok_base;
  const int64_t end = offsets[b + 1] - tok_base;
  len = end - start;
  return start >= 0 && start <= end && end <= n_tokens;
}

// One warp per `per` consecutive requests (lane i < per owns request base + i).  Eight lanes hash a request: four
// requests a step and two steps in flight, each lane eight tokens of each (token 8 j + s by lane s), mixed with their
// positions and summed.  (A request at a time by the whole warp, 32 in series, took 31 us for 65,536 requests and 30
// for 8,191; now 17 and 9.)  Then every distinct key of the warp is looked up or claimed once, by its lowest lane,
// which also lowers the key's leader index to that lane's request (the smallest of the warp's requests with the key).
__global__ void __launch_bounds__(kGroupThreads) group_hash_kernel(
    const int32_t* __restrict__ tokens, int64_t n_tokens, int64_t tok_base, const int64_t* __restrict__ offsets,
    int64_t B, int32_t per, unsigned long long* keys, int32_t* vals, int32_t bits, int32_t* slot_of) {
  static_assert(kGroupHead == 64, "eight tokens for each of eight lanes");
  const int lane = threadIdx.x & 31, sub = lane & 7;
  const int64_t warps = (int64_t)gridDim.x * (kGroupThreads / 32);
  const uint32_t mask = (1u << bits) - 1;
  for (int64_t base = (((int64_t)blockIdx.x * kGroupThreads + threadIdx.x) >> 5) * per; base < B; base += warps * per) {
    int64_t my_start = -1, len;  // -1: the lane's request is not grouped
    if (lane < per && base + lane < B) {
      const bool ok = request_range(offsets, base + lane, tok_base, n_tokens, my_start, len);
      if (!ok || len < kGroupHead) my_start = -1;
    }
    unsigned long long my_h = 0;
    for (int r0 = 0; r0 < per; r0 += 8) {
      unsigned long long h[2];
      int32_t x[2][8];
      int64_t st[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        st[c] = __shfl_sync(kFull, my_start, (r0 + 4 * c + (lane >> 3)) & 31);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[c][j] = st[c] >= 0 ? __ldg(tokens + st[c] + 8 * j + sub) : 0;
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        h[c] = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          h[c] += mix64((unsigned long long)(uint32_t)x[c][j] | ((unsigned long long)(8 * j + sub) << 32));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) h[c] += __shfl_xor_sync(kFull, h[c], o);
        // Lane r0 + 4 c + q owns the request that lanes 8 q .. 8 q + 7 hashed.
        const unsigned long long mine = __shfl_sync(kFull, h[c], (lane & 3) * 8);
        if ((lane >> 2) == (r0 >> 2) + c) my_h = mine | 1ull;  // 0 marks an empty slot
      }
    }
    if (my_start < 0) my_h = 0;
    const unsigned same = __match_any_sync(kFull, my_h);
    const int first = __ffs(same) - 1;
    int32_t slot = -1;
    if (my_h && lane == first) {
      uint32_t sl = (uint32_t)my_h & mask;
      for (uint32_t it = 0; it <= mask; ++it, sl = (sl + 1) & mask) {
        const unsigned long long prev = atomicCAS(&keys[sl], 0ull, my_h);
        if (prev == 0ull || prev == my_h) {
          slot = (int32_t)sl;
          break;
        }
      }
      if (slot >= 0) atomicMin(&vals[slot], (int32_t)(base + lane));
    }
    slot = __shfl_sync(kFull, slot, first);
    if (lane < per && base + lane < B) slot_of[base + lane] = my_h ? slot : -1;
  }
}

// First position in [0, n) where a and b differ, or n (one warp, both in global memory; 32 U tokens per step, and the
// rest in one more: at 32 tokens a round trip it took up to seven, 200,003 requests 152 us instead of 142).
template <int U>
__device__ int64_t lcp_warp(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int64_t n, int lane) {
  int64_t j0 = 0;
  for (; j0 + 32 * U <= n; j0 += 32 * U) {
    int32_t x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = __ldg(a + j0 + u * 32 + lane);
    int32_t diff = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) diff |= x[u] ^ __ldg(b + j0 + u * 32 + lane);
    if (__any_sync(kFull, diff != 0)) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned m = __ballot_sync(kFull, x[u] != __ldg(b + j0 + u * 32 + lane));
        if (m) return j0 + u * 32 + (__ffs(m) - 1);
      }
    }
  }
  if (j0 < n) {  // the rest, less than a step, in one round trip too
    const int32_t left = (int32_t)(n - j0);
    int32_t x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = u * 32 + lane < left;
      x[u] = in ? __ldg(a + j0 + u * 32 + lane) : 0;
      y[u] = in ? __ldg(b + j0 + u * 32 + lane) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned m = __ballot_sync(kFull, x[u] != y[u]);
      if (m) return j0 + u * 32 + (__ffs(m) - 1);
    }
  }
  return n;
}

// One warp per `per` consecutive requests (lane i < per owns request base + i): each request's leader; for each
// follower in turn, the exact common prefix with its leader (the whole warp compares); then the warp's leaders are
// appended to lists[0 ..) with one counter update, and so are its followers to lists[B ..) if `place` is set; if not,
// each follower takes its rank in its group (fcnt[leader] counts them; the rank goes to slot_of[b]) and
// group_ranges_kernel and group_place_kernel make the list.  A leader with followers gets the smallest of their common
// prefixes in cmin and, while rows last, a checkpoint row in gid (one update per distinct leader of the warp's
// followers).  U: 24 for long requests, whose longest compares bound the kernel (8,191 of 11,400 tokens 65 us; 16: 70,
// 32: 75), else 8 and more resident warps (200,003 of 1,250 tokens 142 us; 16: 148) -- but 16 beside a delta, whose
// kernels leave room for few warps (262,144 requests 0.43 ms; 8: 0.53).
template <int U>
__global__ void __launch_bounds__(kGroupThreads) group_resolve_kernel(
    const int32_t* __restrict__ tokens, int64_t n_tokens, int64_t tok_base, const int64_t* __restrict__ offsets,
    int64_t B, int32_t per, bool place, const int32_t* __restrict__ vals, int32_t* slot_of, int32_t* lead,
    int32_t* cpre, int32_t* lists, int32_t* counts, int32_t* gid, int32_t* cmin, int32_t gcap, int32_t* fcnt) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kGroupThreads / 32);
  for (int64_t base = (((int64_t)blockIdx.x * kGroupThreads + threadIdx.x) >> 5) * per; base < B; base += warps * per) {
    const int64_t b = base + lane;
    const bool valid = lane < per && b < B;
    const int32_t s = valid ? slot_of[b] : -1;
    const int32_t l = s >= 0 ? vals[s] : (int32_t)b;
    int32_t my_c = -1;
    for (unsigned fm = __ballot_sync(kFull, valid && l != (int32_t)b); fm; fm &= fm - 1) {
      const int r = __ffs(fm) - 1;
      const int32_t lr = __shfl_sync(kFull, l, r);
      int64_t sb, nb, sl, nl;  // both requests are valid and hold at least kGroupHead tokens
      request_range(offsets, base + r, tok_base, n_tokens, sb, nb);
      request_range(offsets, lr, tok_base, n_tokens, sl, nl);
      int64_t c = lcp_warp<U>(tokens + sb, tokens + sl, min(nb, nl), lane);
      if (c < kGroupHead || c > INT32_MAX) c = -1;
      if (lane == r) my_c = (int32_t)c;
    }
    const bool is_f = my_c >= 0;
    const unsigned lm = __ballot_sync(kFull, valid && !is_f), fm = __ballot_sync(kFull, is_f);
    int32_t at = 0;
    if (lane == 0 && lm) at = atomicAdd(&counts[0], __popc(lm));
    if (lane == 1 && fm) at = atomicAdd(&counts[1], __popc(fm));
    const int32_t lbase = __shfl_sync(kFull, at, 0), fbase = __shfl_sync(kFull, at, 1);
    const unsigned below = (1u << lane) - 1;
    if (valid && !is_f) {
      lead[b] = (int32_t)b;
      lists[lbase + __popc(lm & below)] = (int32_t)b;
    }
    const unsigned same = __match_any_sync(kFull, is_f ? l : -1);
    if (is_f) {
      lead[b] = l;
      cpre[b] = my_c;
      const int32_t c_min = (int32_t)__reduce_min_sync(same, (unsigned)my_c);
      const int first = __ffs(same) - 1;
      int32_t rbase = 0;
      if (lane == first) {
        if (c_min < *(volatile int32_t*)&cmin[l]) atomicMin(&cmin[l], c_min);
        if (!place) rbase = atomicAdd(&fcnt[l], __popc(same));
        if (*(volatile int32_t*)&gid[l] == kNoRow && atomicCAS(&gid[l], kNoRow, -1) == kNoRow) {
          const int32_t row = atomicAdd(&counts[2], 1);  // the leader's first follower gives it a row
          if (row < gcap) atomicExch(&gid[l], row);
        }
      }
      if (place)
        lists[B + fbase + __popc(fm & below)] = (int32_t)b;
      else
        slot_of[b] = __shfl_sync(same, rbase, first) + __popc(same & below);  // rank in the group
    }
  }
}

// Gives every leader with followers a contiguous range of the follower list: fcnt[l] (its follower count)
// becomes the start of the range.  One warp per 32 consecutive requests: an inclusive scan of their counts
// and one counter update per warp (counts[4]).
__global__ void __launch_bounds__(kGroupThreads) group_ranges_kernel(int64_t B, int32_t* fcnt, int32_t* counts) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kGroupThreads / 32);
  for (int64_t base = (((int64_t)blockIdx.x * kGroupThreads + threadIdx.x) >> 5) * 32; base < B; base += warps * 32) {
    const int64_t b = base + lane;
    const int32_t c = b < B ? fcnt[b] : 0;  // zero for every request that leads no follower
    int32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    int32_t off = 0;
    if (lane == 31 && incl) off = atomicAdd(&counts[4], incl);
    off = __shfl_sync(kFull, off, 31);
    if (c) fcnt[b] = off + incl - c;
  }
}

// Places follower b at lists[B + start of its leader's range + its rank in the group].
__global__ void __launch_bounds__(kGroupThreads) group_place_kernel(int64_t B, const int32_t* __restrict__ lead,
                                                                    const int32_t* __restrict__ rank,
                                                                    const int32_t* __restrict__ fcnt, int32_t* lists) {
  const int64_t stride = (int64_t)gridDim.x * kGroupThreads;
  for (int64_t b = (int64_t)blockIdx.x * kGroupThreads + threadIdx.x; b < B; b += stride) {
    const int32_t l = lead[b];
    if (l != (int32_t)b) lists[B + fcnt[l] + rank[b]] = (int32_t)b;
  }
}

}  // namespace

// CTAs a SM of the resolve kernel (by its registers).  A warp gets as many requests as give every resident warp about
// the same (one counter update serves them all): 65,536 requests 65 us, 80 from a work cursor in smaller pieces.
constexpr int64_t kResolveCtas = 6;

// Below this many bytes of match matrix the followers are listed as they come: their leaders' rows, checkpoints and
// tables stay in L2 (126 MB) whatever the order, and two launches are spared (65,536 requests of 1,250 tokens on 16
// trees: the follower pass 24 -> 27 us, 12 us of launches less; 8,191 of 11,400 tokens on 32 trees: 62 -> 65 and 12
// less).  Above it a group's followers lie side by side: the follower pass of 200,003 requests on 64 trees takes 148
// us so and 168 as they come, of 262,144 on 256 trees 0.70 ms and 0.87.  (A single tree's row is 4 bytes and
// its requests have no choice of route: that path is left as it was.)
constexpr int64_t kPlaceBytes = (int64_t)8 << 20;

cudaError_t launch_group(const int32_t* tokens, int64_t n_tokens, int64_t tok_base, const int64_t* offsets, int64_t B,
                         int32_t P, const GroupScratch& g, bool beside, int num_sms, cudaStream_t st, int* launched) {
  *launched = 0;
  if (B <= 0) return cudaSuccess;
  constexpr int kWarps = kGroupThreads / 32;
  const int64_t warps = (int64_t)num_sms * kResolveCtas * kWarps;
  const int32_t per = (int32_t)std::min<int64_t>(32, long_requests(B, n_tokens) ? 1 : (B + warps - 1) / warps);
  const int32_t per_hash = B < 16 * warps ? 8 : 32;  // (eight requests are hashed at a time)
  const bool place = P > 1 && B * P * (int64_t)sizeof(int32_t) <= kPlaceBytes;
  cudaError_t e = cudaMemsetAsync(g.keys, 0, g.n_zero, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(g.vals, 0x7f, g.n_large, st);
  if (e != cudaSuccess) return e;
  auto grid_for = [&](int64_t items, int64_t per_cta, int64_t most = 8) {
    return (int)std::min<int64_t>((items + per_cta - 1) / per_cta, (int64_t)num_sms * most);
  };
  P2P_TIMED(K_GROUP_HASH, st,
            (group_hash_kernel<<<grid_for(B, (int64_t)kWarps * per_hash), kGroupThreads, 0, st>>>(
                tokens, n_tokens, tok_base, offsets, B, per_hash, g.keys, g.vals, g.bits, g.slot_of)));
  const auto resolve = long_requests(B, n_tokens) ? group_resolve_kernel<24>
                       : beside                   ? group_resolve_kernel<16>
                                                  : group_resolve_kernel<8>;
  P2P_TIMED(K_GROUP_RESOLVE, st,
            (resolve<<<grid_for(B, (int64_t)kWarps * per), kGroupThreads, 0, st>>>(
                tokens, n_tokens, tok_base, offsets, B, per, place, g.vals, g.slot_of, g.lead, g.cpre, g.lists,
                g.counts, g.gid, g.cmin, g.gcap, g.fcnt)));
  *launched = 2;
  if (!place) {  // each group's followers side by side in the follower list
    P2P_TIMED(K_GROUP_RANGES, st,
              (group_ranges_kernel<<<grid_for(B, kGroupThreads), kGroupThreads, 0, st>>>(B, g.fcnt, g.counts)));
    P2P_TIMED(K_GROUP_PLACE, st,
              (group_place_kernel<<<grid_for(B, kGroupThreads), kGroupThreads, 0, st>>>(B, g.lead, g.slot_of, g.fcnt,
                                                                                       g.lists)));
    *launched = 4;
  }
  return cudaGetLastError();
}

}  // namespace p2p
