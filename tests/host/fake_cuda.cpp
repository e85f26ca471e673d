// The router's host code without a GPU: the CUDA runtime calls it makes, over host memory, and launchers that do
// nothing or what a test asks for.  Device allocations can be made to fail; the launchers look at the tree states they
// are given and count the arrays that are not live allocations of their stated capacity.
#include <cstdlib>
#include <cstring>
#include <map>

#include "internal.h"

namespace {
std::map<char*, size_t> live;
cudaError_t last = cudaSuccess;
size_t fail_from = 0, fail_to = 0;  // allocations of fail_from .. fail_to bytes fail (0: none)
int fail_after = 0;                 // > 0: the allocation after that many more fails
int ask_node = 0, ask_child = 0, ask_label = 0;  // what the next bulk rounds find no room for
int64_t pool_end = 0;                // of the interned labels that the last upload's edges point at
int32_t pool_at = 0, pool_tok = 0;  // one of them, and its first token
int bad_arrays = 0, bulk_calls = 0, delta_calls = 0;

cudaError_t err(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
bool holds(const void* p, size_t bytes) {
  auto it = live.find((char*)p);
  return it != live.end() && it->second >= bytes;
}
void look(const p2p::TreeState* s, int32_t n) {
  for (int32_t i = 0; i < n; ++i)
    if (!holds(s[i].node, (size_t)s[i].cap_node * 16) || !holds(s[i].child, (size_t)s[i].cap_child * 16) ||
        !holds(s[i].label, (size_t)s[i].cap_label * 4) || (s[i].stamp && !holds(s[i].stamp, (size_t)s[i].cap_node * 4)))
      ++bad_arrays;
}
}  // namespace

extern "C" {
void fake_fail_sizes(int64_t from, int64_t to) { fail_from = (size_t)from, fail_to = (size_t)to; }
void fake_fail_after(int n) { fail_after = n; }
void fake_ask(int node, int child, int label) { ask_node = node, ask_child = child, ask_label = label; }
int fake_bad_arrays() { return bad_arrays; }
int fake_bulk_calls() { return bulk_calls; }
int fake_delta_calls() { return delta_calls; }

cudaError_t CUDARTAPI cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
  const bool turn = fail_after > 0 && --fail_after == 0;
  if (turn || (fail_from && n >= fail_from && n <= fail_to)) return err(cudaErrorMemoryAllocation);
  *p = std::calloc(1, n);
  live[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFreeAsync(void* p, cudaStream_t) {  // (kept mapped: a use after it is counted, not a crash)
  return live.erase((char*)p) ? cudaSuccess : err(cudaErrorInvalidValue);
}
cudaError_t CUDARTAPI cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t CUDARTAPI cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaMallocHost(void** p, size_t n) { return (*p = std::calloc(1, n)) ? cudaSuccess : err(cudaErrorMemoryAllocation); }
cudaError_t CUDARTAPI cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
const char* CUDARTAPI cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t CUDARTAPI cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t CUDARTAPI cudaSetDevice(int) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceGetStreamPriorityRange(int* a, int* b) { return *a = 0, *b = -1, cudaSuccess; }
cudaError_t CUDARTAPI cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return *p = (cudaMemPool_t)&live, cudaSuccess; }
cudaError_t CUDARTAPI cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return *s = nullptr, cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t CUDARTAPI cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t CUDARTAPI cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { return *t = 0, cudaSuccess; }
cudaError_t CUDARTAPI cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { return a->type = cudaMemoryTypeUnregistered, cudaSuccess; }
}

// The launchers end as the real ones do: with the runtime's last error.
namespace p2p {
cudaError_t launch_group(const int32_t*, int64_t, int64_t, const int64_t*, int64_t, int32_t, const GroupScratch&, bool, int,
                         cudaStream_t, int* l) { return *l = 0, cudaGetLastError(); }
cudaError_t launch_decide(const int32_t*, int64_t, int32_t, const int32_t*, int32_t, int32_t*, int32_t*, int, cudaStream_t) {
  return cudaGetLastError();
}
bool route_ungrouped(int64_t, int32_t, int64_t, int) { return true; }
cudaError_t launch_route(const TreeView*, int32_t, const int32_t*, int64_t, int64_t, const int64_t*, int64_t, const int32_t*,
                         int32_t, int32_t*, int32_t*, int32_t*, const GroupScratch*, int, cudaStream_t, int* l, bool, int32_t*) {
  return *l = 0, cudaGetLastError();
}
cudaError_t launch_delta(TreeState* s, uint8_t*, int32_t n, const int32_t*, const int64_t*, const int64_t*, const int32_t*,
                         const int32_t*, int32_t*, int64_t, const int32_t*, cudaStream_t, const GlobalMemo*, const int32_t*,
                         int32_t, int32_t) {
  ++delta_calls;
  look(s, n);
  return cudaGetLastError();
}
size_t bulk_scratch(int64_t, int32_t, void*, BulkArgs&) { return 4096; }
cudaError_t launch_bulk(const BulkArgs& A, int, cudaStream_t, int* l) {
  *l = 0;
  ++bulk_calls;
  look(A.states, A.n_trees);
  if (ask_node || ask_child || ask_label) {
    A.states->status = DELTA_NEED_SPACE | DELTA_NEED_BULK;
    A.states->need_node = ask_node;
    A.states->need_child = ask_child;
    A.states->need_label = ask_label;
    ask_node = ask_child = ask_label = 0;
  }
  return cudaGetLastError();
}
cudaError_t launch_compact(CompactJob*, int32_t, int32_t, int, cudaStream_t) { return cudaGetLastError(); }
cudaError_t launch_upload(const UploadEdge* e, int64_t n, int4*, const int32_t*, int32_t*, int, cudaStream_t) {
  pool_end = 0;
  for (int64_t i = 0; i < n; ++i)
    if (e[i].slot.z < 0 && (int64_t)~e[i].slot.z + e[i].slot.w > pool_end) {
      pool_end = (int64_t)~e[i].slot.z + e[i].slot.w;
      pool_at = ~e[i].slot.z;
      pool_tok = e[i].slot.x;
    }
  return cudaGetLastError();
}
cudaError_t launch_set_tree(TreeState* s, TreeView*, TreeState v, const int32_t* shared, cudaStream_t) {
  *s = v;
  if (pool_end && (!holds(shared, (size_t)pool_end * 4) || shared[pool_at] != pool_tok)) ++bad_arrays;
  pool_end = 0;
  return cudaGetLastError();
}
cudaError_t launch_refresh_views(const TreeState* s, TreeView*, int32_t n, const int32_t*, cudaStream_t) {
  look(s, n);
  return cudaGetLastError();
}
int64_t static_scratch_tokens() { return 0; }
cudaError_t static_scratch(int, int32_t**, int32_t**) { return cudaErrorNotSupported; }
cudaError_t launch_validate(int32_t* h, const p2p_delta* d, int32_t, int32_t, cudaStream_t) {
  std::memset(h, 0, kStaticHeaderInts * 4);
  h[0] = h[3] = 1;
  h[4] = (int32_t)d->seqs.n;
  return cudaGetLastError();
}
cudaError_t launch_init_ranges(TreeState* s, int32_t nt, const int64_t*, int64_t n, cudaStream_t) {
  for (int32_t i = 0; i < nt; ++i) {
    s[i].op_begin = 0, s[i].op_end = n, s[i].status = DELTA_OK, s[i].n_absent = 0;
    s[i].need_node = s[i].need_child = s[i].need_label = s[i].need_root = 0;
  }
  return cudaGetLastError();
}
cudaError_t launch_room(const TreeState*, int32_t nt, const uint8_t*, const int32_t*, const int64_t*, const int32_t*,
                        long long* room, cudaStream_t) { return std::memset(room, 0, (size_t)nt * 16), cudaGetLastError(); }
cudaError_t launch_update_count(const int32_t*, const int64_t*, int64_t, int64_t, int32_t, int32_t*, int32_t*, int, cudaStream_t) {
  return cudaGetLastError();
}
cudaError_t launch_update_scan(const int32_t*, int32_t, int64_t*, int32_t*, int64_t*, int64_t*, cudaStream_t) { return cudaGetLastError(); }
cudaError_t launch_update_scatter(const int32_t*, const int64_t*, int64_t, int64_t, int32_t, int32_t*, int32_t*, int64_t*,
                                  int64_t*, int32_t*, int, cudaStream_t) { return cudaGetLastError(); }
cudaError_t launch_lru_walk(const TreeState& s, const int32_t*, const int32_t*, int64_t, const int64_t*, int64_t, int32_t*,
                            int32_t*, int32_t*, int32_t*, int, cudaStream_t) { return look(&s, 1), cudaGetLastError(); }
cudaError_t launch_lru_stamp(const TreeState& s, TreeState*, const int32_t*, const int32_t*, const int32_t*, int32_t, uint32_t,
                             int, cudaStream_t) { return look(&s, 1), cudaGetLastError(); }
size_t lru_scratch(int64_t, void*, LruScratch&) { return 4096; }
cudaError_t launch_lru_evict(const TreeState&, TreeState*, const LruScratch&, int32_t, unsigned long long, cudaStream_t) {
  return cudaGetLastError();
}
cudaError_t launch_lru_ops(const int64_t*, int64_t, int64_t, int32_t*, int64_t*, int64_t*, int32_t*, int, cudaStream_t) {
  return cudaGetLastError();
}
cudaError_t launch_hit_rate(const int32_t*, int32_t, const int64_t*, int64_t, const int32_t*, float*, int, cudaStream_t) {
  return cudaGetLastError();
}
}  // namespace p2p
