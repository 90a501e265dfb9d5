// One refinement round of k-bisimulation on the GPU, level 0, and the
// once-per-graph relabelling of node ids.
//
// Round i (Algorithm 1, the k > 0 branch; Definition 3; Proposition 2):
//   (a) gather: for every edge e = (u, l, v) of the source-sorted edge table,
//       the element (l, pId_{i-1}(v))  -- Algorithm 1 fills pId_old(tId) by a
//       merge join of the edge and node tables; here it is a direct gather;
//   (b) per source node: drop duplicate elements (the duplicate-free F of
//       Algorithm 1, unsorted), written at the node's CSR offset;
//   (c) a 64-bit hash of (pId_{i-1}(u), the element set)  -- it only routes
//       nodes to candidate groups; it stands in for the signature store S
//       (Section 3, "Data structures for S");
//   (d) group nodes with equal hash in an open-addressing table that keeps the
//       smallest original node id per hash, compare every node's signature
//       with that node's exactly (a hash collision never merges two blocks),
//       repair collisions, and number blocks by their smallest original id;
//   (e) the caller stops when the block count is unchanged.
// Level 0 groups nodes by label the same way (Algorithm 1, k = 0 branch).
//
// Degree tiers of steps (a) to (c): out-degree <= 16 one thread per node with
// its elements in registers, 17..256 one warp and 257..4096 one CTA per node,
// both with a shared-memory hash set; larger "hubs" are partitioned by key bits
// into buckets, each deduplicated by one CTA.  A node's distinct elements are
// kept in any order and compared as sets.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <unordered_map>
#include <vector>

#include "kbisim_internal.cuh"
#include "per_device.h"

namespace kb {

namespace {
constexpr unsigned kFull = 0xFFFFFFFFu;
}  // namespace

// --------------------------------------------------------------------------
// Kernel timing (CUDA events on the handle's stream)
// --------------------------------------------------------------------------
struct KernelTimer {
  struct Rec {
    int cls;
    cudaEvent_t a, b;
  };
  std::vector<cudaEvent_t> pool;
  std::vector<Rec> done;
  cudaEvent_t get() {
    if (!pool.empty()) {
      cudaEvent_t e = pool.back();
      pool.pop_back();
      return e;
    }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
  }
};

Status timer_collect(Store& s) {
  if (!s.timer) return Status::Ok();
  for (auto& r : s.timer->done) {
    cudaEventSynchronize(r.b);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, r.a, r.b);
    s.total_ms[r.cls] += ms;
    s.timer->pool.push_back(r.a);
    s.timer->pool.push_back(r.b);
  }
  s.timer->done.clear();
  return cuda_check(cudaGetLastError(), "timer");
}

void timer_destroy(Store& s) {
  if (!s.timer) return;
  for (auto e : s.timer->pool) cudaEventDestroy(e);
  for (auto& r : s.timer->done) {
    cudaEventDestroy(r.a);
    cudaEventDestroy(r.b);
  }
  delete s.timer;
  s.timer = nullptr;
}

namespace {

// Records one CUDA event pair around the kernels launched in its scope.
// Events around a group of launches of one kernel class; `kernels` is the
// number of this library's kernels the group launches (clears by
// cudaMemsetAsync are not counted).
struct TimedScope {
  Store& s;
  int cls;
  KernelTimer::Rec rec;
  TimedScope(Store& st, int c, int kernels) : s(st), cls(c) {
    s.launches[c] += (uint64_t)kernels;
    if (!s.timing) return;
    if (!s.timer) s.timer = new KernelTimer();
    rec.cls = c;
    rec.a = s.timer->get();
    rec.b = s.timer->get();
    cudaEventRecord(rec.a, s.stream);
  }
  ~TimedScope() {
    if (!s.timing) return;
    cudaEventRecord(rec.b, s.stream);
    s.timer->done.push_back(rec);
  }
};

template <typename T>
T* ptr(Buf& b) { return static_cast<T*>(b.p); }

inline unsigned grid_for(uint64_t work, unsigned per_block) {
  uint64_t g = (work + per_block - 1) / per_block;
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(g, 0x7FFFFFFFull));
}

Status launch_check(const char* what) { return cuda_check(cudaGetLastError(), what); }

int sm_count(int device) {
  static PerDevice known;
  const int v = known.get(device, [&] {
    int sms = 0;
    return cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) == cudaSuccess ? sms : 0;
  });
  return v > 0 ? v : 148;
}

// resident_blocks of one kernel, asked of the runtime once per device (the
// answer depends on the compiled kernel and the device only).
template <typename F>
unsigned resident_grid(F kernel, int threads, size_t dyn_smem, int device, PerDevice& known) {
  const int per_sm = known.get(device, [&] {
    int v = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, threads, dyn_smem) == cudaSuccess ? v : 0;
  });
  return (unsigned)std::max(per_sm, 1) * (unsigned)sm_count(device);
}

// Launch overlap within a round (programmatic dependent launch).  Every
// round kernel lets the next one start as soon as its own blocks are all
// resident (overlap_next).  A kernel that reads what earlier ones of the round
// wrote waits for them first (overlap_wait); the signature kernels do not
// depend on one another, so they run side by side, each waiting only before it
// ends, so that the end of any kernel still means the end of all before it.
// At 1M edges a signature kernel has too few blocks to fill the device and its
// 5 to 10 us are latency; at 256M edges only the tails overlap.
//
// The kernels that wait first (launch_chained) overlap only on small graphs
// (chained): it hides launch latency (100K nodes, 1M edges: 0.38 against 0.49
// ms a refinement of four rounds), but blocks that already hold their place,
// and their shared memory, slow the kernel before.  Whether that costs more is
// decided by the nodes, whose grouping and numbering these kernels do: at 4
// edges a node 1.58 against 1.72 ms with 1.5M nodes but 2.75 against 2.65 with
// 3M and 12.0 against 7.2 with 8.3M; at 8 edges a node 0.91 against 0.96 with
// 1.5M, 1.48 against 1.41 with 2.5M, 2.87 against 2.49 with 4.1M; at 16 edges
// 0.94 against 0.96 with 1.5M, 1.27 against 1.20 with 2.1M.  With few nodes and
// many edges the two are equal from about 32M edges on (1M nodes: 1.11 against
// 1.12 ms).
constexpr uint64_t kChainNodes = 3ull << 19, kChainEdges = 32ull << 20;
inline bool chained(const Store& s) { return s.n <= kChainNodes && s.m <= kChainEdges; }
__device__ __forceinline__ void overlap_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void overlap_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
void launch_if_overlapped(bool on, Store& s, void (*kernel)(P...), unsigned blocks, int threads, size_t smem,
                          A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = smem;
  c.stream = s.stream;
  c.attrs = &at;
  c.numAttrs = on ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, P(args)...);
}

template <typename... P, typename... A>
void launch_chained(Store& s, void (*kernel)(P...), unsigned blocks, int threads, size_t smem, A&&... args) {
  launch_if_overlapped(chained(s), s, kernel, blocks, threads, smem, args...);
}

// --------------------------------------------------------------------------
// Small device helpers
// --------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cas(uint32_t* a, uint32_t c, uint32_t v) { return atomicCAS(a, c, v); }
__device__ __forceinline__ uint64_t cas(uint64_t* a, uint64_t c, uint64_t v) {
  return atomicCAS((unsigned long long*)a, (unsigned long long)c, (unsigned long long)v);
}

// L2 cache policies (sm_90+ createpolicy): streamed edge data and signature
// words are marked evict-first, the gathered identifier array evict-last, so
// the random gathers of pId_{i-1}[dst] keep hitting L2 while the edge table
// streams past.
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// Loads with an L2 policy, predicated (0 when p is false, no access), so
// loads of several items are issued back to back without a branch between them.
__device__ __forceinline__ uint32_t ld_hint_if(const uint32_t* a, uint64_t pol, bool p) {
  uint32_t v;
  asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\tmov.u32 %0, 0;\n\t"
      "@q ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;\n\t}"
      : "=r"(v) : "l"(a), "l"(pol), "r"((uint32_t)p));
  return v;
}
__device__ __forceinline__ uint32_t ld_hint_if(const uint8_t* a, uint64_t pol, bool p) {
  uint32_t v;
  asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\tmov.u32 %0, 0;\n\t"
      "@q ld.global.nc.L2::cache_hint.u8 %0, [%1], %2;\n\t}"
      : "=r"(v) : "l"(a), "l"(pol), "r"((uint32_t)p));
  return v;
}

// Lanes of a sub-warp team (NT < 32) or the whole warp.
template <int NT>
__device__ __forceinline__ unsigned team_mask() {
  if (NT >= 32) return kFull;
  const unsigned lane = threadIdx.x & 31;
  return ((1u << (NT & 31)) - 1u) << (lane & ~(unsigned)(NT - 1));
}

template <int NT>
__device__ __forceinline__ void team_sync() {
  if (NT <= 32) __syncwarp(team_mask<NT>()); else __syncthreads();
}

// --------------------------------------------------------------------------
// Team dedupe in shared memory (no sorting)
// --------------------------------------------------------------------------
// A team (one warp, or one CTA) inserts keys into an open-addressing set in
// shared memory.  The first inserter of a key owns it: it writes the key to
// the node's output at the next free position and adds its hash term.  The
// order of a node's distinct keys is therefore arbitrary: signatures are
// compared as sets (see k_group_verify / k_verify_long).
template <typename K>
struct TeamSet {
  K* set;          // [hcap]
  K* uniq;         // [ucap] distinct keys (hub buckets only)
  uint32_t* sh;    // [4]: distinct count, saw-the-empty-key flag, overflow flag, spare
  uint32_t* red;   // [NT/32] reduction scratch
};

template <typename K>
__host__ __device__ constexpr size_t team_set_bytes(int hcap, int ucap, int nt) {
  return ((size_t)hcap * sizeof(K) + (size_t)ucap * sizeof(K) + 16 + (size_t)(nt / 32) * 8 + 15) / 16 * 16;
}

template <typename K>
__device__ __forceinline__ TeamSet<K> carve_set(char* base, int hcap, int ucap) {
  TeamSet<K> t;
  t.set = reinterpret_cast<K*>(base);
  t.uniq = t.set + hcap;
  t.sh = reinterpret_cast<uint32_t*>(t.uniq + ucap);
  t.red = t.sh + 4;
  return t;
}

// Smallest power of two >= 2 n, clamped to [64, cap].
__device__ __forceinline__ int set_size_for(uint64_t n, int cap) {
  int h = 64;
  while (h < cap && (uint64_t)h < 2 * n) h <<= 1;
  return h;
}

template <int NT, typename K>
__device__ __forceinline__ void set_clear(const TeamSet<K>& ts, int hcap, int rank) {
  for (int i = rank; i < hcap; i += NT) ts.set[i] = KeyOps<K>::kEmpty;
  if (rank < 4) ts.sh[rank] = 0;
}

// Insert k; true if this call inserted it first.  Probing is bounded by the
// set size; a full set raises the overflow flag.
template <typename K>
__device__ __forceinline__ bool set_insert(const TeamSet<K>& ts, int hcap, K k) {
  if (k == KeyOps<K>::kEmpty) return atomicExch(&ts.sh[1], 1u) == 0u;
  volatile K* vset = ts.set;
  const uint32_t hmask = (uint32_t)(hcap - 1);
  uint32_t s = (uint32_t)k & hmask;
  for (int t = 0; t < hcap; ++t) {
    const K cur = vset[s];
    if (cur == k) return false;
    if (cur == KeyOps<K>::kEmpty) {
      const K old = cas(&ts.set[s], KeyOps<K>::kEmpty, k);
      if (old == KeyOps<K>::kEmpty) return true;
      if (old == k) return false;
    }
    s = (s + 1) & hmask;
  }
  ts.sh[2] = 1u;
  return false;
}

// Membership test in a set built by set_insert.
template <typename K>
__device__ __forceinline__ bool set_find(const TeamSet<K>& ts, int hcap, K k) {
  if (k == KeyOps<K>::kEmpty) return ts.sh[1] != 0u;
  const uint32_t hmask = (uint32_t)(hcap - 1);
  uint32_t s = (uint32_t)k & hmask;
  for (int t = 0; t < hcap; ++t) {
    const K cur = ts.set[s];
    if (cur == k) return true;
    if (cur == KeyOps<K>::kEmpty) return false;
    s = (s + 1) & hmask;
  }
  return false;
}

// Sum over the team (modulo 2^32); valid in every lane for NT <= 32, in rank
// 0 otherwise.
template <int NT>
__device__ __forceinline__ uint32_t team_sum(uint32_t t, uint32_t* red, int rank) {
  const unsigned m = team_mask<NT>();
  t = __reduce_add_sync(m, t);
  if (NT <= 32) return t;
  if ((rank & 31) == 0) red[rank >> 5] = t;
  __syncthreads();
  uint32_t tot = 0;
  if (rank == 0)
    for (int w = 0; w < NT / 32; ++w) tot += red[w];
  __syncthreads();
  return tot;
}

// --------------------------------------------------------------------------
// Signature kernels
// --------------------------------------------------------------------------
struct SigArgs {
  const uint64_t* off;
  const uint32_t* dst;
  const void* lab;
  const uint32_t* prev;
  void* sigkey;
  uint32_t* ucnt;
  uint64_t* hash;
  uint64_t seed;
  uint64_t mask;
  int pbits;          // bits of a child identifier in a 32-bit key
  uint32_t* err;
  const uint32_t* fmask;  // bitmap over internal ids of the nodes to sign (NULL = all)
  // nodes alone in their previous block (NULL = not known): they stay alone, so
  // nothing reads their keys or hash, only their number of distinct elements
  const uint8_t* alone;
  // With the edges that repeat an earlier (label, target) of their node marked
  // (dup) and the nodes alone in their block as a bitmap (alone_bits), an
  // unmarked edge to such a node is a distinct element by itself: nothing else
  // of its node can equal it, so a node that only counts needs neither its key
  // nor a place in a set for it.  NULL = not known.
  const uint32_t* dup;
  const uint32_t* alone_bits;
  bool dup_hubs;    // the hubs' edges are marked too
  uint32_t* mark;   // marking pass: output, a bit per edge (prev = identity, every node counts)
};

// The node is to be signed this pass (every node unless a frontier mask is set).
__device__ __forceinline__ bool in_mask(const SigArgs& a, uint64_t p) {
  return !a.fmask || ((a.fmask[p >> 5] >> (p & 31)) & 1u);
}


struct Policies {
  uint64_t stream, keep;
  __device__ __forceinline__ Policies() : stream(policy_evict_first()), keep(policy_evict_last()) {}
};

// Keys of N edges base + i * stride into key[O + i] (i < N; an edge counts
// while it is below end): labels and targets first, then the identifier
// gathers, then the packing, so all loads of the batch are in flight together.
template <int N, int O, int M, typename LabelT, typename K>
__device__ __forceinline__ void edge_keys(const SigArgs& a, uint64_t base, uint32_t stride, uint64_t end,
                                          const Policies& pol, K (&key)[M]) {
  static_assert(O + N <= M, "batch out of range");
  const LabelT* lab = static_cast<const LabelT*>(a.lab);
  uint32_t l[N], t[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint64_t e = base + (uint64_t)i * stride;
    l[i] = ld_hint_if(lab + e, pol.stream, e < end);
    t[i] = ld_hint_if(a.dst + e, pol.stream, e < end);
  }
#pragma unroll
  for (int i = 0; i < N; ++i) t[i] = ld_hint_if(a.prev + t[i], pol.keep, base + (uint64_t)i * stride < end);
#pragma unroll
  for (int i = 0; i < N; ++i) key[O + i] = KeyOps<K>::make(l[i], t[i], a.pbits);
}

// Variants of the kernels for out-degree 17..4096: without marks, with a.dup
// set, and the marking pass itself (each carries only its own code).
enum { kPlain = 0, kWithDup = 1, kMarking = 2 };

__device__ __forceinline__ void mark_dup(const SigArgs& a, uint64_t e) { atomicOr(&a.mark[e >> 5], 1u << (e & 31)); }

// For a node that only counts: of N edges base + i * stride below end, the
// number of unmarked ones to nodes alone in their block, and the keys of the
// other unmarked ones (bits of the returned mask), for a set.  In late rounds
// that is hardly any, and an edge costs its target, two bits and no label.
template <int N, typename LabelT, typename K>
__device__ __forceinline__ uint32_t edge_rest(const SigArgs& a, uint64_t base, uint32_t stride, uint64_t end,
                                              const Policies& pol, K (&key)[N], uint32_t& count) {
  uint32_t t[N], d[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint64_t e = base + (uint64_t)i * stride;
    t[i] = ld_hint_if(a.dst + e, pol.stream, e < end);
    d[i] = ld_hint_if(a.dup + (e >> 5), pol.stream, e < end);
  }
  uint32_t ok = 0, rest = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint64_t e = base + (uint64_t)i * stride;
    if (e < end && !((d[i] >> (e & 31)) & 1u)) ok |= 1u << i;
    d[i] = ld_hint_if(a.alone_bits + (t[i] >> 5), pol.keep, (ok >> i) & 1u);
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (((ok >> i) & 1u) && !((d[i] >> (t[i] & 31)) & 1u)) rest |= 1u << i;
  count += __popc(ok & ~rest);
  if (__any_sync(kFull, rest)) {
    const LabelT* lab = static_cast<const LabelT*>(a.lab);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const bool r = (rest >> i) & 1u;
      d[i] = ld_hint_if(lab + base + (uint64_t)i * stride, pol.stream, r);
      t[i] = ld_hint_if(a.prev + t[i], pol.keep, r);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) key[i] = KeyOps<K>::make(d[i], t[i], a.pbits);
  }
  return rest;
}

// Out-degree <= 16: a thread per node for the 32 nodes of a warp (consecutive
// internal ids, so their edges are one contiguous range of at most 32 * S
// edges), with the edges staged through the warp's shared-memory buffer: the
// warp loads the range coalesced (lane l takes edges l, l + 32, ...) and makes
// the keys, each thread reads its node's keys back into registers (S = 2^c
// slots, S >= out-degree) and keeps a key unless an earlier slot holds it, so
// no sorting or set is needed; it writes the distinct ones over its own keys,
// and the warp stores the whole range coalesced (slots past a node's distinct
// count keep leftovers that nothing reads).  A node alone in its block only
// counts.  Lanes past the class end take part without a node.
// Bound by the L1's data pipe (81% at out-degree <= 8 where every node writes
// its keys: about 0.75 of 1.4 wavefronts per edge are the identifier gather; 67%
// and 1.05 wavefronts in round 2 of the 64M-edge powerlaw graph, where most
// nodes only count).
template <int S, typename LabelT, typename K>
__device__ __forceinline__ void sig_warp_staged(const SigArgs& a, uint64_t p_first, uint32_t nvalid, K* wsm,
                                                const Policies& pol) {
  const uint32_t lane = threadIdx.x & 31;
  const bool valid = lane < nvalid;
  const uint64_t p = p_first + lane;
  if (a.fmask && !__any_sync(0xFFFFFFFFu, valid && in_mask(a, p))) return;
  const uint64_t base = a.off[p_first];
  const uint64_t end = a.off[p_first + nvalid];
  const uint32_t T = (uint32_t)(end - base);  // at most 32 * S
  {
    K kk[S];
    edge_keys<S, 0, S, LabelT, K>(a, base + lane, 32u, end, pol, kk);
#pragma unroll
    for (int t = 0; t < S; ++t)
      if (lane + 32u * t < T) wsm[lane + 32u * t] = kk[t];
  }
  __syncwarp();
  uint32_t r0 = 0, d = 0;
  const bool full = valid && !(a.alone && a.alone[p]);  // its keys and hash are needed
  if (valid) {
    const uint64_t o = a.off[p];
    r0 = (uint32_t)(o - base);
    d = (uint32_t)(a.off[p + 1] - o);
  }
  K k[S];
#pragma unroll
  for (int i = 0; i < S; ++i) k[i] = i < (int)d ? wsm[r0 + i] : (K)0;
  __syncwarp();  // every read is done before the distinct keys go back
  uint64_t term = 0;
  uint32_t U = 0;
#pragma unroll
  for (int i = 0; i < S; ++i) {
    bool keep = i < (int)d;
#pragma unroll
    for (int j = 0; j < i; ++j) keep = keep && k[j] != k[i];
    if (keep) {
      if (full) {
        wsm[r0 + U] = k[i];
        term = term_add(term, elem_term(k[i], a.seed));
      }
      ++U;
    }
  }
  if (__any_sync(kFull, full)) {
    __syncwarp();
    K* out = static_cast<K*>(a.sigkey) + base;
#pragma unroll
    for (int t = 0; t < S; ++t)
      if (lane + 32u * t < T) out[lane + 32u * t] = wsm[lane + 32u * t];
  }
  if (valid) a.ucnt[p] = U;
  if (full) a.hash[p] = node_hash(term, a.prev[p], U, a.seed, a.mask);
}

// Resident CTAs per multiprocessor the small-class kernels are compiled for:
// all 8 (32 registers) for out-degree <= 8 with 32-bit keys, fewer where more
// keys sit in registers.
template <int LAST, typename K>
__host__ __device__ constexpr int small_min_blocks() {
  return LAST <= 4 ? (sizeof(K) == 4 ? 8 : 6) : 4;
}

struct SmallLaunch {
  uint64_t start[kSmallClasses];
  uint64_t count[kSmallClasses];
  uint32_t bstart[kSmallClasses + 1];
};

constexpr int kSmallThreads = 256;

// Class 0 (no out-edges): signature (pId_{i-1}(u), {}); classes 1..5
// (out-degree 1..16): one node per thread.  Classes FIRST..LAST per launch, so
// that each kernel carries only its own unrolled code.
template <int FIRST, int LAST, typename LabelT, typename K>
__device__ __forceinline__ void sig_small_block(const SigArgs& a, const SmallLaunch& L) {
  constexpr int kSLast = LAST == 0 ? 1 : (1 << (LAST - 1));
  __shared__ K stage[kSmallThreads / 32][32 * kSLast];  // per warp, for the largest class of this launch
  int c = FIRST;
  while (c < LAST && blockIdx.x >= L.bstart[c + 1]) ++c;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t idx = (uint64_t)(blockIdx.x - L.bstart[c]) * kSmallThreads + threadIdx.x;
  const uint64_t widx = idx - lane;
  if (widx >= L.count[c]) return;  // the whole warp is past the class end
  const uint64_t left = L.count[c] - widx;
  const uint32_t nvalid = left < 32 ? (uint32_t)left : 32u;
  const uint64_t p = L.start[c] + idx;
  const Policies pol;
  K* wsm = stage[threadIdx.x >> 5];
#define KB_SMALL_CLASS(C, S)                                                                                  \
  case C:                                                                                                     \
    if constexpr (LAST >= C) sig_warp_staged<S, LabelT, K>(a, L.start[c] + widx, nvalid, wsm, pol);            \
    break;
  switch (c) {
    case 0:
      if (idx < L.count[c] && in_mask(a, p)) {
        a.ucnt[p] = 0;
        a.hash[p] = node_hash(0, a.prev[p], 0, a.seed, a.mask);
      }
      break;
    KB_SMALL_CLASS(1, 1)
    KB_SMALL_CLASS(2, 2)
    KB_SMALL_CLASS(3, 4)
    KB_SMALL_CLASS(4, 8)
    KB_SMALL_CLASS(5, 16)
  }
#undef KB_SMALL_CLASS
}

template <int FIRST, int LAST, typename LabelT, typename K>
__global__ void __launch_bounds__(kSmallThreads, small_min_blocks<LAST, K>()) k_sig_small(SigArgs a, SmallLaunch L) {
  overlap_next();
  sig_small_block<FIRST, LAST, LabelT, K>(a, L);
  overlap_wait();
}

// ---- chunk-level sets of the hubs ------------------------------------------
// A region of a shared-memory hash set takes a chunk's keys: the lane whose
// insert puts a key into the set lists it.  The key equal to the empty-slot
// marker is kept as a flag.

template <typename K>
struct ChunkSmem {
  K slot[2 * kHubChunk];
  uint32_t cnt;    // distinct keys listed
  uint32_t empty;  // the key equal to KeyOps<K>::kEmpty was seen
  uint32_t pad[2];
};

__device__ __forceinline__ uint32_t key_h32(uint32_t k) { return k; }
__device__ __forceinline__ uint32_t key_h32(uint64_t k) { return (uint32_t)(k >> 32) ^ (uint32_t)k; }

// Home slot of k in a region of rs slots: monotone in the key's top bits.
template <typename K>
__device__ __forceinline__ uint32_t region_home(K k, uint32_t rs) {
  return (uint32_t)(((uint64_t)key_h32(k) * rs) >> 32);
}

// Shared-memory compare-and-swap by shared-window address (no generic addressing).
__device__ __forceinline__ uint32_t atoms_cas(uint32_t a, uint32_t c, uint32_t v) {
  uint32_t r;
  asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(r) : "r"(a), "r"(c), "r"(v) : "memory");
  return r;
}
__device__ __forceinline__ uint64_t atoms_cas(uint32_t a, uint64_t c, uint64_t v) {
  uint64_t r;
  asm volatile("atom.shared.cas.b64 %0, [%1], %2, %3;" : "=l"(r) : "r"(a), "l"(c), "l"(v) : "memory");
  return r;
}

// Insert k (!= kEmpty) into the set held in slots [rb, rb + rs) of the slot
// array at shared-window address `base`; true iff this call put it there.
// The region has more slots than keys are ever inserted into it, and probing
// is bounded by its size; the compare-and-swap is the probe itself.
template <typename K>
__device__ __forceinline__ bool region_insert(uint32_t base, uint32_t rb, uint32_t rs, K k) {
  uint32_t s = rb + region_home(k, rs);
  const uint32_t re = rb + rs;
  for (uint32_t t = 0; t < rs; ++t) {
    const K cur = atoms_cas(base + s * (uint32_t)sizeof(K), KeyOps<K>::kEmpty, k);
    if (cur == KeyOps<K>::kEmpty) return true;
    if (cur == k) return false;
    if (++s == re) s = rb;
  }
  return false;
}

// All ones into the first `slots` words of a 16-byte aligned array (slots a
// multiple of 16 / sizeof(K)), by NT threads.
template <int NT, typename K>
__device__ __forceinline__ void fill_empty(K* slot, uint32_t slots, uint32_t rank) {
  uint4* s4 = reinterpret_cast<uint4*>(slot);
  const uint4 ones = make_uint4(~0u, ~0u, ~0u, ~0u);
  for (uint32_t i = rank; i < slots * (uint32_t)sizeof(K) / 16; i += NT) s4[i] = ones;
}

template <int NT, typename LabelT, typename K>
__device__ __forceinline__ void chunk_keys(const SigArgs& a, uint64_t ebase, uint32_t E, K (&key)[kChunkItems]) {
  const Policies pol;
  edge_keys<kChunkItems, 0, kChunkItems, LabelT, K>(a, ebase + threadIdx.x, NT, ebase + E, pol, key);
}

// Lanes below `lane`.
__device__ __forceinline__ unsigned lanes_below(uint32_t lane) { return (1u << lane) - 1u; }


// Insert k (!= kEmpty) into a power-of-two set of hmask + 1 slots at
// shared-window address `base`, home slot from the key's low bits (the keys of
// one hub bucket share their top bits).  The compare-and-swap is the probe
// itself: one shared access per probed slot, whether the slot is empty, holds
// k or holds another key.  Returns 1 if this call inserted k, 0 if k was
// present, -1 if the set is full.
template <typename K>
__device__ __forceinline__ int pow2_insert(uint32_t base, uint32_t hmask, K k) {
  uint32_t s = key_h32(k) & hmask;
  for (uint32_t t = 0; t <= hmask; ++t) {
    const K cur = atoms_cas(base + s * (uint32_t)sizeof(K), KeyOps<K>::kEmpty, k);
    if (cur == KeyOps<K>::kEmpty) return 1;
    if (cur == k) return 0;
    s = (s + 1) & hmask;
  }
  return -1;
}

// ---- out-degree 17..256: a warp per node ----------------------------------
// A warp takes `per` consecutive nodes (at most 32; lane j holds the bounds and
// results of node j) and signs them one after the other: the node's edges come
// coalesced, STEPS per lane, their gathers all in flight; every key is inserted
// into the warp's own power-of-two set in shared memory, and the lane whose
// insert was the first writes the key out behind those found before.  Count and
// term sums stay in registers, and the hashes of the warp's nodes are made
// together at the end, a lane per node.
// Bound by instruction issue (57% at out-degree 17..64) and the L1 (47 to 61%).
// Chunks of whole nodes in a CTA-wide set, where a step of 32 edges could meet
// two nodes, spent most of their 239 warp instructions a step on finding the
// node, on two-node sums and on shared atomics; a step that belongs to one node
// takes 130 (out-degree 65..256) to 187 (17..32), with marks 85 to 155.
// Out-degree 17..32 ran one thread per node with 32 keys in registers, whose
// uncoalesced loads kept the L1 at 77%: 155 -> 145 us a round for 18M edges, and
// 625 -> 582 us for a refinement of 1M edges.
constexpr int kNodeWarps = 8;  // per CTA

// Distinct elements of a node that only counts, with its duplicates marked: the
// set (of SLOTS slots) is needed for targets not alone in their block only.
template <uint32_t SLOTS, int PART, typename LabelT, typename K>
__device__ __forceinline__ uint32_t count_one_node(const SigArgs& a, uint64_t e0, uint32_t d, uint32_t sbase, K* set,
                                                   const Policies& pol) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t c = 0;
  bool empty = false, cleared = false;
#pragma unroll 1
  for (uint32_t i0 = 0; i0 < d; i0 += 32 * PART) {
    K key[PART];
    const uint32_t rest = edge_rest<PART, LabelT, K>(a, e0 + i0 + lane, 32u, e0 + d, pol, key, c);
    if (!__any_sync(kFull, rest)) continue;
    if (!cleared) fill_empty<32>(set, SLOTS, lane);
    cleared = true;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < PART; ++t) {
      if (!((rest >> t) & 1u)) continue;
      if (key[t] != KeyOps<K>::kEmpty) c += pow2_insert(sbase, SLOTS - 1, key[t]) > 0 ? 1u : 0u;
      else empty = true;
    }
  }
  return __reduce_add_sync(kFull, c) + (__any_sync(kFull, empty) ? 1u : 0u);
}

template <int STEPS, int MODE, typename LabelT, typename K>
__device__ __forceinline__ void sig_one_node(const SigArgs& a, uint64_t e0, uint32_t d, bool alone, uint32_t sbase,
                                             K* set, const Policies& pol, uint32_t& U, uint32_t& lo, uint32_t& hi) {
  const uint32_t lane = threadIdx.x & 31;
  K key[STEPS];
  edge_keys<STEPS, 0, STEPS, LabelT, K>(a, e0 + lane, 32u, e0 + d, pol, key);
  fill_empty<32>(set, 64u * STEPS, lane);
  __syncwarp();
  K* out = static_cast<K*>(a.sigkey) + e0;
  uint32_t u = 0, l = 0, h = 0;
  bool seen_empty = false;
  if (MODE != kWithDup && alone) {  // only the number of distinct keys is needed (with duplicates marked: count_one_node)
#pragma unroll
    for (int t = 0; t < STEPS; ++t) {
      const K k = key[t];
      const bool valid = lane + 32u * t < d, empty = valid && k == KeyOps<K>::kEmpty;
      bool fresh = false;
      if (valid && !empty) fresh = pow2_insert(sbase, 64u * STEPS - 1, k) > 0;
      const unsigned em = __ballot_sync(kFull, empty);
      if (em) {
        fresh |= !seen_empty && lane == (uint32_t)__ffs(em) - 1u;
        seen_empty = true;
      }
      u += fresh ? 1u : 0u;
      if (MODE == kMarking && valid && !fresh) mark_dup(a, e0 + lane + 32u * t);
    }
    U = __reduce_add_sync(kFull, u);
    return;
  }
#pragma unroll
  for (int t = 0; t < STEPS; ++t) {
    if (STEPS > 2 && 32u * t >= d) break;
    const K k = key[t];
    bool fresh = false;
    const bool valid = lane + 32u * t < d;
    if (valid && k != KeyOps<K>::kEmpty) fresh = pow2_insert(sbase, 64u * STEPS - 1, k) > 0;
    const unsigned em = __ballot_sync(kFull, valid && k == KeyOps<K>::kEmpty);
    if (em) {  // the key that marks empty slots: kept beside the set
      fresh |= !seen_empty && lane == (uint32_t)__ffs(em) - 1u;
      seen_empty = true;
    }
    const unsigned fm = __ballot_sync(kFull, fresh);
    if (fresh) {
      out[u + __popc(fm & lanes_below(lane))] = k;
      const uint64_t tm = elem_term(k, a.seed);
      l += (uint32_t)tm;
      h += (uint32_t)(tm >> 32);
    }
    u += __popc(fm);
  }
  U = u;
  lo = __reduce_add_sync(kFull, l);
  hi = __reduce_add_sync(kFull, h);
}

template <int MAXSTEPS, int MODE, typename LabelT, typename K>
__device__ __forceinline__ void sig_warp_block(const SigArgs& a, uint64_t first, uint64_t count, uint32_t per) {
  __shared__ __align__(16) K sets[kNodeWarps][64 * MAXSTEPS];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t i0 = ((uint64_t)blockIdx.x * kNodeWarps + w) * per;
  if (i0 >= count) return;
  const uint32_t nn = (uint32_t)min((uint64_t)per, count - i0);
  const uint64_t p0 = first + i0, p = p0 + min(lane, nn - 1);
  const uint64_t b = a.off[p];
  const uint32_t d_l = (uint32_t)(a.off[p + 1] - b);
  const uint64_t base = __shfl_sync(kFull, b, 0);
  const uint32_t r_l = (uint32_t)(b - base);
  const bool mine = lane < nn && in_mask(a, p);
  const bool alone_l = a.alone && a.alone[p];
  unsigned todo = __ballot_sync(kFull, mine);
  const unsigned alone_m = __ballot_sync(kFull, alone_l);
  uint32_t U_l = 0, lo_l = 0, hi_l = 0;
  const Policies pol;
  K* set = sets[w];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(set);
  while (todo) {
    __syncwarp();  // the set is cleared for this node after every insert of the one before (votes order no memory)
    const uint32_t j = (uint32_t)__ffs(todo) - 1u;
    todo &= todo - 1;
    const uint64_t e0 = base + __shfl_sync(kFull, r_l, j);
    const uint32_t d = __shfl_sync(kFull, d_l, j);
    const bool alone = (alone_m >> j) & 1u;
    uint32_t U = 0, lo = 0, hi = 0;
    if (MODE == kWithDup && alone) {
      U = count_one_node<64u * MAXSTEPS, (MAXSTEPS < 4 ? MAXSTEPS : 4), LabelT, K>(a, e0, d, sbase, set, pol);
    } else if constexpr (MAXSTEPS == 8) {
      if (d <= 128) sig_one_node<4, MODE, LabelT, K>(a, e0, d, alone, sbase, set, pol, U, lo, hi);
      else sig_one_node<8, MODE, LabelT, K>(a, e0, d, alone, sbase, set, pol, U, lo, hi);
    } else {
      sig_one_node<MAXSTEPS, MODE, LabelT, K>(a, e0, d, alone, sbase, set, pol, U, lo, hi);
    }
    if (lane == j) {
      U_l = U;
      lo_l = lo;
      hi_l = hi;
    }
  }
  if (mine) {
    a.ucnt[p] = U_l;
    if (!alone_l) a.hash[p] = node_hash(((uint64_t)hi_l << 32) | lo_l, a.prev[p], U_l, a.seed, a.mask);
  }
}

template <int MAXSTEPS, int MODE, typename LabelT, typename K>
__global__ void __launch_bounds__(kNodeWarps * 32, sizeof(K) == 4 ? 6 : 4) k_sig_warp(SigArgs a, uint64_t first, uint64_t count,
                                                                uint32_t per) {
  overlap_next();
  sig_warp_block<MAXSTEPS, MODE, LabelT, K>(a, first, count, per);
  overlap_wait();
}

// ---- out-degree 257..4096: a CTA per node ----------------------------------
// As above with one set for the CTA; a warp inserts all its steps, then takes
// the places of its fresh keys with one reservation on the node's count.
constexpr int kCtaNodeItems = 8;  // edges per thread

template <typename K>
struct CtaNodeSmem {
  uint32_t cnt, lo, hi, empty;
  __device__ __forceinline__ K* set() { return reinterpret_cast<K*>(this + 1); }
};

template <int NT, typename K>
__host__ __device__ constexpr size_t cta_node_smem() { return sizeof(CtaNodeSmem<K>) + 2 * (size_t)NT * kCtaNodeItems * sizeof(K); }

template <int NT, int ITEMS, int MODE, typename LabelT, typename K>
__device__ __forceinline__ void sig_cta_node(const SigArgs& a, uint64_t p, uint64_t e0, uint32_t d, CtaNodeSmem<K>& sm) {
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const bool alone = a.alone && a.alone[p];
  const Policies pol;
  K key[ITEMS];
  constexpr uint32_t kSlots = 2 * NT * ITEMS;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm.set());
  if (tid < 4) (&sm.cnt)[tid] = 0;
  if (MODE == kWithDup && alone) {
    uint32_t c = 0;
    const uint32_t rest = edge_rest<ITEMS, LabelT, K>(a, e0 + tid, NT, e0 + d, pol, key, c);
    if (__syncthreads_or(rest != 0)) {
      fill_empty<NT>(sm.set(), kSlots, tid);
      __syncthreads();
#pragma unroll
      for (int t = 0; t < ITEMS; ++t) {
        if (!((rest >> t) & 1u)) continue;
        c += key[t] == KeyOps<K>::kEmpty ? (atomicExch(&sm.empty, 1u) == 0u ? 1u : 0u)
                                         : (pow2_insert(sbase, kSlots - 1, key[t]) > 0 ? 1u : 0u);
      }
    }
    c = __reduce_add_sync(kFull, c);
    if (lane == 0 && c) atomicAdd(&sm.cnt, c);
    __syncthreads();
    if (tid == 0) a.ucnt[p] = sm.cnt;
    return;
  }
  edge_keys<ITEMS, 0, ITEMS, LabelT, K>(a, e0 + tid, NT, e0 + d, pol, key);
  fill_empty<NT>(sm.set(), kSlots, tid);
  __syncthreads();
  if (MODE != kWithDup && alone) {  // only the number of distinct keys is needed
    uint32_t c = 0;
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {
      if (tid + (uint32_t)t * NT >= d) continue;
      const K k = key[t];
      const bool fresh = k == KeyOps<K>::kEmpty ? atomicExch(&sm.empty, 1u) == 0u : pow2_insert(sbase, kSlots - 1, k) > 0;
      c += fresh ? 1u : 0u;
      if (MODE == kMarking && !fresh) mark_dup(a, e0 + tid + (uint32_t)t * NT);
    }
    c = __reduce_add_sync(kFull, c);
    if (lane == 0) atomicAdd(&sm.cnt, c);
    __syncthreads();
    if (tid == 0) a.ucnt[p] = sm.cnt;
    return;
  }
  unsigned fms[ITEMS];
  uint32_t lo = 0, hi = 0, total = 0;
#pragma unroll
  for (int t = 0; t < ITEMS; ++t) {
    fms[t] = 0u;
    if ((uint32_t)t * NT >= d) continue;  // the same for the whole CTA
    const K k = key[t];
    bool fresh = false;
    if (tid + (uint32_t)t * NT < d)
      fresh = k == KeyOps<K>::kEmpty ? atomicExch(&sm.empty, 1u) == 0u : pow2_insert(sbase, kSlots - 1, k) > 0;
    fms[t] = __ballot_sync(kFull, fresh);
    total += __popc(fms[t]);
    if (fresh) {
      const uint64_t tm = elem_term(k, a.seed);
      lo += (uint32_t)tm;
      hi += (uint32_t)(tm >> 32);
    }
  }
  if (total) {
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&sm.cnt, total);
    at = __shfl_sync(kFull, at, 0);
    K* out = static_cast<K*>(a.sigkey) + e0;
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {
      if ((fms[t] >> lane) & 1u) out[at + __popc(fms[t] & lanes_below(lane))] = key[t];
      at += __popc(fms[t]);
    }
    lo = __reduce_add_sync(kFull, lo);
    hi = __reduce_add_sync(kFull, hi);
    if (lane == 0) {
      atomicAdd(&sm.lo, lo);
      atomicAdd(&sm.hi, hi);
    }
  }
  __syncthreads();
  if (tid == 0) {
    a.ucnt[p] = sm.cnt;
    a.hash[p] = node_hash(((uint64_t)sm.hi << 32) | sm.lo, a.prev[p], sm.cnt, a.seed, a.mask);
  }
}

template <int NT, int MODE, typename LabelT, typename K>
__device__ __forceinline__ void sig_cta_block(const SigArgs& a, uint64_t first) {
  extern __shared__ __align__(16) char smem_raw[];
  CtaNodeSmem<K>& sm = *reinterpret_cast<CtaNodeSmem<K>*>(smem_raw);
  const uint64_t p = first + blockIdx.x;
  if (!in_mask(a, p)) return;
  const uint64_t e0 = a.off[p];
  const uint32_t d = (uint32_t)(a.off[p + 1] - e0);
  if (d <= NT * kCtaNodeItems / 2) sig_cta_node<NT, kCtaNodeItems / 2, MODE, LabelT, K>(a, p, e0, d, sm);
  else sig_cta_node<NT, kCtaNodeItems, MODE, LabelT, K>(a, p, e0, d, sm);
}

template <int NT, int MODE, typename LabelT, typename K>
__global__ void __launch_bounds__(NT, sizeof(K) == 4 ? 2048 / NT : 1536 / NT) k_sig_cta(SigArgs a, uint64_t first) {
  overlap_next();
  sig_cta_block<NT, MODE, LabelT, K>(a, first);
  overlap_wait();
}

// ---- hubs: out-degree > kBlockMax ----------------------------------------
// Pass 1 (k_hub_chunk): a CTA takes kHubChunk edges of one hub, deduplicates
// their keys in shared memory as above (one region), listing each distinct
// key once, and appends the list to the hub's buckets; the bucket of a key is
// its top bits, so equal keys from different chunks meet in one bucket.
// Hubs whose keys rarely repeat (k_hub_sample) skip the chunk set
// (k_hub_scatter).  Buckets have a fixed capacity: an append past it flags the
// hub (kErrHubOverflow) and the host repeats the hub passes with larger
// buckets for that hub, or, for a scattering hub whose buckets have grown
// twice already, with the deduplicating pass (a key repeated that often stays
// repeated in later rounds); a bucket with more distinct keys than its set
// (kErrHubSet) gives its hub more buckets.  Pass 2 (k_hub_bucket):
// one CTA per bucket deduplicates across chunks and appends the bucket's
// distinct keys at the hub's CSR offset, adding to the hub's count and term
// sums; the CTA of a hub's last bucket, or k_hub_finish, writes its count and
// hash.
struct HubArgs {
  uint64_t first;           // internal id of hub 0
  const uint32_t* hub_bits;
  const uint64_t* hub_bbase;
  const uint32_t* hub_cap;
  const uint64_t* hub_tbase;
  const uint32_t* bucket_hub;
  const uint4* chunks;
  uint32_t* cursor;              // per bucket: key words appended
  unsigned long long* hub_cur;   // per hub: distinct keys written
  uint32_t* hub_term;            // per hub: term sum halves (low, high)
  uint32_t* done;                // per hub: buckets deduplicated (NULL: k_hub_finish follows)
  void* tmp;
  uint8_t* mode;                 // per hub: 1 = chunks skip their set (few repeated keys)
  const uint8_t* force;          // per hub: 1 = always the deduplicating chunk pass
  uint32_t* hub_err;             // per hub: kErrHubOverflow / kErrHubSet raised for it
};

__device__ __forceinline__ void hub_fail(const SigArgs& a, const HubArgs& h, uint32_t hub, uint32_t e) {
  atomicOr(&h.hub_err[hub], e);
  atomicOr(a.err, e);
}

// Key words a hub bucket holds at most: the sizes options.hub_bucket_keys
// accepts; the first is the size before tuning, and the tuning compares the
// first two (8192 measured slower on every workload here once bucket growth
// had settled, while its first pass, with fewer overflows, times faster).
constexpr int kHubUcaps[3] = {4096, 2048, 8192};
constexpr int kHubSmemBuckets = 1024;  // per-chunk bucket counts in shared memory up to this many buckets
constexpr int kHubSample = 128;        // keys sampled per hub to choose its chunk pass
constexpr int kHubSamplePairs = 16;    // equal sampled pairs from which a hub keeps the chunk set
constexpr uint32_t kHubScatterShiftMax = 2;  // bucket growth of a scattering hub before it takes the set

template <typename K>
__host__ __device__ constexpr size_t hub_chunk_smem() {
  return sizeof(ChunkSmem<K>) + (size_t)kHubChunk * sizeof(K) + 2 * kHubSmemBuckets * sizeof(uint32_t);
}


template <typename K>
__device__ __forceinline__ uint32_t hub_bucket(K k, uint32_t bits) {
  return bits ? (uint32_t)(k >> (KeyOps<K>::kBits - bits)) : 0u;
}

// Keys of a hub piece's edges that go to the hub's buckets (bits of the
// returned mask); a hub that only counts adds its edges to nodes alone in their
// block straight to its count.
template <int MODE, typename LabelT, typename K>
__device__ __forceinline__ uint32_t hub_piece_keys(const SigArgs& a, const HubArgs& h, uint32_t hub, uint64_t ebase,
                                                   uint32_t E, K (&key)[kChunkItems]) {
  const uint32_t tid = threadIdx.x;
  if (MODE == kWithDup && a.alone[h.first + hub]) {
    const Policies pol;
    uint32_t c = 0;
    const uint32_t rest = edge_rest<kChunkItems, LabelT, K>(a, ebase + tid, kChunkThreads, ebase + E, pol, key, c);
    c = __reduce_add_sync(kFull, c);
    if ((tid & 31) == 0 && c) atomicAdd(&h.hub_cur[hub], (unsigned long long)c);
    return rest;
  }
  chunk_keys<kChunkThreads, LabelT, K>(a, ebase, E, key);
  uint32_t m = 0;
#pragma unroll
  for (int t = 0; t < kChunkItems; ++t) m |= tid + t * kChunkThreads < E ? 1u << t : 0u;
  return m;
}

template <int MODE, typename LabelT, typename K>
__device__ __forceinline__ void hub_chunk_block(const SigArgs& a, const HubArgs& h, char* smem_raw) {
  ChunkSmem<K>& sm = *reinterpret_cast<ChunkSmem<K>*>(smem_raw);
  K* list = reinterpret_cast<K*>(smem_raw + sizeof(ChunkSmem<K>));
  uint32_t* bcnt = reinterpret_cast<uint32_t*>(list + kHubChunk);
  uint32_t* bpos = bcnt + kHubSmemBuckets;
  const uint4 c = h.chunks[blockIdx.x];
  const uint32_t hub = c.x;
  if (h.mode[hub]) return;  // this hub's chunks run k_hub_scatter
  if (!in_mask(a, h.first + hub)) return;
  const uint64_t ebase = ((uint64_t)c.z << 32) | c.y;
  const uint32_t E = c.w;
  const uint32_t bits = h.hub_bits[hub];
  const uint32_t nb = 1u << bits;
  const bool in_smem = nb <= (uint32_t)kHubSmemBuckets;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  fill_empty<kChunkThreads>(sm.slot, (2 * E + 3) & ~3u, tid);
  if (tid == 0) sm.cnt = sm.empty = 0;
  if (in_smem)
    for (uint32_t i = tid; i < nb; i += kChunkThreads) bcnt[i] = 0;
  __syncthreads();
  K key[kChunkItems];
  uint32_t todo = hub_piece_keys<MODE, LabelT, K>(a, h, hub, ebase, E, key);
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm.slot);
#pragma unroll 1
  for (int t = 0; t < kChunkItems; ++t) {
    const K kt = key[0];
#pragma unroll
    for (int q = 0; q + 1 < kChunkItems; ++q) key[q] = key[q + 1];
    bool fresh = false;
    if (todo & 1u)
      fresh = kt == KeyOps<K>::kEmpty ? atomicExch(&sm.empty, 1u) == 0u : region_insert(sbase, 0u, 2 * E, kt);
    todo >>= 1;
    const unsigned fm = __ballot_sync(kFull, fresh);
    if (fm == 0u) continue;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(&sm.cnt, (uint32_t)__popc(fm));
    base = __shfl_sync(kFull, base, 0);
    if (fresh) list[base + __popc(fm & lanes_below(lane))] = kt;
  }
  __syncthreads();
  const uint32_t U = sm.cnt;
  const uint32_t cap = h.hub_cap[hub];
  uint32_t* cur = h.cursor + h.hub_bbase[hub];
  K* tmp = static_cast<K*>(h.tmp) + h.hub_tbase[hub];
  if (in_smem) {
    for (uint32_t i = tid; i < U; i += kChunkThreads) atomicAdd(&bcnt[hub_bucket(list[i], bits)], 1u);
    __syncthreads();
    for (uint32_t b = tid; b < nb; b += kChunkThreads) {
      const uint32_t n_b = bcnt[b];
      bpos[b] = n_b ? atomicAdd(&cur[b], n_b) : 0u;
      bcnt[b] = 0;
    }
    __syncthreads();
  }
  for (uint32_t i = tid; i < U; i += kChunkThreads) {
    const K v = list[i];
    const uint32_t b = hub_bucket(v, bits);
    const uint32_t q = in_smem ? bpos[b] + atomicAdd(&bcnt[b], 1u) : atomicAdd(&cur[b], 1u);
    if (q < cap) tmp[(uint64_t)b * cap + q] = v;
    else hub_fail(a, h, hub, kErrHubOverflow);
  }
}

template <int MODE, typename LabelT, typename K>
__global__ void __launch_bounds__(kChunkThreads) k_hub_chunk(SigArgs a, HubArgs h) {
  overlap_next();
  overlap_wait();
  extern __shared__ __align__(16) char smem_raw[];
  hub_chunk_block<MODE, LabelT, K>(a, h, smem_raw);
}

// Hub pieces without the chunk-level set, for hubs whose keys rarely repeat
// (k_hub_sample): the keys of a chunk go straight to the hub's buckets
// (ranked per bucket in shared memory, one global reservation per bucket,
// then ordered by bucket in shared memory so that each bucket's keys are
// stored as one run), and the bucket pass removes every duplicate.

// One warp per hub: kHubSample keys at an even stride over the hub's edges.
// Among S samples from U equally frequent distinct keys about S(S-1)/2 / U
// pairs are equal: kHubSamplePairs or more equal pairs mean about 500
// distinct keys or fewer (the few blocks of an early level), or a key that
// makes up some 5% of the hub's edges or more, and the hub keeps the chunk
// set, which sends each distinct key of a chunk to the buckets once.  Other
// hubs skip it, unless an earlier overflow forced the set on them.
template <typename LabelT, typename K>
__device__ __forceinline__ void hub_sample_block(const SigArgs& a, const HubArgs& h, uint64_t n_hub) {
  constexpr int kPer = kHubSample / 32;
  __shared__ K sk[256 / 32][kHubSample];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t hub = (uint64_t)blockIdx.x * (256 / 32) + w;
  if (hub >= n_hub) return;
  const uint64_t p = h.first + hub;
  const uint64_t e0 = a.off[p], D = a.off[p + 1] - e0;
  const uint32_t st = (uint32_t)(D / kHubSample);  // >= 1: hubs have more than 4096 edges
  const Policies pol;
  K key[kPer];
  edge_keys<kPer, 0, kPer, LabelT, K>(a, e0 + (uint64_t)lane * st, 32u * st, e0 + D, pol, key);
#pragma unroll
  for (int t = 0; t < kPer; ++t) sk[w][lane + 32 * t] = key[t];
  __syncwarp();
  uint32_t pairs = 0;
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    const uint32_t i = lane + 32 * t;
    for (uint32_t j = i + 1; j < (uint32_t)kHubSample; ++j) pairs += sk[w][j] == key[t] ? 1u : 0u;
  }
  pairs = __reduce_add_sync(kFull, pairs);
  if (lane == 0) h.mode[hub] = (!h.force[hub] && pairs < (uint32_t)kHubSamplePairs) ? 1 : 0;
}

template <typename LabelT, typename K>
__global__ void __launch_bounds__(256) k_hub_sample(SigArgs a, HubArgs h, uint64_t n_hub) {
  overlap_next();
  hub_sample_block<LabelT, K>(a, h, n_hub);
  overlap_wait();
}

// Exclusive prefix sums of v[0..n) in place (n <= 2 * NT), by the whole CTA;
// wsum holds NT / 32 words.  Ends with a barrier.
template <int NT>
__device__ __forceinline__ void cta_exclusive_scan(uint32_t* v, uint32_t n, uint32_t* wsum) {
  static_assert(NT % 32 == 0 && NT / 32 <= 32, "one warp scans the warp totals");
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t a = 2 * tid < n ? v[2 * tid] : 0u, b = 2 * tid + 1 < n ? v[2 * tid + 1] : 0u;
  uint32_t x = a + b;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, d);
    if (lane >= (uint32_t)d) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t t = lane < (uint32_t)(NT / 32) ? wsum[lane] : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, t, d);
      if (lane >= (uint32_t)d) t += y;
    }
    if (lane < (uint32_t)(NT / 32)) wsum[lane] = t;
  }
  __syncthreads();
  const uint32_t before = (w ? wsum[w - 1] : 0u) + x - (a + b);
  if (2 * tid < n) v[2 * tid] = before;
  if (2 * tid + 1 < n) v[2 * tid + 1] = before + a;
  __syncthreads();
}

template <typename K>
struct ScatterSmem {
  K stage[kHubChunk];
  uint32_t bcnt[kHubSmemBuckets], bpos[kHubSmemBuckets], lstart[kHubSmemBuckets];
  uint32_t wsum[kChunkThreads / 32];
};

template <int MODE, typename LabelT, typename K>
__device__ __forceinline__ void hub_scatter_block(const SigArgs& a, const HubArgs& h, ScatterSmem<K>& sm) {
  uint32_t *bcnt = sm.bcnt, *bpos = sm.bpos, *lstart = sm.lstart, *wsum = sm.wsum;
  K* stage = sm.stage;
  const uint4 c = h.chunks[blockIdx.x];
  const uint32_t hub = c.x;
  if (!h.mode[hub]) return;  // this hub's chunks run k_hub_chunk
  if (!in_mask(a, h.first + hub)) return;
  const uint64_t ebase = ((uint64_t)c.z << 32) | c.y;
  const uint32_t E = c.w;
  const uint32_t bits = h.hub_bits[hub];
  const uint32_t nb = 1u << bits;
  const bool in_smem = nb <= (uint32_t)kHubSmemBuckets;
  const uint32_t tid = threadIdx.x;
  if (in_smem)
    for (uint32_t i = tid; i < nb; i += kChunkThreads) bcnt[i] = 0;
  __syncthreads();
  K key[kChunkItems];
  const uint32_t todo = hub_piece_keys<MODE, LabelT, K>(a, h, hub, ebase, E, key);
  if (MODE == kWithDup && !__syncthreads_or(todo != 0)) return;
  const uint32_t cap = h.hub_cap[hub];
  uint32_t* cur = h.cursor + h.hub_bbase[hub];
  K* tmp = static_cast<K*>(h.tmp) + h.hub_tbase[hub];
  // rank of each key within its bucket in this chunk (shared counts), then one
  // global reservation per bucket
  uint32_t rank[kChunkItems];
#pragma unroll
  for (int t = 0; t < kChunkItems; ++t) {
    rank[t] = 0;
    if ((todo >> t) & 1u) {
      const uint32_t b = hub_bucket(key[t], bits);
      rank[t] = in_smem ? atomicAdd(&bcnt[b], 1u) : atomicAdd(&cur[b], 1u);
    }
  }
  if (!in_smem) {
#pragma unroll
    for (int t = 0; t < kChunkItems; ++t) {
      if (!((todo >> t) & 1u)) continue;
      const uint32_t b = hub_bucket(key[t], bits);
      if (rank[t] < cap) tmp[(uint64_t)b * cap + rank[t]] = key[t];
      else hub_fail(a, h, hub, kErrHubOverflow);
    }
    return;
  }
  __syncthreads();
  for (uint32_t b = tid; b < nb; b += kChunkThreads) {
    const uint32_t n_b = bcnt[b];
    bpos[b] = n_b ? atomicAdd(&cur[b], n_b) : 0u;
    lstart[b] = n_b;
  }
  __syncthreads();
  // the chunk's keys ordered by bucket in shared memory, so that each
  // bucket's keys leave as one run of consecutive words
  cta_exclusive_scan<kChunkThreads>(lstart, nb, wsum);
#pragma unroll
  for (int t = 0; t < kChunkItems; ++t)
    if ((todo >> t) & 1u) stage[lstart[hub_bucket(key[t], bits)] + rank[t]] = key[t];
  const uint32_t staged = lstart[nb - 1] + bcnt[nb - 1];
  __syncthreads();
  for (uint32_t i = tid; i < staged; i += kChunkThreads) {
    const K k = stage[i];
    const uint32_t b = hub_bucket(k, bits);
    const uint32_t q = bpos[b] + (i - lstart[b]);
    if (q < cap) tmp[(uint64_t)b * cap + q] = k;
    else hub_fail(a, h, hub, kErrHubOverflow);
  }
}

template <int MODE, typename LabelT, typename K>
__global__ void __launch_bounds__(kChunkThreads, sizeof(K) == 4 ? 4 : 3) k_hub_scatter(SigArgs a, HubArgs h) {
  overlap_next();
  overlap_wait();
  __shared__ ScatterSmem<K> sm;
  hub_scatter_block<MODE, LabelT, K>(a, h, sm);
}

// Both kinds of chunk in one launch, for graphs whose rounds are launches and
// latency more than work (chained): one launch less per round (1M nodes, 8
// edges a node, 767 -> 736 us a refinement of four rounds; equal from 2M nodes
// on).  Its shared memory is the chunk set's, which on larger graphs would take
// the L1 from the scatter's gathers.
template <int MODE, typename LabelT, typename K>
__global__ void __launch_bounds__(kChunkThreads, sizeof(K) == 4 ? 4 : 3) k_hub_pieces(SigArgs a, HubArgs h) {
  overlap_next();
  overlap_wait();
  extern __shared__ __align__(16) char smem_raw[];
  static_assert(sizeof(ScatterSmem<K>) <= hub_chunk_smem<K>(), "the scatter fits the chunk set's memory");
  if (h.mode[h.chunks[blockIdx.x].x]) hub_scatter_block<MODE, LabelT, K>(a, h, *reinterpret_cast<ScatterSmem<K>*>(smem_raw));
  else hub_chunk_block<MODE, LabelT, K>(a, h, smem_raw);
}

constexpr int kBucketThreads = 256, kBucketItems = 8;

template <typename K, int UCAP>
struct BucketSmem {
  K set[2 * UCAP];
  uint32_t empty, full, lo, hi;
};

// Count and hash of a hub (of the mask) from its buckets' totals.
__device__ __forceinline__ void hub_finish(const SigArgs& a, const HubArgs& h, uint64_t hub) {
  const uint64_t p = h.first + hub;
  if (!in_mask(a, p)) return;
  const unsigned long long tot = __ldcg(&h.hub_cur[hub]);
  const uint64_t tsum = ((uint64_t)__ldcg(&h.hub_term[2 * hub + 1]) << 32) | __ldcg(&h.hub_term[2 * hub]);
  a.ucnt[p] = (uint32_t)tot;
  a.hash[p] = node_hash(tsum, a.prev[p], tot, a.seed, a.mask);
}

// A bucket of the hub is done (called by one thread of its CTA, after the
// bucket's sums have been added): the hub's last one finishes the hub.  Saves
// a launch per round, but costs a fence and an atomic per bucket (256M edges,
// 40K buckets a round: 9.92 against 9.81 ms), so larger graphs have h.done NULL.
__device__ __forceinline__ void hub_bucket_done(const SigArgs& a, const HubArgs& h, uint32_t hub) {
  if (!h.done) return;
  const uint32_t nb = (uint32_t)(h.hub_bbase[hub + 1] - h.hub_bbase[hub]);
  __threadfence();
  if (atomicAdd(&h.done[hub], 1u) != nb - 1) return;
  __threadfence();
  hub_finish(a, h, hub);
}

__global__ void k_hub_finish(SigArgs a, HubArgs h, uint64_t n_hub) {
  overlap_next();
  overlap_wait();
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n_hub; i += (uint64_t)gridDim.x * blockDim.x)
    hub_finish(a, h, i);
}

// One CTA per hub bucket (grid-stride): distinct keys of the bucket into a
// shared set; a warp appends the keys it finds fresh straight after the
// hub's keys written so far (one reservation per warp step on the hub's
// counter) and adds their term sums to the bucket's, which go to the hub's
// at the end.  If the set fills, the host repeats the hub with more buckets
// (its counter restarts from zero, so the keys written are written again).
template <typename K, int UCAP>
__global__ void __launch_bounds__(kBucketThreads, sizeof(K) == 4 ? 6 : 3) k_hub_bucket(SigArgs a, HubArgs h, uint64_t n_buckets) {
  overlap_next();
  overlap_wait();
  extern __shared__ __align__(16) char smem_raw[];
  BucketSmem<K, UCAP>& sm = *reinterpret_cast<BucketSmem<K, UCAP>*>(smem_raw);
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm.set);
  K* out = static_cast<K*>(a.sigkey);
  // a bucket's hub, key count and first kBucketThreads * kBucketItems keys are
  // loaded one bucket ahead, so that their latency overlaps the work on the
  // bucket before
  uint32_t nx_hub = 0, nx_n = 0;
  bool nx_alone = false;
  const K* nx_tmp = nullptr;
  K kk[kBucketItems];
  auto fetch = [&](uint64_t bb) {
    nx_hub = h.bucket_hub[bb];
    const uint32_t cap = h.hub_cap[nx_hub];
    nx_tmp = static_cast<const K*>(h.tmp) + h.hub_tbase[nx_hub] + (bb - h.hub_bbase[nx_hub]) * cap;
    nx_n = min(h.cursor[bb], cap);
    nx_alone = a.alone && a.alone[h.first + nx_hub];
#pragma unroll
    for (int t = 0; t < kBucketItems; ++t) {
      const uint32_t i = tid + t * kBucketThreads;
      kk[t] = i < nx_n ? nx_tmp[i] : (K)0;
    }
  };
  if (blockIdx.x < n_buckets) fetch(blockIdx.x);
  for (uint64_t b = blockIdx.x; b < n_buckets; b += gridDim.x) {
    const uint32_t hub = nx_hub, n = nx_n;
    const bool alone = nx_alone;  // only the number of distinct keys is needed
    const uint64_t p = h.first + hub;
    const K* tmp = nx_tmp;
    if (n == 0) {  // nothing appended (a hub outside a frontier mask): no barrier, no output
      if (tid == 0) hub_bucket_done(a, h, hub);
      if (b + gridDim.x < n_buckets) fetch(b + gridDim.x);
      continue;
    }
    uint32_t hcap = 64;
    while (hcap < 2 * n && hcap < 2 * UCAP) hcap <<= 1;
    {
      uint4* s4 = reinterpret_cast<uint4*>(sm.set);
      const uint4 ones = make_uint4(~0u, ~0u, ~0u, ~0u);
      for (uint32_t i = tid; i < hcap * sizeof(K) / 16; i += kBucketThreads) s4[i] = ones;
    }
    if (tid == 0) {
      sm.empty = 0;
      sm.full = 0;
      sm.lo = 0;
      sm.hi = 0;
    }
    __syncthreads();
    K* hout = out + a.off[p];
    unsigned long long* hcur = &h.hub_cur[hub];
    for (uint32_t i0 = 0; i0 < n; i0 += kBucketThreads * kBucketItems) {
      if (i0) {
#pragma unroll
        for (int t = 0; t < kBucketItems; ++t) {
          const uint32_t i = i0 + tid + t * kBucketThreads;
          kk[t] = i < n ? tmp[i] : (K)0;
        }
      }
      if (alone) {
        uint32_t c = 0;
#pragma unroll
        for (int t = 0; t < kBucketItems; ++t) {
          const uint32_t i = i0 + tid + t * kBucketThreads;
          const K k = kk[t];
          if (i >= n) continue;
          if (k == KeyOps<K>::kEmpty) {
            c += atomicExch(&sm.empty, 1u) == 0u ? 1u : 0u;
          } else {
            const int r = pow2_insert(sbase, hcap - 1, k);
            c += r > 0 ? 1u : 0u;
            if (r < 0) sm.full = 1u;
          }
        }
        c = __reduce_add_sync(kFull, c);
        if (lane == 0) atomicAdd(&sm.lo, c);
        continue;
      }
      // the keys of kBucketItems steps are inserted first; then the warp
      // takes the places of all its fresh keys with one reservation on the
      // hub's counter (its latency paid once, not per step) and adds their
      // term sums once
      unsigned fms[kBucketItems];
      uint32_t lo = 0, hi = 0, total = 0;
#pragma unroll
      for (int t = 0; t < kBucketItems; ++t) {
        fms[t] = 0u;
        if (i0 + (uint32_t)t * kBucketThreads >= n) continue;  // the same for the whole CTA
        const uint32_t i = i0 + tid + t * kBucketThreads;
        const K k = kk[t];
        bool fresh = false;
        if (i < n) {
          if (k == KeyOps<K>::kEmpty) {
            fresh = atomicExch(&sm.empty, 1u) == 0u;
          } else {
            const int r = pow2_insert(sbase, hcap - 1, k);
            fresh = r > 0;
            if (r < 0) sm.full = 1u;
          }
        }
        fms[t] = __ballot_sync(kFull, fresh);
        total += __popc(fms[t]);
        if (fresh) {
          const uint64_t tm = elem_term(k, a.seed);
          lo += (uint32_t)tm;
          hi += (uint32_t)(tm >> 32);
        }
      }
      if (total) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(hcur, (unsigned long long)total);
        base = __shfl_sync(kFull, base, 0);
#pragma unroll
        for (int t = 0; t < kBucketItems; ++t) {
          if ((fms[t] >> lane) & 1u) hout[base + __popc(fms[t] & lanes_below(lane))] = kk[t];
          base += __popc(fms[t]);
        }
        lo = __reduce_add_sync(kFull, lo);
        hi = __reduce_add_sync(kFull, hi);
        if (lane == 0) {
          atomicAdd(&sm.lo, lo);
          atomicAdd(&sm.hi, hi);
        }
      }
    }
    if (b + gridDim.x < n_buckets) fetch(b + gridDim.x);
    __syncthreads();
    if (tid == 0) {
      if (sm.full) hub_fail(a, h, hub, kErrHubSet);  // more distinct keys than the set holds: the host adds buckets
      // (a failed hub's sums are cleared before its repeat)
      if (alone) {
        atomicAdd(hcur, (unsigned long long)sm.lo);
      } else {
        atomicAdd(&h.hub_term[2 * hub], sm.lo);
        atomicAdd(&h.hub_term[2 * hub + 1], sm.hi);
      }
      hub_bucket_done(a, h, hub);
    }
    // no barrier here: thread 0 alone reads the bucket's totals, and the next
    // bucket's first barrier comes before anything is written to them again
  }
}

// Marks the edges of hubs that repeat an earlier (label, target) of their hub:
// a set in global memory, two 32-bit slots per edge at the hub's place in the
// key buffer (all ones before).  Once per loaded graph; bound by the L2's
// atomics (the word is read first, which spares them for repeats).
template <typename LabelT>
__global__ void __launch_bounds__(kChunkThreads) k_mark_hubs(SigArgs a, uint64_t first, const uint4* chunks,
                                                             uint32_t* empty_seen) {
  const uint4 c = chunks[blockIdx.x];
  const uint64_t p = first + c.x, ebase = ((uint64_t)c.z << 32) | c.y;
  const uint64_t off = a.off[p];
  const uint32_t slots = (uint32_t)min((uint64_t)0xFFFFFFFEu, 2 * (a.off[p + 1] - off));
  uint32_t* set = static_cast<uint32_t*>(a.sigkey) + 2 * off;
  uint32_t key[kChunkItems];
  chunk_keys<kChunkThreads, LabelT, uint32_t>(a, ebase, c.w, key);
#pragma unroll 1
  for (int t = 0; t < kChunkItems; ++t) {
    const uint32_t i = threadIdx.x + t * kChunkThreads;
    if (i >= c.w) break;
    const uint32_t k = key[0];
#pragma unroll
    for (int q = 0; q + 1 < kChunkItems; ++q) key[q] = key[q + 1];
    bool fresh = false;
    if (k == KeyOps<uint32_t>::kEmpty) {
      fresh = atomicExch(&empty_seen[c.x], 1u) == 0u;
    } else {
      uint32_t s = region_home(k, slots);
      for (uint32_t q = 0; q < slots; ++q) {  // at most half full: ends at k or at an empty slot
        uint32_t cur = *(volatile uint32_t*)&set[s];
        if (cur == KeyOps<uint32_t>::kEmpty) cur = atomicCAS(&set[s], KeyOps<uint32_t>::kEmpty, k);
        if (cur == KeyOps<uint32_t>::kEmpty) {
          fresh = true;
          break;
        }
        if (cur == k) break;
        if (++s == slots) s = 0;
      }
    }
    if (!fresh) mark_dup(a, ebase + i);
  }
}

__global__ void k_iota(uint64_t n, uint32_t* a) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    a[i] = (uint32_t)i;
}

// --------------------------------------------------------------------------
// Grouping: equal hashes -> smallest original id; exact verification
// --------------------------------------------------------------------------
// Table slots are 64-bit words (hash fingerprint << 32 | smallest original
// id), empty = all ones.  A slot is claimed by CAS and then lowered with
// atomicMin; different hashes that meet in one slot with the same
// fingerprint are merged here and separated again by exact verification.
struct GroupArgs {
  const uint64_t* hash;
  const uint32_t* p2o;
  const uint32_t* o2p;
  unsigned long long* table;
  uint64_t tmask;   // table capacity - 1
  uint32_t* slot;
  uint32_t* rep;
  uint32_t* err;
  const uint8_t* alone;  // nodes alone in their previous block (may be null): heads, not grouped
  int read_first;        // few distinct hashes shared by many nodes (level 0): read a slot before any atomic
  // number of listed nodes on the device (NULL = the launch's count); the table
  // then has table_slots of it
  const unsigned long long* d_count;
  uint2* seen;           // filter: per 32 bits, (hash seen, hash seen twice); NULL = no filter
  uint64_t seen_mask;    // bits - 1
};

// Slots of a table for n nodes: a power of two, at most half full.
__host__ __device__ __forceinline__ uint64_t table_slots(uint64_t n) {
  uint64_t c = 1024;
  while (c < 2 * n) c <<= 1;
  return c;
}

__device__ __forceinline__ uint32_t table_insert(const GroupArgs& g, uint64_t tmask, uint64_t h, uint32_t minid) {
  const unsigned long long fp = (unsigned long long)(uint32_t)(h >> 32);
  const unsigned long long v = (fp << 32) | minid;
  uint32_t s = (uint32_t)(mix64(h) & tmask);
  for (uint64_t t = 0; t <= tmask; ++t) {
    // a slot already holding this fingerprint with an id no larger needs no atomic
    if (g.read_first) {
      const unsigned long long seen = *(volatile unsigned long long*)&g.table[s];
      if ((seen >> 32) == fp && seen != kEmpty64 && (uint32_t)seen <= minid) return s;
    }
    const unsigned long long cur = atomicCAS(&g.table[s], (unsigned long long)kEmpty64, v);
    if (cur == kEmpty64) return s;
    if ((cur >> 32) == fp) {
      if ((uint32_t)cur > minid) atomicMin(&g.table[s], v);
      return s;
    }
    s = (uint32_t)((s + 1) & tmask);
  }
  atomicOr(g.err, kErrProbe);
  return 0;
}

// Whether the CTA's tile of `tile` nodes from base on (a multiple of 4) holds a
// node not alone in its previous block, by 4 flags a thread; called by the whole
// CTA.  In late rounds most tiles hold none, and the grouping would pass through
// its barriers for nothing (16M nodes, four rounds: 373 -> 252 us).
__device__ __forceinline__ bool tile_has_work(const uint8_t* alone, uint64_t base, uint32_t tile, uint64_t count) {
  if (base + tile > count) return true;
  const bool mine = threadIdx.x * 4 < tile &&
                    (reinterpret_cast<const uint32_t*>(alone + base)[threadIdx.x] & 0x01010101u) != 0x01010101u;
  return __syncthreads_or(mine);
}

// A CTA takes 1024 nodes, combines equal hashes in shared memory (smallest
// original id per hash), then inserts each distinct hash once.
constexpr int kInsThreads = 256, kInsItems = 4, kInsChunk = kInsThreads * kInsItems, kInsSlots = 2 * kInsChunk;

__global__ void __launch_bounds__(kInsThreads) k_group_insert(GroupArgs g, const uint32_t* list, uint64_t count) {
  overlap_next();
  overlap_wait();
  if (g.d_count) count = *g.d_count;
  const uint64_t tmask = g.d_count ? table_slots(count) - 1 : g.tmask;
  __shared__ unsigned long long skey[kInsSlots];
  __shared__ unsigned int smin[kInsSlots];
  __shared__ unsigned int sglob[kInsSlots];
  __shared__ unsigned short used[kInsChunk];  // slots taken in this chunk (one per distinct hash)
  __shared__ unsigned int n_used;
  const uint32_t lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kInsSlots; i += kInsThreads) {
    skey[i] = kEmpty64;
    smin[i] = kNone32;
  }
  if (threadIdx.x == 0) n_used = 0;
  __syncthreads();
  for (uint64_t base = (uint64_t)blockIdx.x * kInsChunk; base < count; base += (uint64_t)gridDim.x * kInsChunk) {
    if (g.alone && !list && !tile_has_work(g.alone, base, kInsChunk, count)) continue;
    // loads of all items first (node ids, then alone flags, then hashes and
    // original ids of the nodes that are grouped), so that they overlap
    uint32_t ls[kInsItems], pp[kInsItems], oo[kInsItems];
    uint64_t hh[kInsItems];
#pragma unroll
    for (int t = 0; t < kInsItems; ++t) {
      const uint64_t i = base + threadIdx.x + (uint64_t)t * kInsThreads;
      pp[t] = i < count ? (list ? list[i] : (uint32_t)i) : kNone32;
    }
#pragma unroll
    for (int t = 0; t < kInsItems; ++t)
      ls[t] = (pp[t] != kNone32 && !(g.alone && g.alone[pp[t]])) ? 0u : kNone32;
#pragma unroll
    for (int t = 0; t < kInsItems; ++t) {
      if (ls[t] != kNone32) {
        hh[t] = g.hash[pp[t]];
        oo[t] = g.p2o[pp[t]];
      }
    }
#pragma unroll
    for (int t = 0; t < kInsItems; ++t) {
      bool took = false;
      if (ls[t] != kNone32) {
        const uint64_t h = hh[t];
        uint32_t s = (uint32_t)(mix64(h) & (kInsSlots - 1));
        for (int q = 0; q < kInsSlots; ++q) {  // at most kInsChunk distinct hashes: always room
          const unsigned long long cur = atomicCAS(&skey[s], (unsigned long long)kEmpty64, (unsigned long long)h);
          if (cur == kEmpty64) { took = true; break; }
          if (cur == h) break;
          s = (s + 1) & (kInsSlots - 1);
        }
        atomicMin(&smin[s], oo[t]);
        ls[t] = s;
      }
      const unsigned tm = __ballot_sync(kFull, took);
      if (tm) {
        uint32_t b0 = 0;
        if (lane == 0) b0 = atomicAdd(&n_used, (unsigned)__popc(tm));
        b0 = __shfl_sync(kFull, b0, 0);
        if (took) used[b0 + __popc(tm & lanes_below(lane))] = (unsigned short)ls[t];
      }
    }
    __syncthreads();
    const uint32_t nu = n_used;
    for (uint32_t i = threadIdx.x; i < nu; i += kInsThreads) {
      const uint32_t sl = used[i];
      sglob[sl] = table_insert(g, tmask, skey[sl], smin[sl]);
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kInsItems; ++t)
      if (ls[t] != kNone32) g.slot[pp[t]] = sglob[ls[t]];
    __syncthreads();
    // only the slots this chunk took are cleared for the next one
    for (uint32_t i = threadIdx.x; i < nu; i += kInsThreads) {
      const uint32_t sl = used[i];
      skey[sl] = kEmpty64;
      smin[sl] = kNone32;
    }
    if (threadIdx.x == 0) n_used = 0;
    __syncthreads();
  }
}

struct VerifyArgs {
  int mode;                 // 0: level 0 (labels), 1: signatures
  int key64;                // signature words are 64-bit
  const uint32_t* nlabel;
  const uint32_t* prev;
  const uint32_t* ucnt;
  const uint64_t* off;
  const void* sigkey;
  uint32_t* out_list;       // unresolved nodes
  unsigned long long* n_out;
  unsigned long long* n_collided;
  // (node, candidate) pairs left to k_verify_long, in one array of pair_cap
  // pairs: up to kMidSig elements from the front, longer ones from the back
  uint32_t* long_list;
  uint64_t pair_cap;
  unsigned long long* n_mid;
  unsigned long long* n_long;
  uint32_t* hbits;          // head bitmap over original ids (canonical numbering)
  uint8_t* member;          // per internal id: this head has other members
  // the marks and representatives of the nodes alone in their previous block
  // stand since the level before (a head stays one: its block only splits)
  bool keep;
};

constexpr uint32_t kShortSig = 8;   // compared by one thread
constexpr uint32_t kMidSig = 64;    // compared by one warp, two elements per lane

// Set equality of two duplicate-free key lists of the same length n <= kShortSig.
template <typename K>
__device__ __forceinline__ bool same_set_short(const K* a, const K* b, uint32_t n) {
  K bk[kShortSig];
#pragma unroll
  for (uint32_t j = 0; j < kShortSig; ++j) bk[j] = j < n ? b[j] : (K)0;
  for (uint32_t i = 0; i < n; ++i) {
    const K x = a[i];
    bool found = false;
#pragma unroll
    for (uint32_t j = 0; j < kShortSig; ++j) found |= (j < n && bk[j] == x);
    if (!found) return false;
  }
  return true;
}

// Marks for the canonical numbering, set where a node's representative is
// settled: a head sets the bit of its original id; a member sets its head's
// member flag (read first: in a large block most members find it set).
__device__ __forceinline__ void mark_head(const VerifyArgs& v, uint32_t o) {
  atomicOr(&v.hbits[o >> 5], 1u << (o & 31));
}
__device__ __forceinline__ void mark_member(const VerifyArgs& v, uint32_t r) {
  if (!*(volatile uint8_t*)&v.member[r]) v.member[r] = 1;
}

// Filter before the table, when the table would not stay in L2.  Where blocks
// are small most hashes occur once, and a node alone with its hash is a head
// that needs neither the table nor a comparison.  One pass notes every hash in
// a bitmap of 8 to 16 bits per node, and in a second one the hashes met before;
// the next pass settles the nodes whose bit was met once and lists the others
// (those that share a hash, and one node in 16 to 8 by chance) for the grouping,
// whose table is sized for them.
// 16M random accesses cost 0.43 ms as compare-and-swaps in a table of 256 MB
// and 0.25 ms as its loads, 0.14 and 0.07 ms in 32 MB.  Grouping and comparison
// of the 16M-node powerlaw graph's four rounds: 1.95 -> 1.55 ms; 25.6M nodes of
// the alpha = 2.0 one, five rounds: 5.2 -> 4.7 ms.  Up to 4M nodes the table
// is as cheap (64 MB) and the two passes only cost.
// They also only cost in round 1 where most nodes share their hash: level 0 has
// few blocks, so a signature of no element or one repeats unless (label, block)
// takes many values (kFilterValues), and where more than a node in 20 has such
// a signature, the others are short too.  Refinement to level 1 with the filter
// against without: 10M nodes of which 55% have two out-edges or more 1,454
// against 1,254 us, 86% 1,710 and 1,622, 98% 1,837 and 1,900, 100% 1,475 to
// 1,962 against 1,497 to 2,054; 10M with 5,000 edge labels 1,494 against 1,696.
constexpr uint64_t kFilterNodes = 4u << 20;  // table above 64 MB
constexpr uint64_t kFilterValues = 1u << 14;
constexpr int kFilThreads = 256, kFilItems = 4, kFilTile = kFilThreads * kFilItems;

__device__ __forceinline__ uint64_t filter_bit(const GroupArgs& g, uint64_t h) { return (mix64(h) >> 32) & g.seen_mask; }

__global__ void __launch_bounds__(kFilThreads) k_group_filter(GroupArgs g, uint64_t count) {
  overlap_next();
  overlap_wait();
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t base = (uint64_t)blockIdx.x * kFilTile; base < count; base += (uint64_t)gridDim.x * kFilTile) {
    uint64_t b[kFilItems];
    bool act[kFilItems];
    uint2 w[kFilItems];
#pragma unroll
    for (int t = 0; t < kFilItems; ++t) {
      const uint64_t p = base + threadIdx.x + (uint64_t)t * kFilThreads;
      act[t] = p < count && !(g.alone && g.alone[p]);
      b[t] = act[t] ? filter_bit(g, g.hash[p]) : ~0ull;
    }
    // bits only get set, so a stale word can only cost an atomic
#pragma unroll
    for (int t = 0; t < kFilItems; ++t)
      w[t] = act[t] ? g.seen[b[t] >> 5] : make_uint2(0u, 0u);
#pragma unroll
    for (int t = 0; t < kFilItems; ++t) {
      // of a run of lanes with one hash, the first notes it as seen and the
      // second as seen twice
      const bool run = __shfl_up_sync(kFull, b[t], 1) == b[t] && lane > 0;
      const bool rest = __shfl_up_sync(kFull, (uint32_t)run, 1) != 0u && lane > 0 && run;
      if (!act[t] || rest) continue;
      const uint32_t bit = 1u << (b[t] & 31);
      uint2* at = &g.seen[b[t] >> 5];
      if (w[t].y & bit) continue;
      if (run || (w[t].x & bit) || (atomicOr(&at->x, bit) & bit)) atomicOr(&at->y, bit);
    }
  }
}

// Nodes alone in their previous block or with their hash: heads.  The others
// are listed (a CTA takes its places together).
__global__ void __launch_bounds__(kFilThreads) k_group_select(GroupArgs g, VerifyArgs v, uint64_t count, uint32_t* list,
                                                              unsigned long long* n_list) {
  overlap_next();
  overlap_wait();
  __shared__ uint32_t n_cta;
  __shared__ unsigned long long at_cta;
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t base = (uint64_t)blockIdx.x * kFilTile; base < count; base += (uint64_t)gridDim.x * kFilTile) {
    if (threadIdx.x == 0) n_cta = 0;
    __syncthreads();
    uint32_t o[kFilItems], at[kFilItems];
    uint64_t h[kFilItems];
    bool act[kFilItems], cand[kFilItems];
#pragma unroll
    for (int t = 0; t < kFilItems; ++t) {
      const uint64_t p = base + threadIdx.x + (uint64_t)t * kFilThreads;
      act[t] = p < count;
      cand[t] = act[t] && !(g.alone && g.alone[p]);
      act[t] = act[t] && !(v.keep && !cand[t]);
      if (act[t]) o[t] = g.p2o[p];
      if (cand[t]) h[t] = g.hash[p];
    }
#pragma unroll
    for (int t = 0; t < kFilItems; ++t) {
      if (cand[t]) {
        const uint64_t b = filter_bit(g, h[t]);
        cand[t] = (__ldcg(&g.seen[b >> 5].y) >> (b & 31)) & 1u;
      }
    }
#pragma unroll
    for (int t = 0; t < kFilItems; ++t) {
      const unsigned m = __ballot_sync(kFull, cand[t]);
      uint32_t q = 0;
      if (lane == 0 && m) q = atomicAdd(&n_cta, (uint32_t)__popc(m));
      at[t] = __shfl_sync(kFull, q, 0) + __popc(m & lanes_below(lane));
      if (act[t] && !cand[t]) {
        g.rep[base + threadIdx.x + (uint64_t)t * kFilThreads] = (uint32_t)(base + threadIdx.x + (uint64_t)t * kFilThreads);
        mark_head(v, o[t]);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && n_cta) at_cta = atomicAdd(n_list, (unsigned long long)n_cta);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kFilItems; ++t)
      if (cand[t]) list[at_cta + at[t]] = (uint32_t)(base + threadIdx.x + (uint64_t)t * kFilThreads);
    __syncthreads();  // the CTA's count and place are read before the next tile's
  }
}

__global__ void __launch_bounds__(kFilThreads) k_table_clear(GroupArgs g) {
  overlap_next();
  overlap_wait();
  const uint64_t units = table_slots(*g.d_count) / 2;  // 16 bytes
  for (uint64_t u = blockIdx.x * (uint64_t)kFilThreads + threadIdx.x; u < units; u += (uint64_t)gridDim.x * kFilThreads)
    reinterpret_cast<uint4*>(g.table)[u] = make_uint4(~0u, ~0u, ~0u, ~0u);
}

constexpr int kMarkSeen = 256;  // heads a verification CTA remembers as marked

__device__ __forceinline__ void mark_unresolved(const VerifyArgs& v, uint32_t* rep, uint32_t p) {
  rep[p] = kNone32;
  const unsigned long long q = atomicAdd(v.n_out, 1ull);
  v.out_list[q] = p;
  atomicAdd(v.n_collided, 1ull);
}

// Each thread takes kVerItems nodes of a tile at a time, and every step's
// loads for all of them are issued together (node ids; alone flags; original
// ids and table slots; representatives; their fields; the short key lists).
constexpr int kVerNodeThreads = 256, kVerItems = 2, kVerTile = kVerNodeThreads * kVerItems;

__global__ void __launch_bounds__(kVerNodeThreads, 6) k_group_verify(GroupArgs g, VerifyArgs v, const uint32_t* list,
                                                                   uint64_t count) {
  overlap_next();
  overlap_wait();
  if (g.d_count) count = *g.d_count;
  // heads this CTA has marked as having members: a block of millions of
  // nodes (level 0) then costs one global access per CTA, not per member
  __shared__ uint32_t seen[kMarkSeen];
  for (int i = threadIdx.x; i < kMarkSeen; i += kVerNodeThreads) seen[i] = kNone32;
  __syncthreads();
  for (uint64_t base = (uint64_t)blockIdx.x * kVerTile; base < count; base += (uint64_t)gridDim.x * kVerTile) {
    uint32_t p[kVerItems], o[kVerItems], x[kVerItems], r[kVerItems], U[kVerItems];
    bool act[kVerItems], eq[kVerItems];
#pragma unroll
    for (int t = 0; t < kVerItems; ++t) {
      const uint64_t i = base + threadIdx.x + (uint64_t)t * kVerNodeThreads;
      p[t] = i < count ? (list ? list[i] : (uint32_t)i) : kNone32;
    }
#pragma unroll
    for (int t = 0; t < kVerItems; ++t) act[t] = p[t] != kNone32 && !(g.alone && g.alone[p[t]]);
    if (v.keep) {  // (most warps of a late round; no barrier: warps go on by themselves)
      bool any = false;
#pragma unroll
      for (int t = 0; t < kVerItems; ++t) any |= act[t];
      if (!__any_sync(kFull, any)) continue;
    }
#pragma unroll
    for (int t = 0; t < kVerItems; ++t) {
      if (!act[t] && v.keep) p[t] = kNone32;
      if (p[t] != kNone32) o[t] = g.p2o[p[t]];
      if (act[t]) x[t] = g.slot[p[t]];
    }
#pragma unroll
    for (int t = 0; t < kVerItems; ++t)
      if (act[t]) x[t] = (uint32_t)g.table[x[t]];  // smallest original id of the node's hash
    // heads: alone in the previous block, or the smallest id of their hash
#pragma unroll
    for (int t = 0; t < kVerItems; ++t) {
      if (p[t] != kNone32 && (!act[t] || x[t] == o[t])) {
        g.rep[p[t]] = p[t];
        mark_head(v, o[t]);
        act[t] = false;
      }
    }
#pragma unroll
    for (int t = 0; t < kVerItems; ++t)
      if (act[t]) r[t] = g.o2p[x[t]];
    if (v.mode == 0) {
#pragma unroll
      for (int t = 0; t < kVerItems; ++t)
        if (act[t]) eq[t] = v.nlabel[p[t]] == v.nlabel[r[t]];
    } else {
#pragma unroll
      for (int t = 0; t < kVerItems; ++t) {
        if (act[t]) {
          U[t] = v.ucnt[p[t]];
          eq[t] = v.prev[p[t]] == v.prev[r[t]] && U[t] == v.ucnt[r[t]];
        }
      }
#pragma unroll
      for (int t = 0; t < kVerItems; ++t) {
        // longer signatures go to k_verify_long (a warp takes its places in a list together)
        const bool lng = act[t] && eq[t] && U[t] > kShortSig;
        if (!__any_sync(kFull, lng)) continue;
        const uint32_t lane = threadIdx.x & 31;
        const unsigned mm = __ballot_sync(kFull, lng && U[t] <= kMidSig), lm = __ballot_sync(kFull, lng && U[t] > kMidSig);
        unsigned long long q = 0;
        if (lane == 0 && mm) q = atomicAdd(v.n_mid, (unsigned long long)__popc(mm));
        if (lane == 1 && lm) q = atomicAdd(v.n_long, (unsigned long long)__popc(lm));
        const unsigned long long qm = __shfl_sync(kFull, q, 0), ql = __shfl_sync(kFull, q, 1);
        if (lng) {
          q = U[t] <= kMidSig ? qm + __popc(mm & lanes_below(lane))
                              : v.pair_cap - 1 - (ql + __popc(lm & lanes_below(lane)));
          v.long_list[2 * q] = p[t];
          v.long_list[2 * q + 1] = r[t];
          act[t] = false;
        }
      }
#pragma unroll
      for (int t = 0; t < kVerItems; ++t) {
        if (act[t] && eq[t]) {
          eq[t] = v.key64 ? same_set_short(static_cast<const uint64_t*>(v.sigkey) + v.off[p[t]],
                                           static_cast<const uint64_t*>(v.sigkey) + v.off[r[t]], U[t])
                          : same_set_short(static_cast<const uint32_t*>(v.sigkey) + v.off[p[t]],
                                           static_cast<const uint32_t*>(v.sigkey) + v.off[r[t]], U[t]);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < kVerItems; ++t) {
      if (!act[t]) continue;
      if (eq[t]) {
        g.rep[p[t]] = r[t];
        if (atomicCAS(&seen[r[t] % kMarkSeen], kNone32, r[t]) != r[t]) mark_member(v, r[t]);
      } else {
        mark_unresolved(v, g.rep, p[t]);
      }
    }
  }
}

// The pairs k_group_verify left, their numbers read from the device, so that
// the host need not wait for them before the next launches.  Lists are
// duplicate-free and of equal length, so the sets are equal iff every one of
// the node's keys is found among the candidate's.
// Up to kMidSig elements (most pairs: the few blocks of level 0 bound the sets
// of level 1): a warp per pair, two keys of each list per lane, the
// candidate's keys handed round by shuffles.  Longer ones: a CTA per pair, the
// candidate's keys in a shared-memory set, chunk by chunk.
constexpr int kVerThreads = 256, kVerChunk = 4096;

template <typename K>
__host__ __device__ constexpr size_t verify_ws_bytes() { return team_set_bytes<K>(2 * kVerChunk, 0, kVerThreads); }

__device__ __forceinline__ void settle_pair(const GroupArgs& g, const VerifyArgs& v, uint32_t p, uint32_t r, bool same) {
  if (same) {
    g.rep[p] = r;
    mark_member(v, r);
  } else {
    mark_unresolved(v, g.rep, p);
  }
}

template <typename K>
__global__ void __launch_bounds__(kVerThreads) k_verify_long(GroupArgs g, VerifyArgs v) {
  overlap_next();
  overlap_wait();
  extern __shared__ __align__(16) char smem[];
  const K* keys = static_cast<const K*>(v.sigkey);
  const uint64_t n_mid = *v.n_mid, n_long = *v.n_long;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * kVerThreads) >> 5;
  for (uint64_t q = ((uint64_t)blockIdx.x * kVerThreads + threadIdx.x) >> 5; q < n_mid; q += warps) {
    const uint2 pr = reinterpret_cast<const uint2*>(v.long_list)[q];
    const uint32_t U = v.ucnt[pr.x];
    const K* ka = keys + v.off[pr.x];
    const K* kb = keys + v.off[pr.y];
    const bool h0 = lane < U, h1 = lane + 32 < U;
    const K a0 = h0 ? ka[lane] : (K)0, a1 = h1 ? ka[lane + 32] : (K)0;
    const K b0 = h0 ? kb[lane] : (K)0, b1 = h1 ? kb[lane + 32] : (K)0;
    bool f0 = !h0, f1 = !h1;
    for (uint32_t j = 0; j < min(U, 32u); ++j) {
      const K x = __shfl_sync(kFull, b0, j);
      f0 |= a0 == x;
      f1 |= a1 == x;
    }
    for (uint32_t j = 32; j < U; ++j) {
      const K x = __shfl_sync(kFull, b1, j - 32);
      f0 |= a0 == x;
      f1 |= a1 == x;
    }
    const bool same = __all_sync(kFull, f0 && f1);
    if (lane == 0) settle_pair(g, v, pr.x, pr.y, same);
  }
  TeamSet<K> ts = carve_set<K>(smem, 2 * kVerChunk, 0);
  for (uint64_t q = blockIdx.x; q < n_long; q += gridDim.x) {
    const uint2 pr = reinterpret_cast<const uint2*>(v.long_list)[v.pair_cap - 1 - q];
    const uint32_t U = v.ucnt[pr.x];
    const K* ka = keys + v.off[pr.x];
    const K* kb = keys + v.off[pr.y];
    uint32_t found = 0;
    for (uint32_t c0 = 0; c0 < U; c0 += kVerChunk) {
      const uint32_t cn = min((uint32_t)kVerChunk, U - c0);
      const int hcap = set_size_for(cn, 2 * kVerChunk);
      set_clear<kVerThreads>(ts, hcap, threadIdx.x);
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < cn; i += kVerThreads) set_insert(ts, hcap, kb[c0 + i]);
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < U; i += kVerThreads) found += set_find(ts, hcap, ka[i]) ? 1 : 0;
      __syncthreads();
    }
    found = team_sum<kVerThreads>(found, ts.red, threadIdx.x);
    if (threadIdx.x == 0) settle_pair(g, v, pr.x, pr.y, found == U);
    __syncthreads();
  }
}

// --------------------------------------------------------------------------
// Canonical renumbering: heads are nodes with rep[p] == p (the node with the
// smallest original id in its block); a block's id is the number of heads
// with a smaller original id.  Heads are marked in a bitmap over original ids
// (n/8 bytes, cache resident); an exclusive scan of the per-word head counts
// then gives each head its rank with one more popcount.
// --------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

struct RankArgs {
  uint64_t n, n_alive;
  const uint32_t* rep;
  const uint32_t* p2o;
  const uint32_t* ucnt;    // may be null (level 0)
  const uint2* hrank;      // [words] head bitmap word and the heads before it in its tile
  const uint32_t* tbase;   // [tiles] heads before each tile of kRankTile words
  uint8_t* member;         // [n] internal order: the head has other members
  uint8_t* alone;          // [n] internal order: output, node alone in its block
  uint32_t* pid;           // output level, internal order
  const uint32_t* err;     // error flags, copied to stats[7]
  unsigned long long* stats;  // [2] key total, [3] max signature, [7] error flags, [8] nodes alone in their block
  unsigned long long* host;   // pinned: all 16 scalars, by the last CTA
  uint32_t* alone_bits;       // [(n + 31) / 32] alone as a bitmap (may be null)
};

// The 16 scalars of a level into pinned host memory (a copy of its own took
// 3.3 us a round).  For the CTA that ends last, after a fence.
__device__ __forceinline__ void publish_scalars(const unsigned long long* stats, unsigned long long* host, uint32_t lane) {
  if (lane < 16) host[lane] = __ldcg(stats + lane);
}

// Heads before every bitmap word, in one pass: a CTA takes a tile of kRankTile
// words and writes each word beside the heads before it in the tile; the CTA
// that finishes last (a ticket, so nothing waits) turns the tile totals into
// heads before each tile and the level's block count.  Word and rank sit in
// one 8-byte entry, so k_pid_fill fetches both with one random access.  One
// launch instead of a word count, two tile passes and a scan of the tiles:
// bound by launch latency (31K words at 1M nodes; 9.5 us for the four before).
constexpr int kRankThreads = 256, kRankItems = 4, kRankTile = kRankThreads * kRankItems;
static_assert(kRankTile * 32 == 1 << kRankTileShift, "tile of original ids");

// Exclusive sum of v over the CTA; *total gets the CTA's sum.  red: NT / 32 words.
template <int NT>
__device__ __forceinline__ uint32_t cta_exclusive_sum(uint32_t v, uint32_t* red, uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  if (lane == 31) red[w] = x;
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (uint32_t i = 0; i < NT / 32; ++i) {
    const uint32_t r = red[i];
    before += i < w ? r : 0u;
    all += r;
  }
  __syncthreads();
  *total = all;
  return before + x - v;
}

__global__ void __launch_bounds__(kRankThreads) k_head_ranks(const uint32_t* hbits, uint64_t words, uint2* hrank,
                                                             uint32_t* tbase, unsigned long long* ticket,
                                                             unsigned long long* total) {
  overlap_next();
  overlap_wait();
  __shared__ uint32_t red[kRankThreads / 32];
  __shared__ uint32_t last;
  const uint64_t w0 = (uint64_t)blockIdx.x * kRankTile + (uint64_t)threadIdx.x * kRankItems;
  uint32_t b[kRankItems], c = 0;
#pragma unroll
  for (int t = 0; t < kRankItems; ++t) {
    b[t] = w0 + t < words ? hbits[w0 + t] : 0u;
    c += __popc(b[t]);
  }
  uint32_t all;
  uint32_t run = cta_exclusive_sum<kRankThreads>(c, red, &all);
#pragma unroll
  for (int t = 0; t < kRankItems; ++t) {
    if (w0 + t < words) hrank[w0 + t] = make_uint2(b[t], run);
    run += __popc(b[t]);
  }
  if (threadIdx.x == 0) {
    tbase[blockIdx.x] = all;
    __threadfence();
    last = atomicAdd(ticket, 1ull) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  uint32_t carry = 0;
  for (uint32_t t0 = 0; t0 < gridDim.x; t0 += kRankThreads) {
    const uint32_t i = t0 + threadIdx.x;
    const uint32_t v = i < gridDim.x ? __ldcg(tbase + i) : 0u;
    const uint32_t before = cta_exclusive_sum<kRankThreads>(v, red, &all);
    if (i < gridDim.x) tbase[i] = carry + before;
    carry += all;
  }
  if (threadIdx.x == 0) *total = carry;
}

// Exclusive scan of bsum[0..nb) in one CTA; total into *total.
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(uint64_t* bsum, uint64_t nb,
                                                              unsigned long long* total) {
  __shared__ unsigned long long wt[kScanThreads / 32];
  __shared__ unsigned long long carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (uint64_t base = 0; base < nb; base += kScanThreads) {
    const uint64_t i = base + threadIdx.x;
    const unsigned long long v = i < nb ? bsum[i] : 0ull;
    unsigned long long x = v;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wt[w] = x;
    __syncthreads();
    if (w == 0) {
      unsigned long long t = wt[lane];
      unsigned long long xx = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(kFull, xx, o);
        if (lane >= o) xx += y;
      }
      wt[lane] = xx - t;
    }
    __syncthreads();
    const unsigned long long c0 = carry;
    if (i < nb) bsum[i] = c0 + wt[w] + x - v;
    __syncthreads();
    if (threadIdx.x == kScanThreads - 1) carry = c0 + wt[w] + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

// Every alive node takes its head's block id; deleted nodes get kDead.  A
// thread takes kFillItems nodes at a time and issues each step's loads for
// all of them together (representatives; their original ids; the bitmap
// words), so the three dependent gathers of a node overlap with the others'.
// The node's own original id is read beside its representative, so that only
// members of a block with another head pay a third dependent gather (16M
// nodes: 97 -> 65 us a call; without any of this 106).
// No load waits behind a store of the item before (the arrays might alias, so
// the compiler keeps that order).  The grid is one resident wave and a CTA adds
// its counts with one atomic per statistic: with one per warp the same-address
// atomics took most of the time at 1M nodes (39 us a call).
// When a hub's buckets overflowed, the groups come from incomplete signatures
// and the round is grouped again: nothing is written then but the scalars,
// since alone and alone_bits still hold the level before, which that grouping
// and the repeated hubs read (the flags are final: every earlier kernel ended).
constexpr int kFillThreads = 256, kFillItems = 4;

__global__ void __launch_bounds__(kFillThreads, 4) k_pid_fill(RankArgs r) {
  overlap_next();
  overlap_wait();
  __shared__ unsigned int s_alone, s_mx;
  __shared__ unsigned long long s_keys;
  if (threadIdx.x == 0) {
    s_alone = s_mx = 0;
    s_keys = 0;
  }
  __syncthreads();
  unsigned int n_alone = 0, mx = 0;
  unsigned long long keys = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t n_fill = *r.err & (kErrHubOverflow | kErrHubSet) ? 0 : r.n;
  // (the whole warp goes through the loop together)
  for (uint64_t p0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p0 - lane < n_fill; p0 += stride * kFillItems) {
    uint32_t h[kFillItems], o[kFillItems], u[kFillItems];
    uint8_t mem[kFillItems];
    uint2 hr[kFillItems];
    bool live[kFillItems];
#pragma unroll
    for (int t = 0; t < kFillItems; ++t) {
      const uint64_t p = p0 + (uint64_t)t * stride;
      live[t] = p < r.n_alive;
      u[t] = 0;
      if (live[t]) {
        h[t] = r.rep[p];
        o[t] = r.p2o[p];  // the head's, unless p is not one
        mem[t] = r.member[p];
        if (r.ucnt) u[t] = r.ucnt[p];
      }
    }
    // a hash collision leaves nodes without a head: the fill runs again once
    // they are settled
#pragma unroll
    for (int t = 0; t < kFillItems; ++t)
      if (live[t] && h[t] != (uint32_t)(p0 + (uint64_t)t * stride)) o[t] = h[t] < r.n_alive ? r.p2o[h[t]] : 0u;
#pragma unroll
    for (int t = 0; t < kFillItems; ++t) {
      if (live[t]) {
        hr[t] = r.hrank[o[t] >> 5];
        hr[t].y += r.tbase[o[t] >> kRankTileShift];
      }
    }
#pragma unroll
    for (int t = 0; t < kFillItems; ++t) {
      const uint64_t p = p0 + (uint64_t)t * stride;
      bool al = false;
      if (live[t]) {
        keys += u[t];
        mx = max(mx, u[t]);
        r.pid[p] = hr[t].y + (uint32_t)__popc(hr[t].x & ((1u << (o[t] & 31)) - 1u));
        al = h[t] == (uint32_t)p && !mem[t];
        r.alone[p] = al ? 1 : 0;
        n_alone += al ? 1u : 0u;
      } else if (p < r.n) {
        r.pid[p] = kDead;
      }
      if (r.alone_bits) {  // a warp's 32 nodes are one word
        const uint32_t bits = __ballot_sync(kFull, al);
        if (lane == 0 && p < r.n) r.alone_bits[p >> 5] = bits;
      }
    }
  }
  n_alone = __reduce_add_sync(kFull, n_alone);
  mx = __reduce_max_sync(kFull, mx);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) keys += __shfl_xor_sync(kFull, keys, o);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_alone, n_alone);
    atomicMax(&s_mx, mx);
    atomicAdd(&s_keys, keys);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_alone) atomicAdd(&r.stats[8], (unsigned long long)s_alone);
    if (r.ucnt) {
      atomicAdd(&r.stats[2], s_keys);
      atomicMax(&r.stats[3], (unsigned long long)s_mx);
    }
    if (blockIdx.x == 0) r.stats[7] = *r.err;
    __threadfence();
    s_mx = atomicAdd(&r.stats[12], 1ull) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (s_mx && threadIdx.x < 32) {
    __threadfence();
    publish_scalars(r.stats, r.host, threadIdx.x);
  }
}

// What a round starts from, cleared by one launch: up to kClearMax arrays of
// 16-byte units, each filled with one word.  Seven cudaMemsetAsync of mostly a
// few KB cost their launches: 1.5 us of device time and 2.5 us of host each.
constexpr int kClearMax = 8, kClearThreads = 256;
struct ClearArgs {
  uint4* p[kClearMax];
  uint64_t units[kClearMax];
  uint32_t word[kClearMax];
  int n = 0;
  void add(void* a, uint64_t bytes, uint32_t w) {  // bytes rounded up: the arrays are allocated so
    if (!bytes) return;
    p[n] = static_cast<uint4*>(a);
    units[n] = (bytes + 15) / 16;
    word[n++] = w;
  }
};

__global__ void __launch_bounds__(kClearThreads) k_clear(ClearArgs c) {
  overlap_next();
  const uint64_t t0 = blockIdx.x * (uint64_t)kClearThreads + threadIdx.x, stride = (uint64_t)gridDim.x * kClearThreads;
  for (int i = 0; i < c.n; ++i) {
    const uint4 v = make_uint4(c.word[i], c.word[i], c.word[i], c.word[i]);
    for (uint64_t u = t0; u < c.units[i]; u += stride) c.p[i][u] = v;
  }
}

// Nodes outside the round's mask keep their block: signature (pId_{i-1}(u), {})
// -- a node of a graph that has stopped (batched build) then stays with the
// nodes it was grouped with at the level before.
__global__ void k_freeze(uint64_t n_alive, const uint32_t* mask, const uint32_t* prev, uint32_t* ucnt,
                         uint64_t* hash, uint64_t seed, uint64_t hmask) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n_alive; p += (uint64_t)gridDim.x * blockDim.x) {
    if ((mask[p >> 5] >> (p & 31)) & 1u) continue;
    ucnt[p] = 0;
    hash[p] = node_hash(0, prev[p], 0, seed, hmask);
  }
}

// Checked mode: every a[i] (i < n) must be below `bound`.  The kernels that
// index with an array run only after this check has passed on it.
__global__ void k_check_below(const uint32_t* a, uint64_t n, uint64_t bound, uint32_t* err) {
  bool bad = false;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    bad |= (uint64_t)a[i] >= bound;
  if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(err, kErrChecked);
}

// Checked mode: offsets non-decreasing from 0 to m.
__global__ void k_check_offsets_mono(const uint64_t* off, uint64_t n, uint64_t m, uint32_t* err) {
  bool bad = false;
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n; p += (uint64_t)gridDim.x * blockDim.x)
    bad |= off[p] > off[p + 1] || off[p + 1] > m || (p == 0 && off[0] != 0);
  if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(err, kErrChecked);
}

// Level 0 hash: the node label.
__global__ void k_label_hash(uint64_t n, const uint32_t* nlabel, uint64_t* hash, uint64_t seed, uint64_t mask) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n;
       p += (uint64_t)gridDim.x * blockDim.x)
    hash[p] = node_hash(0, nlabel[p], 0, seed, mask);
}

// A level in original order: a coalesced read, a gather and a coalesced write
// per node.  Four nodes per thread in flight (one a time left the loads' latency
// bare: 58 us at 16M nodes).
constexpr int kUnpItems = 4, kUnpThreads = 256;

__global__ void __launch_bounds__(kUnpThreads) k_unpermute(uint64_t n, const uint32_t* o2p, const uint32_t* lvl, uint32_t* out) {
  const uint64_t stride = (uint64_t)gridDim.x * kUnpThreads;
  for (uint64_t o0 = blockIdx.x * (uint64_t)kUnpThreads + threadIdx.x; o0 < n; o0 += stride * kUnpItems) {
    uint32_t x[kUnpItems];
#pragma unroll
    for (int t = 0; t < kUnpItems; ++t)
      if (o0 + t * stride < n) x[t] = __ldg(o2p + o0 + t * stride);
#pragma unroll
    for (int t = 0; t < kUnpItems; ++t)
      if (o0 + t * stride < n) x[t] = __ldg(lvl + x[t]);
#pragma unroll
    for (int t = 0; t < kUnpItems; ++t)
      if (o0 + t * stride < n) out[o0 + t * stride] = x[t];
  }
}

// --------------------------------------------------------------------------
// Relabelling (once per graph)
// --------------------------------------------------------------------------
__device__ __forceinline__ int degree_class(uint64_t d) { return degree_class_of(d); }

constexpr int kClassTile = 1024;

__device__ __forceinline__ int node_class(uint64_t o, uint64_t n, const uint64_t* off, const uint8_t* alive) {
  if (o >= n) return -1;
  if (alive && !alive[o]) return kClassDead;
  return degree_class(off[o + 1] - off[o]);
}

// Within a degree class, nodes are ordered by popularity as a target (hot
// first), so the identifiers that most edges gather sit in a few dense cache
// lines.  Popularity is the in-degree counted on every 2^kHotSampleShift-th
// edge, put into kHotBuckets buckets; it affects speed only, never results.
constexpr int kHotBuckets = 8;
constexpr int kNumOrder = kNumClasses * kHotBuckets;
constexpr int kHotSampleShift = 8;

__device__ __forceinline__ int hot_bucket(uint32_t c) {
  return c >= 1024 ? 0 : c >= 256 ? 1 : c >= 64 ? 2 : c >= 16 ? 3 : c >= 4 ? 4 : c >= 2 ? 5 : c >= 1 ? 6 : 7;
}

__device__ __forceinline__ int order_class(uint64_t o, uint64_t n, const uint64_t* off, const uint8_t* alive,
                                           const uint32_t* hot) {
  const int c = node_class(o, n, off, alive);
  if (c < 0) return -1;
  return c * kHotBuckets + (c == kClassDead ? 0 : hot_bucket(hot[o]));
}

__global__ void k_hot_sample(uint64_t m, const uint32_t* dst0, uint32_t* hot) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; (i << kHotSampleShift) < m; i += stride)
    atomicAdd(&hot[dst0[i << kHotSampleShift]], 1u);
}

__global__ void __launch_bounds__(kClassTile)
    k_class_tile_count(uint64_t n, const uint64_t* off, const uint8_t* alive, const uint32_t* hot, uint64_t ntiles,
                       unsigned long long* tcnt) {
  __shared__ unsigned int c[kNumOrder];
  for (int i = threadIdx.x; i < kNumOrder; i += kClassTile) c[i] = 0;
  __syncthreads();
  const int cls = order_class((uint64_t)blockIdx.x * kClassTile + threadIdx.x, n, off, alive, hot);
  if (cls >= 0) atomicAdd(&c[cls], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < kNumOrder; i += kClassTile) tcnt[(uint64_t)i * ntiles + blockIdx.x] = c[i];
}

// Stable scatter: each tile writes its nodes of order class c in id order at
// the (class, tile) base.
__global__ void __launch_bounds__(kClassTile)
    k_class_tile_scatter(uint64_t n, const uint64_t* off, const uint8_t* alive, const uint32_t* hot, uint64_t ntiles,
                         const unsigned long long* tbase, uint32_t* p2o) {
  __shared__ unsigned int wcnt[kClassTile / 32][kNumOrder];
  for (int i = threadIdx.x; i < (kClassTile / 32) * kNumOrder; i += kClassTile) (&wcnt[0][0])[i] = 0;
  const uint64_t o = (uint64_t)blockIdx.x * kClassTile + threadIdx.x;
  const int cls = order_class(o, n, off, alive, hot);
  const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned same = __match_any_sync(kFull, cls);
  __syncthreads();
  if (cls >= 0 && lane == (unsigned)__ffs(same) - 1u) wcnt[w][cls] = __popc(same);
  __syncthreads();
  if (cls >= 0) {
    unsigned before = __popc(same & ((1u << lane) - 1u));
    for (unsigned i = 0; i < w; ++i) before += wcnt[i][cls];
    p2o[tbase[(uint64_t)cls * ntiles + blockIdx.x] + before] = (uint32_t)o;
  }
}

__global__ void k_order_starts(const unsigned long long* tbase, uint64_t ntiles, unsigned long long* out) {
  for (int i = threadIdx.x; i < kNumOrder; i += blockDim.x) out[i] = tbase[(uint64_t)i * ntiles];
}

__global__ void k_invert(uint64_t n, const uint32_t* p2o, uint32_t* o2p) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n;
       p += (uint64_t)gridDim.x * blockDim.x)
    o2p[p2o[p]] = (uint32_t)p;
}

// deg of internal node p into off[p] (then an exclusive scan makes offsets);
// node labels follow their node.
__global__ void k_relabel_nodes(uint64_t n, const uint32_t* p2o, const uint64_t* off0, const uint32_t* nlab0,
                                unsigned long long* deg, uint32_t* nlab) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t o = p2o[p];
    deg[p] = off0[o + 1] - off0[o];
    nlab[p] = nlab0[o];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) deg[n] = 0;
}

// Copy out-edges to the segment of their source's internal id, relabelling
// targets.  Every lane handles kRelItems edges at a time, all their loads in
// flight together (targets and labels, then the identifier gathers).
constexpr int kRelItems = 4;

// Out-degree <= kSmallMax: one warp per 32 consecutive internal nodes, whose
// edges form one contiguous range of the new table.  Lane k copies edges k,
// k + 32, ... of that range; an edge's node is found by a binary search over
// the 32 new offsets the lanes hold, so reads follow each node's edges in
// order and writes fill the range coalesced.
template <typename TI, typename TO>
__global__ void k_relabel_edges_small(uint64_t n_small, const uint32_t* p2o, const uint32_t* o2p,
                                      const uint64_t* off0, const uint32_t* dst0, const TI* lab0, const uint64_t* off,
                                      uint32_t* dst, TO* lab) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 32 < n_small; w += warps) {
    const uint64_t p = w * 32 + lane;
    const uint64_t base = off[w * 32];
    const uint64_t end = off[min(w * 32 + 32, n_small)];
    // lanes past the last node hold the range's end: an empty node there
    const uint32_t r1 = (uint32_t)((p < n_small ? off[p] : end) - base);
    const uint64_t s0 = p < n_small ? off0[p2o[p]] : 0;
    const uint32_t T = (uint32_t)(end - base);  // at most 32 * kSmallMax
    for (uint32_t k0 = 0; k0 < T; k0 += 32 * kRelItems) {
      uint64_t src[kRelItems];
#pragma unroll
      for (int t = 0; t < kRelItems; ++t) {
        const uint32_t k = min(k0 + lane + 32u * t, T - 1);
        uint32_t j = 0;
#pragma unroll
        for (uint32_t step = 16; step; step >>= 1)
          if (__shfl_sync(kFull, r1, j + step) <= k) j += step;
        src[t] = __shfl_sync(kFull, s0, j) + (k - __shfl_sync(kFull, r1, j));
      }
      uint32_t dv[kRelItems];
      TI lv[kRelItems];
#pragma unroll
      for (int t = 0; t < kRelItems; ++t) {
        if (k0 + lane + 32u * t < T) {
          dv[t] = dst0[src[t]];
          lv[t] = lab0[src[t]];
        }
      }
#pragma unroll
      for (int t = 0; t < kRelItems; ++t)
        if (k0 + lane + 32u * t < T) dv[t] = o2p[dv[t]];
#pragma unroll
      for (int t = 0; t < kRelItems; ++t) {
        const uint32_t k = k0 + lane + 32u * t;
        if (k < T) {
          dst[base + k] = dv[t];
          lab[base + k] = (TO)lv[t];
        }
      }
    }
  }
}

// Deleted nodes (their own class, last): one thread per node; those of
// out-degree <= kSmallMax keep their edges in the new table.
template <typename TI, typename TO>
__global__ void k_relabel_edges_dead(uint64_t p_first, uint64_t p_end, const uint32_t* p2o, const uint32_t* o2p,
                                     const uint64_t* off0, const uint32_t* dst0, const TI* lab0, const uint64_t* off,
                                     uint32_t* dst, TO* lab) {
  for (uint64_t p = p_first + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < p_end;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t o = p2o[p];
    const uint64_t s0 = off0[o], d = off0[o + 1] - s0;
    if (d > (uint64_t)kSmallMax) continue;
    const uint64_t s1 = off[p];
    for (uint64_t i = 0; i < d; ++i) {
      dst[s1 + i] = o2p[dst0[s0 + i]];
      lab[s1 + i] = (TO)lab0[s0 + i];
    }
  }
}

// Copy d edges from src to dst_at in the new table, kRelItems per lane at a
// time, `lane` of `lanes` threads.
template <typename TI, typename TO>
__device__ __forceinline__ void relabel_run(uint64_t src, uint64_t at, uint64_t d, uint32_t lane, uint32_t lanes,
                                            const uint32_t* o2p, const uint32_t* dst0, const TI* lab0, uint32_t* dst,
                                            TO* lab) {
  for (uint64_t i0 = 0; i0 < d; i0 += (uint64_t)lanes * kRelItems) {
    uint32_t dv[kRelItems];
    TI lv[kRelItems];
#pragma unroll
    for (int t = 0; t < kRelItems; ++t) {
      const uint64_t i = i0 + lane + (uint64_t)t * lanes;
      if (i < d) {
        dv[t] = dst0[src + i];
        lv[t] = lab0[src + i];
      }
    }
#pragma unroll
    for (int t = 0; t < kRelItems; ++t)
      if (i0 + lane + (uint64_t)t * lanes < d) dv[t] = o2p[dv[t]];
#pragma unroll
    for (int t = 0; t < kRelItems; ++t) {
      const uint64_t i = i0 + lane + (uint64_t)t * lanes;
      if (i < d) {
        dst[at + i] = dv[t];
        lab[at + i] = (TO)lv[t];
      }
    }
  }
}

// Out-degree 65..4096: one warp per node.
template <typename TI, typename TO>
__global__ void k_relabel_edges_large(uint64_t p_first, uint64_t p_end, const uint32_t* p2o, const uint32_t* o2p,
                                      const uint64_t* off0, const uint32_t* dst0, const TI* lab0, const uint64_t* off,
                                      uint32_t* dst, TO* lab) {
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t p = p_first + ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5); p < p_end;
       p += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
    const uint32_t o = p2o[p];
    const uint64_t s0 = off0[o];
    relabel_run(s0, off[p], off0[o + 1] - s0, lane, 32u, o2p, dst0, lab0, dst, lab);
  }
}

// Hub edges: one CTA per chunk of kHubChunk edges (chunks as in the hub
// signature kernels: hub index, first edge in the new table, length).
template <typename TI, typename TO>
__global__ void k_relabel_edges_hub(uint64_t hub_first, const uint4* chunks, const uint32_t* p2o, const uint32_t* o2p,
                                    const uint64_t* off0, const uint32_t* dst0, const TI* lab0, const uint64_t* off,
                                    uint32_t* dst, TO* lab) {
  const uint4 c = chunks[blockIdx.x];
  const uint64_t p = hub_first + c.x;
  const uint64_t begin = ((uint64_t)c.z << 32) | c.y;
  const uint64_t src = off0[p2o[p]] + (begin - off[p]);
  relabel_run(src, begin, c.w, threadIdx.x, blockDim.x, o2p, dst0, lab0, dst, lab);
}

template <typename TI, typename TO>
void relabel_edges(Store& s, const uint64_t* off0, const uint32_t* dst0, const TI* lab0, TO* lab, int sms) {
  const uint64_t n = s.n;
  const uint32_t* o2p = ptr<uint32_t>(s.o2p);
  const uint64_t* off = ptr<uint64_t>(s.offsets);
  uint32_t* dst = ptr<uint32_t>(s.dst);
  const uint64_t n_small = s.class_start[kClassWarp];
  if (n_small) {
    const unsigned g1 = (unsigned)std::min<uint64_t>(grid_for(n_small, 256), (uint64_t)sms * 32);
    k_relabel_edges_small<TI, TO><<<g1, 256, 0, s.stream>>>(n_small, ptr<uint32_t>(s.p2o), o2p, off0, dst0, lab0, off,
                                                           dst, lab);
  }
  const uint64_t dead = s.class_start[kClassDead];
  if (n > dead)
    k_relabel_edges_dead<TI, TO><<<(unsigned)std::min<uint64_t>(grid_for(n - dead, 256), (uint64_t)sms * 8), 256, 0,
                                   s.stream>>>(dead, n, ptr<uint32_t>(s.p2o), o2p, off0, dst0, lab0, off, dst, lab);
  const uint64_t pf = s.class_start[kClassWarp], pe = s.class_start[kClassHub];
  if (pe > pf) {
    const unsigned g2 = (unsigned)std::min<uint64_t>(grid_for((pe - pf) * 32, 256), (uint64_t)sms * 32);
    k_relabel_edges_large<TI, TO><<<g2, 256, 0, s.stream>>>(pf, pe, ptr<uint32_t>(s.p2o), o2p, off0, dst0, lab0, off,
                                                           dst, lab);
  }
  if (s.n_hub_chunks)
    k_relabel_edges_hub<TI, TO><<<(unsigned)s.n_hub_chunks, 256, 0, s.stream>>>(
        s.class_start[kClassHub], ptr<uint4>(s.hub_chunks), ptr<uint32_t>(s.p2o), o2p, off0, dst0, lab0, off, dst, lab);
}

// Exclusive scan of a uint64 array in place, with an optional copy.
__global__ void __launch_bounds__(kScanThreads) k_tile_sum64(const uint64_t* a, uint64_t n, uint64_t* bsum) {
  __shared__ unsigned long long red[kScanThreads / 32];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  unsigned long long c = 0;
#pragma unroll
  for (int t = 0; t < kScanItems; ++t) {
    const uint64_t i = base + (uint64_t)t * kScanThreads + threadIdx.x;
    if (i < n) c += a[i];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) tot += red[w];
    bsum[blockIdx.x] = tot;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_tile_scan64(uint64_t* a, uint64_t n, const uint64_t* bsum,
                                                                uint64_t* copy) {
  __shared__ unsigned long long wt[kScanThreads / 32];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  unsigned long long f[kScanItems];
  unsigned long long c = 0;
#pragma unroll
  for (int t = 0; t < kScanItems; ++t) {
    f[t] = base + t < n ? a[base + t] : 0ull;
    c += f[t];
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned long long y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wt[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned long long t = wt[lane];
    unsigned long long xx = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long y = __shfl_up_sync(kFull, xx, o);
      if (lane >= o) xx += y;
    }
    wt[lane] = xx - t;
  }
  __syncthreads();
  unsigned long long run = bsum[blockIdx.x] + wt[w] + (x - c);
#pragma unroll
  for (int t = 0; t < kScanItems; ++t) {
    if (base + t < n) {
      a[base + t] = run;
      if (copy) copy[base + t] = run;
    }
    run += f[t];
  }
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
Status scan64(Store& s, uint64_t* a, uint64_t n, uint64_t* copy) {
  if (!n) return Status::Ok();
  const uint64_t tiles = (n + kScanTile - 1) / kScanTile;
  Status st = ensure(s, s.bsum, std::max<uint64_t>(tiles, 64) * 8);
  if (!st.ok()) return st;
  uint64_t* bs = ptr<uint64_t>(s.bsum);
  k_tile_sum64<<<(unsigned)tiles, kScanThreads, 0, s.stream>>>(a, n, bs);
  k_scan_tiles<<<1, kScanThreads, 0, s.stream>>>(bs, tiles, ptr<unsigned long long>(s.d_scalars) + 15);
  k_tile_scan64<<<(unsigned)tiles, kScanThreads, 0, s.stream>>>(a, n, bs, copy);
  return launch_check("scan64");
}

template <typename LabelT, typename K>
cudaError_t set_smem_attrs_label() {
  cudaError_t e = cudaSuccess;
  for (auto kernel : {k_sig_cta<kChunkThreads, kPlain, LabelT, K>, k_sig_cta<kChunkThreads, kWithDup, LabelT, K>,
                      k_sig_cta<kChunkThreads, kMarking, LabelT, K>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cta_node_smem<kChunkThreads, K>());
  for (auto kernel : {k_hub_chunk<kPlain, LabelT, K>, k_hub_chunk<kWithDup, LabelT, K>, k_hub_pieces<kPlain, LabelT, K>,
                      k_hub_pieces<kWithDup, LabelT, K>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hub_chunk_smem<K>());
  return e;
}

template <typename K>
Status set_smem_attrs_for() {
  cudaError_t e = set_smem_attrs_label<uint8_t, K>();

  if (e == cudaSuccess) e = set_smem_attrs_label<uint32_t, K>();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hub_bucket<K, kHubUcaps[0]>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(BucketSmem<K, kHubUcaps[0]>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hub_bucket<K, kHubUcaps[1]>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(BucketSmem<K, kHubUcaps[1]>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_hub_bucket<K, kHubUcaps[2]>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(BucketSmem<K, kHubUcaps[2]>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_verify_long<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)verify_ws_bytes<K>());
  return cuda_check(e, "cudaFuncSetAttribute");
}

Status set_smem_attrs(int device) {
  static PerDevice done;
  Status st;
  done.get(device, [&] {
    st = set_smem_attrs_for<uint32_t>();
    if (st.ok()) st = set_smem_attrs_for<uint64_t>();
    return st.ok() ? 1 : 0;
  });
  return st;
}

// Wait for the stream; the scalars are those its last kernel put into pinned memory.
Status await_scalars(Store& s, uint64_t* out) {
  Status st = cuda_check(cudaStreamSynchronize(s.stream), "stream sync");
  if (st.ok()) std::memcpy(out, s.h_scalars.p, 16 * sizeof(uint64_t));
  return st;
}

Status read_scalars(Store& s, uint64_t* out) {
  Status st = cuda_check(cudaMemcpyAsync(s.h_scalars.p, s.d_scalars.p, 16 * sizeof(uint64_t),
                                         cudaMemcpyDeviceToHost, s.stream), "read scalars");
  if (!st.ok()) return st;
  st = cuda_check(cudaStreamSynchronize(s.stream), "stream sync");
  if (!st.ok()) return st;
  std::memcpy(out, s.h_scalars.p, 16 * sizeof(uint64_t));
  return Status::Ok();
}

// Checked mode: bring a check kernel's outcome to the host.  Returns CHECKED if
// an index check failed (the kernels that would use the array are not run).
Status checked_outcome(Store& s, const char* what) {
  uint32_t e = 0;
  Status st = launch_check(what);
  if (st.ok()) st = cuda_check(cudaMemcpyAsync(&e, s.d_err.p, 4, cudaMemcpyDeviceToHost, s.stream), what);
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), what);
  if (!st.ok()) return st;
  if (e & kErrChecked) return Status::Err(KBISIM_ERR_CHECKED, std::string("index check failed: ") + what);
  return Status::Ok();
}

Status check_below(Store& s, const uint32_t* a, uint64_t n, uint64_t bound, const char* what) {
  if (!n) return Status::Ok();
  const unsigned g = (unsigned)std::min<uint64_t>(grid_for(n, 256), (uint64_t)sm_count(s.device) * 16);
  k_check_below<<<g, 256, 0, s.stream>>>(a, n, bound, ptr<uint32_t>(s.d_err));
  return checked_outcome(s, what);
}

uint64_t table_capacity(uint64_t n) { return table_slots(n); }

void launch_insert(Store& s, const GroupArgs& g, const uint32_t* list, uint64_t count) {
  static PerDevice known;
  const unsigned res = resident_grid(k_group_insert, kInsThreads, 0, s.device, known);
  launch_chained(s, k_group_insert, (unsigned)std::min<uint64_t>((count + kInsChunk - 1) / kInsChunk, res),
                    kInsThreads, 0, g, list, count);
}

template <typename K>
void launch_verify_long(Store& s, const GroupArgs& g, const VerifyArgs& v, uint64_t count) {
  static PerDevice known;
  const unsigned res = resident_grid(k_verify_long<K>, kVerThreads, verify_ws_bytes<K>(), s.device, known);
  launch_chained(s, k_verify_long<K>, (unsigned)std::min<uint64_t>((count + 31) / 32, res), kVerThreads,
                    verify_ws_bytes<K>(), g, v);
}

// The pairs k_group_verify left (at most `count`).
Status launch_pairs(Store& s, const GroupArgs& g, const VerifyArgs& v, uint64_t count) {
  if (v.key64) launch_verify_long<uint64_t>(s, g, v, count);
  else launch_verify_long<uint32_t>(s, g, v, count);
  return launch_check("k_verify_long");
}

// Exact comparison of `count` nodes (of `list`, or all) with the head of their
// hash: the short signatures, then (with_pairs) the others.
Status launch_verify(Store& s, const GroupArgs& g, const VerifyArgs& v, const uint32_t* list, uint64_t count,
                     bool with_pairs) {
  static PerDevice known;
  const unsigned res = resident_grid(k_group_verify, kVerNodeThreads, 0, s.device, known);
  launch_chained(s, k_group_verify, (unsigned)std::min<uint64_t>(grid_for(count, kVerTile), res), kVerNodeThreads,
                    0, g, v, list, count);
  Status st = launch_check("k_group_verify");
  return st.ok() && v.mode != 0 && with_pairs ? launch_pairs(s, g, v, count) : st;
}

// After a first insert + verify pass (scalars in h): regroup the nodes a hash
// collision left unresolved until none is left.  The unresolved nodes hold
// whole classes; the smallest unresolved node of each hash group heads its
// class, so every pass settles at least one class per group (a pass that
// settles nothing is an error).
Status settle_unresolved(Store& s, const GroupArgs& g, const VerifyArgs& v, uint64_t* h) {
  Status st;
  unsigned long long* sc = ptr<unsigned long long>(s.d_scalars);
  uint64_t unresolved_n = h[1];
  int cur = 0;
  while (unresolved_n > 0) {
    const uint64_t cap = table_capacity(unresolved_n);
    GroupArgs g2 = g;
    g2.tmask = cap - 1;
    g2.alone = nullptr;  // no listed node is (the flags may be the new level's already)
    VerifyArgs v2 = v;
    v2.out_list = ptr<uint32_t>(s.ulist[cur ^ 1]);
    v2.n_out = sc + 5;
    {
      TimedScope ts(s, KBISIM_KERNEL_OTHER, v.mode ? 3 : 2);
      cudaMemsetAsync(s.table.p, 0xFF, cap * 8, s.stream);
      cudaMemsetAsync(sc + 5, 0, 16, s.stream);   // [5] and [6]
      cudaMemsetAsync(sc + 10, 0, 8, s.stream);
      launch_insert(s, g2, ptr<uint32_t>(s.ulist[cur]), unresolved_n);
      st = launch_verify(s, g2, v2, ptr<uint32_t>(s.ulist[cur]), unresolved_n, true);
    }
    if (!st.ok()) return st;
    if (!(st = read_scalars(s, h)).ok()) return st;
    if (h[5] >= unresolved_n)
      return Status::Err(KBISIM_ERR_TIMEOUT, "collision repair made no progress");
    unresolved_n = h[5];
    cur ^= 1;
  }
  return Status::Ok();
}

// Table slots of a grouping that inserts `ins` nodes.
uint64_t group_slots(const Store& s, uint64_t ins) { return std::min<uint64_t>(s.tcap, table_capacity(ins)); }

// Arguments of a grouping over the stored graph.
GroupArgs group_args(Store& s, uint64_t slots) {
  GroupArgs g;
  g.hash = ptr<uint64_t>(s.hash);
  g.p2o = ptr<uint32_t>(s.p2o);
  g.o2p = ptr<uint32_t>(s.o2p);
  g.table = ptr<unsigned long long>(s.table);
  g.tmask = slots - 1;
  g.slot = ptr<uint32_t>(s.slot);
  g.rep = ptr<uint32_t>(s.rep);
  g.err = ptr<uint32_t>(s.d_err);
  g.alone = nullptr;
  g.read_first = 0;
  g.d_count = nullptr;
  g.seen = nullptr;
  g.seen_mask = 0;
  return g;
}

VerifyArgs verify_args(Store& s, int mode, const uint32_t* prev, bool key64) {
  unsigned long long* sc = ptr<unsigned long long>(s.d_scalars);
  VerifyArgs v;
  v.mode = mode;
  v.key64 = key64 ? 1 : 0;
  v.nlabel = ptr<uint32_t>(s.nlabel);
  v.prev = prev;
  v.ucnt = ptr<uint32_t>(s.ucnt);
  v.off = ptr<uint64_t>(s.offsets);
  v.sigkey = s.sigkey.p;
  v.out_list = ptr<uint32_t>(s.ulist[0]);
  v.n_out = sc + 1;
  v.n_collided = sc + 4;
  v.long_list = ptr<uint32_t>(s.long_pairs);
  v.pair_cap = std::max<uint64_t>(s.n, 1);
  v.n_mid = sc + 10;
  v.n_long = sc + 6;
  v.hbits = ptr<uint32_t>(s.hbits);
  v.member = ptr<uint8_t>(s.member);
  v.keep = false;
  return v;
}

// Bits of the filter before the grouping of `ins` nodes (0 = none): 8 to 16 per
// node, two bitmaps, so at most 4 of the 8 bytes per node of the pair lists,
// which nothing uses before the comparison.  `first`: the grouping of round 1.
uint64_t filter_bits(const Store& s, uint64_t ins, bool first) {
  if (ins <= kFilterNodes) return 0;
  if (first) {
    const bool many_values = s.counts[0] << s.label_bits >= kFilterValues;
    if (s.class_start[many_values ? 1 : 2] > s.n_alive / 20) return 0;  // nodes of out-degree 0, or 0 and 1
  }
  return 4 * table_slots(ins);
}

// Clear what a level's signatures and grouping start from: error flags,
// scalars, the marks of the canonical numbering, the hash table for `ins`
// inserted nodes or the filter of `bits` before it (0 = none), and, with hubs,
// their buckets' cursors and totals.
// `keep`: the head marks of the level before stay.
Status clear_round(Store& s, uint64_t ins, uint64_t bits, bool hubs, bool keep) {
  ClearArgs c;
  c.add(s.d_err.p, 16, 0u);
  c.add(s.d_scalars.p, 16 * 8, 0u);
  if (!keep) c.add(s.hbits.p, (s.n + 31) / 32 * 4, 0u);
  c.add(s.member.p, s.n, 0u);
  if (bits) c.add(s.long_pairs.p, bits / 4, 0u);
  else c.add(s.table.p, group_slots(s, ins) * 8, ~0u);
  if (hubs) {
    c.add(s.hub_cursor.p, s.n_hub_buckets * 4, 0u);
    c.add(s.hub_acc.p, s.n_hub * 24, 0u);
    c.add(s.hub_err.p, s.n_hub * 4, 0u);
  }
  uint64_t units = 0;
  for (int i = 0; i < c.n; ++i) units += c.units[i];
  TimedScope ts(s, KBISIM_KERNEL_OTHER, 1);
  k_clear<<<(unsigned)std::min<uint64_t>(grid_for(units, kClearThreads), (uint64_t)sm_count(s.device) * 8),
            kClearThreads, 0, s.stream>>>(c);
  return launch_check("k_clear");
}

// Nodes a level's grouping inserts: all, or those not alone in their block at
// the level before.
uint64_t insert_count(const Store& s, bool use_alone) {
  return use_alone ? s.n_alive - std::min(s.n_alive, s.n_alone) : s.n_alive;
}

// Group the nodes by exact signature (by label in mode 0) and number the
// blocks, into pid.  clear_round has run.  The host waits once, at the end:
// the comparison of long signatures takes its pairs' number from the device,
// and the numbering is launched before the host knows whether a hash collision
// left nodes unresolved; if one did they are settled and it runs again.
// `first`: a level whose blocks are few, so that long signatures repeat.
// `keep`: hbits and rep hold the level before (Store::heads_level).
// *hub_flags (mode 1): overflow flags of the hub passes before; when set, the
// signatures were incomplete and nothing else is returned.
//
// Scalars used per round (uint64 words of Store::d_scalars):
//  [1] unresolved after the first pass, [2] key total, [3] largest signature,
//  [4] collided nodes, [5] unresolved after a repair pass, [6] and [10] pairs
//  with long and with middle signatures, [7] error flags copy, [8] nodes alone
//  in their block, [9] and [12] tickets of k_head_ranks and k_pid_fill, [11] nodes the filter left to
//  the grouping, [15] the number of blocks.
Status group_and_rank(Store& s, int mode, const uint32_t* prev, bool key64, uint32_t* pid, uint64_t* blocks,
                      uint64_t* collided, bool with_stats, uint64_t* keys, uint64_t* maxsig, bool use_alone,
                      bool first, bool keep, uint32_t* hub_flags) {
  const uint64_t n = s.n, na = s.n_alive;
  Status st;
  unsigned long long* sc = ptr<unsigned long long>(s.d_scalars);
  GroupArgs g = group_args(s, group_slots(s, insert_count(s, use_alone)));
  g.alone = use_alone ? ptr<uint8_t>(s.alone) : nullptr;
  g.read_first = mode == 0 ? 1 : 0;
  VerifyArgs v = verify_args(s, mode, prev, key64);
  v.keep = keep;
  const uint64_t words = (n + 31) / 32;
  // the comparison of longer signatures runs unless the level before had none
  // (the host sees their number at the end, and then compares them and
  // numbers the blocks again)
  const bool with_pairs = first || s.checked || s.pairs_last;
  uint64_t h[16] = {0};
  // canonical renumbering
  RankArgs r;
  r.n = n;
  r.n_alive = na;
  r.rep = g.rep;
  r.p2o = g.p2o;
  r.ucnt = with_stats ? ptr<uint32_t>(s.ucnt) : nullptr;
  r.hrank = ptr<uint2>(s.hword);
  r.tbase = ptr<uint32_t>(s.bsum);
  r.err = ptr<uint32_t>(s.d_err);
  r.member = ptr<uint8_t>(s.member);
  r.alone = ptr<uint8_t>(s.alone);
  r.alone_bits = s.dup_valid ? ptr<uint32_t>(s.alone_bits) : nullptr;
  r.pid = pid;
  r.host = ptr<unsigned long long>(s.h_scalars);
  r.stats = sc;
  auto renumber = [&]() -> Status {
    static PerDevice known;
    TimedScope ts(s, KBISIM_KERNEL_RENUMBER, n ? 2 : 0);
    if (!n) return Status::Ok();
    launch_chained(s, k_head_ranks, (unsigned)((words + kRankTile - 1) / kRankTile), kRankThreads, 0,
                      ptr<uint32_t>(s.hbits), words, ptr<uint2>(s.hword), ptr<uint32_t>(s.bsum), sc + 9, sc + 15);
    launch_chained(s, k_pid_fill,
                      (unsigned)std::min<uint64_t>(grid_for(n, kFillThreads * kFillItems),
                                                   resident_grid(k_pid_fill, kFillThreads, 0, s.device, known)),
                      kFillThreads, 0, r);
    return launch_check("renumber");
  };
  const uint64_t bits = mode ? filter_bits(s, insert_count(s, use_alone), first) : 0;
  if (na) {
    const uint32_t* list = nullptr;
    {
      TimedScope ts(s, KBISIM_KERNEL_GROUP, bits ? 4 : 1);
      if (bits) {
        uint32_t* cand = ptr<uint32_t>(s.ulist[1]);
        static PerDevice known_filter, known_select;
        g.seen = ptr<uint2>(s.long_pairs);
        g.seen_mask = bits - 1;
        const uint64_t tiles = grid_for(na, kFilTile);
        launch_chained(s, k_group_filter,
                       (unsigned)std::min<uint64_t>(tiles, resident_grid(k_group_filter, kFilThreads, 0, s.device, known_filter)),
                       kFilThreads, 0, g, na);
        launch_chained(s, k_group_select,
                       (unsigned)std::min<uint64_t>(tiles, resident_grid(k_group_select, kFilThreads, 0, s.device, known_select)),
                       kFilThreads, 0, g, v, na, cand, sc + 11);
        list = cand;
        g.alone = nullptr;  // none of the listed nodes is
        g.d_count = sc + 11;
        launch_chained(s, k_table_clear, (unsigned)sm_count(s.device) * 8, kFilThreads, 0, g);
      }
      launch_insert(s, g, list, na);
    }
    if (!(st = launch_check("k_group_insert")).ok()) return st;
    TimedScope ts(s, KBISIM_KERNEL_VERIFY, mode && with_pairs ? 2 : 1);
    if (!(st = launch_verify(s, g, v, list, na, with_pairs)).ok()) return st;
    g.d_count = nullptr;
  }
  if (s.checked) {  // representatives are checked before the numbering uses them
    if (!(st = read_scalars(s, h)).ok()) return st;
    if (!(st = settle_unresolved(s, g, v, h)).ok()) return st;
    if (!(st = check_below(s, g.rep, na, n, "block heads")).ok()) return st;
  }
  if (!(st = renumber()).ok()) return st;
  if (!n) {
    *blocks = *collided = s.n_alone = 0;
    return read_scalars(s, h);
  }
  if (!(st = await_scalars(s, h)).ok()) return st;
  if (hub_flags && (*hub_flags = (uint32_t)h[7] & (kErrHubOverflow | kErrHubSet))) return Status::Ok();
  const bool missed = !with_pairs && mode && (h[6] || h[10]);
  s.pairs_last = h[6] || h[10];
  if ((h[1] || missed) && !s.checked) {
    if (missed) {
      TimedScope ts(s, KBISIM_KERNEL_VERIFY, 1);
      if (!(st = launch_pairs(s, g, v, na)).ok()) return st;
      if (!(st = read_scalars(s, h)).ok()) return st;
    }
    if (!(st = settle_unresolved(s, g, v, h)).ok()) return st;
    cudaMemsetAsync(sc + 2, 0, 16, s.stream);      // [2] and [3]
    cudaMemsetAsync(sc + 8, 0, 5 * 8, s.stream);   // [8] .. [12]
    if (!(st = renumber()).ok()) return st;
    if (!(st = await_scalars(s, h)).ok()) return st;
  }
  *collided = h[4];
  *blocks = n ? h[15] : 0;  // heads
  if (s.checked && !(st = check_below(s, pid, na, *blocks, "identifiers")).ok()) return st;
  s.n_alone = h[8];
  if (keys) *keys = h[2];
  if (maxsig) *maxsig = h[3];
  const uint32_t e = (uint32_t)h[7];
  if (e & kErrProbe) return Status::Err(KBISIM_ERR_TIMEOUT, "hash table probe bound exceeded");
  if (e & kErrChecked) return Status::Err(KBISIM_ERR_CHECKED, "device bounds check failed");
  return Status::Ok();
}

// (Re)build the per-hub bucket table for the bucket size s.hub_ucap and the
// current extra bits: hub i has 2^(bits_i + extra) buckets of cap_i key words
// each, bits_i the least with degree <= (hub_ucap / 2) << bits_i, cap_i twice
// the mean bucket load plus a margin (at most hub_ucap).
Status hub_layout(Store& s) {
  Status st;
  std::vector<uint32_t> bits(s.n_hub), cap(s.n_hub);
  std::vector<uint64_t> bbase(s.n_hub + 1, 0), tbase(s.n_hub, 0);
  uint64_t words = 0;
  const uint64_t target = s.hub_ucap / 2;
  for (uint64_t i = 0; i < s.n_hub; ++i) {
    uint32_t db = 0;
    while ((target << db) < s.h_hub_deg[i]) ++db;
    bits[i] = db + s.h_hub_xbits[i];
    const uint64_t nb = 1ull << bits[i];
    bbase[i + 1] = bbase[i] + nb;
    const uint64_t mean = (s.h_hub_deg[i] + nb - 1) / nb;
    cap[i] = (uint32_t)std::min<uint64_t>(s.h_hub_deg[i], std::min<uint64_t>(s.hub_ucap, 2 * mean + 256)
                                                                << s.h_hub_shift[i]);
    tbase[i] = words;
    words += nb * cap[i];
  }
  s.n_hub_buckets = bbase[s.n_hub];
  s.hub_tmp_words = words;
  std::vector<uint32_t> bhub(s.n_hub_buckets);
  for (uint64_t i = 0; i < s.n_hub; ++i)
    for (uint64_t b = bbase[i]; b < bbase[i + 1]; ++b) bhub[b] = (uint32_t)i;
  if (!(st = ensure(s, s.hub_bits, s.n_hub * 4)).ok()) return st;
  if (!(st = ensure(s, s.hub_cap, s.n_hub * 4)).ok()) return st;
  if (!(st = ensure(s, s.hub_bbase, (s.n_hub + 1) * 8)).ok()) return st;
  if (!(st = ensure(s, s.hub_tbase, s.n_hub * 8)).ok()) return st;
  if (!(st = ensure(s, s.bucket_hub, s.n_hub_buckets * 4)).ok()) return st;
  if (!(st = ensure(s, s.hub_cursor, (s.n_hub_buckets * 4 + 15) & ~15ull)).ok()) return st;
  if (!(st = ensure(s, s.hub_acc, (s.n_hub * 24 + 15) & ~15ull)).ok()) return st;
  if (!(st = ensure(s, s.hub_mode, s.n_hub)).ok()) return st;
  if (!(st = ensure(s, s.hub_force, s.n_hub)).ok()) return st;
  if (!(st = ensure(s, s.hub_err, (s.n_hub * 4 + 15) & ~15ull)).ok()) return st;
  cudaMemcpyAsync(s.hub_force.p, s.h_hub_force.data(), s.n_hub, cudaMemcpyHostToDevice, s.stream);
  cudaMemcpyAsync(s.hub_bits.p, bits.data(), s.n_hub * 4, cudaMemcpyHostToDevice, s.stream);
  cudaMemcpyAsync(s.hub_cap.p, cap.data(), s.n_hub * 4, cudaMemcpyHostToDevice, s.stream);
  cudaMemcpyAsync(s.hub_bbase.p, bbase.data(), (s.n_hub + 1) * 8, cudaMemcpyHostToDevice, s.stream);
  cudaMemcpyAsync(s.hub_tbase.p, tbase.data(), s.n_hub * 8, cudaMemcpyHostToDevice, s.stream);
  cudaMemcpyAsync(s.bucket_hub.p, bhub.data(), s.n_hub_buckets * 4, cudaMemcpyHostToDevice, s.stream);
  return cuda_check(cudaStreamSynchronize(s.stream), "hub layout");
}

// The bucket pass with buckets of at most U key words: one resident wave of CTAs.
template <typename K, int U>
void launch_hub_bucket(Store& s, const SigArgs& a, const HubArgs& h) {
  static PerDevice known;
  const unsigned g = (unsigned)std::min<uint64_t>(
      s.n_hub_buckets, resident_grid(k_hub_bucket<K, U>, kBucketThreads, sizeof(BucketSmem<K, U>), s.device, known));
  launch_chained(s, k_hub_bucket<K, U>, g, kBucketThreads, sizeof(BucketSmem<K, U>), a, h, s.n_hub_buckets);
}

// One pass over the hubs of a.fmask (NULL = all).  `cleared`: clear_round has
// cleared the buckets' cursors, totals and flags.
template <typename LabelT, typename K>
Status launch_hubs(Store& s, const SigArgs& a, bool cleared) {
  Status st = ensure(s, s.hub_tmp, s.hub_tmp_words * sizeof(K));
  if (!st.ok()) return st;
  HubArgs h;
  h.first = s.class_start[kClassHub];
  h.hub_bits = ptr<uint32_t>(s.hub_bits);
  h.hub_bbase = ptr<uint64_t>(s.hub_bbase);
  h.hub_cap = ptr<uint32_t>(s.hub_cap);
  h.hub_tbase = ptr<uint64_t>(s.hub_tbase);
  h.bucket_hub = ptr<uint32_t>(s.bucket_hub);
  h.chunks = ptr<uint4>(s.hub_chunks);
  h.cursor = ptr<uint32_t>(s.hub_cursor);
  h.hub_cur = ptr<unsigned long long>(s.hub_acc);
  h.hub_term = reinterpret_cast<uint32_t*>(h.hub_cur + s.n_hub);
  const bool small = chained(s);
  h.done = small ? reinterpret_cast<uint32_t*>(h.hub_cur + 2 * s.n_hub) : nullptr;
  h.tmp = s.hub_tmp.p;
  h.mode = ptr<uint8_t>(s.hub_mode);
  h.force = ptr<uint8_t>(s.hub_force);
  h.hub_err = ptr<uint32_t>(s.hub_err);
  // each hub's chunks run either the deduplicating pass or the plain
  // scatter, as its key sample says; both kernels cover all chunks and
  // skip those of the other kind
  TimedScope ts(s, KBISIM_KERNEL_SIG_HUB, small ? 3 : 5);
  if (!cleared) {
    cudaMemsetAsync(h.cursor, 0, s.n_hub_buckets * 4, s.stream);
    cudaMemsetAsync(s.hub_acc.p, 0, s.n_hub * 24, s.stream);
    cudaMemsetAsync(s.hub_err.p, 0, s.n_hub * 4, s.stream);
  }
  launch_chained(s, k_hub_sample<LabelT, K>, (unsigned)((s.n_hub + 7) / 8), 256, 0, a, h, s.n_hub);
  const bool dup = a.dup && a.dup_hubs;
  const unsigned pieces = (unsigned)s.n_hub_chunks;
  if (small) {
    launch_chained(s, dup ? k_hub_pieces<kWithDup, LabelT, K> : k_hub_pieces<kPlain, LabelT, K>, pieces, kChunkThreads,
                   hub_chunk_smem<K>(), a, h);
  } else {
    launch_chained(s, dup ? k_hub_chunk<kWithDup, LabelT, K> : k_hub_chunk<kPlain, LabelT, K>, pieces, kChunkThreads,
                   hub_chunk_smem<K>(), a, h);
    launch_chained(s, dup ? k_hub_scatter<kWithDup, LabelT, K> : k_hub_scatter<kPlain, LabelT, K>, pieces, kChunkThreads,
                   0, a, h);
  }
  if (s.hub_ucap == (uint32_t)kHubUcaps[1]) launch_hub_bucket<K, kHubUcaps[1]>(s, a, h);
  else if (s.hub_ucap == (uint32_t)kHubUcaps[2]) launch_hub_bucket<K, kHubUcaps[2]>(s, a, h);
  else launch_hub_bucket<K, kHubUcaps[0]>(s, a, h);
  if (!small) launch_chained(s, k_hub_finish, (unsigned)((s.n_hub + 255) / 256), 256, 0, a, h, s.n_hub);
  return launch_check("hub kernels");
}

// After a hub pass with overflow flags: grow the buckets of the hubs it
// raised them for, and make a->fmask the mask of those hubs (the others'
// signatures are written).
Status grow_hubs(Store& s, SigArgs* a) {
  std::vector<uint32_t> herr(s.n_hub);
  std::vector<uint8_t> hmode(s.n_hub);
  Status st = cuda_check(cudaMemcpyAsync(herr.data(), s.hub_err.p, s.n_hub * 4, cudaMemcpyDeviceToHost, s.stream),
                         "hub flags");
  if (st.ok())
    st = cuda_check(cudaMemcpyAsync(hmode.data(), s.hub_mode.p, s.n_hub, cudaMemcpyDeviceToHost, s.stream),
                    "hub modes");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return st;
  s.hub_grew = true;
  for (uint64_t i = 0; i < s.n_hub; ++i) {
    // a bucket overflowed (a key repeated many times): larger buckets for
    // the hub, up to its degree, or, once the scatter has overflowed
    // buckets kHubScatterShiftMax times larger than the first, the
    // deduplicating pass; too many distinct keys in a bucket: more buckets
    if (herr[i] & kErrHubOverflow) {
      if (hmode[i] && s.h_hub_shift[i] >= kHubScatterShiftMax) s.h_hub_force[i] = 1;
      else s.h_hub_shift[i] += 1;
    }
    if (herr[i] & kErrHubSet) s.h_hub_xbits[i] += 1;
  }
  if (!(st = hub_layout(s)).ok()) return st;
  // the repeat's mask: the words of the hub id range, bits of the failed hubs
  const uint64_t first = s.class_start[kClassHub], w0 = first >> 5, w1 = (first + s.n_hub + 31) >> 5;
  std::vector<uint32_t> bits(w1 - w0, 0u);
  for (uint64_t i = 0; i < s.n_hub; ++i)
    if (herr[i]) bits[((first + i) >> 5) - w0] |= 1u << ((first + i) & 31);
  if (!(st = ensure(s, s.hub_retry, (w1 + 1) * 4)).ok()) return st;
  st = cuda_check(cudaMemcpyAsync(ptr<uint32_t>(s.hub_retry) + w0, bits.data(), bits.size() * 4,
                                  cudaMemcpyHostToDevice, s.stream), "hub repeat mask");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "hub repeat mask");  // the host vector goes away
  if (!st.ok()) return st;
  a->fmask = ptr<uint32_t>(s.hub_retry);
  return Status::Ok();
}

constexpr int kHubAttempts = 40;
constexpr uint64_t kHubCalmNodes = 4u << 20;
// Edges from which a graph's duplicates are marked: below, a round is latency
// and the extra words only cost.  The rounds from level 2 on use the marks
// (256M-edge powerlaw graph, five rounds 9.70 against 11.08 ms, three 6.89
// against 7.30, two 5.47 against 5.40; 16M edges, three rounds 0.64 against
// 0.71, two 0.51 against 0.53).  Marking takes about one pass over the edges, so
// a graph refined once is not marked, nor one of more than kMarkEdgesTwoRounds
// edges whose refinement ends after two rounds; and the hubs, the larger half of
// the work (1.4 of 2.4 ms at 256M edges), are marked one refinement later.
constexpr uint64_t kMarkEdges = 8u << 20, kMarkEdgesTwoRounds = 32ull << 20;

// Hub passes until no bucket overflows, the host waiting for each.
template <typename LabelT, typename K>
Status run_hubs(Store& s, const SigArgs& a) {
  SigArgs ah = a;
  for (int attempt = 0;; ++attempt) {
    Status st = launch_hubs<LabelT, K>(s, ah, false);
    if (!st.ok()) return st;
    uint32_t e = 0;
    st = cuda_check(cudaMemcpyAsync(&e, s.d_err.p, 4, cudaMemcpyDeviceToHost, s.stream), "read err");
    if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
    if (!st.ok()) return st;
    if (!(e & (kErrHubOverflow | kErrHubSet))) return Status::Ok();
    if (attempt >= kHubAttempts) return Status::Err(KBISIM_ERR_TIMEOUT, "hub bucket overflow persists");
    if (!(st = grow_hubs(s, &ah)).ok()) return st;
    cudaMemsetAsync(s.d_err.p, 0, 4, s.stream);
  }
}

// Signatures of every node class.  With `defer`, the hubs run one pass over
// what clear_round has cleared, and the caller looks at the overflow flags
// once the round's other kernels have run (group_and_rank, grow_hubs);
// otherwise they are complete on return.
template <typename LabelT, typename K>
Status run_signatures(Store& s, const SigArgs& a, bool defer) {
  Status st;
  // thread-per-node classes: 0..4 (out-degree <= 8) in one launch, 5 (9..16)
  // in another; then a warp per node up to 256 and a CTA per node up to 4096
  auto small_launch = [&](int first, int last) {
    SmallLaunch L;
    uint32_t b = 0;
    for (int c = 0; c < kSmallClasses; ++c) {
      L.start[c] = s.class_start[c];
      L.count[c] = s.class_start[c + 1] - s.class_start[c];
      L.bstart[c] = b;
      if (c >= first && c <= last) b += (uint32_t)((L.count[c] + kSmallThreads - 1) / kSmallThreads);
    }
    L.bstart[kSmallClasses] = b;
    return L;
  };
  const SmallLaunch L04 = small_launch(0, 4), L5 = small_launch(5, 5);
  const uint32_t n04 = a.mark ? 0 : L04.bstart[5], n5 = a.mark ? 0 : L5.bstart[6] - L5.bstart[5];
  // the first kernel starts when all earlier work has ended, clear_round's
  // launch (which starts then and writes nothing these kernels read) excepted
  bool overlapped = defer;
  auto run = [&](auto kernel, unsigned blocks, int threads, size_t smem, auto... args) {
    launch_if_overlapped(overlapped, s, kernel, blocks, threads, smem, args...);
    overlapped = true;
  };
  // nodes a warp takes: up to 32 (one lane each), fewer where that would leave
  // multiprocessors without two full waves of warps
  auto warp_nodes = [&](auto kernel, uint64_t first, uint64_t count) {
    const uint32_t per = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(32, count / ((uint64_t)sm_count(s.device) * 128)));
    run(kernel, grid_for(count, kNodeWarps * per), kNodeWarps * 32, 0, a, first, count, per);
  };
  {
    const uint64_t n32 = s.class_start[kSmallClasses - 1] - s.class_start[kSmallClasses - 2];
    const uint64_t n64 = s.class_start[kClassWarp] - s.class_start[kSmallClasses - 1];
    TimedScope ts(s, a.mark ? KBISIM_KERNEL_OTHER : KBISIM_KERNEL_SIG_SMALL,
                  (n04 ? 1 : 0) + (n5 ? 1 : 0) + (n32 ? 1 : 0) + (n64 ? 1 : 0));
    if (n04) run(k_sig_small<0, 4, LabelT, K>, n04, kSmallThreads, 0, a, L04);
    if (n5) run(k_sig_small<5, 5, LabelT, K>, n5, kSmallThreads, 0, a, L5);
    if (n32)
      warp_nodes(a.mark  ? k_sig_warp<1, kMarking, LabelT, K>
                 : a.dup ? k_sig_warp<1, kWithDup, LabelT, K>
                         : k_sig_warp<1, kPlain, LabelT, K>,
                 s.class_start[kSmallClasses - 2], n32);
    if (n64)
      warp_nodes(a.mark  ? k_sig_warp<2, kMarking, LabelT, K>
                 : a.dup ? k_sig_warp<2, kWithDup, LabelT, K>
                         : k_sig_warp<2, kPlain, LabelT, K>,
                 s.class_start[kSmallClasses - 1], n64);
  }
  if (!(st = launch_check("k_sig_small")).ok()) return st;
  const uint64_t n256 = s.class_start[kClassWarp2] - s.class_start[kClassWarp];
  const uint64_t n1k = s.class_start[kClassBlock] - s.class_start[kClassWarp2];
  const uint64_t n4k = s.class_start[kClassHub] - s.class_start[kClassBlock];
  if (n256 + n1k + n4k) {
    TimedScope ts(s, a.mark ? KBISIM_KERNEL_OTHER : KBISIM_KERNEL_SIG_MEDIUM,
                  (n256 ? 1 : 0) + (n1k ? 1 : 0) + (n4k ? 1 : 0));
    if (n256)
      warp_nodes(a.mark  ? k_sig_warp<8, kMarking, LabelT, K>
                 : a.dup ? k_sig_warp<8, kWithDup, LabelT, K>
                         : k_sig_warp<8, kPlain, LabelT, K>,
                 s.class_start[kClassWarp], n256);
    if (n1k)
      run(a.mark  ? k_sig_cta<kSmallChunkThreads, kMarking, LabelT, K>
          : a.dup ? k_sig_cta<kSmallChunkThreads, kWithDup, LabelT, K>
                  : k_sig_cta<kSmallChunkThreads, kPlain, LabelT, K>,
          (unsigned)n1k, kSmallChunkThreads, cta_node_smem<kSmallChunkThreads, K>(), a, s.class_start[kClassWarp2]);
    if (n4k)
      run(a.mark  ? k_sig_cta<kChunkThreads, kMarking, LabelT, K>
          : a.dup ? k_sig_cta<kChunkThreads, kWithDup, LabelT, K>
                  : k_sig_cta<kChunkThreads, kPlain, LabelT, K>, (unsigned)n4k, kChunkThreads, cta_node_smem<kChunkThreads, K>(), a,
          s.class_start[kClassBlock]);
  }
  if (!(st = launch_check("k_sig_warp")).ok()) return st;
  if (s.n_hub && !a.mark) {
    if (!s.tune_now) return defer ? launch_hubs<LabelT, K>(s, a, true) : run_hubs<LabelT, K>(s, a);
    // tuning (once per handle, on a full round from level 2 on): each bucket
    // size runs the hub pass twice, the sizes alternating, each pass timed
    // with the repeats its overflows need (a repeat runs only the hubs that
    // overflowed).  A size's second pass starts from the bucket growth its
    // first pass learned and finds the round's data in L2 as the first passes
    // left it, so the second passes compare the sizes as the later rounds run
    // them; the first size (the default) is kept unless another is faster by
    // more than kHubTuneMargin.  Every pass writes the same signatures, so the
    // round's result is the last pass's.
    constexpr int kSizes = 2;
    constexpr float kHubTuneMargin = 0.05f;
    // bucket growth is learned per size: each starts from the growth before
    // tuning, and the chosen size keeps its own
    const std::vector<uint32_t> x0 = s.h_hub_xbits, sh0 = s.h_hub_shift;
    const std::vector<uint8_t> f0 = s.h_hub_force;
    std::vector<uint32_t> xs[kSizes], shs[kSizes];
    std::vector<uint8_t> fs[kSizes];
    cudaEvent_t ev[2];
    if (!(st = cuda_check(cudaEventCreate(&ev[0]), "event")).ok()) return st;
    if (!(st = cuda_check(cudaEventCreate(&ev[1]), "event")).ok()) {
      cudaEventDestroy(ev[0]);
      return st;
    }
    for (int rep = 0; rep < 2 && st.ok(); ++rep) {
      for (int c = 0; c < kSizes && st.ok(); ++c) {
        s.h_hub_xbits = rep ? xs[c] : x0;
        s.h_hub_shift = rep ? shs[c] : sh0;
        s.h_hub_force = rep ? fs[c] : f0;
        s.hub_ucap = (uint32_t)kHubUcaps[c];
        if (!(st = hub_layout(s)).ok()) break;
        cudaEventRecord(ev[0], s.stream);
        if (!(st = run_hubs<LabelT, K>(s, a)).ok()) break;
        cudaEventRecord(ev[1], s.stream);
        if (!(st = cuda_check(cudaEventSynchronize(ev[1]), "event")).ok()) break;
        cudaEventElapsedTime(&s.hub_tune_ms[c], ev[0], ev[1]);
        xs[c] = s.h_hub_xbits;
        shs[c] = s.h_hub_shift;
        fs[c] = s.h_hub_force;
      }
    }
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    if (!st.ok()) return st;
    s.hub_tune = 2;
    int best = 0;
    for (int c = 1; c < kSizes; ++c)
      if (s.hub_tune_ms[c] < s.hub_tune_ms[best] * (1.0f - kHubTuneMargin)) best = c;
    if (best != kSizes - 1) {
      s.hub_ucap = (uint32_t)kHubUcaps[best];
      s.h_hub_xbits.swap(xs[best]);
      s.h_hub_shift.swap(shs[best]);
      s.h_hub_force.swap(fs[best]);
      if (!(st = hub_layout(s)).ok()) return st;
    }
  }
  return Status::Ok();
}

Status ensure_round_scratch(Store& s) {
  Status st;
  const uint64_t n = std::max<uint64_t>(s.n, 1), m = std::max<uint64_t>(s.m, 1);
  const uint64_t cap = table_capacity(std::max<uint64_t>(s.n_alive, 1));
  if (!(st = ensure(s, s.sigkey, m * 8)).ok()) return st;
  if (!(st = ensure(s, s.ucnt, n * 4)).ok()) return st;
  if (!(st = ensure(s, s.hash, n * 8)).ok()) return st;
  if (!(st = ensure(s, s.table, cap * 8)).ok()) return st;
  s.tcap = cap;
  if (!(st = ensure(s, s.slot, n * 4)).ok()) return st;
  if (!(st = ensure(s, s.rep, n * 4)).ok()) return st;
  if (!(st = ensure(s, s.ulist[0], n * 4)).ok()) return st;
  if (!(st = ensure(s, s.ulist[1], n * 4)).ok()) return st;
  if (!(st = ensure(s, s.hbits, ((n + 31) / 32) * 4 + 16)).ok()) return st;
  if (!(st = ensure(s, s.hword, std::max<uint64_t>((n + 31) / 32, 1) * 8)).ok()) return st;
  if (!(st = ensure(s, s.member, n + 16)).ok()) return st;
  if (!(st = ensure(s, s.alone, n + 16)).ok()) return st;
  if (!(st = ensure(s, s.long_pairs, n * 8)).ok()) return st;
  const uint64_t tiles = (n + kScanTile - 1) / kScanTile;
  if (!(st = ensure(s, s.bsum, std::max<uint64_t>(tiles, 64) * 8)).ok()) return st;
  return Status::Ok();
}

uint32_t bits_for(uint64_t v) {  // bits needed to represent values 0..v
  uint32_t b = 1;
  while (b < 64 && (v >> b)) ++b;
  return b;
}

}  // namespace

// Bucket growth of the hubs, keyed by original node id: a graph laid out
// again after an update, or loaded again into the same handle, keeps what its
// hubs' buckets learned, instead of overflowing and growing them again in the
// next refinement.  Growth only sizes buckets: a wrong carry costs memory or
// a repeat, never a result.
Status save_hub_growth(Store& s, HubGrowth* g) {
  g->orig.clear();
  g->xbits.clear();
  g->shift.clear();
  g->deg.clear();
  g->force.clear();
  if (!s.has_graph || !s.n_hub || s.h_hub_xbits.size() != s.n_hub) return Status::Ok();
  bool any = false;
  for (uint64_t i = 0; i < s.n_hub && !any; ++i) any = s.h_hub_xbits[i] || s.h_hub_shift[i] || s.h_hub_force[i];
  if (!any) return Status::Ok();
  std::vector<uint32_t> p2o(s.n_hub);
  Status st = cuda_check(cudaMemcpyAsync(p2o.data(), ptr<uint32_t>(s.p2o) + s.class_start[kClassHub], s.n_hub * 4,
                                         cudaMemcpyDeviceToHost, s.stream), "hub ids");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return st;
  for (uint64_t i = 0; i < s.n_hub; ++i)
    if (s.h_hub_xbits[i] || s.h_hub_shift[i] || s.h_hub_force[i]) {
      g->orig.push_back(p2o[i]);
      g->xbits.push_back(s.h_hub_xbits[i]);
      g->shift.push_back(s.h_hub_shift[i]);
      g->deg.push_back(i < s.h_hub_deg.size() ? s.h_hub_deg[i] : 0);
      g->force.push_back(s.h_hub_force[i]);
    }
  return Status::Ok();
}

Status restore_hub_growth(Store& s, const HubGrowth& g, bool same_degree) {
  if (g.orig.empty() || !s.has_graph || !s.n_hub) return Status::Ok();
  std::vector<uint32_t> p2o(s.n_hub);
  Status st = cuda_check(cudaMemcpyAsync(p2o.data(), ptr<uint32_t>(s.p2o) + s.class_start[kClassHub], s.n_hub * 4,
                                         cudaMemcpyDeviceToHost, s.stream), "hub ids");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return st;
  std::unordered_map<uint32_t, size_t> at;
  at.reserve(g.orig.size() * 2);
  for (size_t j = 0; j < g.orig.size(); ++j) at[g.orig[j]] = j;
  s.h_hub_xbits.resize(s.n_hub, 0);
  s.h_hub_shift.resize(s.n_hub, 0);
  s.h_hub_force.resize(s.n_hub, 0);
  bool changed = false;
  for (uint64_t i = 0; i < s.n_hub; ++i) {
    const auto it = at.find(p2o[i]);
    if (it == at.end()) continue;
    if (same_degree && (i >= s.h_hub_deg.size() || s.h_hub_deg[i] != g.deg[it->second])) continue;
    s.h_hub_xbits[i] = std::max(s.h_hub_xbits[i], g.xbits[it->second]);
    s.h_hub_shift[i] = std::max(s.h_hub_shift[i], g.shift[it->second]);
    s.h_hub_force[i] = std::max(s.h_hub_force[i], g.force[it->second]);
    changed = true;
  }
  return changed ? hub_layout(s) : Status::Ok();
}

// ---------------------------------------------------------------------------
// Relabelling and degree classes (once per graph)
// ---------------------------------------------------------------------------
// Work lists made from the hubs' offsets: their chunks and bucket layout.
// `fresh`: a new graph (bucket growth learned on the previous one is dropped).
Status build_chunk_lists(Store& s, bool fresh) {
  Status st;
  s.dup_valid = false;  // another edge table
  s.refined = false;
  // hubs: a contiguous internal id range; their offsets come in one copy
  s.n_hub = s.class_start[kClassHub + 1] - s.class_start[kClassHub];
  if (fresh || s.h_hub_xbits.size() != s.n_hub) {  // bucket growth learned on this graph is kept otherwise
    s.h_hub_xbits.assign(s.n_hub, 0);
    s.h_hub_shift.assign(s.n_hub, 0);
    s.h_hub_force.assign(s.n_hub, 0);
    s.hub_calm = false;
  }
  s.h_hub_deg.assign(s.n_hub, 0);
  s.hub_edges = 0;
  s.n_hub_chunks = 0;
  s.n_hub_buckets = 0;
  if (s.n_hub) {
    std::vector<uint64_t> hoff(s.n_hub + 1);
    st = cuda_check(cudaMemcpyAsync(hoff.data(), ptr<uint64_t>(s.offsets) + s.class_start[kClassHub],
                                    (s.n_hub + 1) * 8, cudaMemcpyDeviceToHost, s.stream), "hub offsets");
    if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
    if (!st.ok()) return st;
    s.hub_edge0 = hoff[0];
    std::vector<uint4> chunks;
    std::vector<uint32_t> cstart(s.n_hub + 1, 0);
    for (uint64_t i = 0; i < s.n_hub; ++i) {
      cstart[i] = (uint32_t)chunks.size();
      const uint64_t d = hoff[i + 1] - hoff[i];
      s.h_hub_deg[i] = d;
      s.hub_edges += d;
      for (uint64_t b = 0; b < d; b += kHubChunk) {
        const uint64_t e = hoff[i] + b;
        uint4 q;
        q.x = (uint32_t)i;
        q.y = (uint32_t)(e & 0xFFFFFFFFu);
        q.z = (uint32_t)(e >> 32);
        q.w = (uint32_t)std::min<uint64_t>(kHubChunk, d - b);
        chunks.push_back(q);
      }
    }
    s.n_hub_chunks = chunks.size();
    cstart[s.n_hub] = (uint32_t)chunks.size();
    if (!(st = ensure(s, s.hub_chunks, chunks.size() * sizeof(uint4))).ok()) return st;
    if (!(st = ensure(s, s.hub_cstart, (s.n_hub + 1) * 4)).ok()) return st;
    st = cuda_check(cudaMemcpyAsync(s.hub_chunks.p, chunks.data(), chunks.size() * sizeof(uint4),
                                    cudaMemcpyHostToDevice, s.stream), "hub chunks");
    if (st.ok())
      st = cuda_check(cudaMemcpyAsync(s.hub_cstart.p, cstart.data(), (s.n_hub + 1) * 4, cudaMemcpyHostToDevice,
                                      s.stream), "hub chunks");
    if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "hub chunks");
    if (!st.ok()) return st;
    if (!(st = hub_layout(s)).ok()) return st;
  }
  return Status::Ok();
}

Status scan_u64(Store& s, uint64_t* a, uint64_t n) { return scan64(s, a, n, nullptr); }

Status clear_arrays(Store& s, std::initializer_list<ClearRange> ranges) {
  ClearArgs c;
  uint64_t units = 0;
  for (const ClearRange& r : ranges) {
    c.add(r.p, r.bytes, r.word);
    units += (r.bytes + 15) / 16;
  }
  k_clear<<<(unsigned)std::min<uint64_t>(grid_for(units, kClearThreads), (uint64_t)sm_count(s.device) * 8),
            kClearThreads, 0, s.stream>>>(c);
  return launch_check("k_clear");
}

Status rank_heads(Store& s, const uint32_t* hbits, uint64_t words, uint2* hrank, unsigned long long* ticket_total) {
  const uint64_t tiles = (words + kRankTile - 1) / kRankTile;
  Status st = ensure(s, s.bsum, std::max<uint64_t>(tiles, 64) * 8);
  if (!st.ok()) return st;
  launch_chained(s, k_head_ranks, (unsigned)tiles, kRankThreads, 0, hbits, words, hrank, ptr<uint32_t>(s.bsum),
                 ticket_total, ticket_total + 1);
  return launch_check("k_head_ranks");
}

Status relabel_graph(Store& s, const uint64_t* off0, const uint32_t* dst0, const void* lab0,
                     const uint32_t* nlab0, const uint8_t* alive0, uint32_t lab_bytes) {
  Status st = set_smem_attrs(s.device);
  if (!st.ok()) return st;
  const uint64_t n = s.n, m = s.m;
  const int sms = sm_count(s.device);
  const uint64_t ntiles = std::max<uint64_t>(1, (n + kClassTile - 1) / kClassTile);
  // temporaries of the relabelling (kept between loads)
  InUse use(s, kCacheRelabel);
  Buf &tcnt = s.rl_tcnt, &hot = s.rl_hot, &ost = s.rl_ost;
  auto fail = [&](Status e) { return e; };
  if (!(st = ensure(s, tcnt, ntiles * kNumOrder * 8)).ok()) return fail(st);
  if (!(st = ensure(s, hot, std::max<uint64_t>(1, n) * 4)).ok()) return fail(st);
  if (!(st = ensure(s, ost, kNumOrder * 8)).ok()) return fail(st);
  cudaMemsetAsync(tcnt.p, 0, ntiles * kNumOrder * 8, s.stream);
  cudaMemsetAsync(hot.p, 0, std::max<uint64_t>(1, n) * 4, s.stream);
  if (m >> kHotSampleShift)
    k_hot_sample<<<(unsigned)std::min<uint64_t>(grid_for(m >> kHotSampleShift, 256), (uint64_t)sms * 32), 256, 0,
                   s.stream>>>(m, dst0, ptr<uint32_t>(hot));
  if (n)
    k_class_tile_count<<<(unsigned)ntiles, kClassTile, 0, s.stream>>>(n, off0, alive0, ptr<uint32_t>(hot), ntiles,
                                                                      ptr<unsigned long long>(tcnt));
  if (!(st = launch_check("k_class_tile_count")).ok()) return fail(st);
  if (!(st = scan64(s, ptr<uint64_t>(tcnt), ntiles * kNumOrder, nullptr)).ok()) return fail(st);
  k_order_starts<<<1, 128, 0, s.stream>>>(ptr<unsigned long long>(tcnt), ntiles, ptr<unsigned long long>(ost));
  std::vector<uint64_t> hs(kNumOrder);
  st = cuda_check(cudaMemcpyAsync(hs.data(), ost.p, kNumOrder * 8, cudaMemcpyDeviceToHost, s.stream), "class starts");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return fail(st);
  for (int c = 0; c < kNumClasses; ++c) s.class_start[c] = hs[(size_t)c * kHotBuckets];
  s.class_start[kNumClasses] = n;
  s.n_alive = s.class_start[kClassDead];
  if (st.ok()) st = ensure(s, s.p2o, std::max<uint64_t>(1, n) * 4);
  if (st.ok()) st = ensure(s, s.o2p, std::max<uint64_t>(1, n) * 4);
  if (st.ok()) st = ensure(s, s.offsets, (n + 1) * 8);
  if (st.ok()) st = ensure(s, s.nlabel, std::max<uint64_t>(1, n) * 4);
  if (st.ok()) st = ensure(s, s.dst, std::max<uint64_t>(1, m) * 4);
  if (!st.ok()) return fail(st);
  const unsigned gb = (unsigned)std::min<uint64_t>(grid_for(n, 256), (uint64_t)sms * 32);
  if (n) {
    k_class_tile_scatter<<<(unsigned)ntiles, kClassTile, 0, s.stream>>>(n, off0, alive0, ptr<uint32_t>(hot), ntiles,
                                                                        ptr<unsigned long long>(tcnt),
                                                                        ptr<uint32_t>(s.p2o));
    k_invert<<<gb, 256, 0, s.stream>>>(n, ptr<uint32_t>(s.p2o), ptr<uint32_t>(s.o2p));
  }
  k_relabel_nodes<<<gb, 256, 0, s.stream>>>(n, ptr<uint32_t>(s.p2o), off0, nlab0,
                                            ptr<unsigned long long>(s.offsets), ptr<uint32_t>(s.nlabel));
  st = launch_check("relabel nodes");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  fail(Status::Ok());  // the class scatter has finished with the tile bases and counts
  if (!st.ok()) return st;
  if (!(st = scan64(s, ptr<uint64_t>(s.offsets), n + 1, nullptr)).ok()) return st;
  s.n_alone = 0;
  if (!(st = build_chunk_lists(s, true)).ok()) return st;
  // the edge labels (and with them the label width) from here on
  if (s.await_labels && !(st = s.await_labels(s)).ok()) return st;
  if (!(st = ensure(s, s.elabel, std::max<uint64_t>(1, m) * (s.label8 ? 1 : 4))).ok()) return st;
  if (n && m) {
    if (s.label8) {
      uint8_t* lab = ptr<uint8_t>(s.elabel);
      if (lab_bytes == 1) relabel_edges(s, off0, dst0, static_cast<const uint8_t*>(lab0), lab, sms);
      else if (lab_bytes == 2) relabel_edges(s, off0, dst0, static_cast<const uint16_t*>(lab0), lab, sms);
      else relabel_edges(s, off0, dst0, static_cast<const uint32_t*>(lab0), lab, sms);
    } else {
      uint32_t* lab = ptr<uint32_t>(s.elabel);
      if (lab_bytes == 2) relabel_edges(s, off0, dst0, static_cast<const uint16_t*>(lab0), lab, sms);
      else relabel_edges(s, off0, dst0, static_cast<const uint32_t*>(lab0), lab, sms);
    }
  }
  st = launch_check("relabel edges");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  return st;
}

// ---- level 0 when few labels occur (Definition 2: pId_0 groups nodes by
// label) ------------------------------------------------------------------
// A table of kL0Slots 64-bit slots (label << 32 | smallest original id) and a
// node count per slot.  Each CTA first gathers the labels of its node range in
// a shared copy, so the global table sees one update per label per CTA.  If a
// shared or the global table fills (more labels than it holds) the general
// path (hash, grouping, exact check, renumbering) computes the level instead.
// The host waits once, for the block count.
constexpr int kL0Slots = 4096;        // global table: labels at most kL0Slots / 2
constexpr int kL0SmemSlots = 1024;    // per CTA
constexpr int kL0Threads = 256;
constexpr unsigned long long kL0Empty = ~0ull;  // (0xFFFFFFFF, 0xFFFFFFFF): no original id is 0xFFFFFFFF

__device__ __forceinline__ uint32_t l0_home(uint32_t label, uint32_t mask) {
  return (label * 0x9E3779B1u >> 7) & mask;  // Fibonacci hashing, then the slot bits
}

// Insert (label, id) into a table of 64-bit slots: the slot of the label keeps
// the smallest id; returns the slot, or -1 if the table is full (shared or
// global memory, through generic addressing).
__device__ __forceinline__ int l0_insert(unsigned long long* tab, uint32_t mask, uint32_t label, uint32_t id) {
  const unsigned long long v = ((unsigned long long)label << 32) | id;
  uint32_t at = l0_home(label, mask);
  for (uint32_t t = 0; t <= mask; ++t) {
    const unsigned long long cur = atomicCAS(tab + at, kL0Empty, v);
    if (cur == kL0Empty) return (int)at;
    if ((uint32_t)(cur >> 32) == label) {
      if ((uint32_t)cur > id) atomicMin(tab + at, v);
      return (int)at;
    }
    at = (at + 1) & mask;
  }
  return -1;
}

__global__ void __launch_bounds__(kL0Threads) k_l0_collect(uint64_t n_alive, const uint32_t* nlabel, const uint32_t* p2o,
                                                           unsigned long long* gtab, uint32_t* gcnt, uint32_t* err) {
  overlap_next();
  overlap_wait();
  __shared__ unsigned long long tab[kL0SmemSlots];
  __shared__ uint32_t cnt[kL0SmemSlots];
  __shared__ uint32_t full;
  for (uint32_t i = threadIdx.x; i < (uint32_t)kL0SmemSlots; i += kL0Threads) {
    tab[i] = kL0Empty;
    cnt[i] = 0;
  }
  if (threadIdx.x == 0) full = 0;
  __syncthreads();
  const uint64_t per = (n_alive + gridDim.x - 1) / gridDim.x;
  const uint64_t lo0 = (uint64_t)blockIdx.x * per;
  const uint64_t lo = lo0 < n_alive ? lo0 : n_alive, hi = lo + per < n_alive ? lo + per : n_alive;
  for (uint64_t p = lo + threadIdx.x; p < hi; p += kL0Threads) {
    const int at = l0_insert(tab, kL0SmemSlots - 1, nlabel[p], p2o[p]);
    if (at < 0) full = 1;
    else atomicAdd(&cnt[at], 1u);
  }
  __syncthreads();
  if (full) {
    if (threadIdx.x == 0) atomicOr(err, 1u);
    return;
  }
  for (uint32_t i = threadIdx.x; i < (uint32_t)kL0SmemSlots; i += kL0Threads) {
    const unsigned long long v = tab[i];
    if (v == kL0Empty) continue;
    const int at = l0_insert(gtab, kL0Slots - 1, (uint32_t)(v >> 32), (uint32_t)v);
    if (at < 0) atomicOr(err, 1u);
    else atomicAdd(&gcnt[at], cnt[i]);
  }
}

// Block ids of the table's labels, ranked by smallest original id, by one CTA:
// a label's rank is the number of labels with a smaller id (up to
// kL0Slots / 2 of them, listed in shared memory; more set err).  On the device,
// so that level 0 needs no copies of the table (three, a host sort and one copy
// back took 50 us).  stats: [7] err, [8] nodes alone, [15] blocks.
constexpr int kL0RankThreads = 1024;

__global__ void __launch_bounds__(kL0RankThreads) k_l0_rank(const unsigned long long* gtab, const uint32_t* gcnt,
                                                            uint32_t* rank, uint32_t* err, unsigned long long* stats) {
  // stats: pinned host memory
  overlap_next();
  overlap_wait();
  __shared__ uint32_t ids[kL0Slots / 2];
  __shared__ uint32_t n, alone;
  if (threadIdx.x == 0) n = alone = 0;
  __syncthreads();
  constexpr int kPer = kL0Slots / kL0RankThreads;
  unsigned long long v[kPer];
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    v[t] = gtab[threadIdx.x + t * kL0RankThreads];
    if (v[t] == kL0Empty) continue;
    const uint32_t at = atomicAdd(&n, 1u);
    if (at < (uint32_t)kL0Slots / 2) ids[at] = (uint32_t)v[t];
    if (gcnt[threadIdx.x + t * kL0RankThreads] == 1u) atomicAdd(&alone, 1u);
  }
  __syncthreads();
  const uint32_t found = n;
  if (found > (uint32_t)kL0Slots / 2) {  // long probe runs: the general path
    if (threadIdx.x == 0) {
      *err = 1u;
      stats[7] = 1ull;
    }
    return;
  }
#pragma unroll
  for (int t = 0; t < kPer; ++t) {
    if (v[t] == kL0Empty) continue;
    uint32_t r = 0;
    for (uint32_t j = 0; j < found; ++j) r += ids[j] < (uint32_t)v[t] ? 1u : 0u;
    rank[threadIdx.x + t * kL0RankThreads] = r;
  }
  if (threadIdx.x == 0) {
    stats[7] = *err;
    stats[8] = alone;
    stats[15] = found;
  }
}

// pId_0 of every node from the ranked table: rank[slot] = block id, and the
// node is alone in its block when its label's count is 1.
__global__ void __launch_bounds__(kL0Threads) k_l0_fill(uint64_t n, uint64_t n_alive, const uint32_t* nlabel,
                                                        const unsigned long long* gtab, const uint32_t* rank,
                                                        const uint32_t* gcnt, const uint32_t* err, uint32_t* pid,
                                                        uint8_t* alone) {
  overlap_next();
  overlap_wait();
  if (*err) return;  // too many labels
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n; p += (uint64_t)gridDim.x * blockDim.x) {
    if (p >= n_alive) {
      pid[p] = kDead;
      continue;
    }
    const uint32_t label = nlabel[p];
    uint32_t at = l0_home(label, kL0Slots - 1);
    for (uint32_t t = 0; t < (uint32_t)kL0Slots; ++t) {  // the label is in the table: the loop ends at its slot
      const unsigned long long v = __ldg(gtab + at);
      if (v != kL0Empty && (uint32_t)(v >> 32) == label) break;
      at = (at + 1) & (kL0Slots - 1);
    }
    pid[p] = __ldg(rank + at);
    alone[p] = __ldg(gcnt + at) == 1u ? 1 : 0;
  }
}

// Level 0 by the label table; *done = false when there are too many labels
// (the general path then runs).
Status level0_few_labels(Store& s, bool* done) {
  *done = false;
  const uint64_t n = s.n, na = s.n_alive;
  if (!na) return Status::Ok();
  Status st;
  // the table, counts and ranks in the grouping table's buffer (sized for n
  // nodes, so large enough whenever there are nodes)
  const size_t bytes = kL0Slots * 8 + kL0Slots * 4 + kL0Slots * 4 + 16;
  if (s.table.cap < bytes) return Status::Ok();
  unsigned long long* gtab = ptr<unsigned long long>(s.table);
  uint32_t* gcnt = reinterpret_cast<uint32_t*>(gtab + kL0Slots);
  uint32_t* grank = gcnt + kL0Slots;
  uint32_t* err = grank + kL0Slots;
  const int sms = sm_count(s.device);
  unsigned long long* sc = ptr<unsigned long long>(s.d_scalars);
  {
    TimedScope ts(s, KBISIM_KERNEL_LABEL_GROUP, 3);
    ClearArgs c;
    c.add(s.d_err.p, 16, 0u);
    c.add(sc, 16 * 8, 0u);
    c.add(gtab, kL0Slots * 8, ~0u);
    c.add(gcnt, kL0Slots * 4 * 2 + 16, 0u);
    k_clear<<<8, kClearThreads, 0, s.stream>>>(c);
    const unsigned g = (unsigned)std::min<uint64_t>(grid_for(na, 2048), (uint64_t)sms * 8);
    launch_chained(s, k_l0_collect, g, kL0Threads, 0, na, ptr<uint32_t>(s.nlabel), ptr<uint32_t>(s.p2o), gtab, gcnt, err);
    launch_chained(s, k_l0_rank, 1, kL0RankThreads, 0, gtab, gcnt, grank, err,
                   ptr<unsigned long long>(s.h_scalars));
  }
  if (!(st = launch_check("k_l0_collect")).ok()) return st;
  {
    TimedScope ts(s, KBISIM_KERNEL_RENUMBER, 1);
    const unsigned g = (unsigned)std::min<uint64_t>(grid_for(n, kL0Threads), (uint64_t)sms * 16);
    launch_chained(s, k_l0_fill, g, kL0Threads, 0, n, na, ptr<uint32_t>(s.nlabel), gtab, grank, gcnt, err,
                   ptr<uint32_t>(s.level[0]), ptr<uint8_t>(s.alone));
  }
  if (!(st = launch_check("k_l0_fill")).ok()) return st;
  uint64_t h[16];
  if (!(st = await_scalars(s, h)).ok()) return st;
  if (h[7]) return Status::Ok();  // too many labels: the general path
  if (s.checked && !(st = check_below(s, ptr<uint32_t>(s.level[0]), na, h[15], "identifiers")).ok()) return st;
  s.counts[0] = h[15];
  s.n_alone = h[8];
  *done = true;
  return Status::Ok();
}

Status compute_level0(Store& s) {
  Status st = ensure_round_scratch(s);
  if (!st.ok()) return st;
  bool done = false;
  if (!(st = level0_few_labels(s, &done)).ok()) return st;
  if (done) return Status::Ok();
  const int sms = sm_count(s.device);
  const unsigned blocks = (unsigned)std::min<uint64_t>(grid_for(s.n_alive, 256), (uint64_t)sms * 16);
  if (!(st = clear_round(s, s.n_alive, 0, false, false)).ok()) return st;
  {
    TimedScope ts(s, KBISIM_KERNEL_LABEL_GROUP, s.n_alive ? 1 : 0);
    if (s.n_alive)
      k_label_hash<<<blocks, 256, 0, s.stream>>>(s.n_alive, ptr<uint32_t>(s.nlabel), ptr<uint64_t>(s.hash),
                                                 s.seed, s.hash_mask);
  }
  if (!(st = launch_check("k_label_hash")).ok()) return st;
  uint64_t blocks_out = 0, coll = 0;
  st = group_and_rank(s, 0, nullptr, false, ptr<uint32_t>(s.level[0]), &blocks_out, &coll, false, nullptr,
                      nullptr, false, true, false, nullptr);
  if (!st.ok()) return st;
  s.counts[0] = blocks_out;
  return Status::Ok();
}

// Checked mode, before a round: the edge table's offsets and targets and the
// previous level's identifiers (the indices and the packed values of the
// signature kernels).  With the KBISIM_FAULT_CORRUPT_DST test hook one target
// is set to n first (and put back after the check reports it).
Status check_round_inputs(Store& s, uint32_t i) {
  Status st;
  uint32_t saved = 0;
  const uint64_t at = s.m / 2;
  uint32_t* dst = ptr<uint32_t>(s.dst);
  if (s.fault_corrupt_dst && s.m) {
    const uint32_t bad = (uint32_t)s.n;
    st = cuda_check(cudaMemcpyAsync(&saved, dst + at, 4, cudaMemcpyDeviceToHost, s.stream), "corrupt");
    if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "corrupt");
    if (st.ok()) st = cuda_check(cudaMemcpyAsync(dst + at, &bad, 4, cudaMemcpyHostToDevice, s.stream), "corrupt");
    if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "corrupt");
    if (!st.ok()) return st;
  }
  if (s.n) {
    const unsigned g = (unsigned)std::min<uint64_t>(grid_for(s.n, 256), (uint64_t)sm_count(s.device) * 16);
    k_check_offsets_mono<<<g, 256, 0, s.stream>>>(ptr<uint64_t>(s.offsets), s.n, s.m, ptr<uint32_t>(s.d_err));
    st = checked_outcome(s, "edge offsets");
  }
  if (st.ok()) st = check_below(s, dst, s.m, s.n, "edge targets");
  if (s.fault_corrupt_dst && s.m) {
    Status st2 = cuda_check(cudaMemcpyAsync(dst + at, &saved, 4, cudaMemcpyHostToDevice, s.stream), "restore");
    if (st2.ok()) st2 = cuda_check(cudaStreamSynchronize(s.stream), "restore");
    if (!st2.ok()) return st2;
  }
  if (st.ok()) st = check_below(s, ptr<uint32_t>(s.level[i - 1]), s.n_alive, s.counts[i - 1], "previous level");
  return st;
}

Status compute_round(Store& s, uint32_t i) {
  if (s.fault_timeout_round && i == s.fault_timeout_round)
    return Status::Err(KBISIM_ERR_TIMEOUT, "injected timeout (KBISIM_FAULT_TIMEOUT_ROUND)");
  Status st = ensure_round_scratch(s);
  if (!st.ok()) return st;
  bool keep = s.heads_level == (int64_t)i - 1;
  s.heads_level = -1;
  const uint64_t ins = insert_count(s, true), filter = filter_bits(s, ins, i <= 1);
  if (!(st = clear_round(s, ins, filter, s.n_hub != 0, keep)).ok()) return st;
  if (s.checked && !(st = check_round_inputs(s, i)).ok()) return st;
  SigArgs a;
  a.off = ptr<uint64_t>(s.offsets);
  a.dst = ptr<uint32_t>(s.dst);
  a.lab = s.elabel.p;
  a.prev = ptr<uint32_t>(s.level[i - 1]);
  a.sigkey = s.sigkey.p;
  a.ucnt = ptr<uint32_t>(s.ucnt);
  a.hash = ptr<uint64_t>(s.hash);
  a.seed = s.seed;
  a.mask = s.hash_mask;
  a.err = ptr<uint32_t>(s.d_err);
  a.fmask = s.round_mask;
  a.alone = ptr<uint8_t>(s.alone);
  a.dup = s.dup_valid && keep ? ptr<uint32_t>(s.dup) : nullptr;  // (keep: alone_bits is the level before's)
  a.alone_bits = ptr<uint32_t>(s.alone_bits);
  a.dup_hubs = s.dup_hubs;
  a.mark = nullptr;
  // 32-bit signature words when (label, child id) fits in 32 bits
  const uint32_t pbits = bits_for(s.counts[i - 1] ? s.counts[i - 1] - 1 : 0);
  const bool key64 = pbits + s.label_bits > 32;
  a.pbits = (int)pbits;
  s.tune_now = s.hub_tune == 1 && i >= 2 && !s.round_mask && s.n_hub;
  // the hubs' overflow flags are read with the round's result; a round whose
  // hubs overflowed signs those again and groups again (seldom: the growth is
  // kept).  Checked mode and the tuning wait for complete signatures first, and
  // so does a large graph until a round has passed without growth: a repeated
  // grouping costs it more than the wait (200M edges: 1 ms of the first pass).
  const bool defer = !s.checked && !s.tune_now && (s.hub_calm || s.n_alive <= kHubCalmNodes);
  s.hub_grew = false;
  auto signatures = [&](auto label, auto key) {
    return run_signatures<decltype(label), decltype(key)>(s, a, defer);
  };
  auto hubs_again = [&](auto label, auto key) { return launch_hubs<decltype(label), decltype(key)>(s, a, true); };
  auto typed = [&](auto&& f) {
    if (s.label8) return key64 ? f(uint8_t(), uint64_t()) : f(uint8_t(), uint32_t());
    return key64 ? f(uint32_t(), uint64_t()) : f(uint32_t(), uint32_t());
  };
  st = typed(signatures);
  s.tune_now = false;
  if (!st.ok()) return st;
  if (s.round_mask && s.n_alive) {
    const int sms = sm_count(s.device);
    k_freeze<<<(unsigned)std::min<uint64_t>(grid_for(s.n_alive, 256), (uint64_t)sms * 16), 256, 0, s.stream>>>(
        s.n_alive, s.round_mask, a.prev, a.ucnt, a.hash, s.seed, s.hash_mask);
    if (!(st = launch_check("k_freeze")).ok()) return st;
  }
  uint64_t blocks = 0, coll = 0, keys = 0, maxsig = 0;
  // nodes alone in their block at level i-1 stay alone (Proposition 1): they
  // are heads of level i without a table lookup
  for (int attempt = 0;; ++attempt) {
    uint32_t hub_flags = 0;
    st = group_and_rank(s, 1, a.prev, key64, ptr<uint32_t>(s.level[i]), &blocks, &coll, true, &keys, &maxsig, true,
                        i <= 1, keep, &hub_flags);
    if (!st.ok()) return st;
    if (!hub_flags) break;
    if (attempt >= kHubAttempts) return Status::Err(KBISIM_ERR_TIMEOUT, "hub bucket overflow persists");
    if (!(st = grow_hubs(s, &a)).ok()) return st;
    keep = false;  // heads were marked with incomplete signatures
    if (!(st = clear_round(s, ins, filter, true, false)).ok()) return st;
    if (!(st = typed(hubs_again)).ok()) return st;
  }
  s.heads_level = i;
  if (i >= 2) s.hub_calm = !s.hub_grew;  // (level 1 has few distinct keys)
  s.counts[i] = blocks;
  kbisim_round_stats rs;
  rs.blocks = blocks;
  rs.unique_keys = keys;
  rs.max_signature = maxsig;
  rs.collided_nodes = coll;
  rs.hub_nodes = s.n_hub;
  if (s.stats.size() < i) s.stats.resize(i);
  s.stats[i - 1] = rs;
  return Status::Ok();
}

// The edges of hubs into the marks: their set in the key buffer has 32-bit slots.
template <typename LabelT>
Status mark_hub_edges(Store& s, const SigArgs& a) {
  TimedScope ts(s, KBISIM_KERNEL_OTHER, 1);
  cudaMemsetAsync(static_cast<char*>(s.sigkey.p) + s.hub_edge0 * 8, 0xFF, s.hub_edges * 8, s.stream);
  cudaMemsetAsync(s.hub_err.p, 0, s.n_hub * 4, s.stream);
  k_mark_hubs<LabelT><<<(unsigned)s.n_hub_chunks, kChunkThreads, 0, s.stream>>>(
      a, s.class_start[kClassHub], ptr<uint4>(s.hub_chunks), ptr<uint32_t>(s.hub_err));
  return launch_check("k_mark_hubs");
}

Status mark_duplicates(Store& s, uint32_t rounds) {
  if (!s.n || s.m < kMarkEdges || s.budget || s.checked) return Status::Ok();
  if (rounds < (s.m > kMarkEdgesTwoRounds ? 3u : 2u)) return Status::Ok();
  const uint32_t pbits = bits_for(s.n - 1);
  const bool key64 = pbits + s.label_bits > 32, hubs = s.dup_valid;  // (the hubs' turn)
  if (hubs && (s.dup_hubs || !s.n_hub || key64)) return Status::Ok();
  Status st = ensure_round_scratch(s);
  if (!st.ok()) return st;
  const uint64_t words = s.m / 32 + 1;
  if (!hubs && (!ensure(s, s.dup, words * 4 + 16).ok() || !ensure(s, s.alone_bits, s.n / 32 * 4 + 16).ok())) {
    release(s, s.dup);
    return Status::Ok();  // no room: every round runs without the marks
  }
  SigArgs a = {};
  a.off = ptr<uint64_t>(s.offsets);
  a.dst = ptr<uint32_t>(s.dst);
  a.lab = s.elabel.p;
  a.prev = ptr<uint32_t>(s.slot);     // the identity
  a.alone = ptr<uint8_t>(s.member);   // every node only counts
  a.sigkey = s.sigkey.p;
  a.ucnt = ptr<uint32_t>(s.ucnt);
  a.hash = ptr<uint64_t>(s.hash);
  a.pbits = (int)pbits;
  a.err = ptr<uint32_t>(s.d_err);
  a.mark = ptr<uint32_t>(s.dup);
  {
    TimedScope ts(s, KBISIM_KERNEL_OTHER, 1);
    k_iota<<<(unsigned)std::min<uint64_t>(grid_for(s.n, 256), (uint64_t)sm_count(s.device) * 16), 256, 0, s.stream>>>(
        s.n, ptr<uint32_t>(s.slot));
  }
  if (!(st = launch_check("mark duplicates")).ok()) return st;
  s.dup_valid = false;  // (until the marks are whole)
  if (hubs) {
    st = s.label8 ? mark_hub_edges<uint8_t>(s, a) : mark_hub_edges<uint32_t>(s, a);
  } else {
    cudaMemsetAsync(s.dup.p, 0, words * 4, s.stream);
    cudaMemsetAsync(s.member.p, 1, s.n, s.stream);
    if (s.label8)
      st = key64 ? run_signatures<uint8_t, uint64_t>(s, a, false) : run_signatures<uint8_t, uint32_t>(s, a, false);
    else
      st = key64 ? run_signatures<uint32_t, uint64_t>(s, a, false) : run_signatures<uint32_t, uint32_t>(s, a, false);
  }
  if (!st.ok()) return st;
  s.dup_hubs = hubs;
  s.dup_valid = true;
  return Status::Ok();
}

Status masked_signatures(Store& s, const uint32_t* prev, const uint32_t* fmask) {
  Status st = ensure_round_scratch(s);
  if (!st.ok()) return st;
  cudaMemsetAsync(s.d_err.p, 0, 4, s.stream);
  SigArgs a;
  a.off = ptr<uint64_t>(s.offsets);
  a.dst = ptr<uint32_t>(s.dst);
  a.lab = s.elabel.p;
  a.prev = prev;
  a.sigkey = s.sigkey.p;
  a.ucnt = ptr<uint32_t>(s.ucnt);
  a.hash = ptr<uint64_t>(s.hash);
  a.seed = s.seed;
  a.mask = s.hash_mask;
  a.err = ptr<uint32_t>(s.d_err);
  a.fmask = fmask;
  a.alone = nullptr;
  a.dup = a.alone_bits = nullptr;
  a.dup_hubs = false;
  a.mark = nullptr;
  if (s.mt.key32) {  // labels below 2^pbits (the stores' width)
    a.pbits = (int)s.mt.pbits;
    return s.label8 ? run_signatures<uint8_t, uint32_t>(s, a, false) : run_signatures<uint32_t, uint32_t>(s, a, false);
  }
  a.pbits = 32;
  return s.label8 ? run_signatures<uint8_t, uint64_t>(s, a, false) : run_signatures<uint32_t, uint64_t>(s, a, false);
}

Status group_list(Store& s, const uint32_t* list, uint64_t count, const uint32_t* prev) {
  Status st = ensure_round_scratch(s);
  if (!st.ok() || !count) return st;
  const uint64_t slots = group_slots(s, count);
  const GroupArgs g = group_args(s, slots);
  // (the marks of the canonical numbering are not used here)
  const VerifyArgs v = verify_args(s, 1, prev, !s.mt.key32);
  cudaMemsetAsync(s.d_scalars.p, 0, 15 * 8, s.stream);
  cudaMemsetAsync(s.table.p, 0xFF, slots * 8, s.stream);
  {
    TimedScope ts(s, KBISIM_KERNEL_GROUP, 3);
    launch_insert(s, g, list, count);
    st = launch_verify(s, g, v, list, count, true);
  }
  if (!st.ok()) return st;
  uint64_t h[16];
  if (!(st = read_scalars(s, h)).ok()) return st;
  if (!(st = settle_unresolved(s, g, v, h)).ok()) return st;
  uint32_t e = 0;
  st = cuda_check(cudaMemcpyAsync(&e, s.d_err.p, 4, cudaMemcpyDeviceToHost, s.stream), "group list");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "group list");
  if (st.ok() && (e & kErrProbe)) return Status::Err(KBISIM_ERR_TIMEOUT, "hash table probe bound exceeded");
  return st;
}

Status unpermute_level(Store& s, uint32_t level, uint32_t* dst) {
  if (!s.n) return Status::Ok();
  const int sms = sm_count(s.device);
  const unsigned gb = (unsigned)std::min<uint64_t>(grid_for(s.n, kUnpThreads * kUnpItems), (uint64_t)sms * 8);
  k_unpermute<<<gb, kUnpThreads, 0, s.stream>>>(s.n, ptr<uint32_t>(s.o2p), ptr<uint32_t>(s.level[level]), dst);
  return launch_check("k_unpermute");
}

}  // namespace kb
