// Batched build: many independent graphs refined together.
//
// The graphs arrive as one graph whose node ids are grouped by graph (graph j
// owns ids start[j] .. start[j+1]-1) with no edge between two graphs.  The
// library refines this disjoint union with its usual kernels, one launch
// sequence per round for all graphs.  k-bisimilarity of two nodes of one graph
// depends only on that graph (Definition 1 follows out-edges, which stay in
// the graph), so the union's partition at every level, restricted to graph j,
// is graph j's own partition.  After each level, the blocks are renumbered
// per graph: the block of (graph j, union block b) gets the rank of its
// smallest node id within graph j, which is the canonical numbering graph j
// would get alone.  Per-graph block counts give each graph its own early stop.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "kbisim_internal.cuh"

namespace kb {
namespace {

constexpr unsigned kFullMask = 0xFFFFFFFFu;
constexpr int kThreads = 256;
constexpr int kAggItems = 4, kAggChunk = kThreads * kAggItems, kAggSlots = 2 * kAggChunk;

template <typename T>
T* ptr(const Buf& b) {
  return static_cast<T*>(b.p);
}

unsigned grid_for(uint64_t n, int threads, int cap) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + threads - 1) / threads, (uint64_t)cap));
}

// Graph of each original node: the largest j with start[j] <= o.
__global__ void k_many_gid(uint64_t n, const uint64_t* start, uint32_t G, uint32_t* gid) {
  for (uint64_t o = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; o < n; o += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = G;  // start[lo] <= o < start[hi]
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) / 2;
      if (start[mid] <= o) lo = mid; else hi = mid;
    }
    gid[o] = lo;
  }
}

// gidp[p] = graph of internal node p.
__global__ void k_many_gidp(uint64_t n, const uint32_t* p2o, const uint32_t* gid, uint32_t* gidp) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < n; p += (uint64_t)gridDim.x * blockDim.x)
    gidp[p] = gid[p2o[p]];
}

// Every edge must stay in its graph.  Bound by the gather of the target's
// graph: one per edge, kCheckItems of a lane in flight.  (A warp per node,
// whatever its degree, with two gathers per edge took 790 us for 4.6M nodes
// and 37M edges.)
constexpr int kCheckItems = 4;

__device__ __forceinline__ bool check_run(uint64_t b, uint64_t e, uint32_t g, uint32_t rank, uint32_t threads,
                                          const uint32_t* dst, const uint32_t* gidp) {
  bool bad = false;
  for (uint64_t i0 = b + rank; i0 < e; i0 += (uint64_t)threads * kCheckItems) {
    uint32_t v[kCheckItems];
#pragma unroll
    for (int t = 0; t < kCheckItems; ++t)
      if (i0 + (uint64_t)t * threads < e) v[t] = dst[i0 + (uint64_t)t * threads];
#pragma unroll
    for (int t = 0; t < kCheckItems; ++t)
      if (i0 + (uint64_t)t * threads < e) bad |= gidp[v[t]] != g;
  }
  return bad;
}

// Out-degree <= 64: a warp per 32 consecutive nodes, whose edges are one
// contiguous range; an edge's node by binary search over the lanes' offsets.
__global__ void k_many_check_small(uint64_t n, const uint64_t* off, const uint32_t* dst, const uint32_t* gidp,
                                   uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  bool bad = false;
  for (uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 32 < n; w += warps) {
    const uint64_t p = w * 32 + lane;
    const uint64_t base = off[w * 32], end = off[min(w * 32 + 32, n)];
    const uint32_t r = (uint32_t)((p < n ? off[p] : end) - base), T = (uint32_t)(end - base);
    const uint32_t g = p < n ? gidp[p] : 0u;
    for (uint32_t k0 = 0; k0 < T; k0 += 32 * kCheckItems) {
      uint32_t v[kCheckItems], ge[kCheckItems];
#pragma unroll
      for (int t = 0; t < kCheckItems; ++t) {
        const uint32_t k = min(k0 + 32 * t + lane, T - 1);
        v[t] = dst[base + k];
        uint32_t j = 0;
#pragma unroll
        for (uint32_t step = 16; step; step >>= 1)
          if (__shfl_sync(kFullMask, r, j + step) <= k) j += step;
        ge[t] = __shfl_sync(kFullMask, g, j);
      }
#pragma unroll
      for (int t = 0; t < kCheckItems; ++t) bad |= gidp[v[t]] != ge[t];
    }
  }
  if (__any_sync(kFullMask, bad) && lane == 0) atomicOr(err, kErrBadInput);
}

// Larger nodes p0 .. p1-1: a warp per node; hubs: a CTA per chunk.
__global__ void k_many_check_large(uint64_t p0, uint64_t p1, const uint64_t* off, const uint32_t* dst,
                                   const uint32_t* gidp, uint32_t* err) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  bool bad = false;
  for (uint64_t p = p0 + (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); p < p1; p += warps)
    bad |= check_run(off[p], off[p + 1], gidp[p], lane, 32u, dst, gidp);
  if (__any_sync(kFullMask, bad) && lane == 0) atomicOr(err, kErrBadInput);
}

__global__ void k_many_check_hub(uint64_t hub_first, const uint4* chunks, const uint32_t* dst, const uint32_t* gidp,
                                 uint32_t* err) {
  const uint4 c = chunks[blockIdx.x];
  const uint64_t b = ((uint64_t)c.z << 32) | c.y;
  const bool bad = check_run(b, b + c.w, gidp[hub_first + c.x], threadIdx.x, blockDim.x, dst, gidp);
  if (__any_sync(kFullMask, bad) && (threadIdx.x & 31) == 0) atomicOr(err, kErrBadInput);
}

struct ManyArgs {
  uint64_t n_alive;
  const uint32_t* lvl;     // union level, internal order
  const uint8_t* alone;    // union level: node alone in its block
  const uint32_t* p2o;
  const uint32_t* o2p;
  const uint32_t* gid;     // graph of each original node
  const uint32_t* gidp;    // graph of each internal node
  unsigned long long* tkey;  // (graph << 32 | union block), empty = all ones
  uint32_t* tmin;            // smallest original id of the key
  uint64_t tmask;
  uint32_t* slot;          // per internal node: its key's slot
  uint32_t* hbits;         // head bitmap over original ids
  const uint2* hrank;      // (bitmap word, heads before it in its tile)
  const uint32_t* tbase;   // heads before each tile
  uint32_t* err;
};

__device__ __forceinline__ uint32_t many_insert(const ManyArgs& a, unsigned long long key, uint32_t o) {
  uint32_t s = (uint32_t)(mix64(key) & a.tmask);
  for (uint64_t t = 0; t <= a.tmask; ++t) {
    const unsigned long long cur = atomicCAS(&a.tkey[s], (unsigned long long)kEmpty64, key);
    if (cur == kEmpty64 || cur == key) {
      atomicMin(&a.tmin[s], o);
      return s;
    }
    s = (uint32_t)((s + 1) & a.tmask);
  }
  atomicOr(a.err, kErrProbe);
  return 0;
}

// Nodes not alone in their union block: key (graph, block) -> smallest
// original id.  A CTA combines equal keys of its 1024 nodes first.
__global__ void __launch_bounds__(kThreads) k_many_insert(ManyArgs a) {
  __shared__ unsigned long long skey[kAggSlots];
  __shared__ unsigned int smin[kAggSlots];
  __shared__ unsigned int sglob[kAggSlots];
  for (uint64_t base = (uint64_t)blockIdx.x * kAggChunk; base < a.n_alive; base += (uint64_t)gridDim.x * kAggChunk) {
    uint32_t ls[kAggItems], oo[kAggItems];
    uint64_t pp[kAggItems];
    unsigned long long kk[kAggItems];
    bool any = false;
#pragma unroll
    for (int t = 0; t < kAggItems; ++t) {
      const uint64_t p = base + threadIdx.x + (uint64_t)t * kThreads;
      ls[t] = p < a.n_alive && !a.alone[p] ? 0u : kNone32;
      pp[t] = p;
      any |= ls[t] == 0u;
    }
    if (!__syncthreads_or(any)) continue;  // (most chunks of a late level)
#pragma unroll
    for (int t = 0; t < kAggItems; ++t) {
      if (ls[t] == kNone32) continue;
      kk[t] = ((unsigned long long)a.gidp[pp[t]] << 32) | a.lvl[pp[t]];
      oo[t] = a.p2o[pp[t]];
    }
    for (int i = threadIdx.x; i < kAggSlots; i += kThreads) {
      skey[i] = kEmpty64;
      smin[i] = kNone32;
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kAggItems; ++t) {
      if (ls[t] == kNone32) continue;
      uint32_t s = (uint32_t)(mix64(kk[t]) & (kAggSlots - 1));
      for (int q = 0; q < kAggSlots; ++q) {  // at most kAggChunk distinct keys: always room
        const unsigned long long cur = atomicCAS(&skey[s], (unsigned long long)kEmpty64, kk[t]);
        if (cur == kEmpty64 || cur == kk[t]) break;
        s = (s + 1) & (kAggSlots - 1);
      }
      atomicMin(&smin[s], oo[t]);
      ls[t] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kAggSlots; i += kThreads)
      if (skey[i] != kEmpty64) sglob[i] = many_insert(a, skey[i], smin[i]);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kAggItems; ++t)
      if (ls[t] != kNone32) a.slot[pp[t]] = sglob[ls[t]];
    __syncthreads();
  }
}

// Heads: nodes alone in their union block, and the smallest node of each key.
__global__ void k_many_heads(ManyArgs a) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < a.n_alive;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t o = a.p2o[p];
    if (a.alone[p] || a.tmin[a.slot[p]] == o) atomicOr(&a.hbits[o >> 5], 1u << (o & 31));
  }
}

__device__ __forceinline__ uint64_t heads_before(const ManyArgs& a, uint64_t x) {
  const uint2 r = a.hrank[x >> 5];
  return (uint64_t)a.tbase[x >> kRankTileShift] + r.y + (uint64_t)__popc(r.x & ((1u << (x & 31)) - 1u));
}

// Per-graph identifier of every node (original order): rank of its head
// among the heads of its graph.
__global__ void k_many_pid(ManyArgs a, uint64_t n, const uint64_t* start, uint32_t* out) {
  for (uint64_t o = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; o < n; o += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t p = a.o2p[o];
    if (p >= a.n_alive) {
      out[o] = kDead;
      continue;
    }
    const uint32_t head = a.alone[p] ? (uint32_t)o : a.tmin[a.slot[p]];
    out[o] = (uint32_t)(heads_before(a, head) - heads_before(a, start[a.gid[o]]));
  }
}

// cnt[j] = heads before start[j] (j <= G); cnt[G + 1] = the error flags.
__global__ void k_many_counts(ManyArgs a, const uint64_t* start, uint32_t G, unsigned long long* cnt) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j <= G; j += gridDim.x * blockDim.x)
    cnt[j] = heads_before(a, start[j]);
  if (blockIdx.x == 0 && threadIdx.x == 0) cnt[G + 1] = *a.err;
}

// Work list of the next round: nodes of the graphs still refined after level l
// (l < k, and with early stop the level before had fewer blocks), from the
// counts of this level and the one before, so that the host need not be asked.
__global__ void k_many_live_mask(uint64_t n_alive, const uint32_t* gidp, const uint32_t* k, uint32_t l, bool early_stop,
                                 const unsigned long long* cnt, const unsigned long long* cnt_before, uint32_t* mask) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 32 < n_alive; w += warps) {
    const uint64_t p = w * 32 + lane;
    bool live = false;
    if (p < n_alive) {
      const uint32_t g = gidp[p];
      live = l < k[g] && !(early_stop && l >= 1 && cnt[g + 1] - cnt[g] == cnt_before[g + 1] - cnt_before[g]);
    }
    const uint32_t bits = __ballot_sync(kFullMask, live);
    if (lane == 0) mask[w] = bits;
  }
}

}  // namespace

// Per-graph renumbering of level l (called right after the union computed it).
Status many_level(Store& s, uint32_t l) {
  ManyState& m = s.many;
  const uint64_t n = s.n, na = s.n_alive;
  const uint64_t words = n / 32 + 1;  // one spare word: heads_before(n) stays in range
  Status st;
  if (m.lvl.size() < (size_t)l + 1) m.lvl.resize(l + 1);
  if (!(st = ensure(s, m.lvl[l], std::max<uint64_t>(n, 1) * 4)).ok()) return st;
  if (!(st = ensure(s, m.hbits, words * 4 + 16)).ok()) return st;
  if (!(st = ensure(s, m.hword, words * 8)).ok()) return st;
  const uint64_t per = m.G + 4;  // counts of a level: [G + 1], error flags, ticket, number of heads
  if (!(st = ensure(s, m.cnt, 2 * per * 8)).ok()) return st;
  if (!(st = ensure(s, m.live_mask, (na / 32 + 1) * 4)).ok()) return st;
  const uint64_t ins = na - std::min(na, s.n_alone);
  uint64_t cap = 1024;
  while (cap < 2 * ins) cap <<= 1;
  if (!(st = ensure(s, m.tkey, cap * 8)).ok()) return st;
  if (!(st = ensure(s, m.tmin, cap * 4)).ok()) return st;
  if (!(st = ensure(s, m.slot, std::max<uint64_t>(na, 1) * 4)).ok()) return st;
  unsigned long long* cnt = ptr<unsigned long long>(m.cnt) + (l & 1) * per;
  const unsigned long long* cnt_before = ptr<unsigned long long>(m.cnt) + ((l + 1) & 1) * per;
  ManyArgs a;
  a.n_alive = na;
  a.lvl = ptr<uint32_t>(s.level[l]);
  a.alone = ptr<uint8_t>(s.alone);
  a.p2o = ptr<uint32_t>(s.p2o);
  a.o2p = ptr<uint32_t>(s.o2p);
  a.gid = ptr<uint32_t>(m.gid);
  a.gidp = ptr<uint32_t>(m.gidp);
  a.tkey = ptr<unsigned long long>(m.tkey);
  a.tmin = ptr<uint32_t>(m.tmin);
  a.tmask = cap - 1;
  a.slot = ptr<uint32_t>(m.slot);
  a.hbits = ptr<uint32_t>(m.hbits);
  a.hrank = ptr<uint2>(m.hword);
  a.err = ptr<uint32_t>(s.d_err);
  cudaMemsetAsync(cnt + m.G + 2, 0, 8, s.stream);  // the ranks' ticket
  if (!(st = clear_arrays(s, {{m.tkey.p, cap * 8, ~0u}, {m.tmin.p, cap * 4, ~0u}, {m.hbits.p, words * 4, 0u}})).ok())
    return st;
  if (na) {
    k_many_insert<<<grid_for(na, kAggChunk, (int)resident_blocks(k_many_insert, kThreads, 0, s.sms)), kThreads, 0,
                    s.stream>>>(a);
    k_many_heads<<<grid_for(na, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(a);
  }
  if (!(st = rank_heads(s, ptr<uint32_t>(m.hbits), words, ptr<uint2>(m.hword), cnt + m.G + 2)).ok()) return st;
  a.tbase = ptr<uint32_t>(s.bsum);
  k_many_counts<<<grid_for(m.G + 1, kThreads, 64), kThreads, 0, s.stream>>>(a, ptr<uint64_t>(m.dstart), m.G, cnt);
  if (n)
    k_many_pid<<<grid_for(n, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(a, n, ptr<uint64_t>(m.dstart),
                                                                             ptr<uint32_t>(m.lvl[l]));
  // the next round's work list, used while some graphs have stopped and others
  // go on: the nodes of the others keep their blocks
  if (na)
    k_many_live_mask<<<grid_for(na, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(
        na, ptr<uint32_t>(m.gidp), ptr<uint32_t>(m.live), l, s.early_stop, cnt, cnt_before, ptr<uint32_t>(m.live_mask));
  if (!(st = cuda_check(cudaGetLastError(), "per-graph renumbering")).ok()) return st;
  std::vector<uint64_t> c(m.G + 2);
  st = cuda_check(cudaMemcpyAsync(c.data(), cnt, (m.G + 2) * 8, cudaMemcpyDeviceToHost, s.stream), "counts");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return st;
  if (c[m.G + 1] & kErrProbe) return Status::Err(KBISIM_ERR_TIMEOUT, "hash table probe bound exceeded");
  if (m.counts.size() < (size_t)l + 1) m.counts.resize(l + 1);
  m.counts[l].resize(m.G);
  for (uint32_t j = 0; j < m.G; ++j) m.counts[l][j] = c[j + 1] - c[j];
  m.levels = l + 1;
  uint64_t nlive = 0;
  for (uint32_t j = 0; j < m.G; ++j)
    nlive += l < m.k[j] && !(s.early_stop && l >= 1 && m.counts[l][j] == m.counts[l - 1][j]) ? 1 : 0;
  m.live_graphs = nlive;
  s.round_mask = nlive && nlive < m.G ? ptr<uint32_t>(m.live_mask) : nullptr;
  return Status::Ok();
}

Status many_check_args(const kbisim_graph* g, const uint64_t* start, uint32_t G, const uint32_t* k,
                       uint32_t* kmax_out) {
  if (!g || !start || !k || G == 0) return Status::Err(KBISIM_ERR_INVALID_ARG, "graph, starts and k are required");
  if (start[0] != 0 || start[G] != g->num_nodes)
    return Status::Err(KBISIM_ERR_INVALID_ARG, "graph_start must run from 0 to num_nodes");
  uint32_t kmax = 0;
  for (uint32_t j = 0; j < G; ++j) {
    if (start[j + 1] < start[j]) return Status::Err(KBISIM_ERR_INVALID_ARG, "graph_start must not decrease");
    if (k[j] > KBISIM_MAX_K) return Status::Err(KBISIM_ERR_INVALID_ARG, "k too large");
    kmax = std::max(kmax, k[j]);
  }
  *kmax_out = kmax;
  return Status::Ok();
}

// After the union is loaded: graph of every node, and no edge between graphs.
Status many_setup(Store& s, const uint64_t* start, uint32_t G, const uint32_t* k) {
  ManyState& m = s.many;
  m.valid = false;
  m.levels = 0;
  m.counts.clear();
  m.G = G;
  m.start.assign(start, start + G + 1);
  m.k.assign(k, k + G);
  const uint64_t n = s.n;
  Status st;
  if (!(st = ensure(s, m.dstart, (G + 1) * 8)).ok()) return st;
  if (!(st = ensure(s, m.gid, std::max<uint64_t>(n, 1) * 4)).ok()) return st;
  if (!(st = ensure(s, m.gidp, std::max<uint64_t>(n, 1) * 4)).ok()) return st;
  cudaMemcpyAsync(m.dstart.p, m.start.data(), (G + 1) * 8, cudaMemcpyHostToDevice, s.stream);
  cudaMemsetAsync(s.d_err.p, 0, 4, s.stream);
  if (!(st = ensure(s, m.live, G * 4)).ok()) return st;
  cudaMemcpyAsync(m.live.p, m.k.data(), G * 4, cudaMemcpyHostToDevice, s.stream);
  if (n) {
    const uint32_t* gidp = ptr<uint32_t>(m.gidp);
    const uint64_t* off = ptr<uint64_t>(s.offsets);
    const uint32_t* dst = ptr<uint32_t>(s.dst);
    uint32_t* err = ptr<uint32_t>(s.d_err);
    k_many_gid<<<grid_for(n, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(n, ptr<uint64_t>(m.dstart), G,
                                                                             ptr<uint32_t>(m.gid));
    k_many_gidp<<<grid_for(n, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(n, ptr<uint32_t>(s.p2o),
                                                                              ptr<uint32_t>(m.gid), ptr<uint32_t>(m.gidp));
    const uint64_t small = s.class_start[kClassWarp], hub = s.class_start[kClassHub];
    if (small) k_many_check_small<<<grid_for(small, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(small, off, dst, gidp, err);
    if (hub > small)
      k_many_check_large<<<grid_for((hub - small) * 32, kThreads, s.sms * 16), kThreads, 0, s.stream>>>(small, hub, off,
                                                                                                        dst, gidp, err);
    if (s.n_hub_chunks)
      k_many_check_hub<<<(unsigned)s.n_hub_chunks, kThreads, 0, s.stream>>>(hub, ptr<uint4>(s.hub_chunks), dst, gidp, err);
  }
  uint32_t e = 0;
  st = cuda_check(cudaGetLastError(), "graph ids");
  if (st.ok()) st = cuda_check(cudaMemcpyAsync(&e, s.d_err.p, 4, cudaMemcpyDeviceToHost, s.stream), "check");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  if (!st.ok()) return st;
  if (e) return Status::Err(KBISIM_ERR_INVALID_ARG, "an edge joins two graphs of the batch");
  return Status::Ok();
}

// Per-graph rounds (early stop on the graph's own counts) after the union run.
void many_finish(Store& s) {
  ManyState& m = s.many;
  m.rounds.assign(m.G, 0);
  for (uint32_t j = 0; j < m.G; ++j) {
    uint32_t r = m.k[j];
    if (s.early_stop)
      for (uint32_t i = 1; i <= m.k[j] && i < m.levels; ++i)
        if (m.counts[i][j] == m.counts[i - 1][j]) {
          r = i;
          break;
        }
    m.rounds[j] = r;
  }
  m.valid = true;
}

Status many_pids(Store& s, uint32_t j, uint32_t level, uint32_t* dst, bool dst_on_device) {
  const ManyState& m = s.many;
  if (!m.valid) return Status::Err(KBISIM_ERR_STATE, "no batched result");
  if (j >= m.G || level > m.k[j] || !dst) return Status::Err(KBISIM_ERR_INVALID_ARG, "bad graph or level");
  const uint32_t l = std::min<uint32_t>(std::min(level, m.rounds[j]), m.levels - 1);
  const uint64_t nj = m.start[j + 1] - m.start[j];
  if (!nj) return Status::Ok();
  Status st = cuda_check(cudaMemcpyAsync(dst, ptr<uint32_t>(m.lvl[l]) + m.start[j], nj * 4,
                                         dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                         s.stream), "copy out");
  if (st.ok()) st = cuda_check(cudaStreamSynchronize(s.stream), "sync");
  return st;
}

Status many_info(const Store& s, uint32_t j, uint32_t* rounds_run, uint64_t* counts) {
  const ManyState& m = s.many;
  if (!m.valid) return Status::Err(KBISIM_ERR_STATE, "no batched result");
  if (j >= m.G) return Status::Err(KBISIM_ERR_INVALID_ARG, "bad graph");
  if (rounds_run) *rounds_run = m.rounds[j];
  if (counts)
    for (uint32_t l = 0; l <= m.k[j]; ++l)
      counts[l] = m.counts[std::min<uint32_t>(std::min(l, m.rounds[j]), m.levels - 1)][j];
  return Status::Ok();
}

void many_release(Store& s) {
  ManyState& m = s.many;
  for (Buf& b : m.lvl) release(s, b);
  m.lvl.clear();
  Buf* bufs[] = {&m.dstart, &m.gid, &m.gidp, &m.tkey, &m.tmin, &m.slot, &m.hbits, &m.hword, &m.cnt, &m.live,
                 &m.live_mask};
  for (Buf* b : bufs) release(s, *b);
  m.valid = false;
}

}  // namespace kb
