// Label partition (identifier level 0) without any device allocation.
//
// Some callers cannot allocate device memory when they need this result:
// a serving loop whose device memory is fully reserved up front by another
// allocator (a framework's caching pool, a fixed arena), or code that must
// not risk the implicit device-wide synchronisation that cudaMalloc and
// cudaFree may perform.  For them, kbisim_label_partition_noalloc computes
// the same level 0 as kbisim_refine (blocks of equal node labels, numbered by
// their smallest node id) using only the caller's input and output buffers
// and a fixed scratch area that lives in this library's static device memory.
//
// The scratch area below is allocated when the library is loaded onto a
// device and stays there until the process exits (every GPU that loads the
// library holds it).  It bounds the input size: num_nodes <= kMaxNodes.
// All calls share it and it keeps the last call's contents, so each call
// clears what must start empty, and calls that overlap on the GPU (different
// streams, or different host threads without ordering) race on it.
//
// Host code only ever sees a host-side stand-in for the array's name, so the
// device address is looked up with cudaGetSymbolAddress once per device (with
// that device current) on the first call, which should therefore come before
// any stream capture.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "kbisim.h"

namespace {

constexpr uint64_t kMaxNodes = 1ull << 18;          // 262,144 nodes
constexpr uint64_t kSlots = 2 * kMaxNodes;          // hash table slots (power of two)
constexpr int kThreads = 1024;                      // head kernel: one node per thread
static_assert(kThreads == 1024, "one warp sums the warps");
constexpr uint64_t kTiles = kMaxNodes / kThreads;   // 256
constexpr unsigned long long kEmptySlot = ~0ull;

struct Scratch {
  unsigned long long table[kSlots];  // (label << 32) | smallest node id with that label
  uint32_t rank[kMaxNodes];          // of a head: heads before it in its tile
  uint32_t tile[kTiles];             // heads per tile, then heads before the tile
  uint32_t ticket;                   // tiles counted
};

static __device__ __align__(256) Scratch g_scratch;

constexpr int kMaxDevices = 64;
Scratch* g_dev_ptr[kMaxDevices] = {nullptr};
std::mutex g_mu;

__device__ __forceinline__ uint32_t home_slot(uint32_t label, uint64_t mask) {
  uint32_t x = label;  // MurmurHash3 32-bit finalizer spreads labels over the table
  x ^= x >> 16;
  x *= 0x85ebca6bu;
  x ^= x >> 13;
  x *= 0xc2b2ae35u;
  x ^= x >> 16;
  return (uint32_t)(x & mask);
}

// The slot of `label`, inserting (label, u) on the way when `insert` is set.
// An empty slot reads as label 0xFFFFFFFF, which a node with that label then
// claims with the same atomicMin; probing is bounded by the table size.
__device__ __forceinline__ int64_t find_slot(Scratch* sc, uint32_t label, uint32_t u, uint64_t mask, bool insert) {
  uint64_t s = home_slot(label, mask);
  const unsigned long long v = ((unsigned long long)label << 32) | u;
  for (uint64_t t = 0; t <= mask; ++t) {
    unsigned long long cur = *(volatile unsigned long long*)&sc->table[s];
    if (cur == kEmptySlot && insert) {
      cur = atomicCAS(&sc->table[s], kEmptySlot, v);
      if (cur == kEmptySlot) return (int64_t)s;
    }
    if ((uint32_t)(cur >> 32) == label) {
      if (insert && (uint32_t)cur > u) atomicMin(&sc->table[s], v);
      return (int64_t)s;
    }
    s = (s + 1) & mask;
  }
  return -1;
}

// Four launches, each started while the one before still runs
// (programmatic dependent launch) and waiting for it before its first access:
// at 262,144 nodes the work is a few microseconds a step, and six launches in
// a row (with the tile scan and the ranks in launches of their own) took 33 us.
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__global__ void k_na_clear(Scratch* sc, uint64_t slots) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  ulonglong2* t = reinterpret_cast<ulonglong2*>(sc->table);
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < slots / 2; i += (uint64_t)gridDim.x * blockDim.x)
    t[i] = make_ulonglong2(kEmptySlot, kEmptySlot);
  if (blockIdx.x == 0 && threadIdx.x == 0) sc->ticket = 0;
}

__global__ void k_na_insert(Scratch* sc, const uint32_t* label, uint64_t n, uint64_t mask) {
  after_previous();
  for (uint64_t u = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; u < n; u += (uint64_t)gridDim.x * blockDim.x)
    find_slot(sc, label[u], (uint32_t)u, mask, true);
}

// Exclusive sum of v over the CTA of kThreads; *total gets the CTA's sum.
__device__ __forceinline__ uint32_t cta_before(uint32_t v, uint32_t* warp_sum, uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  if (lane == 31) warp_sum[w] = x;
  __syncthreads();
  const uint32_t s = warp_sum[lane];  // kThreads / 32 = 32 warps
  *total = __reduce_add_sync(0xFFFFFFFFu, s);
  const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < w ? s : 0u);
  __syncthreads();
  return before + x - v;
}

// Heads (the smallest node of each label): their rank in their tile; the CTA
// that comes last (a ticket: nothing waits) turns the tiles' head counts into
// heads before each tile and writes the block count.
__global__ void __launch_bounds__(kThreads) k_na_heads(Scratch* sc, const uint32_t* label, uint64_t n, uint64_t mask,
                                                       uint32_t* count_out) {
  after_previous();
  __shared__ uint32_t warp_sum[kThreads / 32];
  __shared__ uint32_t last;
  const uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
  uint32_t head = 0, total;
  if (u < n) {
    const int64_t s = find_slot(sc, label[u], (uint32_t)u, mask, false);
    head = (s >= 0 && (uint32_t)sc->table[s] == (uint32_t)u) ? 1u : 0u;
  }
  const uint32_t before = cta_before(head, warp_sum, &total);
  if (head) sc->rank[u] = before;
  if (threadIdx.x == 0) {
    sc->tile[blockIdx.x] = total;
    __threadfence();
    last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const uint32_t t = threadIdx.x;
  const uint32_t v = t < gridDim.x ? __ldcg(&sc->tile[t]) : 0u;
  const uint32_t tb = cta_before(v, warp_sum, &total);
  if (t < gridDim.x) sc->tile[t] = tb;
  if (t == 0 && count_out) *count_out = total;
}

__global__ void k_na_assign(Scratch* sc, const uint32_t* label, uint64_t n, uint64_t mask, uint32_t* pid0) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (uint64_t u = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; u < n; u += (uint64_t)gridDim.x * blockDim.x) {
    const int64_t s = find_slot(sc, label[u], (uint32_t)u, mask, false);
    const uint32_t head = s >= 0 ? (uint32_t)sc->table[s] : 0u;
    pid0[u] = s >= 0 ? sc->tile[head / kThreads] + sc->rank[head] : KBISIM_DELETED;
  }
}

template <typename... P, typename... A>
cudaError_t launch_after(cudaStream_t st, bool overlap, void (*kernel)(P...), unsigned blocks, unsigned threads, A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(threads);
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace

extern "C" int kbisim_label_partition_noalloc(const uint32_t* node_label, uint64_t num_nodes, uint32_t* pid0,
                                              uint32_t* block_count, void* stream) {
  if (num_nodes > kMaxNodes) return KBISIM_ERR_INVALID_ARG;
  if (num_nodes && (!node_label || !pid0)) return KBISIM_ERR_INVALID_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return KBISIM_ERR_CUDA;
  }
  Scratch* sc = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_dev_ptr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) {
        cudaGetLastError();
        return KBISIM_ERR_CUDA;
      }
      g_dev_ptr[dev] = static_cast<Scratch*>(p);
    }
    sc = g_dev_ptr[dev];
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (num_nodes == 0) {
    if (block_count && cudaMemsetAsync(block_count, 0, sizeof(uint32_t), st) != cudaSuccess) return KBISIM_ERR_CUDA;
    return KBISIM_OK;
  }
  uint64_t slots = 1024;
  while (slots < 2 * num_nodes) slots <<= 1;
  const uint64_t mask = slots - 1;
  const uint64_t ntiles = (num_nodes + kThreads - 1) / kThreads;
  const unsigned g = (unsigned)((num_nodes + 255) / 256);
  launch_after(st, false, k_na_clear, (unsigned)((slots / 2 + 255) / 256), 256, sc, slots);
  launch_after(st, true, k_na_insert, g, 256, sc, node_label, num_nodes, mask);
  launch_after(st, true, k_na_heads, (unsigned)ntiles, kThreads, sc, node_label, num_nodes, mask, block_count);
  launch_after(st, true, k_na_assign, g, 256, sc, node_label, num_nodes, mask, pid0);
  return cudaGetLastError() == cudaSuccess ? KBISIM_OK : KBISIM_ERR_CUDA;
}
