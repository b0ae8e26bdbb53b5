// truss_support_noalloc: per-row edge support for small graphs without any
// memory allocation.
//
// Some callers cannot allocate device memory at the time they need a result:
// code running inside a memory pool or allocator callback, a host that has
// handed the whole device to another allocator, or a section that must not
// enter the CUDA allocator (and so must not synchronise with it).  For them,
// this entry point keeps all of its working memory in one fixed array that
// lives in the library's device image (file-scope `static __device__`),
// reserved on every GPU that loads the library until the process exits.
// The caller passes device-accessible input and output buffers; nothing else
// is allocated, neither here nor in a library routine.
//
// The work is the support computation of truss_support (Definition 1):
// distinct edges through an open-addressing hash table, degrees, out-lists
// (every edge points from its end of lower degree to the other), then for
// each edge (u, v) the entries w of out(u) with (v, w) in the table: the
// triangles whose lowest vertex is u.  Both (u, v) and (u, w) find the
// triangle on their own walk, and the one with v < w adds it to (v, w).
// Finally a per-row lookup.  Out-lists keep the walks short next to hubs and
// spare the hubs' counters (whole lists, walked from the shorter end: support
// step 47 us and list step 12 us of 60,001 R-MAT rows, now 17 us and 6 us).
// Each step is a kernel over the whole chip; the launch order separates them.
// What bounds it are the dependent L2 round trips of each step and six
// launches.  One block did all of it before, on one SM of 152: 60,001 R-MAT
// rows took 6,406 us a call, now 76 us.
#include <mutex>

#include "engine.h"

namespace {

constexpr int kMaxRows = TRUSS_NOALLOC_MAX_ROWS;
constexpr int kMaxN = TRUSS_NOALLOC_MAX_N;
constexpr int kSlots = 4 * kMaxRows;  // hash slots (load <= 1/4)
constexpr int kThreads = 256;
constexpr int kGroup = 16;  // lanes that walk the out-list of one edge's lower end
constexpr unsigned long long kEmpty = ~0ull;

// Layout of the scratch array (element counts).
constexpr size_t kKeysBytes = sizeof(unsigned long long) * kSlots;
constexpr size_t kIntsCount = (size_t)kSlots      // edge id per slot
                              + 3 * (size_t)(kMaxN + 1)  // degree, offset, cursor
                              + 2 * (size_t)kMaxRows     // edge endpoints
                              + 2 * (size_t)kMaxRows     // adjacency
                              + (size_t)kMaxRows         // support per edge
                              + 3;                       // edges, adjacency entries, error flag
constexpr size_t kScratchBytes = kKeysBytes + sizeof(int32_t) * kIntsCount;

// The only working memory of truss_support_noalloc.  Shared by every call on
// a device: each call re-initialises what it reads before using it.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// The parts of the scratch array, for a table of `mask` + 1 slots.
struct Scratch {
  unsigned long long *keys;
  int32_t *ids, *deg, *off, *cur, *eu, *ev, *adj, *sup;
  int32_t *ctr;  // [0] distinct edges, [1] adjacency entries, [2] invalid-id flag
  unsigned mask;
};

Scratch scratch_parts(unsigned char *base, unsigned mask) {
  Scratch a;
  a.keys = (unsigned long long *)base;
  a.ids = (int32_t *)(base + kKeysBytes);
  a.deg = a.ids + kSlots;
  a.off = a.deg + (kMaxN + 1);
  a.cur = a.off + (kMaxN + 1);
  a.eu = a.cur + (kMaxN + 1);
  a.ev = a.eu + kMaxRows;
  a.adj = a.ev + kMaxRows;
  a.sup = a.adj + 2 * kMaxRows;
  a.ctr = a.sup + kMaxRows;
  a.mask = mask;
  return a;
}

__device__ __forceinline__ unsigned slot_of(unsigned long long key, unsigned mask) {
  return (unsigned)((key * 0x9E3779B97F4A7C15ull) >> 40) & mask;
}

__device__ __forceinline__ unsigned long long edge_key(int u, int v) {
  return ((unsigned long long)(unsigned)min(u, v) << 32) | (unsigned)max(u, v);
}

__device__ __forceinline__ int find_slot(const Scratch &a, unsigned long long key) {
  unsigned h = slot_of(key, a.mask);
  for (unsigned probe = 0; probe <= a.mask; probe++) {
    const unsigned long long k = __ldg(&a.keys[h]);
    if (k == key) return (int)h;
    if (k == kEmpty) return -1;
    h = (h + 1) & a.mask;
  }
  return -1;
}

// 0. clear what this call reads (the array keeps the last call's data)
__global__ void __launch_bounds__(kThreads) k_na_clear(int n, int rows, Scratch a) {
  const int i0 = blockIdx.x * kThreads + threadIdx.x, step = gridDim.x * kThreads;
  ulonglong2 *k2 = (ulonglong2 *)a.keys;
  for (int i = i0; i < (int)((a.mask + 1) / 2); i += step) k2[i] = make_ulonglong2(kEmpty, kEmpty);
  for (int i = i0; i <= n; i += step) {
    a.deg[i] = 0;
    a.cur[i] = 0;
  }
  for (int i = i0; i < rows; i += step) a.sup[i] = 0;
  if (i0 < 3) a.ctr[i0] = 0;
}

// 1. distinct undirected edges into the hash table; the thread that fills a
// slot gives the edge its id and counts its degrees
__global__ void __launch_bounds__(kThreads) k_na_insert(int n, int rows, const int32_t *src,
                                                        const int32_t *dst, Scratch a) {
  const int step = gridDim.x * kThreads;
  for (int r0 = blockIdx.x * kThreads; r0 < rows; r0 += step) {  // whole warps stay together
    const int r = r0 + threadIdx.x;
    int u = 0, v = 0;
    bool fresh = false;
    unsigned h = 0;
    if (r < rows) {
      u = src[r];
      v = dst[r];
      if (u < 0 || u >= n || v < 0 || v >= n) {
        atomicExch(&a.ctr[2], 1);  // the host reports it
      } else if (u != v) {
        const unsigned long long key = edge_key(u, v);
        h = slot_of(key, a.mask);
        for (;;) {
          const unsigned long long prev = atomicCAS(&a.keys[h], kEmpty, key);
          fresh = prev == kEmpty;
          if (fresh || prev == key) break;
          h = (h + 1) & a.mask;
        }
      }
    }
    const int id = tr::warp_append(fresh, &a.ctr[0]);
    if (fresh) {
      a.ids[h] = id;
      a.eu[id] = u;
      a.ev[id] = v;
      atomicAdd(&a.deg[u], 1);
      atomicAdd(&a.deg[v], 1);
    }
  }
}

// 2. a stretch of the adjacency array for each vertex (its degree bounds its
// out-list), in any order
__global__ void __launch_bounds__(kThreads) k_na_offsets(int n, Scratch a) {
  const int step = gridDim.x * kThreads, lane = tr::lane_id();
  for (int v0 = blockIdx.x * kThreads; v0 < n; v0 += step) {
    const int v = v0 + threadIdx.x;
    const int d = v < n ? a.deg[v] : 0;
    const int P = tr::warp_incl_scan(d);
    int base = 0;
    if (lane == 31 && P > 0) base = atomicAdd(&a.ctr[1], P);
    base = __shfl_sync(TR_FULL, base, 31);
    if (v < n) a.off[v] = base + P - d;
  }
}

// 3. out-lists: an edge's end of lower (degree, id) lists the other
__global__ void __launch_bounds__(kThreads) k_na_fill(Scratch a) {
  const int m = a.ctr[0], step = gridDim.x * kThreads;
  for (int id = blockIdx.x * kThreads + threadIdx.x; id < m; id += step) {
    int u = a.eu[id], v = a.ev[id];
    const int du = a.deg[u], dv = a.deg[v];
    if (dv < du || (dv == du && v < u)) {
      const int t = u;
      u = v;
      v = t;
      a.eu[id] = u;
      a.ev[id] = v;
    }
    a.adj[a.off[u] + atomicAdd(&a.cur[u], 1)] = v;
  }
}

// 4. support: kGroup lanes walk out(u) for one edge (u, v)
__global__ void __launch_bounds__(kThreads) k_na_support(Scratch a) {
  const int m = a.ctr[0], step = gridDim.x * (kThreads / kGroup);
  const int j = threadIdx.x % kGroup, first = (threadIdx.x % 32) / kGroup;
  // whole warps stay together: i0 - first is the warp's first edge
  for (int i0 = (blockIdx.x * kThreads + threadIdx.x) / kGroup; i0 - first < m; i0 += step) {
    int c = 0;
    if (i0 < m) {
      const int u = a.eu[i0], v = a.ev[i0];
      const int d = a.cur[u], o = a.off[u];
      for (int i = j; i < d; i += kGroup) {
        const int w = __ldg(&a.adj[o + i]);
        if (w == v) continue;
        const int sl = find_slot(a, edge_key(v, w));
        if (sl < 0) continue;
        c++;
        if (v < w) atomicAdd(&a.sup[a.ids[sl]], 1);
      }
    }
#pragma unroll
    for (int o = kGroup / 2; o >= 1; o >>= 1) c += __shfl_xor_sync(TR_FULL, c, o);
    if (i0 < m && j == 0 && c > 0) atomicAdd(&a.sup[i0], c);
  }
}

// 5. per-row output
__global__ void __launch_bounds__(kThreads) k_na_rows(int rows, const int32_t *src,
                                                      const int32_t *dst, int32_t *support_out,
                                                      Scratch a) {
  if (a.ctr[2] != 0) return;  // vertex id out of range: the host reports it
  const int step = gridDim.x * kThreads;
  for (int r = blockIdx.x * kThreads + threadIdx.x; r < rows; r += step) {
    const int u = src[r], v = dst[r];
    int out = -1;
    if (u != v) {
      const int sl = find_slot(a, edge_key(u, v));
      out = sl >= 0 ? a.sup[a.ids[sl]] : -1;
    }
    support_out[r] = out;
  }
}

// Device address of the scratch array, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_setup_mu;
unsigned char *g_scratch_addr[kMaxDevices] = {};

int scratch_for_current_device(unsigned char **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return TRUSS_ECUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) return TRUSS_EINVAL;
  std::lock_guard<std::mutex> lk(g_setup_mu);
  if (!g_scratch_addr[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
      cudaGetLastError();
      return TRUSS_ECUDA;
    }
    g_scratch_addr[dev] = (unsigned char *)p;
  }
  *out = g_scratch_addr[dev];
  return TRUSS_OK;
}

// True if the kernel, launched on device `dev`, may dereference p as given:
// memory of that same device, managed memory, or pinned host memory mapped
// at the same address.  Memory of another GPU is refused (without peer
// access a kernel reading it would fault), and so is pageable host memory.
bool device_accessible(const void *p, int dev) {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  switch (at.type) {
    case cudaMemoryTypeDevice: return at.device == dev;
    case cudaMemoryTypeManaged: return true;
    case cudaMemoryTypeHost: return at.devicePointer == p;
    default: return false;
  }
}

}  // namespace

extern "C" int truss_support_noalloc(int64_t n, int64_t rows, const int32_t *src,
                                     const int32_t *dst, int32_t *support_out,
                                     void *cuda_stream) {
  if (n < 0 || rows < 0 || n > kMaxN || rows > kMaxRows) return TRUSS_EINVAL;
  if (rows == 0) return TRUSS_OK;
  if (!src || !dst || !support_out || n == 0) return TRUSS_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return TRUSS_ECUDA;
  }
  if (!device_accessible(src, dev) || !device_accessible(dst, dev) ||
      !device_accessible(support_out, dev))
    return TRUSS_EINVAL;
  unsigned char *scratch = nullptr;
  TR_TRY(scratch_for_current_device(&scratch));
  cudaStream_t s = (cudaStream_t)cuda_stream;
  // table of at least 4 slots per row: load at most 1/4
  unsigned slots = 1024;
  while (slots < 4u * (unsigned)rows) slots *= 2;
  const Scratch a = scratch_parts(scratch, slots - 1);
  const int nn = (int)n, nr = (int)rows;
  auto grid = [](int64_t threads) { return tr::grid_for(threads, kThreads, 152 * 8); };
  k_na_clear<<<grid(slots / 2 > (unsigned)n + 1 ? slots / 2 : n + 1), kThreads, 0, s>>>(nn, nr, a);
  k_na_insert<<<grid(rows), kThreads, 0, s>>>(nn, nr, src, dst, a);
  k_na_offsets<<<grid(n), kThreads, 0, s>>>(nn, a);
  k_na_fill<<<grid(rows), kThreads, 0, s>>>(a);
  k_na_support<<<grid(rows * kGroup), kThreads, 0, s>>>(a);
  k_na_rows<<<grid(rows), kThreads, 0, s>>>(nr, src, dst, support_out, a);
  if (cudaGetLastError() != cudaSuccess) return TRUSS_ECUDA;
  // the invalid-id flag lives in the scratch array; read it back
  int32_t flag = 0;
  const size_t flag_off = kKeysBytes + sizeof(int32_t) * (kIntsCount - 1);
  if (cudaMemcpyAsync(&flag, scratch + flag_off, sizeof(int32_t), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return TRUSS_ECUDA;
  }
  return flag != 0 ? TRUSS_EINVAL : TRUSS_OK;
}
