// Small graphs: the CSR build with everything the support walk needs from it,
// and the list offsets, each in one cooperative launch.
//
// The general path (build.cu, run_support, run_lists) sorts and scans with
// device-wide passes: about 45 launches around the walk and the peel, 2 to 11
// us each whatever the size, which is most of a small call.  Here the steps
// are phases of one kernel and no step needs a sort:
//  * distinct edges through a hash table (load at most 1/2);
//  * rank by (degree, id): a stable counting sort of the low degrees, the few
//    vertices of higher degree by counting those before them;
//  * each edge goes to its tail's list through a cursor, and its place in the
//    list is the number of heads below its own, counted against the list
//    itself (sum of squared out-degrees, about the work of the support walk);
//    lists of more than kLongList are sorted first, by a block each;
//  * the edges grouped by head take a cursor per head, once per group of
//    lanes with the same head.
// What bounds it: a few dependent L2 round trips (540 clocks each) and a grid
// barrier (1.3 us) per phase, then the hash table's and the cursors' atomics.
//
// Decompose, general path / here (ms): 1.5 M R-MAT rows over 262,144 vertices
// 5.87 / 5.60, 2.1 M 7.97 / 7.71, 2.6 M 9.54 / 9.59; 2.6 M Chung-Lu rows over
// 1,048,576 vertices 8.19 / 8.42, random rows 1.40 / 1.28.  Support alone: 65 K
// R-MAT rows over 16,384 vertices 0.46 / 0.17, 262 K 0.53 / 0.27, 1.05 M 0.98 /
// 0.86.  Above kSmallRows rows the table and the lists leave L2, and the sorts,
// which stream, are faster.
#include <climits>
#include <cstdlib>

#include "engine.h"

namespace tr {

namespace {

constexpr int kBlock = 512;
constexpr unsigned long long kEmpty = ~0ull;

// Grid-wide exclusive prefix sums of K values per element, i = 0 .. N-1: put
// receives each element's prefixes, total the sums.  Every block takes one
// contiguous chunk; part holds gridDim.x sums per value.  A tile's sums fit 31
// bits (the callers' values are below 2^22).  Ends without a barrier.
template <int K, class Get, class Put>
__device__ __forceinline__ bool grid_scan(unsigned long long *bar, int *err, long long wait_ns,
                                          int64_t N, int64_t *part, int64_t (&total)[K], Get get,
                                          Put put) {
  __shared__ int s_w[K][kBlock / 32];
  __shared__ int64_t s_base[K], s_tot[K];
  const int lane = lane_id(), wib = threadIdx.x >> 5;
  const int64_t chunk = (N + gridDim.x - 1) / gridDim.x;
  const int64_t i0 = min(N, chunk * blockIdx.x), i1 = min(N, i0 + chunk);
  int64_t sum[K];
#pragma unroll
  for (int q = 0; q < K; q++) sum[q] = 0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kBlock) {
    int v[K];
    get(i, v);
#pragma unroll
    for (int q = 0; q < K; q++) sum[q] += v[q];
  }
  if (threadIdx.x < K) s_base[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < K; q++) {
    for (int o = 16; o >= 1; o >>= 1) sum[q] += __shfl_down_sync(TR_FULL, sum[q], o);
    if (lane == 0 && sum[q]) atomicAdd((unsigned long long *)&s_base[q], (unsigned long long)sum[q]);
  }
  __syncthreads();
  if (threadIdx.x < K) part[threadIdx.x * gridDim.x + blockIdx.x] = s_base[threadIdx.x];
  if (!grid_barrier(bar, err, wait_ns)) return false;
  // a warp per value: sums of the blocks before this one, and of all
  for (int q = wib; q < K; q += kBlock / 32) {
    int64_t before = 0, all = 0;
    for (int j = lane; j < (int)gridDim.x; j += 32) {
      const int64_t x = __ldcg(&part[q * gridDim.x + j]);
      all += x;
      if (j < (int)blockIdx.x) before += x;
    }
    for (int o = 16; o >= 1; o >>= 1) {
      before += __shfl_down_sync(TR_FULL, before, o);
      all += __shfl_down_sync(TR_FULL, all, o);
    }
    if (lane == 0) {
      s_base[q] = before;
      s_tot[q] = all;
    }
  }
  __syncthreads();
  int64_t base[K];
#pragma unroll
  for (int q = 0; q < K; q++) {
    base[q] = s_base[q];
    total[q] = s_tot[q];
  }
  for (int64_t t0 = i0; t0 < i1; t0 += kBlock) {
    const int64_t i = t0 + threadIdx.x;
    int v[K], P[K];
    if (i < i1) {
      get(i, v);
    } else {
#pragma unroll
      for (int q = 0; q < K; q++) v[q] = 0;
    }
#pragma unroll
    for (int q = 0; q < K; q++) {
      P[q] = warp_incl_scan(v[q]);
      if (lane == 31) s_w[q][wib] = P[q];
    }
    __syncthreads();
    int64_t ex[K];
#pragma unroll
    for (int q = 0; q < K; q++) {
      const int w = lane < kBlock / 32 ? s_w[q][lane] : 0;
      const int S = warp_incl_scan(w);
      const int before = __shfl_sync(TR_FULL, S - w, wib);
      ex[q] = base[q] + before + P[q] - v[q];
      base[q] += __shfl_sync(TR_FULL, S, 31);
    }
    if (i < i1) put(i, ex, v);
    __syncthreads();
  }
  return true;
}

// The lanes with this lane's key (only itself if not ok); a key is not negative.
// RUNS: looked for only where two neighbouring lanes share one, which is enough
// against the hot counters of hubs and repeated rows; a match by every warp
// lengthens each of the steps that use it by 3 to 8 % on random rows.
template <bool RUNS, class K>
__device__ __forceinline__ unsigned lanes_alike(bool ok, K key) {
  const K k = ok ? key : ~(K)lane_id();
  if (RUNS) {
    const K left = __shfl_up_sync(TR_FULL, k, 1);
    if (!__any_sync(TR_FULL, lane_id() > 0 && left == k)) return 1u << lane_id();
  }
  return __match_any_sync(TR_FULL, k);
}

// One atomic per group of lanes with the same key: the group's total is added
// to ctr[key]; returns this lane's slot.  All lanes call it (ok masks).
template <bool RUNS>
__device__ __forceinline__ int grouped_slot(bool ok, int key, int *ctr) {
  const unsigned peers = lanes_alike<RUNS>(ok, key);
  const int first = __ffs(peers) - 1;
  int c = 0;
  if (ok && lane_id() == first) c = atomicAdd(&ctr[key], __popc(peers));
  c = __shfl_sync(TR_FULL, c, first);
  return c + __popc(peers & ((1u << lane_id()) - 1u));
}

// The same without the slots.  (A counter per lane serialises on hubs: support
// of 2.4 M edges of four of them 2.58 ms, now 0.78; of K_1200, where a tail's
// edges come together, 1.79, now 1.22.)
__device__ __forceinline__ void grouped_add(bool ok, int key, int *ctr) {
  const unsigned peers = lanes_alike<true>(ok, key);
  if (ok && lane_id() == __ffs(peers) - 1) atomicAdd(&ctr[key], __popc(peers));
}

constexpr int kLow = 256;       // degrees sorted by counting
// Out-lists of more than kLongList entries are sorted by a block each, shorter
// ones by counting (262 K edges of lists of 512: support 0.23 -> 0.20 ms).
// kSortCap: an out-list of d heads, each of degree d or more, needs d * d <= 2 m.
constexpr int kLongList = 384;
constexpr int kSortCap = 2304;

// Sort d keys in shared memory by the whole block: a bitonic network whose
// merges all ascend (each begins by comparing mirrored positions), so that
// positions from d on, which would hold the largest keys, need no memory.
__device__ __forceinline__ void block_sort(unsigned long long *x, int d) {
  int N = 2;
  while (N < d) N *= 2;
  for (int k = 2; k <= N; k *= 2)
    for (int j = k / 2; j > 0; j /= 2) {
      __syncthreads();
      for (int i = threadIdx.x; i < N / 2; i += kBlock) {
        const int r = i & (j - 1), lo = 2 * i - r;
        const int hi = j == k / 2 ? lo + k - 1 - 2 * r : lo + j;
        if (hi < d) {
          const unsigned long long a = x[lo], b = x[hi];
          if (a > b) {
            x[lo] = b;
            x[hi] = a;
          }
        }
      }
    }
  __syncthreads();
}

struct SmallCtl {
  unsigned long long bar;
  int err;       // barrier time-out
  int m, bad;    // distinct edges; non-zero: a vertex id out of range
  int high;      // vertices of degree kLow or more
  int longs;     // out-lists of more than kLongList entries
  int64_t W, R;  // walk cost, record slots
  int64_t P;     // walk ranges
};

struct SmallArgs {
  RowsIn in;
  SmallCtl *ctl;
  long long wait_ns;
  int64_t *part;
  unsigned long long *keys;  // mask + 1 slots
  unsigned mask;
  int32_t *slot_id, *row_slot;
  int32_t *eu, *ev;        // [rows] ends of edge id (after the ranks: tail, head)
  int32_t *deg, *hist;     // [n], [kLow * blocks]
  int2 *high;              // (degree, vertex) of the high degrees; then the long out-lists
  int32_t *outc, *curo, *curi;  // [n]
  int32_t *lt, *lh, *lid;  // [rows] unsorted lists: tail, head, edge id
  int32_t *newid, *lex2e;
  // results
  int32_t *sdeg, *order;
  int64_t *offp, *inoff;
  int32_t *adjp, *esrc, *row2e, *inedge, *ihead;
  int64_t *wcost, *bound, *wpre, *tbpre;
  int32_t *supA, *supB, *cuv;  // zeroed here for the walk (cuv: with records)
  int ecost;
  int64_t range_work, warps;  // how the walk is cut into ranges
  int64_t *rb;
};

__global__ void __launch_bounds__(kBlock, 2) k_small_build(SmallArgs a) {
  SmallCtl *ctl = a.ctl;
  const int64_t n = a.in.n, rows = a.in.rows;
  const int64_t tid = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * kBlock;
  auto sync = [&]() { return grid_barrier(&ctl->bar, &ctl->err, a.wait_ns); };
  if (a.wait_ns < 0 && tid == 0) raise_error(&ctl->bar, &ctl->err, TRUSS_ETIMEOUT);
  // 0. clear
  {
    ulonglong2 *k2 = (ulonglong2 *)a.keys;
    for (int64_t i = tid; i < ((int64_t)a.mask + 1) / 2; i += nt)
      k2[i] = make_ulonglong2(kEmpty, kEmpty);
    for (int64_t v = tid; v < n; v += nt) {
      a.deg[v] = 0;
      a.outc[v] = 0;
      a.curo[v] = 0;
      a.curi[v] = 0;
    }
    for (int64_t e = tid; e < rows; e += nt) {
      a.supA[e] = 0;
      a.supB[e] = 0;
      if (a.cuv) a.cuv[e] = 0;
    }
  }
  if (!sync()) return;
  // 1. distinct edges; the thread that fills a slot gives the edge its id
  for (int64_t r0 = (int64_t)blockIdx.x * kBlock; r0 < rows; r0 += nt) {
    const int64_t r = r0 + threadIdx.x;
    int64_t u = 0, v = 0;
    bool ok = false, fresh = false;
    unsigned h = 0;
    unsigned long long key = kEmpty;
    if (r < rows) {
      u = a.in.src[r];
      v = a.in.dst[r];
      int64_t lo = 0, hi = n;
      if (a.in.voff != nullptr) {
        int g = 0, top = a.in.graphs - 1;
        while (g < top) {
          const int mid = (g + top + 1) >> 1;
          if (a.in.row_off[mid] <= r) g = mid; else top = mid - 1;
        }
        lo = a.in.voff[g];
        hi = a.in.voff[g + 1];
        u += lo;
        v += lo;
      }
      if (u < lo || u >= hi || v < lo || v >= hi) {
        atomicExch(&ctl->bad, 1);
      } else if (u != v) {
        ok = true;
        key = (unsigned long long)(u < v ? u : v) << 32 | (unsigned long long)(u < v ? v : u);
      }
    }
    // one lane per edge looks it up (2.6 M rows of one edge, each with a compare
    // and swap on its slot: support 1.85 ms, now 0.22)
    const int first = __ffs(lanes_alike<true>(ok, key)) - 1;
    if (ok && lane_id() == first) {
      h = (unsigned)((key * 0x9E3779B97F4A7C15ull) >> 40) & a.mask;
      for (;;) {
        const unsigned long long prev = atomicCAS(&a.keys[h], kEmpty, key);
        fresh = prev == kEmpty;
        if (fresh || prev == key) break;
        h = (h + 1) & a.mask;
      }
    }
    const int slot = __shfl_sync(TR_FULL, (int)h, first);
    if (r < rows) a.row_slot[r] = ok ? slot : -1;
    const int id = warp_append(fresh, &ctl->m);
    if (fresh) {
      a.slot_id[h] = id;
      a.eu[id] = (int32_t)u;
      a.ev[id] = (int32_t)v;
    }
    grouped_add(fresh, (int)u, a.deg);
    grouped_add(fresh, (int)v, a.deg);
  }
  if (!sync()) return;
  if (__ldcg(&ctl->bad)) return;  // the same in every block
  const int64_t m = __ldcg(&ctl->m);
  // 2. each block counts the vertices of its stretch by degree below kLow; the
  // few of higher degree (at most 2m / kLow) are listed
  __shared__ int s_cnt[kLow];
  __shared__ unsigned short s_warp[kBlock / 32][kLow];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t c0 = min(n, chunk * blockIdx.x), c1 = min(n, c0 + chunk);
  for (int d = threadIdx.x; d < kLow; d += kBlock) {
    s_cnt[d] = 0;
    for (int w = 0; w < kBlock / 32; w++) s_warp[w][d] = 0;
  }
  __syncthreads();
  for (int64_t v0 = c0; v0 < c1; v0 += kBlock) {
    const int64_t v = v0 + threadIdx.x;
    const int d = v < c1 ? __ldcg(&a.deg[v]) : -1;
    const unsigned peers = __match_any_sync(TR_FULL, d);
    if (d >= 0 && d < kLow && lane_id() == __ffs(peers) - 1) atomicAdd(&s_cnt[d], __popc(peers));
    const int at = warp_append(d >= kLow, &ctl->high);
    if (d >= kLow) a.high[at] = make_int2(d, (int)v);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kLow; d += kBlock)
    a.hist[(int64_t)d * gridDim.x + blockIdx.x] = s_cnt[d];
  if (!sync()) return;
  // 3. first rank of each degree and block
  {
    int64_t tot[1];
    if (!grid_scan<1>(
            &ctl->bar, &ctl->err, a.wait_ns, (int64_t)kLow * gridDim.x, a.part, tot,
            [&](int64_t i, int (&v)[1]) { v[0] = __ldcg(&a.hist[i]); },
            [&](int64_t i, const int64_t (&ex)[1], const int (&)[1]) { a.hist[i] = (int)ex[0]; }))
      return;
  }
  if (!sync()) return;
  // 4. ranks by (degree, id): low degrees in the order of the stretch, high
  // ones by the number of high vertices before them
  auto put_rank = [&](int64_t v, int d, int r) {
    a.newid[v] = r;
    a.order[r] = (int32_t)v;
    a.sdeg[r] = d;
  };
  for (int d = threadIdx.x; d < kLow; d += kBlock)
    s_cnt[d] = __ldcg(&a.hist[(int64_t)d * gridDim.x + blockIdx.x]);
  __syncthreads();
  for (int64_t v0 = c0; v0 < c1; v0 += kBlock) {
    const int64_t v = v0 + threadIdx.x;
    const int d = v < c1 ? __ldcg(&a.deg[v]) : INT_MAX;
    const int wib = threadIdx.x >> 5;
    const unsigned peers = __match_any_sync(TR_FULL, d);
    const bool low = d < kLow;
    if (low && lane_id() == __ffs(peers) - 1) s_warp[wib][d] = (unsigned short)__popc(peers);
    __syncthreads();
    if (low) {
      int r = s_cnt[d] + __popc(peers & ((1u << lane_id()) - 1u));
      for (int w = 0; w < wib; w++) r += s_warp[w][d];
      put_rank(v, d, r);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < kLow; x += kBlock) {
      int sum = 0;
      for (int w = 0; w < kBlock / 32; w++) {
        sum += s_warp[w][x];
        s_warp[w][x] = 0;
      }
      s_cnt[x] += sum;
    }
    __syncthreads();
  }
  {
    // a warp per high vertex: with most vertices high (10,000 of degree 512) a
    // thread each was a chain of 10,000 L2 loads (support 3.49 ms; with a warp
    // each 3.28, this step 73 us)
    const int nh = __ldcg(&ctl->high);
    for (int i = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < nh;
         i += gridDim.x * (kBlock / 32)) {
      const int2 x = a.high[i];
      int before = 0;
#pragma unroll 4
      for (int j = lane_id(); j < nh; j += 32) {
        const int2 y = a.high[j];
        before += y.x < x.x || (y.x == x.x && y.y < x.y);
      }
      before = __reduce_add_sync(TR_FULL, before);
      if (lane_id() == 0) put_rank(x.y, x.x, (int)n - nh + before);
    }
  }
  if (!sync()) return;
  // 5. orientation, out-degrees
  for (int64_t e0 = (int64_t)blockIdx.x * kBlock; e0 < m; e0 += nt) {
    const int64_t e = e0 + threadIdx.x;
    const bool ok = e < m;
    int t = 0;
    if (ok) {
      const int x = __ldcg(&a.newid[__ldcg(&a.eu[e])]), y = __ldcg(&a.newid[__ldcg(&a.ev[e])]);
      t = min(x, y);
      a.eu[e] = t;
      a.ev[e] = max(x, y);
    }
    grouped_add(ok, t, a.outc);
  }
  if (!sync()) return;
  // 6. offsets of the out-lists and of the groups by head
  {
    int64_t tot[2];
    if (!grid_scan<2>(
            &ctl->bar, &ctl->err, a.wait_ns, n, a.part, tot,
            [&](int64_t i, int (&v)[2]) {
              v[0] = __ldcg(&a.outc[i]);
              v[1] = __ldcg(&a.sdeg[i]) - v[0];
            },
            [&](int64_t i, const int64_t (&ex)[2], const int (&v)[2]) {
              a.offp[i] = ex[0];
              a.inoff[i] = ex[1];
              if (v[0] > kLongList) a.high[atomicAdd(&ctl->longs, 1)] = make_int2((int)i, v[0]);
            }))
      return;
    if (tid == 0) {
      a.offp[n] = tot[0];
      a.inoff[n] = tot[1];
    }
  }
  if (!sync()) return;
  // 7. edges to their tail's list
  for (int64_t e0 = (int64_t)blockIdx.x * kBlock; e0 < m; e0 += nt) {
    const int64_t e = e0 + threadIdx.x;
    const bool ok = e < m;
    const int t = ok ? __ldcg(&a.eu[e]) : 0;
    const int c = grouped_slot<true>(ok, t, a.curo);
    if (ok) {
      const int64_t p = __ldcg(&a.offp[t]) + c;
      a.lt[p] = t;
      a.lh[p] = __ldcg(&a.ev[e]);
      a.lid[p] = (int32_t)e;
    }
  }
  if (!sync()) return;
  // long out-lists, sorted where they lie: counting is quadratic (2 M edges of
  // lists of 1,000: 825 us, now 148 and 94 for the pass)
  if (const int longs = __ldcg(&ctl->longs)) {
    __shared__ unsigned long long s_sort[kSortCap];
    for (int i = blockIdx.x; i < longs; i += gridDim.x) {
      const int2 l = __ldcg(&a.high[i]);
      const int64_t beg = __ldcg(&a.offp[l.x]);
      const int d = min(l.y, kSortCap);
      for (int q = threadIdx.x; q < d; q += kBlock)
        s_sort[q] = (unsigned long long)(unsigned)__ldcg(&a.lh[beg + q]) << 32 |
                    (unsigned)__ldcg(&a.lid[beg + q]);
      block_sort(s_sort, d);
      for (int q = threadIdx.x; q < d; q += kBlock) {
        a.lh[beg + q] = (int)(s_sort[q] >> 32);
        a.lid[beg + q] = (int)(unsigned)s_sort[q];
      }
      __syncthreads();
    }
    if (!sync()) return;
  }
  // 8. place within the list; groups by head, walk costs and record bounds
  for (int64_t p0 = (int64_t)blockIdx.x * kBlock; p0 < m; p0 += nt) {
    const int64_t p = p0 + threadIdx.x;
    const bool ok = p < m;
    int h = 0, t = 0;
    int64_t e = 0, end = 0;
    if (ok) {
      t = __ldcg(&a.lt[p]);
      h = __ldcg(&a.lh[p]);
      const int64_t beg = __ldcg(&a.offp[t]);
      end = __ldcg(&a.offp[t + 1]);
      int c = 0;
      if (end - beg > kLongList) {
        c = (int)(p - beg);
      } else {
#pragma unroll 4
        for (int64_t q = beg; q < end; q++) c += a.lh[q] < h;
      }
      e = beg + c;
      a.adjp[e] = h;
      a.esrc[e] = t;
      a.lex2e[__ldcg(&a.lid[p])] = (int32_t)e;
    }
    const int g = grouped_slot<false>(ok, h, a.curi);
    if (ok) {
      const int64_t i = __ldcg(&a.inoff[h]) + g;
      const int64_t after = end - e - 1;
      const int64_t dv = __ldcg(&a.offp[h + 1]) - __ldcg(&a.offp[h]);
      a.inedge[i] = (int32_t)e;
      a.ihead[i] = h;
      a.wcost[i] = after + a.ecost;
      a.bound[e] = dv < after ? dv : after;
    }
  }
  if (!sync()) return;
  // 9. rows, prefix sums of the costs and bounds
  for (int64_t r = tid; r < rows; r += nt) {
    const int sl = a.row_slot[r];
    a.row2e[r] = sl < 0 ? -1 : __ldcg(&a.lex2e[__ldcg(&a.slot_id[sl])]);
  }
  int64_t tot[2];
  if (!grid_scan<2>(
          &ctl->bar, &ctl->err, a.wait_ns, m, a.part, tot,
          [&](int64_t i, int (&v)[2]) {
            v[0] = (int)__ldcg(&a.wcost[i]);
            v[1] = (int)__ldcg(&a.bound[i]);
          },
          [&](int64_t i, const int64_t (&ex)[2], const int (&)[2]) {
            a.wpre[i] = ex[0];
            a.tbpre[i] = ex[1];
          }))
    return;
  int64_t P = tot[0] / a.range_work;
  if (P < a.warps) P = a.warps;
  if (P > m) P = m > 0 ? m : 1;
  if (tid == 0) {
    a.wpre[m] = tot[0];
    a.tbpre[m] = tot[1];
    ctl->W = tot[0];
    ctl->R = tot[1];
    ctl->P = P;
  }
  if (!sync()) return;
  // 10. rb[r] = first position whose cost prefix reaches r W / P: position i
  // takes the r with prefix(i - 1) < r W / P <= prefix(i)
  const int64_t W = tot[0];
  for (int64_t i = tid; i <= m; i += nt) {
    const int64_t x = __ldcg(&a.wpre[i]);
    int64_t r = 0;
    if (i > 0) {
      const int64_t y = __ldcg(&a.wpre[i - 1]);
      // least r with point(r) > y (W, P and their product stay below 2^63)
      r = W > 0 ? y * P / W : 0;
      while (r > 0 && range_point(W, P, r - 1) > y) r--;
      while (r <= P && range_point(W, P, r) <= y) r++;
    }
    for (; r <= P && range_point(W, P, r) <= x; r++) a.rb[r] = i;
  }
}

struct OffsetCtl {
  unsigned long long bar;
  int err;
  int pad;
  int64_t total;
};

struct OffsetArgs {
  int64_t n, m;
  OffsetCtl *ctl;
  long long wait_ns;
  int64_t *part;
  const int32_t *supA, *supB;
  const int32_t *cuv;  // null: supports only
  const int32_t *inedge;
  const int64_t *offp, *inoff;
  int32_t *sup;
  int64_t *toff;
  unsigned long long *cur;
  int64_t *p1, *p2, *vb1, *vb2;
};

// Vertex ranges: vb[r] = first vertex v with cost(v) >= r * rc, for r < nr, and
// vb[nr] = n.  Vertex v (cost c, its predecessor's c0) takes r with c0 < r rc <= c.
__device__ __forceinline__ void put_ranges(int64_t v, int64_t n, int64_t c0, int64_t c, int64_t rc,
                                           int64_t nr, int64_t *vb) {
  if (v < n) {
    for (int64_t r = v == 0 ? 0 : c0 / rc + 1; r <= c / rc && r < nr; r++) vb[r] = v;
  } else {
    for (int64_t r = n == 0 ? 0 : c0 / rc + 1; r <= nr; r++) vb[r] = n;
  }
}

__global__ void __launch_bounds__(kBlock, 2) k_small_offsets(OffsetArgs a) {
  OffsetCtl *ctl = a.ctl;
  const int64_t tid = (int64_t)blockIdx.x * kBlock + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * kBlock, m = a.m, n = a.n;
  if (a.wait_ns < 0 && tid == 0) raise_error(&ctl->bar, &ctl->err, TRUSS_ETIMEOUT);
  int64_t tot[3];
  if (!grid_scan<3>(
          &ctl->bar, &ctl->err, a.wait_ns, m, a.part, tot,
          [&](int64_t i, int (&v)[3]) {
            v[0] = a.supA[i] + a.supB[i];
            v[1] = a.cuv ? a.cuv[i] + kListEdgeCost : 0;
            v[2] = a.cuv ? a.cuv[a.inedge[i]] + kListEdgeCost : 0;
          },
          [&](int64_t i, const int64_t (&ex)[3], const int (&v)[3]) {
            a.sup[i] = v[0];
            a.toff[i] = ex[0];
            if (a.cuv) {
              a.cur[i] = (unsigned long long)(ex[0] + v[1] - kListEdgeCost);
              a.p1[i] = ex[1];
              a.p2[i] = ex[2];
            }
          }))
    return;
  if (tid == 0) {
    a.toff[m] = tot[0];
    ctl->total = tot[0];
    if (a.cuv) {
      a.p1[m] = tot[1];
      a.p2[m] = tot[2];
    }
  }
  if (!a.cuv) return;
  if (!grid_barrier(&ctl->bar, &ctl->err, a.wait_ns)) return;
  const ListRanges lr = list_ranges(tot[0] / 3, m);
  for (int64_t v = tid; v <= n; v += nt) {
    auto c1 = [&](int64_t x) { return __ldcg(&a.p1[a.offp[x]]); };
    auto c2 = [&](int64_t x) { return __ldcg(&a.p2[a.inoff[x]]) + kListEdgeCost * a.offp[x]; };
    put_ranges(v, n, v > 0 ? c1(v - 1) : 0, v < n ? c1(v) : 0, lr.cost, lr.n1, a.vb1);
    put_ranges(v, n, v > 0 ? c2(v - 1) : 0, v < n ? c2(v) : 0, lr.cost, lr.n2, a.vb2);
  }
}

// Rows and vertices up to which the small paths are taken (see the top).  Above
// kSmallAnyRows rows, only with at most kSmallPerVertex rows per vertex: where
// few vertices share the rows the sorts take fewer passes (a key is two vertex
// ids), and here more atomics meet and more out-lists are long.  Support,
// general path / here (ms): random rows, 1.05 M over 4,096 vertices (256 rows
// each) 1.28 / 1.23; 1.5 M over 8,192 (183) 1.61 / 1.64; 2.1 M over 16,384 (128)
// 1.62 / 1.65, over 8,192 (256) 2.26 / 2.40; 2.6 M over 16,384 (160) 2.07 / 2.52;
// Chung-Lu of 2.6 M over 16,384 1.59 / 1.93; cliques K_1000 1.02 / 0.84, K_1200
// 1.35 / 1.22, fifty of K_300 (2.2 M rows) 1.45 / 1.71.  (Rows that repeat few
// edges are better off here at any density: 1,000 times 2,600 edges of 3,000
// vertices 0.44 / 0.21; their sizes do not tell them from the dense ones.)
constexpr int64_t kSmallRows = 5 << 19;
static_assert((int64_t)kSortCap * kSortCap >= 2 * kSmallRows, "the longest out-list fits");
constexpr int64_t kSmallAnyRows = 1 << 20;
constexpr int64_t kSmallPerVertex = 128;
constexpr long long kWaitNs = 4000000000LL;

// Limit of a launch's barriers; testing: from the environment, so that the
// blocks give up and the general path takes over (a negative one has run out
// before the first barrier).
long long wait_limit(const char *name) {
  const char *v = getenv(name);
  return v ? atoll(v) : kWaitNs;
}

// Blocks of a cooperative launch for about `work` elements: one per SM, fewer
// for small graphs (two elements per thread).
int small_grid(int64_t work, int sms, int *out) {
  if (sms <= 0) {
    int dev = 0;
    TR_CUDA(cudaGetDevice(&dev));
    TR_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  }
  int64_t grid = (work + 2 * kBlock - 1) / (2 * kBlock);
  if (grid > sms) grid = sms;
  if (grid < 8) grid = sms < 8 ? sms : 8;
  *out = (int)grid;
  return TRUSS_OK;
}

template <class Args>
int launch_small(void (*kern)(Args), int grid, Args a, cudaStream_t s) {
  int occ = 0;
  TR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kBlock, 0));
  if (occ < 1) return TRUSS_ECUDA;
  void *args[] = {&a};
  TR_CUDA(cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(kBlock), args,
                                      0, s));
  count_launches(1);
  return TRUSS_OK;
}

int build_small(Arena &A, const RowsIn &in, const SupportCfg &cfg, Csr *out, SupportPrep *prep,
                cudaStream_t s) {
  const int64_t rows = in.rows, n = in.n;
  // sized to the graph throughout: a run of the server has little more than
  // the rows' share of the workspace
  int64_t slots = 64;
  while (slots < 2 * rows) slots *= 2;
  int grid = 0;
  TR_TRY(small_grid(rows > n ? rows : n, cfg.sms, &grid));
  SmallArgs a{};
  a.in = in;
  a.wait_ns = wait_limit("TRUSS_SMALL_BUILD_WAIT_NS");
  a.mask = (unsigned)(slots - 1);
  static_assert(sizeof(SmallCtl) <= ZeroBlock::kCtl && sizeof(OffsetCtl) <= ZeroBlock::kCtl,
                "control words fit the zero block");
  a.ctl = (SmallCtl *)out->zero->build;
  a.keys = A.get<unsigned long long>(slots);
  a.slot_id = A.get<int32_t>(slots);
  a.row_slot = A.get<int32_t>(rows);
  a.eu = A.get<int32_t>(rows);
  a.ev = A.get<int32_t>(rows);
  a.deg = A.get<int32_t>(n);
  a.part = A.get<int64_t>(2 * (int64_t)grid);
  a.hist = A.get<int32_t>((int64_t)kLow * grid);
  a.high = A.get<int2>(2 * rows / kLow + 1);
  a.outc = A.get<int32_t>(n);
  a.curo = A.get<int32_t>(n);
  a.curi = A.get<int32_t>(n);
  a.lt = A.get<int32_t>(rows);
  a.lh = A.get<int32_t>(rows);
  a.lid = A.get<int32_t>(rows);
  a.newid = A.get<int32_t>(n);
  a.lex2e = A.get<int32_t>(rows);
  a.sdeg = A.get<int32_t>(n);
  a.order = A.get<int32_t>(n);
  a.offp = A.get<int64_t>(n + 1);
  a.inoff = A.get<int64_t>(n + 1);
  a.adjp = A.get<int32_t>(rows);
  a.esrc = A.get<int32_t>(rows);
  a.row2e = A.get<int32_t>(rows);
  a.inedge = A.get<int32_t>(rows);
  a.ihead = A.get<int32_t>(rows);
  a.wcost = A.get<int64_t>(rows + 1);
  a.bound = A.get<int64_t>(rows + 1);
  a.wpre = A.get<int64_t>(rows + 1);
  a.tbpre = A.get<int64_t>(rows + 1);
  a.supA = A.get<int32_t>(rows);
  a.supB = A.get<int32_t>(rows);
  a.cuv = cfg.records ? A.get<int32_t>(rows) : nullptr;
  a.rb = A.get<int64_t>(rows + 2);
  if (!a.keys || !a.slot_id || !a.row_slot || !a.eu || !a.ev || !a.deg || !a.part || !a.hist ||
      !a.high ||
      !a.outc || !a.curo || !a.curi || !a.lt || !a.lh || !a.lid || !a.newid || !a.lex2e ||
      !a.sdeg || !a.order || !a.offp || !a.inoff || !a.adjp || !a.esrc || !a.row2e || !a.inedge ||
      !a.ihead || !a.wcost || !a.bound || !a.wpre || !a.tbpre || !a.supA || !a.supB || !a.rb ||
      (cfg.records && !a.cuv))
    return TRUSS_ENOMEM;
  a.ecost = walk_edge_cost(cfg);
  a.range_work = walk_range_work(cfg);
  TR_TRY(walk_warps(cfg, &a.warps));
  TR_TRY(launch_small(k_small_build, grid, a, s));
  SmallCtl h{};
  TR_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  if (h.err != 0) return h.err;
  if (h.bad != 0) return TRUSS_EINVAL;
  out->n = n;
  out->rows = rows;
  out->m = h.m;
  out->offp = a.offp;
  out->adjp = a.adjp;
  out->esrc = a.esrc;
  out->row2e = a.row2e;
  out->order = a.order;
  out->sdeg = a.sdeg;
  prep->valid = true;
  prep->supA = a.supA;
  prep->supB = a.supB;
  prep->cuv = a.cuv;
  prep->inedge = a.inedge;
  prep->ihead = a.ihead;
  prep->inoff = a.inoff;
  prep->wcost = a.wcost;
  prep->wpre = a.wpre;
  prep->tbpre = a.tbpre;
  prep->rb = a.rb;
  prep->W = h.W;
  prep->R = h.R;
  prep->P = h.P;
  return TRUSS_OK;
}

}  // namespace

int build_graph(Arena &A, const RowsIn &in, const SupportCfg &cfg, Csr *out, SupportPrep *prep,
                int32_t *d_err, cudaStream_t s) {
  *prep = SupportPrep{};
  out->zero = A.get<ZeroBlock>(1);
  if (!out->zero) return TRUSS_ENOMEM;
  TR_CUDA(cudaMemsetAsync(out->zero, 0, sizeof(ZeroBlock), s));
  // the scans add up tiles of edge costs in 31 bits
  if (cfg.small_paths && in.rows > 0 && in.rows <= kSmallRows && in.n <= kSmallRows &&
      (in.rows <= kSmallAnyRows || in.rows <= kSmallPerVertex * in.n) &&
      walk_edge_cost(cfg) <= kSmallRows / 2) {
    const std::vector<size_t> mk = A.mark();
    const int rc = build_small(A, in, cfg, out, prep, s);
    // its blocks could not meet in time (the device is taken by other work), or
    // its arrays, sized by rows where the general path's shrink to the distinct
    // edges, do not fit: the general path waits for nothing and starts over
    // with the workspace
    if (rc != TRUSS_ETIMEOUT && rc != TRUSS_ENOMEM) return rc;
    A.rewind(mk);
    *prep = SupportPrep{};
  }
  return build_csr(A, in, out, d_err, s);
}

int small_offsets(Arena &A, const Csr &g, const SupportPrep &prep, const int32_t *cuv, int sms,
                  int32_t *sup, int64_t *toff, int64_t *total, SmallLists *lists,
                  cudaStream_t s) {
  const int64_t m = g.m, n = g.n;
  OffsetArgs a{};
  a.n = n;
  a.m = m;
  a.wait_ns = wait_limit("TRUSS_SMALL_OFFSETS_WAIT_NS");
  a.ctl = (OffsetCtl *)g.zero->offsets;
  a.supA = prep.supA;
  a.supB = prep.supB;
  a.cuv = cuv;
  a.inedge = prep.inedge;
  a.offp = g.offp;
  a.inoff = prep.inoff;
  a.sup = sup;
  a.toff = toff;
  if (cuv) {
    const int64_t cap = list_ranges_most(prep.R, m) + 1;  // at most as many triangles as slots
    a.cur = A.get<unsigned long long>(m);
    a.p1 = A.get<int64_t>(m + 1);
    a.p2 = A.get<int64_t>(m + 1);
    a.vb1 = A.get<int64_t>(cap);
    a.vb2 = A.get<int64_t>(cap);
    if (!a.cur || !a.p1 || !a.p2 || !a.vb1 || !a.vb2) return TRUSS_ENOMEM;
    lists->cur = a.cur;
    lists->p1 = a.p1;
    lists->p2 = a.p2;
    lists->vb1 = a.vb1;
    lists->vb2 = a.vb2;
  }
  int grid = 0;
  TR_TRY(small_grid(m > n ? m : n, sms, &grid));
  a.part = A.get<int64_t>(3 * (int64_t)grid);
  if (!a.part) return TRUSS_ENOMEM;
  TR_TRY(launch_small(k_small_offsets, grid, a, s));
  OffsetCtl h{};
  TR_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  if (h.err != 0) return h.err;
  *total = h.total;
  return TRUSS_OK;
}

}  // namespace tr
