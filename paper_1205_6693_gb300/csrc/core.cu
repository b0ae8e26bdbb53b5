// Vertex core numbers on the truss library's CSR.  The paper places the
// k-truss inside the (k-1)-core (Section 1) and compares the k_max-truss with
// the c_max-core (Section 7, Table 6); its edge bins reuse the core
// decomposition's bin-sorted degree array (Section 3.2).
//
// core(v) is the largest k such that v lies in the k-core, the largest
// subgraph whose vertices all have degree >= k in it.  Like the edge peel,
// this runs level-synchronously in one persistent cooperative launch:
//
//  scan (level k):  F = {alive v : deg(v) <= k}; the minimum degree of the
//        other alive vertices lets an empty level jump to k = that minimum.
//        The alive list is rewritten without removed vertices only when at
//        most half of it is still alive.
//  sub-round:  every v in F gets core k and is removed; each neighbour w
//        still alive loses one degree, and a w whose degree crosses from
//        k+1 to k joins the next frontier (it now has degree <= k, so it is
//        not in the k+1-core).  Vertices removed together need no exchange:
//        a neighbour in the same frontier is simply skipped.
//
// Vertex state is one word, the current degree, with the top bit set once the
// vertex is removed.  A removed vertex takes one from the word of each of its
// neighbours, alive or not, without reading it first: the low part of a
// removed vertex's word is the number of its neighbours still alive, each of
// which takes one from it once, so it never runs into the mark.
// Neighbours come from a symmetric adjacency built from the oriented CSR.  A
// frontier vertex is split into work items of kItem neighbours, as in the
// edge peel, so a warp's share of a sub-round is bounded whatever the degrees.
// Phases end as in the edge peel (phase_end).  R-MAT scale 20: 5.15 ms with
// phase counters read by every warp and a state read before each decrement,
// 5.04 with the counters passed on, 4.47 without the state read, 4.35 with
// vertices staged and expanded at the flush.
#include <climits>

#include "engine.h"

namespace tr {

namespace {

constexpr int kBlock = 512;
constexpr int kWarps = kBlock / 32;
constexpr int kItem = 16;  // neighbours per work item (8 lanes x 2)
constexpr int kWP = 32;    // pushed vertices staged per warp (one per lane)
constexpr int kWA = 128;   // alive-list entries staged per warp

struct CoreCtl : PhaseCtl {
  int levels, subrounds, kmax, pad1;
};

struct CoreArgs {
  int64_t n;
  const int64_t *soff;  // [n+1] symmetric adjacency offsets
  const int32_t *sadj;  // [2m]
  uint32_t *word;       // current degree; kGone set once removed
  int32_t *core;
  int32_t *alive0, *alive1;
  int4 *Q0, *Q1;  // work items (v, cnt | first << 8, offset lo, hi)
  uint32_t item_cap;
  CoreCtl *ctl;
  long long wait_ns;
};

constexpr uint32_t kGone = 0x80000000u;

__device__ __forceinline__ int items_of(int len) { return len > 0 ? (len + kItem - 1) / kItem : 1; }

// Per-warp staging buffers in shared memory (counts are warp-uniform).
struct WarpBuf {
  int32_t *push;  // vertices pushed to the next frontier, not yet expanded
  int np;
  int32_t *alive;
  int na;
};

__device__ __forceinline__ int4 make_item(int v, int64_t lb, int L, int it) {
  const int64_t off = lb + (int64_t)it * kItem;
  const int cnt = min(kItem, L - it * kItem);
  return make_int4(v, max(cnt, 0) | ((it == 0) << 8), (int)(uint32_t)off,
                   (int)(uint32_t)((uint64_t)off >> 32));
}

// Expand the staged vertices into work items and append them to queue Q with
// one reservation; their offsets are loaded together here, not one dependent
// round trip per push.  A single one, as most flushes have, needs no scan.
__device__ __forceinline__ void flush_push(const CoreArgs &a, WarpBuf &wb, int4 *Q,
                                           unsigned long long *qctr) {
  const int np = wb.np;
  if (np == 0) return;
  const int lane = lane_id();
  const bool v = lane < np;
  const int p = v ? wb.push[lane] : 0;
  const int64_t lb = v ? __ldg(&a.soff[p]) : 0;
  const int L = v ? (int)(__ldg(&a.soff[p + 1]) - lb) : 0;
  const int n = v ? items_of(L) : 0;
  if (np == 1) {
    const int tot = __shfl_sync(TR_FULL, n, 0);
    uint32_t at = 0;
    if (lane == 0) at = reserve_items(qctr, tot);
    at = __shfl_sync(TR_FULL, at, 0);
    const int po = __shfl_sync(TR_FULL, p, 0), Lo = __shfl_sync(TR_FULL, L, 0);
    const int64_t lbo = __shfl_sync(TR_FULL, lb, 0);
    for (int it = lane; it < tot; it += 32)
      if (at + it < a.item_cap) Q[at + it] = make_item(po, lbo, Lo, it);
  } else {
    const int P = warp_incl_scan(n);
    uint32_t b = 0;
    if (lane == 31) b = reserve_items(qctr, P);
    const int tot = __shfl_sync(TR_FULL, P, 31);
    const uint32_t base = __shfl_sync(TR_FULL, b, 31);
    for (int u0 = 0; u0 < tot; u0 += 32) {
      const int t = u0 + lane;
      const int o = warp_owner(P, t < tot ? t : tot - 1);
      const int po = __shfl_sync(TR_FULL, p, o), i0 = __shfl_sync(TR_FULL, P - n, o);
      const int Lo = __shfl_sync(TR_FULL, L, o);
      const int64_t lbo = __shfl_sync(TR_FULL, lb, o);
      const uint32_t idx = base + t;
      if (t < tot && idx < a.item_cap) Q[idx] = make_item(po, lbo, Lo, t - i0);
    }
  }
  __syncwarp();
  wb.np = 0;
}

__device__ __forceinline__ void flush_alive(const CoreArgs &a, WarpBuf &wb, int32_t *A2,
                                            int *actr) {
  if (wb.na == 0) return;
  const int lane = lane_id();
  int b = 0;
  if (lane == 0) b = atomicAdd(actr, wb.na);
  const int b0 = __shfl_sync(TR_FULL, b, 0);
  for (int t = lane; t < wb.na; t += 32)
    if (b0 + t < a.n) A2[b0 + t] = wb.alive[t];
  __syncwarp();
  wb.na = 0;
}

__device__ __forceinline__ void push_alive(const CoreArgs &a, bool keep, int v, WarpBuf &wb,
                                           int32_t *A2, int *actr) {
  const unsigned mask = __ballot_sync(TR_FULL, keep);
  if (mask == 0) return;
  const int tot = __popc(mask);
  if (wb.na + tot > kWA) flush_alive(a, wb, A2, actr);
  if (keep) wb.alive[wb.na + __popc(mask & ((1u << lane_id()) - 1u))] = v;
  __syncwarp();
  wb.na += tot;
}

// Stage vertex p (for each lane with `push`) for expansion into work items of
// the next frontier.  All lanes call it.
__device__ __forceinline__ void push_items(const CoreArgs &a, bool push, int p, WarpBuf &wb,
                                           int4 *Q, unsigned long long *qctr) {
  const unsigned mask = __ballot_sync(TR_FULL, push);
  if (mask == 0) return;
  const int tot = __popc(mask);
  if (wb.np + tot > kWP) flush_push(a, wb, Q, qctr);
  if (push) wb.push[wb.np + __popc(mask & ((1u << lane_id()) - 1u))] = p;
  __syncwarp();
  wb.np += tot;
}

__global__ void __launch_bounds__(kBlock, 2) k_core(CoreArgs a) {
  const int lane = lane_id();
  const int wib = threadIdx.x >> 5;
  // consecutive warps of the launch sit in different blocks, so a phase with
  // little work spreads it over all SMs
  const uint32_t gwarp = wib * gridDim.x + blockIdx.x;
  const uint32_t twarps = gridDim.x * kWarps;
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  CoreCtl *ctl = a.ctl;
  __shared__ int32_t s_push[kWarps][kWP];
  __shared__ int32_t s_alive[kWarps][kWA];
  __shared__ int s_minres, s_live, s_any;
  WarpBuf wb{s_push[wib], 0, s_alive[wib], 0};
  if (threadIdx.x == 0) {
    s_minres = INT_MAX;
    s_live = 0;
    s_any = 0;
  }
  __syncthreads();

  int k = 0, sc = 0;
  unsigned ph = 0;
  int32_t *alive = a.alive0, *alive2 = a.alive1;
  int4 *F = a.Q0, *N = a.Q1;
  int nAlive = (int)a.n;
  bool compact = false;
  auto clamp = [&](uint32_t n) {
    if (n <= a.item_cap) return n;
    // appends beyond the queue were dropped
    if (leader) raise_error(&ctl->phase[ph % 3], &ctl->err, TRUSS_ECHECK);
    return a.item_cap;
  };

  for (;;) {
    // ------------------------------------------------------------ scan ---
    ScanOut *scan = &ctl->scan[sc % 3];
    unsigned long long *qf = &ctl->phase[ph % 3];
    if (leader) {
      *(int4 *)&ctl->scan[(sc + 1) % 3] = make_int4(INT_MAX, 0, 0, 0);
      ctl->phase[(ph + 1) % 3] = 0;
    }
    int lmin = INT_MAX, llive = 0;  // of this lane
    bool lany = false;
    // 4 x 32 entries per warp iteration, all loads before any decision
    constexpr int kScanU = 4;
    for (int64_t base = (int64_t)gwarp * 32 * kScanU; base < nAlive;
         base += (int64_t)twarps * 32 * kScanU) {
      int v[kScanU];
      uint32_t w[kScanU];
#pragma unroll
      for (int u = 0; u < kScanU; u++) {
        const int64_t i = base + u * 32 + lane;
        v[u] = i < nAlive ? __ldcg(&alive[i]) : -1;
      }
#pragma unroll
      for (int u = 0; u < kScanU; u++) w[u] = v[u] >= 0 ? __ldcg(&a.word[v[u]]) : kGone;
      unsigned pend = 0;  // entries of this lane that join the frontier
#pragma unroll
      for (int u = 0; u < kScanU; u++) {
        const bool live = (int32_t)w[u] >= 0;
        const bool toF = live && (int)w[u] <= k;
        const bool keep = live && !toF;
        if (toF) {
          a.word[v[u]] = kGone | w[u];
          lany = true;
          if (w[u] == 0) a.core[v[u]] = k;  // no neighbour left: no item
          else pend |= 1u << u;
        }
        if (compact) push_alive(a, keep, v[u], wb, alive2, &scan->listed);
        if (keep) {
          lmin = min(lmin, (int)w[u]);
          llive++;
        }
      }
      while (__any_sync(TR_FULL, pend != 0)) {
        int q = 0;
        const bool has = pend != 0;
        if (has) {
          const int b = __ffs(pend) - 1;
          pend &= pend - 1;
#pragma unroll
          for (int u = 0; u < kScanU; u++)
            if (b == u) q = v[u];
        }
        push_items(a, has, q, wb, F, qf);
      }
    }
    flush_push(a, wb, F, qf);
    if (compact) flush_alive(a, wb, alive2, &scan->listed);
    if ((int64_t)gwarp * 32 * kScanU < nAlive) {
      lmin = __reduce_min_sync(TR_FULL, lmin);
      llive = __reduce_add_sync(TR_FULL, llive);
      const bool wany = __any_sync(TR_FULL, lany);
      if (lane == 0) {
        if (lmin != INT_MAX) atomicMin(&s_minres, lmin);
        if (llive) atomicAdd(&s_live, llive);
        if (wany) s_any = 1;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (s_minres != INT_MAX) atomicMin(&scan->minres, s_minres);
      if (s_live) atomicAdd(&scan->live, s_live);
      if (s_any) scan->any = 1;
      s_minres = INT_MAX;
      s_live = 0;
      s_any = 0;
    }
    uint32_t nCur;  // items of the frontier
    ScanOut found;
    if (!phase_end(ctl, a.wait_ns, ph, &nCur, scan, &found)) return;
    ph++;
    if (compact) {
      nAlive = found.listed;
      int32_t *t = alive;
      alive = alive2;
      alive2 = t;
    }
    compact = 2 * (int64_t)found.live <= nAlive;
    sc++;
    if (found.any && leader) {
      ctl->levels++;
      ctl->kmax = k;
    }
    if (nCur == 0) {
      // nothing removed had a neighbour left, so the degrees stand; what went
      // counts as one sub-round
      if (found.any && leader) ctl->subrounds++;
      if (found.live == 0) break;
      k = found.minres;  // every alive vertex has degree >= k+1: skip empty levels
      continue;
    }
    // --------------------------------------------------------- sub-rounds ---
    nCur = clamp(nCur);
    for (;;) {
      unsigned long long *qn = &ctl->phase[ph % 3];
      if (leader) ctl->phase[(ph + 1) % 3] = 0;
      const int grp = lane >> 3, j = lane & 7;
      for (uint32_t base = gwarp * 4; base < nCur; base += twarps * 4) {
        const uint32_t it = base + grp;
        int v = 0, cnt = 0;
        int64_t lb = 0;
        if (it < nCur) {
          const int4 item = __ldcg(&F[it]);
          v = item.x;
          cnt = item.y & 0xFF;
          lb = (int64_t)(((uint64_t)(uint32_t)item.w << 32) | (uint32_t)item.z);
          if ((item.y >> 8) && j == 0) a.core[v] = k;
        }
        int w[2];
        uint32_t x[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
          const int jj = j + 8 * q;
          w[q] = jj < cnt ? __ldg(&a.sadj[lb + jj]) : -1;
          if (w[q] >= 0 && (uint32_t)w[q] >= (uint32_t)a.n) {
            raise_error(&ctl->phase[ph % 3], &ctl->err, TRUSS_ECHECK);
            w[q] = -1;
          }
        }
#pragma unroll
        for (int q = 0; q < 2; q++) x[q] = w[q] >= 0 ? atomicSub(&a.word[w[q]], 1u) : kGone;
        // one push_items site: each step pushes one pending neighbour per lane
        unsigned pend = (x[0] == (uint32_t)(k + 1) ? 1u : 0u) | (x[1] == (uint32_t)(k + 1) ? 2u : 0u);
        while (__any_sync(TR_FULL, pend != 0)) {
          const bool has = pend != 0;
          const int b = has ? __ffs(pend) - 1 : 0;
          pend &= pend - 1;
          const int q = b ? w[1] : w[0];
          if (has) atomicOr(&a.word[q], kGone);  // others may still decrement it
          push_items(a, has, q, wb, N, qn);
        }
      }
      flush_push(a, wb, N, qn);
      if (!phase_end(ctl, a.wait_ns, ph, &nCur, nullptr, nullptr)) return;
      ph++;
      if (leader) ctl->subrounds++;
      if (nCur == 0) break;
      { int4 *t = F; F = N; N = t; }
      nCur = clamp(nCur);
    }
    k++;
  }
}

__global__ void k_widen(int64_t n, const int32_t *x, int64_t *y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = i < n ? x[i] : 0;
}

// sadj[soff[v] ..) = v's out-neighbours, then its in-neighbours in any order.
// Out-neighbours are where they are in adjp; in-neighbours take a cursor, one
// atomic per group of lanes of a warp with the same head (one per edge and
// end, hubs included, took 574 us on R-MAT scale 20, now 540 us).
__global__ void k_sym_fill(int64_t m, const int64_t *offp, const int32_t *esrc,
                           const int32_t *adjp, const int64_t *soff, int32_t *cur,
                           int32_t *sadj) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const unsigned lt = (1u << lane_id()) - 1u;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < m; b += stride) {
    const int64_t e = b + threadIdx.x;
    const bool ok = e < m;
    const int u = ok ? esrc[e] : 0, v = ok ? adjp[e] : -1;
    if (ok) sadj[soff[u] + (e - offp[u])] = v;
    const unsigned peers = __match_any_sync(TR_FULL, v);
    const int first = __ffs(peers) - 1;
    int c = 0;
    if (ok && lane_id() == first) c = atomicAdd(&cur[v], __popc(peers));
    c = __shfl_sync(TR_FULL, c, first);
    if (ok) sadj[soff[v] + (offp[v + 1] - offp[v]) + c + __popc(peers & lt)] = u;
  }
}

__global__ void k_core_init(int64_t n, const int32_t *sdeg, uint32_t *word, int32_t *alive,
                            CoreCtl *ctl) {
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->scan[0].minres = INT_MAX;  // first scan's slot
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    word[v] = (uint32_t)sdeg[v];
    alive[v] = (int32_t)v;
  }
}

// core_out[order[r]] = core[r]: back from ranks to input vertex ids.
__global__ void k_core_out(int64_t n, const int32_t *order, const int32_t *core,
                           int32_t *core_out) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x)
    core_out[order[r]] = core[r];
}

}  // namespace

int run_core(Arena &A, const Csr &g, int sms, long long wait_ns, int32_t *core_out,
             int32_t *kmax, int32_t *levels, int32_t *subrounds, cudaStream_t s) {
  const int64_t n = g.n, m = g.m;
  *kmax = 0;
  *levels = *subrounds = 0;
  if (n == 0) return TRUSS_OK;
  int32_t *cur = A.get<int32_t>(n);
  int64_t *deg64 = A.get<int64_t>(n + 1), *soff = A.get<int64_t>(n + 1);
  int32_t *sadj = A.get<int32_t>(2 * m);
  uint32_t *word = A.get<uint32_t>(n);
  int32_t *core = A.get<int32_t>(n);
  int32_t *al0 = A.get<int32_t>(n), *al1 = A.get<int32_t>(n);
  // every vertex is pushed at most once; its items number at most
  // deg / kItem + 1, so 2m / kItem + n items bound any frontier (below 2^32)
  const int64_t item_cap = 2 * m / kItem + n + 1;
  int4 *Q0 = A.get<int4>(item_cap), *Q1 = A.get<int4>(item_cap);
  CoreCtl *ctl = A.get<CoreCtl>(1);
  if (!cur || !deg64 || !soff || !sadj || !word || !core || !al0 || !al1 || !Q0 || !Q1 || !ctl)
    return TRUSS_ENOMEM;
  k_widen<<<grid_for(n + 1, 256, 152 * 16), 256, 0, s>>>(n, g.sdeg, deg64);
  TR_LAUNCHED();
  size_t tb = 0;
  TR_TRY(exclusive_sum_i64(nullptr, &tb, deg64, soff, n + 1, s));
  void *tmp = A.alloc(tb);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(exclusive_sum_i64(tmp, &tb, deg64, soff, n + 1, s));
  TR_CUDA(cudaMemsetAsync(cur, 0, sizeof(int32_t) * n, s));
  if (m > 0) {
    k_sym_fill<<<grid_for(m, 256, 152 * 16), 256, 0, s>>>(m, g.offp, g.esrc, g.adjp, soff, cur,
                                                           sadj);
    TR_LAUNCHED();
  }
  TR_CUDA(cudaMemsetAsync(ctl, 0, sizeof(CoreCtl), s));
  k_core_init<<<grid_for(n, 256, 152 * 16), 256, 0, s>>>(n, g.sdeg, word, al0, ctl);
  TR_LAUNCHED();
  int occ = 0;
  TR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_core, kBlock, 0));
  if (occ < 1) return TRUSS_ECUDA;
  if (occ > 2) occ = 2;
  CoreArgs a{};
  a.n = n;
  a.soff = soff;
  a.sadj = sadj;
  a.word = word;
  a.core = core;
  a.alive0 = al0;
  a.alive1 = al1;
  a.Q0 = Q0;
  a.Q1 = Q1;
  a.item_cap = (uint32_t)item_cap;
  a.ctl = ctl;
  a.wait_ns = wait_ns;
  void *args[] = {&a};
  TR_CUDA(cudaLaunchCooperativeKernel((const void *)k_core, dim3(sms * occ), dim3(kBlock), args,
                                      0, s));
  count_launches(1);
  k_core_out<<<grid_for(n, 256, 152 * 16), 256, 0, s>>>(n, g.order, core, core_out);
  TR_LAUNCHED();
  CoreCtl h{};
  TR_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(CoreCtl), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  if (h.err != 0) return h.err;
  *kmax = h.kmax;
  *levels = h.levels;
  *subrounds = h.subrounds;
  return TRUSS_OK;
}

}  // namespace tr
