// Level-synchronous edge peeling (Algorithm 2 steps 3-16) in one persistent
// cooperative launch.
//
// Algorithm 2 removes, for k = 2, 3, ..., the lowest-support edge while its
// support is <= k-2, decrementing the support of the other two edges of each
// triangle it destroys (steps 7-10) and assigning it to Phi_k (step 11).  The
// order in which edges of one level are removed does not change the result
// (T_k is unique, Definition 2), so here every level is processed in
// sub-rounds: all alive edges whose residual support res is <= k-2 form the
// frontier F and are removed together.
//
//  scan (per level k):  F = {alive e : res[e] <= k-2}; the minimum residual
//        of the other alive edges is taken, so an empty level jumps straight
//        to k = min res + 2.  The list of alive edges scanned is rewritten
//        without the removed ones once at least a quarter of it is dead.
//  sub-round:  for every e in F and every triangle {e, e1, e2} on e's list
//        whose edges are all still alive, the triangle is charged exactly
//        once, by the lowest-id edge among those of its edges that are in F:
//        that edge decrements the residual of each partner not in F.  A
//        partner whose residual crosses from k-1 to k-2 joins the next
//        frontier (warp-aggregated append).  F edges get truss number k.
//
// Load balance inside a sub-round (its time is that of the slowest warp):
// an edge that joins a frontier is staged by the warp that pushed it and
// expanded, when that warp flushes, into work items, the aligned 16-entry
// blocks that its list touches; an item carries its edge, its block number
// and the part of the block that is the list's, so a warp goes from the item
// straight to the list.  Every warp takes 4 items per iteration, 8 lanes per
// item and 2 entries per lane (one 16-byte load).  A warp's share of a
// sub-round is then at most ceil(items / (4 * warps)) iterations, whatever
// the lengths of the lists, and the warps that share a small sub-round sit on
// different SMs.
// Appends are staged per warp in shared memory and flushed with one atomic
// reservation per buffer (the list lengths and offsets of a buffer's pushed
// edges are loaded together at the flush, those of an edge whose residual
// already stood at k-1 together with the decrement that removes it), and
// per-level reductions (minimum residual, alive count) are combined per block
// first: a single global counter hit by every warp would serialise the whole
// grid on one L2 address.
//
// What bounds it: below about 16 K items a sub-round is a chain of dependent
// L2 round trips (about 540 clocks each, 900 from HBM): item, list entries,
// partners' words, decrement, reservation, the release of the barrier's
// arrival and its polling; above, the random word reads and decrements.  So
// each step of the chain that can share a load with another does: an edge's
// state and its residual are one word, the count of a phase's items rides on
// its barrier's word, and one thread per block reads it.  Sub-rounds of at
// most 64 items 5.5 -> 4.2 us, scans of short alive lists 8.7 -> 5.0 us; the
// peel of R-MAT scale 20 27.4 -> 25.6 ms, of a 40 M-edge Chung-Lu graph 77.7
// -> 72.1 ms, of 4,096 small graphs 10.4 -> 7.6 ms, of the 4,096-vertex graph
// 0.205 -> 0.131 ms.  Kept in registers, the rarely used state spilled, and
// every reload after a barrier was one more round trip: it lives in shared
// memory or is derived.
// Every scan and every sub-round is one phase, ended by one grid barrier.
// Appends of phase p reserve space through counter slot p % 3, which is read
// by the barrier that ends p.  The leader zeroes slot (p+1) % 3 during phase
// p: that slot was last read at the end of phase p-2, and every block has
// passed the barrier ending p-1 before the leader can be in phase p.  A block
// that leaves a barrier early therefore never appends to a counter that a
// slow block has still to read.
//
// Edge state is one 32-bit word per edge: an alive edge's word is its
// residual (below 2^31); a removed one's has the top bit set, a 16-bit tag
// and, below it, the residual it was removed with.  tag(s) = in the frontier
// of sub-round s, any other tag = removed earlier.  An edge whose residual
// crosses in sub-round s is marked by adding the top bit and tag(s+1) to its
// word, so that decrements of the same sub-round still land in the residual;
// marked or not yet, it reads as alive during s, so one grid barrier per
// sub-round suffices.  Tags repeat every 65,534 sub-rounds, so at least every
// 32,768 sub-rounds one extra grid-wide pass rewrites every tag but the
// current frontier's to kDead.  The residual of a frontier edge is never
// touched during its sub-round and equals the number of its still-alive
// triangles, so a frontier edge with residual 0 skips its list (one found by
// the scan is not even queued).
//
// Every grid barrier waits at most `wait_ns` (globaltimer); on timeout the
// kernel records TRUSS_ETIMEOUT and all blocks return at their next barrier.
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "engine.h"

namespace tr {

namespace {

constexpr int kPeelBlock = 512;
constexpr int kWarps = kPeelBlock / 32;
constexpr int kItem = 16;  // list entries per work item (8 lanes x 2)
constexpr int kWP = 32;    // pushed edges staged per warp (one per lane)
constexpr int kWA = 128;   // alive-list entries staged per warp

struct PeelCtl : PhaseCtl {
  int levels, subrounds, kmax, ntrace;
  unsigned long long entries, decrements, scanned;
  unsigned long long dead, dead_earlier;  // counting runs
};

struct PeelArgs {
  int64_t m;
  const int32_t *sup;
  // list of e: own[own_off[e] ..] (own_cnt[e] entries), then rest[off[e] ..]
  const int2 *own;
  const int64_t *own_off;
  const int32_t *own_cnt;  // null: no own parts
  const int2 *rest;
  const int64_t *off;
  uint32_t *word;  // state of each edge (alive: its residual; else kGone | tag | residual)
  int retag;       // sub-rounds between tag rewrites (1 .. kRetagMax)
  int32_t *truss;
  int32_t *alive0, *alive1;
  // frontier work items (make_item): one queue grows from the front of Q, the
  // other from its end; every edge is pushed once, so the two never meet
  int4 *Q;
  uint32_t item_cap;  // capacity of Q
  int4 *trace;        // optional: per phase (k, items or -1 for a scan, globaltimer lo/hi)
  int trace_cap;
  PeelCtl *ctl;
  long long wait_ns;
  int k_stop;  // last level to run (0 = all)
  // counting runs (the COUNT kernel): removal sub-round of every edge, and
  // per level k < lvl_cap the entries read, those of destroyed triangles, and
  // those of triangles destroyed in an earlier level (lvl[3k .. 3k+2])
  int32_t *when;
  unsigned long long *lvl;
  int lvl_cap;
};

__device__ __forceinline__ void prefetch_l1(const void *p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

constexpr int kTagMod = 65534;
constexpr int kRetagMax = 32768;
constexpr uint32_t kDead = 0xFFFF;
// Tag of sub-round s >= 1: 1 .. kTagMod.
__device__ __forceinline__ uint32_t tag_of(int s) { return (uint32_t)(1 + (s - 1) % kTagMod); }

// A removed edge's word: kGone, its tag in bits 15 .. 30, its residual (at
// most k - 2, so levels end at kResMax + 2) in the low 15 bits.
constexpr uint32_t kGone = 0x80000000u;
constexpr int kTagShift = 15;
constexpr uint32_t kResMax = (1u << kTagShift) - 1;
__device__ __forceinline__ uint32_t gone_tag(uint32_t tag) { return kGone | (tag << kTagShift); }

// A work item is one aligned block of kItem list entries of one edge, the
// entries [lo, hi) of block `blk` of the own parts or of the rest array: x =
// edge, y = blk, z = lo | hi << 8 | own << 16 | first << 17 (the item that
// records the edge's truss number).  Aligned blocks put an item in
// one 128-byte line and let a lane load its two entries as one 16-byte word.
constexpr int64_t kOffLimit = (int64_t)kItem << 32;

// Blocks that [off, off + len) touches.
__device__ __forceinline__ int blocks_of(int64_t off, int len) {
  return len > 0 ? (int)(((off + len + kItem - 1) >> 4) - (off >> 4)) : 0;
}

__device__ __forceinline__ int4 make_item(int e, int64_t off, int len, int b, bool own,
                                          bool first) {
  const int64_t blk = (off >> 4) + b;
  const int lo = b == 0 ? (int)(off & (kItem - 1)) : 0;
  const int64_t left = off + len - (blk << 4);
  const int hi = left < kItem ? (int)left : kItem;
  return make_int4(e, (int)(uint32_t)blk, lo | (hi << 8) | ((int)own << 16) | ((int)first << 17),
                   0);
}

// Per-warp staging buffers in shared memory (counts are warp-uniform).
struct WarpBuf {
  int4 *push;  // pushed edges not yet expanded: edge, list length (-1: not known yet), offset
  int np;
  int32_t *alive;
  int na;
};

// One of the two item queues: item i is at p[i] (d = 1) or p[-i] (d = -1).
struct Queue {
  int4 *Q;
  uint32_t cap;
  bool rev;
  __device__ __forceinline__ int4 *at(uint32_t i) const { return Q + (rev ? cap - 1 - i : i); }
};

// Expand the staged pushed edges into work items and append them to queue Q
// with one reservation.  The list length and offsets of all staged edges
// are loaded together here, once per flush, instead of one dependent round
// trip per push inside the sub-round's loop.
__device__ __forceinline__ void flush_push(const PeelArgs &a, WarpBuf &wb, const Queue &Q,
                                           unsigned long long *qctr) {
  const int np = wb.np;
  if (np == 0) return;
  const int lane = lane_id();
  const bool v = lane < np;
  const int4 st = v ? wb.push[lane] : make_int4(0, 0, 0, 0);
  const int p = st.x;
  int L = st.y;
  int64_t lb = (int64_t)((uint64_t)(uint32_t)st.w << 32 | (uint32_t)st.z);
  if (L < 0) {
    L = __ldg(&a.sup[p]);
    lb = __ldg(&a.off[p]);
  }
  const bool own = a.own_cnt != nullptr;
  const int cA = (own && v) ? __ldg(&a.own_cnt[p]) : 0;
  const int64_t la = (own && v) ? __ldg(&a.own_off[p]) : 0;
  L -= cA;  // the rest part
  const int nA = blocks_of(la, cA);
  const int n = nA + blocks_of(lb, L);
  if (np == 1) {
    // one push, as most flushes have: no scan, no search for each item's edge
    // (for up to four or eight pushes one after another it lost again; peel of
    // R-MAT scale 20 26.2 -> 25.5 ms, 40 M-edge Chung-Lu 72.7 -> 71.8 ms, 4,096
    // small graphs 7.8 -> 7.5 ms)
    const int tot = __shfl_sync(TR_FULL, n, 0);
    uint32_t at = 0;
    if (lane == 0) at = reserve_items(qctr, tot);
    at = __shfl_sync(TR_FULL, at, 0);
    const int po = __shfl_sync(TR_FULL, p, 0), Lo = __shfl_sync(TR_FULL, L, 0);
    const int64_t lbo = __shfl_sync(TR_FULL, lb, 0);
    const int nAo = own ? __shfl_sync(TR_FULL, nA, 0) : 0;
    const int cAo = own ? __shfl_sync(TR_FULL, cA, 0) : 0;
    const int64_t lao = own ? __shfl_sync(TR_FULL, la, 0) : 0;
    for (int it = lane; it < tot; it += 32)
      if (at + it < a.item_cap)
        *Q.at(at + it) = it < nAo ? make_item(po, lao, cAo, it, true, it == 0)
                                  : make_item(po, lbo, Lo, it - nAo, false, it == 0);
    __syncwarp();
    wb.np = 0;
    return;
  }
  const int P = warp_incl_scan(n);
  uint32_t b = 0;
  if (lane == 31) b = reserve_items(qctr, P);
  const int tot = __shfl_sync(TR_FULL, P, 31);
  const uint32_t base = __shfl_sync(TR_FULL, b, 31);
  for (int u0 = 0; u0 < tot; u0 += 32) {
    const int t = u0 + lane;
    const int o = warp_owner(P, t < tot ? t : tot - 1);
    const int po = __shfl_sync(TR_FULL, p, o);
    const int i0 = __shfl_sync(TR_FULL, P - n, o);
    const int Lo = __shfl_sync(TR_FULL, L, o);
    const int64_t lbo = __shfl_sync(TR_FULL, lb, o);
    int nAo = 0, cAo = 0;
    int64_t lao = 0;
    if (own) {
      nAo = __shfl_sync(TR_FULL, nA, o);
      cAo = __shfl_sync(TR_FULL, cA, o);
      lao = __shfl_sync(TR_FULL, la, o);
    }
    const uint32_t idx = base + t;
    if (t < tot && idx < a.item_cap) {
      const int it = t - i0;
      *Q.at(idx) = it < nAo ? make_item(po, lao, cAo, it, true, it == 0)
                            : make_item(po, lbo, Lo, it - nAo, false, it == 0);
    }
  }
  __syncwarp();
  wb.np = 0;
}

__device__ __forceinline__ void flush_alive(const PeelArgs &a, WarpBuf &wb, int32_t *A2,
                                            int *actr) {
  if (wb.na == 0) return;
  const int lane = lane_id();
  int b = 0;
  if (lane == 0) b = atomicAdd(actr, wb.na);
  const int b0 = __shfl_sync(TR_FULL, b, 0);
  for (int t = lane; t < wb.na; t += 32)
    if (b0 + t < a.m) A2[b0 + t] = wb.alive[t];
  __syncwarp();
  wb.na = 0;
}

// Queue the alive edges of the lanes with `keep` for the rewritten list.
__device__ __forceinline__ void push_alive(const PeelArgs &a, bool keep, int e, WarpBuf &wb,
                                           int32_t *A2, int *actr) {
  const unsigned mask = __ballot_sync(TR_FULL, keep);
  if (mask == 0) return;
  const int tot = __popc(mask);
  if (wb.na + tot > kWA) flush_alive(a, wb, A2, actr);
  if (keep) wb.alive[wb.na + __popc(mask & ((1u << lane_id()) - 1u))] = e;
  __syncwarp();
  wb.na += tot;
}

__device__ __forceinline__ void prefetch_list(const PeelArgs &a, int p) {
  prefetch_l1(a.sup + p);
  prefetch_l1(a.off + p);
  if (a.own_cnt) {
    prefetch_l1(a.own_cnt + p);
    prefetch_l1(a.own_off + p);
  }
}

// Stage edge p (for each lane with `push`) for expansion into work items of
// the next frontier.  All lanes call it.
__device__ __forceinline__ void push_items(const PeelArgs &a, bool push, int4 p, WarpBuf &wb,
                                           const Queue &Q, unsigned long long *qctr) {
  const unsigned mask = __ballot_sync(TR_FULL, push);
  if (mask == 0) return;
  const int tot = __popc(mask);
  if (wb.np + tot > kWP) flush_push(a, wb, Q, qctr);
  if (push) {
    wb.push[wb.np + __popc(mask & ((1u << lane_id()) - 1u))] = p;
    if (p.y < 0) prefetch_list(a, p.x);  // the flush reads its list length and offsets
  }
  __syncwarp();
  wb.np += tot;
}

// What a partner's word says in the sub-round whose frontier carries word
// prefix fs (gone_tag(tag(s)) >> kTagShift) and whose pushes carry fn.
__device__ __forceinline__ bool in_front(uint32_t w, uint32_t fs) { return (w >> kTagShift) == fs; }
__device__ __forceinline__ bool is_dead(uint32_t w, uint32_t fs, uint32_t fn) {
  const uint32_t h = w >> kTagShift;
  return (int32_t)w < 0 && h != fs && h != fn;
}

// MINB = resident blocks per SM the register budget is sized for (1: up to
// 128 registers per thread, 2: 64); G = work items per 8-lane group per
// iteration (2 entries per lane per item).
template <int MINB, int G, bool COUNT = false>
__global__ void __launch_bounds__(kPeelBlock, MINB) k_peel(PeelArgs a) {
  const int lane = lane_id();
  const int wib = threadIdx.x >> 5;
  // consecutive warps of the launch sit in different blocks, so a phase with
  // little work spreads it over all SMs
  const int gwarp = wib * gridDim.x + blockIdx.x;
  const int twarps = gridDim.x * kWarps;
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  PeelCtl *ctl = a.ctl;
  __shared__ int4 s_push[kWarps][kWP];
  __shared__ int32_t s_alive[kWarps][kWA];
  __shared__ int s_minres, s_live, s_any;
  WarpBuf wb{s_push[wib], 0, s_alive[wib], 0};
  if (threadIdx.x == 0) {
    s_minres = INT_MAX;
    s_live = 0;
    s_any = 0;
  }
  __syncthreads();

  int k = 2, s = 1, sc = 0;
  unsigned ph = 0;  // phase index (scans and sub-rounds)
  bool odd = false;  // which alive list is current
  bool rev = false;  // which queue is the current frontier's
  int nAlive = (int)a.m;
  bool compact = false;  // rewrite the alive list during this scan
  // work counts of each thread, in shared memory: registers are short (32-bit:
  // a lane's share of even 2^33 list entries over the grid's 150 K lanes stays
  // far below 2^32)
  __shared__ uint2 s_work[kPeelBlock];  // entries read, decrements
  s_work[threadIdx.x] = make_uint2(0, 0);
  unsigned n_dead = 0, n_early = 0;  // counting runs: totals so far
  auto clamp = [&](uint32_t n) {
    if (n <= a.item_cap) return n;
    // appends beyond the queue were dropped
    if (leader) raise_error(&ctl->phase[ph % 3], &ctl->err, TRUSS_ECHECK);
    return a.item_cap;
  };
  // Every a.retag sub-rounds (checked at the start of each phase, the same in
  // every block): tags other than the current frontier's become kDead.  A
  // tag left on a removed edge is then from the last a.retag sub-rounds, so
  // it never equals tag(s) or tag(s+1) of a later sub-round by wrapping.
  int last_retag = 0;
  auto retag = [&]() -> bool {
    if (s - last_retag < a.retag) return true;
    last_retag = s;
    if (leader) ctl->phase[(ph + 1) % 3] = 0;
    const uint32_t keep = gone_tag(tag_of(s)) >> kTagShift;
    const int64_t nt = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < a.m; e += nt) {
      const uint32_t w = __ldcg(&a.word[e]);
      if ((int32_t)w < 0 && (w >> kTagShift) != keep)
        a.word[e] = gone_tag(kDead) | (w & kResMax);
    }
    uint32_t items;
    const bool ok = phase_end(ctl, a.wait_ns, ph, &items, nullptr, nullptr);
    ph++;
    return ok;
  };

  for (;;) {
    if (a.k_stop > 0 && k > a.k_stop) break;  // k is the same in every block
    if (k - 2 > (int)kResMax) {
      // no graph whose lists fit the device has a truss this deep
      if (leader) raise_error(&ctl->phase[ph % 3], &ctl->err, TRUSS_ECHECK);
      break;
    }
    if (!retag()) return;
    // ------------------------------------------------------------ scan ---
    if (leader && a.trace && ctl->ntrace < a.trace_cap) {
      const unsigned long long t = global_ns();
      a.trace[ctl->ntrace++] = make_int4(k, -1, (int)(uint32_t)t, (int)(uint32_t)(t >> 32));
    }
    ScanOut *scan = &ctl->scan[sc % 3];
    unsigned long long *qf = &ctl->phase[ph % 3];
    if (leader) {
      *(int4 *)&ctl->scan[(sc + 1) % 3] = make_int4(INT_MAX, 0, 0, 0);
      ctl->phase[(ph + 1) % 3] = 0;
    }
    const int32_t *alive = odd ? a.alive1 : a.alive0;
    int32_t *alive2 = odd ? a.alive0 : a.alive1;
    const Queue F{a.Q, a.item_cap, rev};
    int lmin = INT_MAX, llive = 0;  // of this lane
    bool lany = false;
    // 4 x 32 entries per warp iteration: all loads are issued before any
    // decision, so one dependent round trip covers 4 entries per lane
    constexpr int kScanU = 4;
    for (int64_t base = (int64_t)gwarp * 32 * kScanU; base < nAlive;
         base += (int64_t)twarps * 32 * kScanU) {
      int e[kScanU];
      uint32_t w[kScanU];
#pragma unroll
      for (int u = 0; u < kScanU; u++) {
        const int64_t i = base + u * 32 + lane;
        e[u] = i < nAlive ? __ldcg(&alive[i]) : -1;
      }
#pragma unroll
      for (int u = 0; u < kScanU; u++) w[u] = e[u] >= 0 ? __ldcg(&a.word[e[u]]) : kGone;
      unsigned pend = 0;  // entries of this lane that join the frontier
#pragma unroll
      for (int u = 0; u < kScanU; u++) {
        const bool live = (int32_t)w[u] >= 0;
        const bool toF = live && (int)w[u] <= k - 2;
        const bool keep = live && !toF;
        if (toF) {
          // removed at this level; without triangles left it needs no item
          a.word[e[u]] = gone_tag(tag_of(s)) | w[u];
          if (w[u] > 0) {
            pend |= 1u << u;
          } else {
            a.truss[e[u]] = k;
            if (COUNT) a.when[e[u]] = s;
          }
          lany = true;
        }
        if (compact) push_alive(a, keep, e[u], wb, alive2, &scan->listed);
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
            if (b == u) q = e[u];
        }
        push_items(a, has, make_int4(q, -1, 0, 0), wb, F, qf);
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
    const int minres = found.minres, live = found.live, any = found.any;
    if (leader) ctl->scanned += (unsigned)nAlive;
    if (compact) {
      nAlive = found.listed;
      odd = !odd;
    }
    compact = 4 * (int64_t)live <= 3 * (int64_t)nAlive;  // rewrite the list once a quarter of it is dead
    sc++;
    if (any && leader) {
      ctl->levels++;
      ctl->kmax = k;
    }
    if (nCur == 0) {
      // nothing removed had a triangle left, so the residuals stand; what went
      // counts as one sub-round
      if (any) {
        s++;
        if (leader) ctl->subrounds++;
      }
      if (live == 0) break;
      k = minres + 2;  // every alive edge has res >= k-1: skip empty levels
      continue;
    }
    // --------------------------------------------------------- sub-rounds ---
    nCur = clamp(nCur);
    const int s_lvl0 = s;  // first sub-round of this level
    for (;;) {
      const unsigned c_ent = COUNT ? s_work[threadIdx.x].x : 0, c_dead = n_dead, c_early = n_early;
      if (!retag()) return;
      const uint32_t fs = gone_tag(tag_of(s)) >> kTagShift, pushw = gone_tag(tag_of(s + 1)),
                     fn = pushw >> kTagShift;
      if (leader && a.trace && ctl->ntrace < a.trace_cap) {
        const unsigned long long t = global_ns();
        a.trace[ctl->ntrace++] = make_int4(k, (int)min(nCur, (uint32_t)INT_MAX),
                                           (int)(uint32_t)t, (int)(uint32_t)(t >> 32));
      }
      unsigned long long *qn = &ctl->phase[ph % 3];
      if (leader) ctl->phase[(ph + 1) % 3] = 0;
      const int grp = lane >> 3, j = lane & 7;
      const uint32_t stride = (uint32_t)twarps * 4 * G;
      const Queue F{a.Q, a.item_cap, rev}, N{a.Q, a.item_cap, !rev};
      // Items are loaded two iterations ahead and their list entries and
      // edge words one ahead, so that an iteration waits only for its
      // partners' words and decrements.
      int4 cur[G], nxt[G], ent[G], entn[G];  // ent: two list entries of this lane per item
      uint32_t we[G], wen[G];
      auto load_item = [&](int4 *it, uint32_t base) {
#pragma unroll
        for (int g = 0; g < G; g++)
          it[g] = base + g * 4 + grp < nCur ? __ldcg(F.at(base + g * 4 + grp))
                                            : make_int4(0, 0, 0, 0);
      };
      auto load_entries = [&](const int4 *it, int4 *en, uint32_t *w) {
#pragma unroll
        for (int g = 0; g < G; g++) {
          const int lo = it[g].z & 0xFF, hi = (it[g].z >> 8) & 0xFF;
          const bool any2 = 2 * j + 1 >= lo && 2 * j < hi;
          w[g] = any2 ? __ldcg(&a.word[it[g].x]) : 0u;
          // list entries are read once: evict-first, so that the words
          // (re-read at random) keep their place in L2
          const int4 *blk = (const int4 *)(((it[g].z >> 16) & 1) ? a.own : a.rest) +
                            (int64_t)(uint32_t)it[g].y * 8;
          en[g] = any2 ? __ldcs(blk + j) : make_int4(0, 0, 0, 0);
        }
      };
      uint32_t base = (uint32_t)gwarp * 4 * G;
      if (base < nCur) {
        load_item(cur, base);
        load_item(nxt, base + stride);
        load_entries(cur, ent, we);
      }
      for (; base < nCur; base += stride) {
        load_entries(nxt, entn, wen);
        int4 nxt2[G];
        load_item(nxt2, base + 2 * stride);
        bool v0[G], v1[G];
#pragma unroll
        for (int g = 0; g < G; g++) {
          const int lo = cur[g].z & 0xFF, hi = (cur[g].z >> 8) & 0xFF;
          if ((cur[g].z >> 17) && j == 0) {
            a.truss[cur[g].x] = k;
            if (COUNT) a.when[cur[g].x] = s;
          }
          v0[g] = 2 * j >= lo && 2 * j < hi;
          v1[g] = 2 * j + 1 >= lo && 2 * j + 1 < hi;
        }
        // Charge: a triangle of frontier edge e and partners p1, p2, none
        // of them removed earlier, is charged by the lowest-id frontier edge
        // among the three, which decrements the partners not in the frontier.
        uint2 work = make_uint2(0, 0);
        uint32_t s1[2 * G], s2[2 * G];
        bool d1[2 * G], d2[2 * G];
#pragma unroll
        for (int i = 0; i < 2 * G; i++) {
          const int g = i >> 1;
          const int p1 = (i & 1) ? ent[g].z : ent[g].x, p2 = (i & 1) ? ent[g].w : ent[g].y;
          bool v = ((i & 1) ? v1[g] : v0[g]) && (we[g] & kResMax) != 0;
          if (v && ((uint32_t)p1 >= (uint32_t)a.m || (uint32_t)p2 >= (uint32_t)a.m)) {
            raise_error(&ctl->phase[ph % 3], &ctl->err, TRUSS_ECHECK);  // corrupt list entry: skip it
            v = false;
          }
          work.x += v;
          // a masked entry reads as dead
          s1[i] = v ? __ldcg(&a.word[p1]) : gone_tag(0);
          s2[i] = v ? __ldcg(&a.word[p2]) : gone_tag(0);
        }
#pragma unroll
        for (int i = 0; i < 2 * G; i++) {
          const int g = i >> 1, e = cur[g].x;
          const int p1 = (i & 1) ? ent[g].z : ent[g].x, p2 = (i & 1) ? ent[g].w : ent[g].y;
          const bool dead = is_dead(s1[i], fs, fn) || is_dead(s2[i], fs, fn);
          const bool in1 = in_front(s1[i], fs), in2 = in_front(s2[i], fs);
          d1[i] = !dead && !in1 && (!in2 || e < p2);
          d2[i] = !dead && !in2 && (!in1 || e < p1);
          if (COUNT) {
            // a destroyed triangle lost its first edge when the earlier-
            // removed of its removed partners went
            const bool v = ((i & 1) ? v1[g] : v0[g]) && (we[g] & kResMax) != 0;
            if (v && dead && (uint32_t)p1 < (uint32_t)a.m && (uint32_t)p2 < (uint32_t)a.m) {
              const int w1 = __ldcg(&a.when[p1]), w2 = __ldcg(&a.when[p2]);
              n_dead++;
              n_early += min(w1, w2) < s_lvl0;
            }
          }
        }
        // a partner that a decrement should remove: fetch its list's place now
        int cand = -1, candL = 0;
        int64_t candO = 0;
#pragma unroll
        for (int i = 0; i < 2 * G; i++) {
          const int g = i >> 1;
          const int p1 = (i & 1) ? ent[g].z : ent[g].x, p2 = (i & 1) ? ent[g].w : ent[g].y;
          if (d1[i] && s1[i] == (uint32_t)(k - 1)) cand = p1;
          if (d2[i] && s2[i] == (uint32_t)(k - 1)) cand = p2;
        }
        if (cand >= 0) {
          candL = __ldg(&a.sup[cand]);
          candO = __ldg(&a.off[cand]);
        }
        unsigned pend = 0;  // pending pushes, bit 2i (p1) and 2i+1 (p2)
#pragma unroll
        for (int i = 0; i < 2 * G; i++) {
          const int g = i >> 1;
          const int p1 = (i & 1) ? ent[g].z : ent[g].x, p2 = (i & 1) ? ent[g].w : ent[g].y;
          // s1 / s2 take the residuals before the decrements
          s1[i] = d1[i] ? atomicSub(&a.word[p1], 1u) : 0u;
          s2[i] = d2[i] ? atomicSub(&a.word[p2], 1u) : 0u;
          work.y += (unsigned)(d1[i] + d2[i]);
        }
        s_work[threadIdx.x].x += work.x;
        s_work[threadIdx.x].y += work.y;
#pragma unroll
        for (int i = 0; i < 2 * G; i++) {
          // k >= 3 here, so a lane without a decrement (0) never matches
          pend |= (s1[i] == (uint32_t)(k - 1) ? 1u : 0u) << (2 * i) |
                  (s2[i] == (uint32_t)(k - 1) ? 1u : 0u) << (2 * i + 1);
        }
        // the warp pushes one partner per lane per step through one site
        while (__any_sync(TR_FULL, pend != 0)) {
          int q = 0;
          const bool has = pend != 0;
          if (has) {
            const int b = __ffs(pend) - 1;
            pend &= pend - 1;
#pragma unroll
            for (int i = 0; i < 2 * G; i++) {
              const int g = i >> 1;
              if ((b >> 1) == i)
                q = (b & 1) ? ((i & 1) ? ent[g].w : ent[g].y) : ((i & 1) ? ent[g].z : ent[g].x);
            }
            // others may still decrement q's residual: add the mark to it
            atomicAdd(&a.word[q], pushw);
          }
          const bool known = q == cand;
          push_items(a, has,
                     make_int4(q, known ? candL : -1, (int)(uint32_t)candO,
                               (int)(uint32_t)((uint64_t)candO >> 32)),
                     wb, N, qn);
        }
#pragma unroll
        for (int g = 0; g < G; g++) {
          cur[g] = nxt[g];
          nxt[g] = nxt2[g];
          ent[g] = entn[g];
          we[g] = wen[g];
        }
      }
      flush_push(a, wb, N, qn);
      if (COUNT && k < a.lvl_cap) {
        unsigned x0 = s_work[threadIdx.x].x - c_ent, x1 = n_dead - c_dead, x2 = n_early - c_early;
        for (int o = 16; o >= 1; o >>= 1) {
          x0 += __shfl_down_sync(TR_FULL, x0, o);
          x1 += __shfl_down_sync(TR_FULL, x1, o);
          x2 += __shfl_down_sync(TR_FULL, x2, o);
        }
        if (lane == 0 && (x0 | x1 | x2)) {
          atomicAdd(&a.lvl[3 * k], (unsigned long long)x0);
          atomicAdd(&a.lvl[3 * k + 1], (unsigned long long)x1);
          atomicAdd(&a.lvl[3 * k + 2], (unsigned long long)x2);
        }
      }
      if (!phase_end(ctl, a.wait_ns, ph, &nCur, nullptr, nullptr)) return;
      ph++;
      s++;
      if (leader) ctl->subrounds++;
      if (nCur == 0) break;
      rev = !rev;
      nCur = clamp(nCur);
    }
    k++;
  }
  if (leader && a.trace && ctl->ntrace < a.trace_cap) {
    const unsigned long long t = global_ns();
    a.trace[ctl->ntrace++] = make_int4(k, -2, (int)(uint32_t)t, (int)(uint32_t)(t >> 32));
  }
  // totals (one atomic per warp)
  unsigned n_entries = s_work[threadIdx.x].x, n_dec = s_work[threadIdx.x].y;
  for (int o = 16; o >= 1; o >>= 1) {
    n_entries += __shfl_down_sync(TR_FULL, n_entries, o);
    n_dec += __shfl_down_sync(TR_FULL, n_dec, o);
    if (COUNT) {
      n_dead += __shfl_down_sync(TR_FULL, n_dead, o);
      n_early += __shfl_down_sync(TR_FULL, n_early, o);
    }
  }
  if (lane == 0) {
    atomicAdd(&ctl->entries, (unsigned long long)n_entries);
    atomicAdd(&ctl->decrements, (unsigned long long)n_dec);
    if (COUNT) {
      atomicAdd(&ctl->dead, (unsigned long long)n_dead);
      atomicAdd(&ctl->dead_earlier, (unsigned long long)n_early);
    }
  }
}

// Residual given to pinned edges: no level ever reaches it, and the
// decrements it can receive (at most its support) leave it out of reach.
constexpr int kPinnedRes = INT_MAX / 4;

__global__ void k_peel_init(int64_t m, const int32_t *sup, const uint8_t *pinned, uint32_t *word,
                            int32_t *alive, int32_t *truss, const int *list_err, PeelCtl *ctl) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    word[e] = (uint32_t)((pinned && pinned[e]) ? kPinnedRes : sup[e]);
    alive[e] = (int32_t)e;
    truss[e] = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int i = 0; i < 3; i++) ctl->scan[i].minres = INT_MAX;
    ctl->err = *list_err;  // a list builder's error is reported with the peel's result
  }
}

// Removal-order figures of a counting run (PeelResult): min alive degrees
// from the removal sub-rounds, the edges present at each level that removes
// one (from the truss-number histogram), and the per-level entry counts,
// written to the file named by TRUSS_LEVEL_STATS if set.
__global__ void k_truss_hist(int64_t m, const int32_t *truss, int cap,
                             unsigned long long *cnt) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int k = truss[e];
    if (k >= 0 && k < cap) atomicAdd(&cnt[k], 1ull);
  }
}

int count_run(Arena &A, const Csr &g, const SupportOut &so, const PeelArgs &a, const PeelCtl &h,
              const int32_t *truss, PeelResult *out, cudaStream_t s) {
  const int cap = h.kmax + 2 < a.lvl_cap ? h.kmax + 2 : a.lvl_cap;
  unsigned long long *cnt = A.get<unsigned long long>(cap);
  if (!cnt) return TRUSS_ENOMEM;
  TR_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * cap, s));
  k_truss_hist<<<grid_for(g.m, 256, 152 * 16), 256, 0, s>>>(g.m, truss, cap, cnt);
  TR_LAUNCHED();
  std::vector<unsigned long long> hc((size_t)cap), hl((size_t)3 * cap);
  TR_CUDA(cudaMemcpyAsync(hc.data(), cnt, sizeof(unsigned long long) * cap,
                          cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaMemcpyAsync(hl.data(), a.lvl, sizeof(unsigned long long) * 3 * cap,
                          cudaMemcpyDeviceToHost, s));
  unsigned long long sums[2] = {0, 0};
  TR_TRY(count_min_alive(A, g, so, a.when, sums, s));
  TR_CUDA(cudaStreamSynchronize(s));
  // edges present when level k starts: truss number >= k
  std::vector<unsigned long long> alive((size_t)cap + 1, 0);
  for (int k = cap - 1; k >= 0; k--) alive[k] = alive[k + 1] + hc[k];
  out->alive_levels = 0;
  for (int k = 0; k < cap; k++)
    if (hc[k] > 0) out->alive_levels += alive[k];
  out->sum_min_alive = sums[0];
  out->sum_min_alive_start = sums[1];
  out->dead = h.dead;
  out->dead_earlier = h.dead_earlier;
  if (const char *path = getenv("TRUSS_LEVEL_STATS")) {
    if (FILE *f = fopen(path, "w")) {
      fprintf(f, "k,removed,present,entries,dead,dead_earlier\n");
      for (int k = 0; k < cap; k++)
        if (hc[k] > 0 || hl[3 * k] > 0)
          fprintf(f, "%d,%llu,%llu,%llu,%llu,%llu\n", k, hc[k], alive[k], hl[3 * k],
                  hl[3 * k + 1], hl[3 * k + 2]);
      fclose(f);
    }
  }
  return TRUSS_OK;
}

// Keys (endpoint, removal sub-round) of both endpoints of every edge.
__global__ void k_when_keys(int64_t m, const int32_t *esrc, const int32_t *adjp,
                            const int32_t *when, uint64_t *keys) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t w = (uint32_t)when[e];
    keys[2 * e] = (uint64_t)(uint32_t)esrc[e] << 32 | w;
    keys[2 * e + 1] = (uint64_t)(uint32_t)adjp[e] << 32 | w;
  }
}

// Degree of every vertex (out-edges + in-edges); entry n is 0.
__global__ void k_sym_degree(int64_t n, const int64_t *offp, const int64_t *inoff,
                             int64_t *deg) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= n;
       u += (int64_t)gridDim.x * blockDim.x)
    deg[u] = u < n ? (offp[u + 1] - offp[u]) + (inoff[u + 1] - inoff[u]) : 0;
}

// Entries of the sorted run keys[lo, hi) that are >= key.
__device__ __forceinline__ int64_t count_ge(const uint64_t *keys, int64_t lo, int64_t hi,
                                            uint64_t key) {
  const int64_t end = hi;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (keys[mid] < key) lo = mid + 1; else hi = mid;
  }
  return end - lo;
}

// acc[0] += min over e's endpoints x of (1 + x's edges removed in a later
// sub-round than e); acc[1] += the same with every edge not removed before
// e's sub-round (e's co-frontier edges included).
__global__ void k_min_alive(int64_t m, const int32_t *esrc, const int32_t *adjp,
                            const int32_t *when, const int64_t *soff, const uint64_t *keys,
                            unsigned long long *acc) {
  unsigned long long lo = 0, hi = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int u = esrc[e], v = adjp[e];
    const uint64_t w = (uint32_t)when[e];
    const uint64_t ku = (uint64_t)(uint32_t)u << 32 | w, kv = (uint64_t)(uint32_t)v << 32 | w;
    const int64_t su = count_ge(keys, soff[u], soff[u + 1], ku);
    const int64_t sv = count_ge(keys, soff[v], soff[v + 1], kv);
    const int64_t au = 1 + count_ge(keys, soff[u], soff[u + 1], ku + 1);
    const int64_t av = 1 + count_ge(keys, soff[v], soff[v + 1], kv + 1);
    hi += (unsigned long long)(su < sv ? su : sv);
    lo += (unsigned long long)(au < av ? au : av);
  }
  for (int o = 16; o >= 1; o >>= 1) {
    lo += __shfl_down_sync(TR_FULL, lo, o);
    hi += __shfl_down_sync(TR_FULL, hi, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (lo) atomicAdd(&acc[0], lo);
    if (hi) atomicAdd(&acc[1], hi);
  }
}

}  // namespace

int count_min_alive(Arena &A, const Csr &g, const SupportOut &so, const int32_t *when,
                    unsigned long long *sum, cudaStream_t s) {
  const int64_t m = g.m, n = g.n;
  sum[0] = sum[1] = 0;
  if (m == 0) return TRUSS_OK;
  if (!so.inoff) return TRUSS_EINVAL;
  uint64_t *k0 = A.get<uint64_t>(2 * m), *k1 = A.get<uint64_t>(2 * m);
  int64_t *deg = A.get<int64_t>(n + 1), *soff = A.get<int64_t>(n + 1);
  unsigned long long *acc = A.get<unsigned long long>(2);
  if (!k0 || !k1 || !deg || !soff || !acc) return TRUSS_ENOMEM;
  k_when_keys<<<grid_for(m, 256, 152 * 16), 256, 0, s>>>(m, g.esrc, g.adjp, when, k0);
  TR_LAUNCHED();
  k_sym_degree<<<grid_for(n + 1, 256, 152 * 16), 256, 0, s>>>(n, g.offp, so.inoff, deg);
  TR_LAUNCHED();
  const int end_bit = 32 + bits_for((uint64_t)(n > 0 ? n - 1 : 0));
  size_t tb = 0, tb2 = 0;
  TR_TRY(sort_keys_u64(nullptr, &tb, k0, k1, 2 * m, 0, end_bit, s));
  TR_TRY(exclusive_sum_i64(nullptr, &tb2, deg, soff, n + 1, s));
  void *tmp = A.alloc(tb > tb2 ? tb : tb2);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(sort_keys_u64(tmp, &tb, k0, k1, 2 * m, 0, end_bit, s));
  TR_TRY(exclusive_sum_i64(tmp, &tb2, deg, soff, n + 1, s));
  TR_CUDA(cudaMemsetAsync(acc, 0, 2 * sizeof(unsigned long long), s));
  k_min_alive<<<grid_for(m, 256, 152 * 16), 256, 0, s>>>(m, g.esrc, g.adjp, when, soff, k1, acc);
  TR_LAUNCHED();
  TR_CUDA(cudaMemcpyAsync(sum, acc, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  return TRUSS_OK;
}

int run_peel(Arena &A, const Csr &g, const SupportOut &so, const TriLists &L, const PeelCfg &cfg,
             int32_t *truss, PeelResult *out, cudaStream_t s) {
  const int64_t m = g.m;
  *out = PeelResult{};
  if (m == 0) return cfg.then ? cfg.then() : TRUSS_OK;
  // items carry 32-bit block numbers
  if (so.entries >= kOffLimit || (L.own_cnt && so.records >= kOffLimit)) return TRUSS_EINVAL;
  if (so.entries > 0 && (!L.rest || !L.off || (L.own_cnt && (!L.own || !L.own_off))))
    return TRUSS_EINVAL;
  // Items of all edges: the lists in `rest` follow one another, so they touch
  // at most one block each beyond the array's own; an own part of c entries
  // touches at most c / kItem + 2.
  const bool own = L.own_cnt != nullptr;
  const int64_t item_cap = so.entries / kItem + (own ? 3 : 1) * m + 64;
  // items are counted in 32 bits: beyond that their queue alone takes 34 GB
  // and the lists 275 GB or more
  if (item_cap > (int64_t)UINT32_MAX / 2) return TRUSS_ENOMEM;
  uint32_t *word = A.get<uint32_t>(m);
  int32_t *al0 = A.get<int32_t>(m), *al1 = A.get<int32_t>(m);
  int4 *Q = A.get<int4>(item_cap);
  static_assert(sizeof(PeelCtl) <= ZeroBlock::kCtl, "control words fit the zero block");
  PeelCtl *ctl = (PeelCtl *)g.zero->peel;
  if (!word || !al0 || !al1 || !Q) return TRUSS_ENOMEM;
  k_peel_init<<<grid_for(m, 256, 152 * 16), 256, 0, s>>>(m, so.sup, cfg.pinned, word, al0, truss,
                                                          &g.zero->list_err, ctl);
  TR_LAUNCHED();

  int dev = 0, sms = cfg.sms;
  TR_CUDA(cudaGetDevice(&dev));
  if (sms <= 0) TR_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // variant 1: 128-register kernel taking 2 items per lane group, one block
  // per SM; 3: 1 item per group, one block per SM; otherwise (0, 2) the
  // 64-register kernel with 1 item per group and two blocks per SM
  const int variant = cfg.variant == 1 ? 1 : (cfg.variant == 3 ? 3 : 2);
  const void *kern = cfg.count      ? (const void *)k_peel<2, 1, true>
                     : variant == 1 ? (const void *)k_peel<1, 2>
                     : variant == 3 ? (const void *)k_peel<1, 1>
                                    : (const void *)k_peel<2, 1>;
  int occ = 0;
  TR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kPeelBlock, 0));
  if (occ < 1) return TRUSS_ECUDA;
  if (variant != 2 && !cfg.count && occ > 1) occ = 1;
  if (variant == 2) sms = peel_sms(so.entries + 8 * m, sms);
  sms = peel_share(so.entries + 8 * m, sms, cfg.max_sms);
  PeelArgs a{};
  a.m = m;
  a.sup = so.sup;
  a.own = L.own;
  a.own_off = L.own_off;
  a.own_cnt = L.own_cnt;
  a.rest = L.rest;
  a.off = L.off ? L.off : so.toff;
  a.word = word;
  a.retag = kRetagMax;
  if (const char *rt = getenv("TRUSS_PEEL_RETAG")) {  // testing: rewrite tags more often
    const int v = atoi(rt);
    a.retag = v < 1 ? 1 : v > kRetagMax ? kRetagMax : v;
  }
  a.truss = truss;
  a.alive0 = al0;
  a.alive1 = al1;
  a.Q = Q;
  a.item_cap = (uint32_t)item_cap;
  a.ctl = ctl;
  a.wait_ns = cfg.wait_ns;
  a.k_stop = cfg.k_stop;
  constexpr int kLvlCap = 1 << 16;
  if (cfg.count) {
    a.when = A.get<int32_t>(m);
    a.lvl = A.get<unsigned long long>(3 * (int64_t)kLvlCap);
    if (!a.when || !a.lvl) return TRUSS_ENOMEM;
    a.lvl_cap = kLvlCap;
    TR_CUDA(cudaMemsetAsync(a.when, 0x7F, sizeof(int32_t) * m, s));  // never removed
    TR_CUDA(cudaMemsetAsync(a.lvl, 0, sizeof(unsigned long long) * 3 * kLvlCap, s));
  }
  const char *trace_path = getenv("TRUSS_TRACE");
  const int trace_cap = 1 << 20;
  if (trace_path) {
    a.trace = A.get<int4>(trace_cap);
    a.trace_cap = a.trace ? trace_cap : 0;
  }
  void *args[] = {&a};
  TR_CUDA(cudaLaunchCooperativeKernel(kern, dim3(sms * occ), dim3(kPeelBlock), args, 0, s));
  count_launches(1);
  if (cfg.then) TR_TRY(cfg.then());
  PeelCtl h{};
  TR_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(PeelCtl), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  out->err = h.err;
  out->kmax = h.kmax;
  out->levels = h.levels;
  out->subrounds = h.subrounds;
  out->entries = h.entries;
  out->decrements = h.decrements;
  out->scanned = h.scanned;
  if (trace_path && a.trace) {
    const int nt = h.ntrace < trace_cap ? h.ntrace : trace_cap;
    std::vector<int4> t((size_t)nt);
    TR_CUDA(cudaMemcpy(t.data(), a.trace, sizeof(int4) * nt, cudaMemcpyDeviceToHost));
    if (FILE *f = fopen(trace_path, "w")) {
      fprintf(f, "k,items,t_ns\n");  // items: -1 = level scan, -2 = end
      for (auto &x : t)
        fprintf(f, "%d,%d,%llu\n", x.x, x.y,
                ((unsigned long long)(uint32_t)x.w << 32) | (uint32_t)x.z);
      fclose(f);
    }
  }
  if (h.err != 0) return h.err;
  if (cfg.count) TR_TRY(count_run(A, g, so, a, h, truss, out, s));
  return TRUSS_OK;
}

}  // namespace tr
