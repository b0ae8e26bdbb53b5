// Shared device/host helpers of the truss library (sm_103a).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/truss.h"

#define TR_FULL 0xffffffffu

namespace tr {

// ------------------------------------------------------------------ host ---
// Evaluate a CUDA runtime call; on failure return TRUSS_ECUDA from the
// enclosing function (remembering the message for diagnostics).
void note_cuda_error(cudaError_t e, const char *what, const char *file, int line);
void count_launches(int k);

#define TR_CUDA(call)                                             \
  do {                                                            \
    cudaError_t e_ = (call);                                      \
    if (e_ != cudaSuccess) {                                      \
      ::tr::note_cuda_error(e_, #call, __FILE__, __LINE__);       \
      return e_ == cudaErrorMemoryAllocation ? TRUSS_ENOMEM : TRUSS_ECUDA; \
    }                                                             \
  } while (0)

// After a kernel launch: count it and check the launch error.
#define TR_LAUNCHED()                  \
  do {                                 \
    ::tr::count_launches(1);           \
    TR_CUDA(cudaGetLastError());       \
  } while (0)

#define TR_TRY(expr)          \
  do {                        \
    int rc_ = (expr);         \
    if (rc_ != TRUSS_OK) return rc_; \
  } while (0)

inline int grid_for(int64_t work, int block, int max_blocks) {
  int64_t g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > max_blocks) g = max_blocks;
  return (int)g;
}

inline int bits_for(uint64_t maxval) {  // number of bits to represent maxval
  int b = 0;
  while (b < 64 && (maxval >> b) != 0) b++;
  return b;
}

// ---------------------------------------------------------------- device ---
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Inclusive prefix sum across the warp.
__device__ __forceinline__ int warp_incl_scan(int x) {
  const int l = lane_id();
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(TR_FULL, x, o);
    if (l >= o) x += y;
  }
  return x;
}

// Smallest lane o such that P[o] > t, for a non-decreasing per-lane value P
// with t < P[31].  All 32 lanes must call it.
__device__ __forceinline__ int warp_owner(int P, int t) {
  int o = 0;
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    int pv = __shfl_sync(TR_FULL, P, o + s - 1);
    if (pv <= t) o += s;
  }
  return o;
}

// Position of the r-th set bit of m (r from 0, below the number of set bits).
__device__ __forceinline__ int nth_set_bit(unsigned m, int r) {
  int pos = 0;
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const int low = __popc(m & ((1u << s) - 1u));
    if (r >= low) {
      r -= low;
      pos += s;
      m >>= s;
    }
  }
  return pos;
}

// Work of different lengths spread over a warp: lane l < n (n non-empty
// pieces) holds piece l, which takes the steps [S, S + len) of all pieces laid
// end to end.  owner() finds the piece of each lane's step of the window
// [tr, tr + 32), for consecutive windows from 0 on: the pieces that start in
// the window set one bit each, so it takes one warp reduction and a bit count
// where a search through the prefix takes five dependent shuffles.
struct FlatWork {
  int S, len;
  int before = 0;  // pieces that started before the window
  __device__ __forceinline__ int owner(int tr) {
    const int rel = S - tr;
    const unsigned bit = len > 0 && (unsigned)rel < 32u ? 1u << rel : 0u;
    const unsigned mask = __reduce_or_sync(TR_FULL, bit);
    const int o = before + __popc(mask & (0xFFFFFFFFu >> (31 - lane_id()))) - 1;
    before += __popc(mask);
    return o;
  }
};

// Warp-aggregated append: every lane with `pred` gets a distinct slot in a
// buffer whose fill counter is *cnt; returns the slot (or -1).  All lanes of
// the warp must call it.
__device__ __forceinline__ int warp_append(bool pred, int *cnt) {
  unsigned mask = __ballot_sync(TR_FULL, pred);
  if (mask == 0) return -1;
  int leader = __ffs(mask) - 1;
  int base = 0;
  if (lane_id() == leader) base = atomicAdd(cnt, __popc(mask));
  base = __shfl_sync(TR_FULL, base, leader);
  if (!pred) return -1;
  return base + __popc(mask & ((1u << lane_id()) - 1u));
}

// As warp_append, for a monotonically increasing 64-bit counter: returns the
// counter value reserved for this lane (the caller subtracts its base).
__device__ __forceinline__ long long warp_append64(bool pred, unsigned long long *cnt) {
  unsigned mask = __ballot_sync(TR_FULL, pred);
  if (mask == 0) return -1;
  int leader = __ffs(mask) - 1;
  unsigned long long base = 0;
  if (lane_id() == leader) base = atomicAdd(cnt, (unsigned long long)__popc(mask));
  base = __shfl_sync(TR_FULL, base, leader);
  if (!pred) return -1;
  return (long long)(base + __popc(mask & ((1u << lane_id()) - 1u)));
}

// Acquire-release atomic add and acquire load at GPU scope.
__device__ __forceinline__ unsigned long long atom_add_acq_rel_gpu(unsigned long long *p,
                                                                   unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;"
               : "=l"(old)
               : "l"(p), "l"(v)
               : "memory");
  return old;
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Top bit of a barrier counter: some block has recorded an error.
constexpr unsigned long long kBarErr = 1ull << 63;

// Record an error and make every block leave at its next barrier.
__device__ __forceinline__ void raise_error(unsigned long long *bar, int *err, int code) {
  atomicExch(err, code);
  atomicOr(bar, kBarErr);
}

// Grid-wide barrier of a cooperative launch, with a time limit.  Arrival is
// one atomic increment of `bar`, a counter that is never reset: the block
// whose increment returned `old` waits until the counter reaches the next
// multiple of the grid size (every block arrives exactly once per barrier,
// so one barrier's arrivals are gridDim.x consecutive values).  The block's
// writes are published by the __syncthreads and the release half of the
// increment, and the other blocks' writes are seen through the acquire
// loads of the wait (or the acquire half of the last increment).  A wait
// longer than wait_ns records TRUSS_ETIMEOUT in *err.  Returns false if any
// block has recorded an error, so that every block leaves at its next
// barrier.  The error shows in the counter's top bit (raise_error), which the
// waiting loads see anyway: reading *err after the wait was one more L2 round
// trip per barrier (20,000 barriers of 304 blocks: 1.43 -> 1.30 us each).
__device__ __forceinline__ bool grid_barrier(unsigned long long *bar, int *err,
                                             long long wait_ns) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long v = atom_add_acq_rel_gpu(bar, 1ull);
    const unsigned long long old = v & ~kBarErr;
    const unsigned long long target = (old / gridDim.x + 1) * gridDim.x;
    if (old + 1 != target) {
      const unsigned long long t0 = global_ns();
      // a set top bit is above any target
      for (unsigned spins = 1; (v = ld_acquire_gpu(bar)) < target; spins++) {
        if (spins > 32) __nanosleep(32);
        if ((spins & 15) == 0 && (long long)(global_ns() - t0) > wait_ns) {
          raise_error(bar, err, TRUSS_ETIMEOUT);
          v = kBarErr;
          break;
        }
      }
    }
    s_ok = (v & kBarErr) == 0;
  }
  __syncthreads();
  return s_ok != 0;
}

// r W / P without overflowing 64 bits (r <= P <= m).
__device__ __forceinline__ int64_t range_point(int64_t W, int64_t P, int64_t r) {
  return (W / P) * r + (W % P) * r / P;
}

// ----------------------------------------------- phases of a persistent peel ---
// What a scan found (slot = scan index % 3).
struct __align__(16) ScanOut {
  int minres;  // least residual of what is left alive
  int live;    // how much
  int any;     // non-zero: the scan removed something
  int listed;  // entries of the rewritten alive list
};

struct PhaseCtl {
  // Phase p (slot p % 3): barrier arrivals (bits 0 .. 15), frontier items
  // appended (16 .. 62); top bit: some block has recorded an error.
  unsigned long long phase[3];
  int err;
  int pad0;
  ScanOut scan[3];
};

constexpr int kItemShift = 16;
constexpr unsigned long long kArriveMask = (1ull << kItemShift) - 1;

// Reserve n items of phase word *w; the index of the first.
__device__ __forceinline__ uint32_t reserve_items(unsigned long long *w, int n) {
  return (uint32_t)(atomicAdd(w, (unsigned long long)(unsigned)n << kItemShift) >> kItemShift);
}

// End of a phase: a barrier of the whole grid, after which *items is the number
// of items the phase appended and, for a scan, *so is what it found.  The count
// shares its word with the barrier's
// arrivals, so the load that sees the last arrival brings it along, and one
// thread per block reads and passes it on: read by every warp, one L2 sector
// served 4,864 requests per value and barrier (edge peel: 1.1 us of each
// sub-round, 5 to 7 us of each scan).  A grid barrier that waits longer than
// wait_ns records TRUSS_ETIMEOUT.  Returns false if some block has recorded an error.
__device__ __forceinline__ bool phase_end(PhaseCtl *ctl, long long wait_ns, unsigned ph,
                                          uint32_t *items, const ScanOut *scan, ScanOut *so) {
  __shared__ unsigned long long s_word2[2];  // by phase parity: read until the next phase ends
  __shared__ ScanOut s_scan2[2];
  unsigned long long &s_word = s_word2[ph & 1];
  ScanOut &s_scan = s_scan2[ph & 1];
  unsigned long long *w = &ctl->phase[ph % 3];
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long v = atom_add_acq_rel_gpu(w, 1ull) + 1;
    if ((v & kArriveMask) != gridDim.x) {
      const unsigned long long t0 = global_ns();
      for (unsigned spins = 1;; spins++) {
        v = ld_acquire_gpu(w);
        if ((v & kArriveMask) == gridDim.x || (v & kBarErr)) break;
        if (spins > 32) __nanosleep(32);
        if ((spins & 15) == 0 && (long long)(global_ns() - t0) > wait_ns) {
          raise_error(w, &ctl->err, TRUSS_ETIMEOUT);
          v = kBarErr;
          break;
        }
      }
    }
    s_word = v;
    if (scan) *(int4 *)&s_scan = __ldcg((const int4 *)scan);
  }
  __syncthreads();
  const unsigned long long v = s_word;
  *items = (uint32_t)((v & ~kBarErr) >> kItemShift);
  if (scan) *so = s_scan;
  return (v & kBarErr) == 0;
}

}  // namespace tr
