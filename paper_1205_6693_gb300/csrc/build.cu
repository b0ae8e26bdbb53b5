// CSR build: from an edge list of rows to the degree-ordered oriented CSR.
//
// The paper assumes adjacency lists already exist (Section 2) and bounds the
// work of Algorithm 2 through the degree order of Theorem 1: orienting every
// edge from its lower-degree to its higher-degree endpoint bounds each vertex's
// out-list by 2*sqrt(m).  Steps:
//   1. canonical key (min, max) per row; self-loops and invalid rows get a
//      sentinel key; radix sort (key, row);
//   2. run heads -> distinct edges in lexicographic order, row -> lex id;
//   3. degrees; rank = position in ascending (degree, id) (stable radix sort
//      by degree over ids in order), vertices relabelled by rank; the vertices
//      of a batch in ascending (graph, degree, id), so that each graph's
//      edges, words and lists stay together (a batch of 4,096 small graphs,
//      mixed by degree / graph by graph: support stage 4.38 / 4.10 ms, lists
//      2.68 / 2.22, orientation 0.58 / 0.28);
//   4. oriented keys (rank tail, rank head), radix sort -> canonical edge id =
//      position; out-degree count + exclusive scan -> offsets;
//   5. row -> canonical edge id.
// The sorts are bound by the bytes that each 8-bit pass moves, so a key's low
// part is local to its graph (the batch's keys 46 -> 37 bits, six passes to
// five).  (Key and row number packed into one 64-bit word, 16 bytes moved per
// element and pass instead of 24, were slower all the same: 96 against 84 us a
// pass over 10 M rows.)
#include "engine.h"

namespace tr {

namespace {

constexpr int kBlock = 256;

// Graph of row r in a batch (row_off has G+1 entries).
__device__ __forceinline__ int graph_of_row(const int64_t *row_off, int G, int64_t r) {
  int lo = 0, hi = G - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (row_off[mid] <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Keys (u, v), u < v, with v in the low lb bits; local: v less its graph's first
// vertex.
__global__ void k_make_keys(RowsIn in, int lb, bool local, uint64_t sentinel, uint64_t *keys,
                            int32_t *vals, int32_t *err) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < in.rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    int64_t u = in.src[r], v = in.dst[r];
    int64_t lo = 0, hi = in.n;
    if (in.graphs > 1 || in.voff != nullptr) {
      int g = graph_of_row(in.row_off, in.graphs, r);
      lo = in.voff[g];
      hi = in.voff[g + 1];
      u += lo;
      v += lo;
    }
    uint64_t key = sentinel;
    if (u < lo || u >= hi || v < lo || v >= hi) {
      atomicExch(err, TRUSS_EINVAL);
    } else if (u != v) {
      const uint64_t a = (uint64_t)(u < v ? u : v), c = (uint64_t)(u < v ? v : u);
      key = (a << lb) | (local ? c - (uint64_t)lo : c);
    }
    keys[r] = key;
    vals[r] = (int32_t)r;
  }
}

__global__ void k_run_heads(int64_t rows, const uint64_t *sk, uint64_t sentinel, int32_t *flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = sk[i];
    flag[i] = (k != sentinel && (i == 0 || sk[i - 1] != k)) ? 1 : 0;
  }
}

// Distinct edges in lexicographic order (U, V) from the sorted row keys;
// runid[i] becomes the 1-based edge id of sorted row i, 0 for a self-loop.
// vbase[x] (null: 0) is the first vertex of x's graph.
__global__ void k_lex_edges(int64_t rows, int lb, const uint64_t *sk, int32_t *runid,
                            uint64_t sentinel, const int32_t *vbase, int32_t *U, int32_t *V) {
  const uint64_t mask = (1ull << lb) - 1;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = sk[i];
    if (k == sentinel) {
      runid[i] = 0;
      continue;
    }
    const int32_t id = runid[i] - 1;
    if (i == 0 || sk[i - 1] != k) {
      const int32_t u = (int32_t)(k >> lb);
      U[id] = u;
      V[id] = (int32_t)(k & mask) + (vbase ? vbase[u] : 0);
    }
  }
}

// First vertex of each vertex's graph.
__global__ void k_vertex_base(int64_t n, int G, const int64_t *voff, int32_t *vbase) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    vbase[v] = (int32_t)voff[graph_of_row(voff, G, v)];
}

// Sort key of each vertex: its degree, behind its graph's number in a batch
// (recovered from the order of the first vertices: vertices are numbered graph
// by graph, so the stable sort only needs graphs to differ).
// The keys take the place of the degrees.
__global__ void k_degree_keys(int64_t n, int db, int G, const int64_t *voff, uint32_t *deg,
                              int32_t *id) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    if (db < 32) deg[v] |= (uint32_t)graph_of_row(voff, G, v) << db;
    id[v] = (int32_t)v;
  }
}

// U is sorted (edges in lexicographic order), so each run of equal tails
// adds its length once: minus its first index at its first edge, its end at
// its last (int32 wrap-around cancels).  Heads V are added once per group of
// lanes of a warp that hold the same vertex.
__global__ void k_degree(int64_t m, const int32_t *U, const int32_t *V, int32_t *deg) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x; b < m; b += stride) {
    const int64_t e = b + threadIdx.x;
    const bool ok = e < m;
    if (ok) {
      const int u = U[e];
      if (e == 0 || U[e - 1] != u) atomicAdd(&deg[u], -(int)e);
      if (e + 1 == m || U[e + 1] != u) atomicAdd(&deg[u], (int)(e + 1));
    }
    const int v = ok ? V[e] : -1;
    const unsigned peers = __match_any_sync(TR_FULL, v);
    if (ok && lane_id() == __ffs(peers) - 1) atomicAdd(&deg[v], __popc(peers));
  }
}

__global__ void k_iota(int64_t n, int32_t *x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = (int32_t)i;
}

// Ranks of the sorted vertices, and their degrees (the low db bits of the
// sorted keys) in the place of the keys.
__global__ void k_newid(int64_t n, int db, const int32_t *order, int32_t *newid, uint32_t *skey) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    newid[order[i]] = (int32_t)i;
    if (db < 32) skey[i] &= (1u << db) - 1u;
  }
}

__global__ void k_orient_keys(int64_t m, int lb, const int32_t *U, const int32_t *V,
                              const int32_t *newid, const int32_t *vbase, uint64_t *keys,
                              int32_t *vals) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = newid[U[e]], y = newid[V[e]];
    const int32_t lo = x < y ? x : y, hi = x < y ? y : x;
    // ranks keep the vertices of a graph together: its first rank is its first vertex
    keys[e] = ((uint64_t)lo << lb) | (uint64_t)(hi - (vbase ? vbase[lo] : 0));
    vals[e] = (int32_t)e;
  }
}

// The oriented edges are sorted by tail, so each run of equal tails adds
// its length to outdeg once: minus its first index at its first edge, its
// end at its last.
__global__ void k_oriented(int64_t m, int lb, const uint64_t *ok, const int32_t *olex,
                           const int32_t *vbase, int32_t *adjp, int32_t *esrc, int32_t *lex2e,
                           int64_t *outdeg) {
  const uint64_t mask = (1ull << lb) - 1;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < m;
       p += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = ok[p];
    const int32_t x = (int32_t)(k >> lb);
    adjp[p] = (int32_t)(k & mask) + (vbase ? vbase[x] : 0);
    esrc[p] = x;
    lex2e[olex[p]] = (int32_t)p;
    if (p == 0 || (int32_t)(ok[p - 1] >> lb) != x)
      atomicAdd((unsigned long long *)&outdeg[x], (unsigned long long)(-p));
    if (p + 1 == m || (int32_t)(ok[p + 1] >> lb) != x)
      atomicAdd((unsigned long long *)&outdeg[x], (unsigned long long)(p + 1));
  }
}

// Row srow[i] (sorted row i) -> its canonical edge: the lexicographic id is
// runid[i] - 1 (0: a self-loop), read in order, so lex2e is read in order
// and only the write to row2e lands at random.
__global__ void k_row2e(int64_t rows, const int32_t *srow, const int32_t *runid,
                        const int32_t *lex2e, int32_t *row2e) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t l = runid[i];
    row2e[srow[i]] = l > 0 ? lex2e[l - 1] : -1;
  }
}

}  // namespace

int build_csr(Arena &A, const RowsIn &in, Csr *out, int32_t *d_err, cudaStream_t s) {
  const int64_t rows = in.rows, n = in.n;
  const int maxg = 152 * 16;
  out->n = n;
  out->rows = rows;
  const int b = bits_for(n > 1 ? (uint64_t)(n - 1) : 1);
  // a batch whose graph numbers and degrees fit 32 bits together is ranked
  // graph by graph, with heads local to their graph, unless its vertices
  // outnumber its rows: each is looked up in its graph twice (1,000 graphs of
  // 5,000 vertices and 100 rows: 0.83 ms so, 0.75 mixed; of 4,000 vertices and
  // 3,000 rows 1.68 / 1.66)
  const int gb = bits_for((uint64_t)(in.graphs > 1 ? in.graphs - 1 : 0));
  const int nb = bits_for(in.max_n > 1 ? (uint64_t)(in.max_n - 1) : 1);
  const bool local = in.graphs > 1 && in.max_n > 0 && n <= rows && gb + nb < 32;
  const int lb = local ? nb : b, kbits = b + lb;
  const uint64_t sentinel = kbits >= 64 ? ~0ull : ((1ull << kbits) - 1);

  int32_t *row2e = A.get<int32_t>(rows);
  int64_t *offp = A.get<int64_t>(n + 1);
  if (!row2e || !offp) return TRUSS_ENOMEM;
  out->row2e = row2e;
  out->offp = offp;

  if (rows == 0) {
    // no edges: empty out-lists, and every vertex keeps its id as its rank
    int32_t *order = A.get<int32_t>(n);
    if (!order) return TRUSS_ENOMEM;
    TR_CUDA(cudaMemsetAsync(offp, 0, sizeof(int64_t) * (n + 1), s));
    if (n > 0) {
      k_iota<<<grid_for(n, kBlock, maxg), kBlock, 0, s>>>(n, order);
      TR_LAUNCHED();
    }
    out->m = 0;
    out->order = order;
    out->sdeg = A.get<int32_t>(n);
    if (!out->sdeg) return TRUSS_ENOMEM;
    TR_CUDA(cudaMemsetAsync(out->sdeg, 0, sizeof(int32_t) * (n > 0 ? n : 1), s));
    out->adjp = A.get<int32_t>(1);
    out->esrc = A.get<int32_t>(1);
    return TRUSS_OK;
  }

  // 1. keys + sort
  uint64_t *keys = A.get<uint64_t>(rows), *skeys = A.get<uint64_t>(rows);
  int32_t *vals = A.get<int32_t>(rows), *srow = A.get<int32_t>(rows);
  int32_t *flag = A.get<int32_t>(rows), *runid = A.get<int32_t>(rows);
  int32_t *vbase = local ? A.get<int32_t>(n) : nullptr;
  if (!keys || !skeys || !vals || !srow || !flag || !runid || (local && !vbase))
    return TRUSS_ENOMEM;
  if (local) {
    k_vertex_base<<<grid_for(n, kBlock, maxg), kBlock, 0, s>>>(n, in.graphs, in.voff, vbase);
    TR_LAUNCHED();
  }
  k_make_keys<<<grid_for(rows, kBlock, maxg), kBlock, 0, s>>>(in, lb, local, sentinel, keys, vals,
                                                              d_err);
  TR_LAUNCHED();
  size_t tb = 0;
  TR_TRY(sort_pairs_u64(nullptr, &tb, keys, skeys, vals, srow, rows, 0, kbits, s));
  void *tmp = A.alloc(tb);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(sort_pairs_u64(tmp, &tb, keys, skeys, vals, srow, rows, 0, kbits, s));

  // 2. distinct edges
  k_run_heads<<<grid_for(rows, kBlock, maxg), kBlock, 0, s>>>(rows, skeys, sentinel, flag);
  TR_LAUNCHED();
  tb = 0;
  TR_TRY(inclusive_sum_i32(nullptr, &tb, flag, runid, rows, s));
  tmp = A.alloc(tb);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(inclusive_sum_i32(tmp, &tb, flag, runid, rows, s));
  int32_t h_m = 0, h_err = 0;
  TR_CUDA(cudaMemcpyAsync(&h_m, runid + rows - 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaMemcpyAsync(&h_err, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  TR_CUDA(cudaStreamSynchronize(s));
  if (h_err != 0) return TRUSS_EINVAL;
  const int64_t m = h_m;
  out->m = m;
  int32_t *U = A.get<int32_t>(m), *V = A.get<int32_t>(m);
  if (!U || !V) return TRUSS_ENOMEM;
  k_lex_edges<<<grid_for(rows, kBlock, maxg), kBlock, 0, s>>>(rows, lb, skeys, runid, sentinel,
                                                               vbase, U, V);
  TR_LAUNCHED();

  // 3. degrees and rank
  int32_t *deg = A.get<int32_t>(n), *sdeg = A.get<int32_t>(n);
  int32_t *ids = A.get<int32_t>(n), *order = A.get<int32_t>(n), *newid = A.get<int32_t>(n);
  if (!deg || !sdeg || !ids || !order || !newid) return TRUSS_ENOMEM;
  TR_CUDA(cudaMemsetAsync(deg, 0, sizeof(int32_t) * n, s));
  if (m > 0) {
    k_degree<<<grid_for(m, kBlock, maxg), kBlock, 0, s>>>(m, U, V, deg);
    TR_LAUNCHED();
  }
  // degrees are below the vertices of a graph, and at most the edges
  const int db = local ? nb : 32;
  const int mb = bits_for((uint64_t)(m > 0 ? m : 1));
  const int dbits = local ? nb + gb : (b < mb ? b : mb);
  uint32_t *dkey = (uint32_t *)deg, *skey = (uint32_t *)sdeg;
  k_degree_keys<<<grid_for(n, kBlock, maxg), kBlock, 0, s>>>(n, db, in.graphs, in.voff, dkey, ids);
  TR_LAUNCHED();
  tb = 0;
  TR_TRY(sort_pairs_u32(nullptr, &tb, dkey, skey, ids, order, n, 0, dbits, s));
  tmp = A.alloc(tb);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(sort_pairs_u32(tmp, &tb, dkey, skey, ids, order, n, 0, dbits, s));
  out->order = order;
  out->sdeg = sdeg;
  k_newid<<<grid_for(n, kBlock, maxg), kBlock, 0, s>>>(n, db, order, newid, skey);
  TR_LAUNCHED();

  // 4. orientation
  int32_t *adjp = A.get<int32_t>(m), *esrc = A.get<int32_t>(m), *lex2e = A.get<int32_t>(m);
  int64_t *outdeg = A.get<int64_t>(n + 1);
  if (!adjp || !esrc || !lex2e || !outdeg) return TRUSS_ENOMEM;
  out->adjp = adjp;
  out->esrc = esrc;
  TR_CUDA(cudaMemsetAsync(outdeg, 0, sizeof(int64_t) * (n + 1), s));
  if (m > 0) {
    // reuse the row-sized key/value buffers (m <= rows); srow and runid
    // stay for the row -> edge map, flag (dead) takes the sorted values
    int32_t *olex = flag;
    k_orient_keys<<<grid_for(m, kBlock, maxg), kBlock, 0, s>>>(m, lb, U, V, newid, vbase, keys,
                                                               vals);
    TR_LAUNCHED();
    tb = 0;
    TR_TRY(sort_pairs_u64(nullptr, &tb, keys, skeys, vals, olex, m, 0, kbits, s));
    tmp = A.alloc(tb);
    if (!tmp) return TRUSS_ENOMEM;
    TR_TRY(sort_pairs_u64(tmp, &tb, keys, skeys, vals, olex, m, 0, kbits, s));
    k_oriented<<<grid_for(m, kBlock, maxg), kBlock, 0, s>>>(m, lb, skeys, olex, vbase, adjp, esrc,
                                                             lex2e, outdeg);
    TR_LAUNCHED();
  }
  tb = 0;
  TR_TRY(exclusive_sum_i64(nullptr, &tb, outdeg, offp, n + 1, s));
  tmp = A.alloc(tb);
  if (!tmp) return TRUSS_ENOMEM;
  TR_TRY(exclusive_sum_i64(tmp, &tb, outdeg, offp, n + 1, s));

  // 5. rows -> canonical edge ids
  k_row2e<<<grid_for(rows, kBlock, maxg), kBlock, 0, s>>>(rows, srow, runid, lex2e, row2e);
  TR_LAUNCHED();
  return TRUSS_OK;
}

}  // namespace tr
