// Graph upload: canonical-CSR validation on the GPU and, for directed graphs,
// the in-arc CSR (a stable sort of arcs by head keeps each row ascending).
#include <algorithm>

#include "job.cuh"

namespace cen {

// Canonical-CSR validation in three passes (each *bad |= 1 on a violation):
// offsets that rise from 0 to nnz, with the first arc of every non-empty row
// marked; every head in [0, n) and above the arc before it unless it starts
// its row (so rows are strictly ascending: no repeats); and no row that holds
// its own node (a binary search, exact once the rows are ascending).
__global__ void k_mark_starts(const int64_t *__restrict__ off, int32_t n, int64_t nnz, uint8_t *start, int *bad) {
  if (blockIdx.x == 0 && threadIdx.x == 0)
    if (off[0] != 0 || off[n] != nnz) atomicOr(bad, 1);
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = off[v], e = off[v + 1];
    if (b > e || b < 0 || e > nnz)
      atomicOr(bad, 1);
    else if (b < e)
      start[b] = 1;
  }
}

__global__ void k_check_arcs(const int32_t *__restrict__ col, int32_t n, int64_t nnz,
                             const uint8_t *__restrict__ start, int *bad) {
  bool ok = true;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = col[i];
    ok &= c >= 0 && c < n;
    if (i > 0 && !start[i]) ok &= col[i - 1] < c;
  }
  if (!__all_sync(0xffffffffu, ok) && (threadIdx.x & 31) == 0) atomicOr(bad, 1);
}

__global__ void k_check_loops(const int64_t *__restrict__ off, const int32_t *__restrict__ col, int32_t n,
                              int64_t nnz, int *bad) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = off[v], hi = off[v + 1];
    if (lo < 0 || hi > nnz || lo >= hi) continue;  // bad offsets are flagged by k_mark_starts
    while (lo < hi) {
      const int64_t mid = lo + ((hi - lo) >> 1);
      const int32_t c = col[mid];
      if (c == (int32_t)v) {
        atomicOr(bad, 1);
        break;
      }
      if (c < (int32_t)v)
        lo = mid + 1;
      else
        hi = mid;
    }
  }
}

// Calls f(e, u) for every arc e with its row u.  A warp takes kArcRun
// consecutive arcs, finds the rows of the first and the last, and each lane
// searches its arcs' rows between them, so that work follows arcs and not
// rows (a warp per row took 0.87 ms for 15.6 million R-MAT arcs, waiting on
// the hubs' rows; this takes 0.10).
constexpr int kArcRun = 256;
template <class F>
__device__ __forceinline__ void for_arcs(const int64_t *__restrict__ off, int32_t n, int64_t nnz, F &&f) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kArcRun; b < nnz; b += nwarps * kArcRun) {
    const int64_t end = b + kArcRun < nnz ? b + kArcRun : nnz;
    int32_t lo = (int32_t)warp_upper(off, (int64_t)n + 1, b);  // the row of arc b: the last that starts at or before it
    const int32_t last = (int32_t)warp_upper(off, (int64_t)n + 1, end - 1);
    for (int64_t e = b + lane; e < end; e += 32) {
      int32_t hi = last;  // off[lo] <= e
      while (lo < hi) {
        const int32_t mid = lo + ((hi - lo + 1) >> 1);
        if (off[mid] <= e)
          lo = mid;
        else
          hi = mid - 1;
      }
      f(e, lo);
    }
  }
}

// Arc list in CSR order: key = head, value = tail.
__global__ void __launch_bounds__(256) k_arcs_by_tail(const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                                      int32_t n, int64_t nnz, uint32_t *key, uint32_t *val) {
  for_arcs(off, n, nnz, [&](int64_t e, int32_t u) {
    key[e] = (uint32_t)col[e];
    val[e] = (uint32_t)u;
  });
}

// Sets roff[w] = at for the rows w in (lo, hi]: a lane's own when they are
// few, else with its whole warp.  Called by whole warps.
__device__ __forceinline__ void fill_rows(int64_t lo, int64_t hi, int64_t at, int64_t *roff) {
  const int lane = threadIdx.x & 31;
  const bool wide = hi - lo > 32;
  if (!wide)
    for (int64_t w = lo + 1; w <= hi; ++w) roff[w] = at;
  for (unsigned m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1) {
    const int src = __ffs(m) - 1;
    const int64_t a = __shfl_sync(0xffffffffu, lo, src), b = __shfl_sync(0xffffffffu, hi, src);
    const int64_t x = __shfl_sync(0xffffffffu, at, src);
    for (int64_t w = a + 1 + lane; w <= b; w += 32) roff[w] = x;
  }
}

// In-CSR offsets from the heads sorted ascending (nnz >= 1): roff[w] is the
// first position whose head is >= w.  Position i sets it for the heads w in
// (key[i-1], key[i]], with key[-1] = -1 and key[nnz] = n, so every w in
// [0, n] is set exactly once (roff[n] = nnz).
__global__ void __launch_bounds__(256) k_in_offsets(const uint32_t *__restrict__ key, int64_t nnz, int32_t n,
                                                    int64_t *roff) {
  const int64_t span = (nnz + 32) & ~(int64_t)31;  // positions 0 .. nnz, in whole warps
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < span; i += (int64_t)gridDim.x * 256) {
    int64_t lo = 0, hi = 0;
    if (i <= nnz) {
      lo = i == 0 ? -1 : (int64_t)key[i - 1];
      hi = i == nnz ? (int64_t)n : (int64_t)key[i];
    }
    fill_rows(lo, hi, i, roff);
  }
}

// Chunk table of the rows longer than kHeavyRow: row v contributes
// ceil(deg/kChunk) chunks starting at off[v], off[v]+kChunk, ...
__global__ void k_chunk_count(const int64_t *off, int32_t n, int32_t *cnt) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const int64_t d = off[v + 1] - off[v];
    cnt[v] = d > kHeavyRow ? (int32_t)((d + kChunk - 1) / kChunk) : 0;
  }
}
__global__ void k_chunk_fill(const int64_t *off, int32_t n, const int64_t *coff, int32_t *cw, int64_t *cbeg) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    for (int64_t c = coff[v]; c < coff[v + 1]; ++c) {
      cw[c] = v;
      cbeg[c] = off[v] + (c - coff[v]) * kChunk;
    }
  }
}

static void build_chunks(const int64_t *off, int32_t n, ChunkTable &T, cudaStream_t st, Stats *S) {
  DevBuf cnt, coff, tmp;
  cnt.ensure(4 * (size_t)n, st);
  coff.ensure(8 * ((size_t)n + 1), st);
  launch(S, K_GRAPH, st, [&] { k_chunk_count<<<grid_for(n, 256), 256, 0, st>>>(off, n, cnt.as<int32_t>()); });
  counts_to_offsets(cnt.as<int32_t>(), coff.as<int64_t>(), (size_t)n, tmp, st, S);
  int64_t total = 0;
  CEN_CK(cudaMemcpyAsync(&total, coff.as<int64_t>() + n, 8, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  T.count = total;
  T.w.ensure(4 * (size_t)(total + 1), st);
  T.beg.ensure(8 * (size_t)(total + 1), st);
  if (total)
    launch(S, K_GRAPH, st, [&] {
      k_chunk_fill<<<grid_for(n, 256), 256, 0, st>>>(off, n, coff.as<int64_t>(), T.w.as<int32_t>(),
                                                     T.beg.as<int64_t>());
    });
  CEN_CK(cudaStreamSynchronize(st));
}

// ------------------------------------------------------- canonical form
// Offsets non-decreasing from 0 to nnz and every id in [0, n): else *bad = 1.
__global__ void k_check_ids(const int64_t *__restrict__ off, const int32_t *__restrict__ col, int32_t n, int64_t nnz,
                            int *bad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= (int64_t)n; i += (int64_t)gridDim.x * blockDim.x)
    if ((i == 0 && off[0] != 0) || (i == n && off[n] != nnz) || (i > 0 && off[i] < off[i - 1])) *bad = 1;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
    if (col[e] < 0 || col[e] >= n) *bad = 1;
}

// Arc list of the input rows (u, v), and with `both` also (v, u).
__global__ void __launch_bounds__(256) k_arc_list(const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                                  int32_t n, int64_t nnz, bool both, uint32_t *tail, uint32_t *head) {
  for_arcs(off, n, nnz, [&](int64_t e, int32_t u) {
    const uint32_t v = (uint32_t)col[e];
    tail[e] = (uint32_t)u;
    head[e] = v;
    if (both) {
      tail[nnz + e] = v;
      head[nnz + e] = (uint32_t)u;
    }
  });
}

// The arcs of the list sorted by (tail, head) that stay (not a self-loop, not a
// repeat of the arc before) in two passes over tiles of kKeepTile: their number in
// each tile, then (after a scan of the numbers) their heads in place and the
// row offsets, which come from the same positions: row w starts at the number
// of arcs kept before the first arc of a tail >= w.  (Counting rows by atomics
// waited on the hubs' counters: 0.57 ms for 16.8 million arcs, and flags and
// positions of 8 bytes an arc went through memory; both passes take 0.10.)
constexpr int kKeepItems = 8, kKeepTile = 256 * kKeepItems;  // consecutive arcs a thread, and a block

// The thread's arcs (base .. base + kKeepItems - 1) and the one before them;
// bit i of the result: arc base + i stays.
__device__ __forceinline__ unsigned keep_load(const uint32_t *__restrict__ tail, const uint32_t *__restrict__ head,
                                              int64_t A, int64_t base, uint32_t *t, uint32_t *h) {
  t[0] = base > 0 && base <= A ? tail[base - 1] : 0xFFFFFFFFu;
  h[0] = base > 0 && base <= A ? head[base - 1] : 0xFFFFFFFFu;
  if (base + kKeepItems <= A && (((uintptr_t)tail | (uintptr_t)head) & 15) == 0) {
#pragma unroll
    for (int i = 0; i < kKeepItems; i += 4) {
      const uint4 a = *(const uint4 *)(tail + base + i), b = *(const uint4 *)(head + base + i);
      t[i + 1] = a.x, t[i + 2] = a.y, t[i + 3] = a.z, t[i + 4] = a.w;
      h[i + 1] = b.x, h[i + 2] = b.y, h[i + 3] = b.z, h[i + 4] = b.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kKeepItems; ++i) {
      t[i + 1] = base + i < A ? tail[base + i] : 0u;
      h[i + 1] = base + i < A ? head[base + i] : 0u;
    }
  }
  unsigned k = 0;
#pragma unroll
  for (int i = 0; i < kKeepItems; ++i)  // (no arc before the first: its ids are out of range)
    if (base + i < A && t[i + 1] != h[i + 1] && (t[i + 1] != t[i] || h[i + 1] != h[i])) k |= 1u << i;
  return k;
}

__global__ void __launch_bounds__(256) k_keep_count(const uint32_t *__restrict__ tail,
                                                    const uint32_t *__restrict__ head, int64_t A, int64_t *cnt) {
  __shared__ uint32_t wc[8];
  uint32_t t[kKeepItems + 1], h[kKeepItems + 1];
  const int64_t base = (int64_t)blockIdx.x * kKeepTile + threadIdx.x * kKeepItems;
  const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(keep_load(tail, head, A, base, t, h)));
  if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t s = 0;
    for (int w = 0; w < 8; ++w) s += wc[w];
    cnt[blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(256) k_keep_pack(const uint32_t *__restrict__ tail,
                                                   const uint32_t *__restrict__ head, int64_t A,
                                                   const int64_t *__restrict__ tile_pos, int32_t n, int32_t *col,
                                                   int64_t *off) {
  __shared__ uint32_t wc[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t t[kKeepItems + 1], h[kKeepItems + 1];
  const int64_t base = (int64_t)blockIdx.x * kKeepTile + threadIdx.x * kKeepItems;
  const unsigned k = keep_load(tail, head, A, base, t, h);
  uint32_t inc = (uint32_t)__popc(k);
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wc[wid] = inc;
  __syncthreads();
  int64_t at = tile_pos[blockIdx.x] + (inc - (uint32_t)__popc(k));
  for (int w = 0; w < wid; ++w) at += wc[w];
#pragma unroll
  for (int i = 0; i < kKeepItems; ++i) {
    // rows that start here: those in (the tail before, this tail], and at position A all that are left
    int64_t lo = 0, hi = 0;
    if (base + i <= A) {
      lo = base + i == 0 ? -1 : (int64_t)t[i];
      hi = base + i == A ? (int64_t)n : (int64_t)t[i + 1];
    }
    if (__any_sync(0xffffffffu, hi > lo)) fill_rows(lo, hi, at, off);
    if ((k >> i) & 1u) col[at++] = (int32_t)h[i + 1];
  }
}

// Canonical CSR of the input rows on the device: rows sorted, repeated arcs and
// self-loops dropped, and with `symmetrize` the reverse of every arc added
// first.  Sets g->off, g->col and g->nnz.  Ids out of [0, n) or malformed
// offsets give CEN_EINVAL.
void graph_canonicalize(cen_graph *g, const int64_t *off, const int32_t *col, int64_t nnz, bool on_device,
                        bool symmetrize, Stats *S) {
  cudaStream_t st = g->st;
  const int32_t n = g->n;
  DevBuf ioff, icol, bad;
  ioff.ensure(8 * ((size_t)n + 1), st);
  icol.ensure(4 * (size_t)(nnz > 0 ? nnz : 1), st);
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  CEN_CK(cudaMemcpyAsync(ioff.p, off, 8 * ((size_t)n + 1), kind, st));
  if (nnz) CEN_CK(cudaMemcpyAsync(icol.p, col, 4 * (size_t)nnz, kind, st));
  bad.ensure(4, st);
  CEN_CK(cudaMemsetAsync(bad.p, 0, 4, st));
  launch(S, K_GRAPH, st, [&] {
    k_check_ids<<<grid_for((size_t)std::max<int64_t>(nnz, n + 1), 256), 256, 0, st>>>(
        ioff.as<int64_t>(), icol.as<int32_t>(), n, nnz, bad.as<int>());
  });
  int hbad = 0;
  CEN_CK(cudaMemcpyAsync(&hbad, bad.p, 4, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  CEN_REQUIRE(hbad == 0, CEN_EINVAL, "cen_graph_load: offsets must rise from 0 to nnz and ids lie in [0, n)");
  const int64_t A = symmetrize ? 2 * nnz : nnz;
  CEN_REQUIRE(A < ((int64_t)1 << 32), CEN_EINVAL, "cen_graph_load: too many arcs to canonicalize");
  g->off.ensure(8 * ((size_t)n + 1), st);
  g->col.ensure(4 * (size_t)(A > 0 ? A : 1), st);
  if (A == 0) {
    CEN_CK(cudaMemsetAsync(g->off.p, 0, 8 * ((size_t)n + 1), st));
    g->nnz = 0;
    return;
  }
  DevBuf tail, head, k2, v2, hist, tmp, pos;
  tail.ensure(4 * (size_t)A, st);
  head.ensure(4 * (size_t)A, st);
  launch(S, K_GRAPH, st, [&] {
    k_arc_list<<<grid_for((size_t)nnz, 8 * kArcRun, sm_count() * 64), 256, 0, st>>>(
        ioff.as<int64_t>(), icol.as<int32_t>(), n, nnz, symmetrize, tail.as<uint32_t>(), head.as<uint32_t>());
  });
  int bits = 1;
  while (bits < 31 && (1u << bits) < (uint32_t)n) ++bits;
  // by head, then (stably) by tail: the arcs end up sorted by (tail, head)
  radix_sort_pairs(head.as<uint32_t>(), tail.as<uint32_t>(), (size_t)A, bits, k2, v2, hist, tmp, st, S);
  radix_sort_pairs(tail.as<uint32_t>(), head.as<uint32_t>(), (size_t)A, bits, k2, v2, hist, tmp, st, S);
  // tiles cover positions 0 .. A: position A closes the last rows
  const int64_t tiles = A / kKeepTile + 1;
  pos.ensure(8 * (size_t)(tiles + 1), st);
  launch(S, K_GRAPH, st, [&] {
    k_keep_count<<<(unsigned)tiles, 256, 0, st>>>(tail.as<uint32_t>(), head.as<uint32_t>(), A, pos.as<int64_t>());
  });
  exclusive_scan_i64(pos.as<int64_t>(), pos.as<int64_t>(), (size_t)tiles, pos.as<int64_t>() + tiles, tmp, st, S);
  launch(S, K_GRAPH, st, [&] {
    k_keep_pack<<<(unsigned)tiles, 256, 0, st>>>(tail.as<uint32_t>(), head.as<uint32_t>(), A, pos.as<int64_t>(), n,
                                                 g->col.as<int32_t>(), g->off.as<int64_t>());
  });
  int64_t kept = 0;
  CEN_CK(cudaMemcpyAsync(&kept, pos.as<int64_t>() + tiles, 8, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  g->nnz = kept;
}

// Sums of d and d^2 over the rows of off (one pass, double sums, two atomics a block).
__global__ void __launch_bounds__(256) k_degree_moments(const int64_t *__restrict__ off, int32_t n, double *sums) {
  __shared__ double sa[8], sb[8];
  double a = 0.0, b = 0.0;
  for (int64_t v = (int64_t)blockIdx.x * 256 + threadIdx.x; v < n; v += (int64_t)gridDim.x * 256) {
    const double d = (double)(off[v + 1] - off[v]);
    a += d;
    b += d * d;
  }
  a = warp_sum(a);
  b = warp_sum(b);
  if ((threadIdx.x & 31) == 0) {
    sa[threadIdx.x >> 5] = a;
    sb[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      a += sa[w];
      b += sb[w];
    }
    atomicAdd(&sums[0], a);
    atomicAdd(&sums[1], b);
  }
}

// The chunk tables of the bit-parallel sampler's long rows, built on their
// first use (on `st`, synchronized; released later on the graph's stream).
static void graph_chunks_ready(const cen_graph *g, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g->chunks_mu);
  if (g->chunks_built) return;
  build_chunks(g->off.as<int64_t>(), g->n, g->out_chunks, st, nullptr);
  if (g->directed) build_chunks(g->roff.as<int64_t>(), g->n, g->in_chunks_own, st, nullptr);
  for (DevBuf *b : {&g->out_chunks.w, &g->out_chunks.beg, &g->in_chunks_own.w, &g->in_chunks_own.beg}) b->st = g->st;
  g->chunks_built = true;
}

const ChunkTable &graph_out_chunks(const cen_graph *g, cudaStream_t st) {
  graph_chunks_ready(g, st);
  return g->out_chunks;
}

const ChunkTable &graph_in_chunks(const cen_graph *g, cudaStream_t st) {
  graph_chunks_ready(g, st);
  return g->directed ? g->in_chunks_own : g->out_chunks;
}

double graph_branching(const cen_graph *g, cudaStream_t st) {
  std::lock_guard<std::mutex> lk(g->branching_mu);
  if (g->branching >= 0.0) return g->branching;
  DevBuf sums;
  sums.ensure(4 * sizeof(double), st);
  CEN_CK(cudaMemsetAsync(sums.p, 0, 4 * sizeof(double), st));
  const int blocks = grid_for((size_t)g->n, 256, sm_count() * 4);
  k_degree_moments<<<blocks, 256, 0, st>>>(g->off.as<int64_t>(), g->n, sums.as<double>());
  if (g->directed) k_degree_moments<<<blocks, 256, 0, st>>>(g->in_off(), g->n, sums.as<double>() + 2);
  CEN_CK(cudaGetLastError());
  double h[4] = {0, 0, 0, 0};
  CEN_CK(cudaMemcpyAsync(h, sums.p, sizeof(h), cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  const double out = h[0] > 0 ? h[1] / h[0] : 0.0, in = h[2] > 0 ? h[3] / h[2] : 0.0;
  g->branching = out > in ? out : in;
  return g->branching;
}

void graph_build(cen_graph *g, const int64_t *off, const int32_t *col, bool on_device, Stats *S) {
  cudaStream_t st = g->st;
  const int32_t n = g->n;
  const int64_t nnz = g->nnz;
  if (off) {  // null: g->off / g->col already hold the graph (see graph_canonicalize)
    g->off.ensure(sizeof(int64_t) * ((size_t)n + 1), st);
    g->col.ensure(sizeof(int32_t) * (size_t)(nnz > 0 ? nnz : 1), st);
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    CEN_CK(cudaMemcpyAsync(g->off.p, off, sizeof(int64_t) * ((size_t)n + 1), kind, st));
    if (nnz) CEN_CK(cudaMemcpyAsync(g->col.p, col, sizeof(int32_t) * (size_t)nnz, kind, st));
  }
  // the validation flag and the degree moments (sums of d and d^2 over the
  // out-rows, then the in-rows) come back in one copy
  struct Check {
    double sums[4];
    int bad;
  };
  DevBuf chk;
  chk.ensure(sizeof(Check), st);
  CEN_CK(cudaMemsetAsync(chk.p, 0, sizeof(Check), st));
  Check *dchk = chk.as<Check>();
  DevBuf start;
  start.ensure((size_t)(nnz > 0 ? nnz : 1), st);
  CEN_CK(cudaMemsetAsync(start.p, 0, (size_t)(nnz > 0 ? nnz : 1), st));
  launch(S, K_GRAPH, st, [&] {
    k_mark_starts<<<grid_for((size_t)n, 256), 256, 0, st>>>(g->off.as<int64_t>(), n, nnz, start.as<uint8_t>(),
                                                           &dchk->bad);
  });
  if (nnz)
    launch(S, K_GRAPH, st, [&] {
      k_check_arcs<<<grid_for((size_t)nnz, 256), 256, 0, st>>>(g->col.as<int32_t>(), n, nnz, start.as<uint8_t>(),
                                                                &dchk->bad);
    });
  launch(S, K_GRAPH, st, [&] {
    k_check_loops<<<grid_for((size_t)n, 256), 256, 0, st>>>(g->off.as<int64_t>(), g->col.as<int32_t>(), n, nnz,
                                                           &dchk->bad);
  });
  const int mblocks = grid_for((size_t)n, 256, sm_count() * 4);
  launch(S, K_GRAPH, st,
         [&] { k_degree_moments<<<mblocks, 256, 0, st>>>(g->off.as<int64_t>(), n, dchk->sums); });
  Check h{};
  CEN_CK(cudaMemcpyAsync(&h, chk.p, sizeof(Check), cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  CEN_REQUIRE(h.bad == 0, CEN_EINVAL,
              "cen_graph_load: CSR is not canonical (offsets, ids in [0,n), no self-loops, rows strictly ascending)");
  const double bout = h.sums[0] > 0 ? h.sums[1] / h.sums[0] : 0.0;
  if (!g->directed || nnz == 0) {
    if (g->directed) {  // no arcs: in-CSR is all zeros
      g->roff.ensure(sizeof(int64_t) * ((size_t)n + 1), st);
      CEN_CK(cudaMemsetAsync(g->roff.p, 0, sizeof(int64_t) * ((size_t)n + 1), st));
      g->rcol.ensure(4, st);
      CEN_CK(cudaStreamSynchronize(st));
    }
    g->branching = bout;
    return;
  }
  // arcs (head, tail) in CSR order, stably sorted by head: the tails of each
  // head stay ascending, so rcol rows are ascending; the tails are sorted in
  // place in rcol
  DevBuf key, k2, v2, hist, tmp;
  key.ensure(4 * (size_t)nnz, st);
  g->rcol.ensure(4 * (size_t)nnz, st);
  launch(S, K_GRAPH, st, [&] {
    k_arcs_by_tail<<<grid_for((size_t)nnz, 8 * kArcRun, sm_count() * 64), 256, 0, st>>>(
        g->off.as<int64_t>(), g->col.as<int32_t>(), n, nnz, key.as<uint32_t>(), g->rcol.as<uint32_t>());
  });
  int bits = 1;
  while (bits < 31 && (1u << bits) < (uint32_t)n) ++bits;
  radix_sort_pairs(key.as<uint32_t>(), g->rcol.as<uint32_t>(), (size_t)nnz, bits, k2, v2, hist, tmp, st, S);
  g->roff.ensure(sizeof(int64_t) * ((size_t)n + 1), st);
  launch(S, K_GRAPH, st, [&] {
    k_in_offsets<<<grid_for((size_t)nnz + 1, 256), 256, 0, st>>>(key.as<uint32_t>(), nnz, n, g->roff.as<int64_t>());
  });
  launch(S, K_GRAPH, st,
         [&] { k_degree_moments<<<mblocks, 256, 0, st>>>(g->roff.as<int64_t>(), n, dchk->sums + 2); });
  CEN_CK(cudaMemcpyAsync(&h, chk.p, sizeof(Check), cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  const double bin = h.sums[2] > 0 ? h.sums[3] / h.sums[2] : 0.0;
  g->branching = bout > bin ? bout : bin;
}

}  // namespace cen
