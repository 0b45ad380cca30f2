// Hyper-edge spaces other than set betweenness (Sec. 2): kappa-path and
// triangle centralities.  CentRA is oblivious to sampleHEs (Sec. 4.2), so only
// the sampler changes; greedyCover, AMCERA and the bounds run as they are.
//
// kappa-path: s uniform (purpose 0), a length l uniform in 1..kappa (purpose
// 1), then a random simple walk of up to l steps: step i moves to the r-th
// (ascending id) out-neighbour of the current node that is not yet on the
// walk, r uniform below their number (purpose 2 + i); the walk stops early
// when there is none.  The hyper-edge is the nodes after s in walk order.
//
// Triangle: on an undirected graph, triangles {u < v < w} are ranked in
// (u, v, w) order: tri_off[e] (an exclusive prefix over arcs e = (u, v) in CSR
// order of the number of common neighbours w > v of u and v, counted only when
// v > u) ranks the first triangle on arc e, and within the arc the common
// neighbours ascend.  A rank r uniform below the total (purpose 0) is unranked
// and the three nodes, ascending, are the hyper-edge.
#include "job.cuh"

namespace cen {

namespace {

constexpr int kWalkThreads = 128;  // block of the walk kernel
constexpr int kMaxKappa = 1024;

// First position in the sorted c[lo, hi) whose value is >= w.
__device__ __forceinline__ int64_t lower_bound32(const int32_t *__restrict__ c, int64_t lo, int64_t hi, int32_t w) {
  while (lo < hi) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (c[mid] < w)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// GS lanes per sample.  The walk (at most kappa nodes after s) sits in shared
// memory.  At a step the lanes look the walk's nodes up in the current node's
// sorted row: the row less those found are the free out-neighbours, and the
// r-th of them is the least position i with i = r + (found positions <= i),
// reached from i = r by repetition.  So a step costs a binary search per walk
// node, side by side, where counting and finding the free arcs one by one
// reads a hub's row of thousands twice (R-MAT 18, kappa = 8, 65,536 walks:
// 2.0 -> 0.10 ms).  Bound by the latency of a step's chain of loads; 8 lanes
// hold all nodes of a walk of kappa <= 8, so four walks share a warp.
template <int GS>
__global__ void __launch_bounds__(kWalkThreads) k_kpath(uint64_t j0, uint64_t count, int32_t n, int kappa,
                                                        const int64_t *__restrict__ off,
                                                        const int32_t *__restrict__ col, SampleKey key, int32_t *ps,
                                                        int32_t *pt, int32_t *pd, int32_t *out,
                                                        const int64_t *__restrict__ hoff, int *bmax,
                                                        unsigned long long *units) {
  extern __shared__ int32_t walk_sh[];
  constexpr int kGroups = kWalkThreads / GS;
  const int gl = threadIdx.x & (GS - 1), gib = threadIdx.x / GS, lane = threadIdx.x & 31;
  const unsigned gmask = GS == 32 ? 0xffffffffu : ((1u << GS) - 1u) << (lane & ~(GS - 1));
  int32_t *walk = walk_sh + (size_t)gib * 2 * kappa;  // then the found positions
  int32_t *found = walk + kappa;
  const uint64_t ng = (uint64_t)gridDim.x * kGroups;
  unsigned long long probes = 0;
  int mymax = 0;
  for (uint64_t i = (uint64_t)blockIdx.x * kGroups + gib; i < count; i += ng) {
    const uint64_t j = j0 + i;
    int32_t draw = 0;  // lane 0 draws s, lane 1 the length
    if (gl < 2)
      draw = (int32_t)uniform_below64(key.seed, key.id(j), gl ? kPurposeT : kPurposeS, (uint64_t)(gl ? kappa : n));
    const int32_t s = __shfl_sync(gmask, draw, 0, GS);
    const int32_t l = 1 + __shfl_sync(gmask, draw, 1, GS);
    int32_t cur = s, len = 0;
    for (int32_t step = 0; step < l; ++step) {
      const int64_t e0 = off[cur];
      const int32_t deg = (int32_t)(off[cur + 1] - e0);
      const int32_t *__restrict__ row = col + e0;
      int32_t nfound = 0;  // of s and the walk's nodes, in the row
      for (int q = gl; q - gl <= len; q += GS) {
        int32_t at = -1;
        if (q <= len) {
          const int32_t w = q ? walk[q - 1] : s;
          const int32_t p = (int32_t)lower_bound32(row, 0, deg, w);
          if (p < deg && row[p] == w) at = p;
        }
        const unsigned m = __ballot_sync(gmask, at >= 0);
        if (at >= 0) found[nfound + __popc(m & ((1u << lane) - 1u))] = at;
        nfound += __popc(m);
      }
      probes += (unsigned long long)(len + 1);
      if (nfound == deg) break;
      const int32_t r =
          (int32_t)uniform_below64(key.seed, key.id(j), kPurposeWalk0 + (uint32_t)step, (uint64_t)(deg - nfound));
      __syncwarp(gmask);
      int32_t at = r;
      for (;;) {
        int32_t below = 0;
        for (int q = gl; q - gl < nfound; q += GS)
          below += __popc(__ballot_sync(gmask, q < nfound && found[q] <= at));
        if (r + below == at) break;
        at = r + below;
      }
      cur = row[at];
      if (gl == 0) walk[len] = cur;
      __syncwarp(gmask);
      ++len;
    }
    if (out) {  // members at stride kappa, or at their place in the store when hoff is given
      int32_t *dst = hoff ? out + hoff[j] : out + (size_t)i * kappa;
      for (int q = gl; q < len; q += GS) dst[q] = walk[q];
    }
    if (gl == 0) {
      ps[j] = s;
      pt[j] = l;
      pd[j] = len;
    }
    mymax = max(mymax, len);
    __syncwarp(gmask);
  }
  mymax = __reduce_max_sync(0xffffffffu, mymax);
  probes = warp_sum(gl == 0 ? probes : 0ull);
  if (lane == 0) {
    if (mymax) atomicMax(bmax, mymax);
    if (probes) atomicAdd(units, probes * 4ull);
  }
}

// Common neighbours w > v of u and v, ascending: the shorter row's entries
// above v, 128 at a time, are looked up in the longer row by binary search
// (both rows are sorted, so either order of the two rows gives the same
// ascending w).  A lane's four searches go side by side, so that their loads
// overlap.  Returns how many there are; with want >= 0, stops at the one of
// that rank and returns it in *w_out.  Called by a whole warp.
__device__ __forceinline__ int32_t common_above(const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                                int32_t u, int32_t v, int64_t want, int32_t *w_out) {
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const int64_t u0 = off[u], v0 = off[v];
  int32_t na = (int32_t)(off[u + 1] - u0), nb = (int32_t)(off[v + 1] - v0);
  const int32_t *__restrict__ A = col + u0, *__restrict__ B = col + v0;
  if (na > nb) {
    const int32_t *t = A;
    A = B;
    B = t;
    const int32_t nt = na;
    na = nb;
    nb = nt;
  }
  int32_t c = 0;
  for (int32_t a = (int32_t)lower_bound32(A, 0, na, v + 1); a < na && nb > 0; a += 32 * U) {
    int32_t w[U], p[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      w[i] = a + 32 * i + lane < na ? A[a + 32 * i + lane] : 0x7fffffff;
      p[i] = 0;
    }
    int32_t len = nb;
    while (len > 1) {
      const int32_t half = len >> 1;
#pragma unroll
      for (int i = 0; i < U; ++i)
        if (B[p[i] + half - 1] < w[i]) p[i] += half;
      len -= half;
    }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int32_t x = B[p[i]];  // the first entry >= w, or the last
      unsigned m = __ballot_sync(0xffffffffu, x == w[i] && a + 32 * i + lane < na);
      const int found = __popc(m);
      if (want >= 0 && want < c + found) {
        for (int64_t q = c; q < want; ++q) m &= m - 1;
        *w_out = __shfl_sync(0xffffffffu, w[i], __ffs(m) - 1);
        return (int32_t)want;
      }
      c += found;
    }
  }
  return c;
}

// The same count (want < 0) by one thread: a search in the longer row for each entry of the shorter one, from where
// the last ended.
__device__ __forceinline__ int32_t common_above_thread(const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                                       int32_t u, int32_t v) {
  int64_t a = off[u], a1 = off[u + 1], b = off[v], b1 = off[v + 1];
  if (a1 - a > b1 - b) {
    const int64_t t = a, t1 = a1;
    a = b;
    a1 = b1;
    b = t;
    b1 = t1;
  }
  int32_t c = 0;
  for (a = lower_bound32(col, a, a1, v + 1); a < a1 && b < b1; ++a) {
    const int32_t w = col[a];
    b = lower_bound32(col, b, b1, w);
    c += b < b1 && col[b] == w;
  }
  return c;
}

// Warp per `run` (at most 32) arcs: each arc's triangle count (0 unless col > row).  A lane
// counts its arc where the shorter of the two rows is short; the warp shares the
// entries of the others', so that a hub's arcs do not run on in one thread.  First
// job on a graph, a thread for every arc, a warp for every arc, and as it is, ms: ring
// lattice of 100,000 nodes, 20 neighbours each, 0.38, 0.77, 0.32; 2 million random
// arcs of 200,000 nodes 0.56, 1.37, 0.52; BA n = 200,000 4.5, 1.12, 0.69; R-MAT 18
// 524, 5.13, 4.73; R-MAT 12 4.3, 0.174, 0.171 (0.256 with runs of 32).
constexpr int kTriShort = 32;
constexpr int64_t kTriFew = (int64_t)1 << 19;  // fewer arcs are dealt to more warps, eight each
__global__ void __launch_bounds__(256) k_tri_count(int32_t n, int64_t nnz, int run, const int64_t *__restrict__ off,
                                                   const int32_t *__restrict__ col, int64_t *cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * 8;
  for (int64_t b = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * run; b < nnz; b += nwarps * run) {
    const int64_t end = b + run < nnz ? b + run : nnz, e = b + lane;
    int32_t u = (int32_t)warp_upper(off, (int64_t)n + 1, b), last = (int32_t)warp_upper(off, (int64_t)n + 1, end - 1);
    int32_t v = -1;
    if (e < end) {
      while (u < last) {  // off[u] <= e
        const int32_t mid = u + ((last - u + 1) >> 1);
        if (off[mid] <= e)
          u = mid;
        else
          last = mid - 1;
      }
      v = col[e];
    }
    int64_t mine = 0;
    bool wide = false;
    if (v > u) {
      const int64_t du = off[u + 1] - off[u], dv = off[v + 1] - off[v];
      wide = (du < dv ? du : dv) > kTriShort;
      if (!wide) mine = common_above_thread(off, col, u, v);
    }
    for (unsigned m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int32_t c = common_above(off, col, __shfl_sync(0xffffffffu, u, src), __shfl_sync(0xffffffffu, v, src), -1,
                                     nullptr);
      if (lane == src) mine = c;
    }
    if (e < end) cnt[e] = mine;
  }
}

// Warp per sample: rank r -> arc e (the last with tri_off[e] <= r) -> (u, v)
// -> the common neighbour of rank r - tri_off[e].  Bound by the latency of its
// searches, 33-way for the arc and its row, and a binary search per lane among
// the common neighbours.  R-MAT 16, 65,536 samples: 4.0 ms with a thread per
// sample -> 0.21 ms
__global__ void __launch_bounds__(256) k_tri_sample(uint64_t j0, uint64_t count, int32_t n, int64_t nnz,
                                                    const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                                    const int64_t *__restrict__ tri_off, SampleKey key, int32_t *ps,
                                                    int32_t *pt, int32_t *pd, const int64_t *__restrict__ hoff,
                                                    int32_t *hmem) {
  const int lane = threadIdx.x & 31;
  const uint64_t T = (uint64_t)tri_off[nnz];
  const uint64_t nwarps = (uint64_t)gridDim.x * 8;
  for (uint64_t i = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5); i < count; i += nwarps) {
    const uint64_t j = j0 + i;
    const int64_t r = (int64_t)uniform_below64(key.seed, key.id(j), kPurposeS, T);
    const int64_t e = warp_upper(tri_off, nnz + 1, r);
    const int32_t u = (int32_t)warp_upper(off, (int64_t)n + 1, e), v = col[e];
    int32_t w = -1;
    common_above(off, col, u, v, r - tri_off[e], &w);
    if (lane < 3) {
      const int32_t x = lane == 0 ? u : lane == 1 ? v : w;
      (lane == 0 ? ps : lane == 1 ? pt : pd)[j] = x;
      hmem[hoff[j] + lane] = x;
    }
  }
}

}  // namespace

// Writes ps/pt/pd of the new samples and their members: to `out` at stride
// kappa, or, with hoff, into the store at hoff[j]; none when out is null.
void kpath_sample(cen_job *job, uint64_t j0, uint64_t count, int32_t *out, const int64_t *hoff) {
  const cen_graph *g = job->g;
  cudaStream_t st = job->st;
  auto go = [&](auto kernel, int gs) {
    const int groups = kWalkThreads / gs;
    const size_t smem = 2 * sizeof(int32_t) * (size_t)job->kappa * groups;
    launch(&job->stats, K_SPACE, st, [&] {
      kernel<<<grid_for(count, groups, sm_count() * 16), kWalkThreads, smem, st>>>(
          j0, count, g->n, job->kappa, g->off.as<int64_t>(), g->col.as<int32_t>(), job->key(), job->ps.as<int32_t>(),
          job->pt.as<int32_t>(), job->pd.as<int32_t>(), out, hoff, job->bmax.as<int>(),
          (unsigned long long *)(job->stats.d_units + K_SPACE));
    });
  };
  if (job->kappa <= 8)
    go(k_kpath<8>, 8);
  else
    go(k_kpath<32>, 32);
}

// Triangle ranks of the graph (kept on the graph), and their total.
int64_t triangle_index(cen_job *job) {
  cen_graph *g = const_cast<cen_graph *>(job->g);
  std::lock_guard<std::mutex> lk(g->tri_mu);
  if (g->tri_total < 0) {
    cudaStream_t st = job->st;
    DevBuf cnt;
    cnt.ensure(8 * (size_t)(g->nnz + 1), st);
    g->tri_off.ensure(8 * (size_t)(g->nnz + 1), st);
    launch(&job->stats, K_SPACE, st, [&] {
      const int run = g->nnz < kTriFew ? 8 : 32;
      k_tri_count<<<grid_for((size_t)g->nnz, 8 * run, sm_count() * 64), 256, 0, st>>>(
          g->n, g->nnz, run, g->off.as<int64_t>(), g->col.as<int32_t>(), cnt.as<int64_t>());
    });
    exclusive_scan_i64(cnt.as<int64_t>(), g->tri_off.as<int64_t>(), (size_t)g->nnz, g->tri_off.as<int64_t>() + g->nnz,
                       job->scan_tmp, st, &job->stats);
    int64_t *h = (int64_t *)host_staging(job, 8);
    CEN_CK(cudaMemcpyAsync(h, g->tri_off.as<int64_t>() + g->nnz, 8, cudaMemcpyDeviceToHost, st));
    CEN_CK(cudaStreamSynchronize(st));
    cnt.release();
    CEN_CK(cudaStreamSynchronize(st));
    g->tri_total = *h;
  }
  return g->tri_total;
}

// Members of samples j0 .. j0+count-1 straight into the store (3 each; hoff set).
void triangle_sample(cen_job *job, uint64_t j0, uint64_t count) {
  const cen_graph *g = job->g;
  cudaStream_t st = job->st;
  launch(&job->stats, K_SPACE, st, [&] {
    k_tri_sample<<<grid_for(count, 8), 256, 0, st>>>(j0, count, g->n, g->nnz, g->off.as<int64_t>(),
                                                         g->col.as<int32_t>(), g->tri_off.as<int64_t>(), job->key(),
                                                         job->ps.as<int32_t>(), job->pt.as<int32_t>(),
                                                         job->pd.as<int32_t>(), job->hoff.as<int64_t>(),
                                                         job->hmem.as<int32_t>());
  });
}

int max_kappa() { return kMaxKappa; }

}  // namespace cen
