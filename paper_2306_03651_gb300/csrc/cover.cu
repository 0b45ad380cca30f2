// Node -> sample incidence and greedyCover(k, H) (Sec. 3.1; Alg. 1 line "greedyCover").
#include <cooperative_groups.h>

#include <algorithm>
#include <cstddef>
#include <cstdlib>
#include <map>
#include <mutex>

#include "heavy.cuh"

namespace cg = cooperative_groups;

namespace cen {

// ------------------------------------------------------- incidence
constexpr int kRankThreads = 512;
// Members from which a thread takes eight, below it two (more blocks); the time
// of all rounds of a run, two against eight: BA n = 2,000 up to 0.6M members
// 75 and 81 us, R-MAT 18 up to 3M members 165 and 120 us.
constexpr size_t kRankWide = (size_t)1 << 19;

// Counts every node's members in c (zero before) and gives each member its
// place among its node's (in no particular order).  A block's members meet in
// a table of as many slots in shared memory, and each node found there takes
// one atomic on its count for the whole block; a node that finds no slot within
// kRankProbes takes one per member.  The counts of hub nodes are what bounds
// this: with one atomic a member to count it and another to place it, all on a
// few addresses at L2, a run's rounds took 256 + 225 us on BA n = 2,000 (0.6M
// members at the end) and 489 + 511 us on R-MAT 18 (3M); they take 75 + 29 and
// 120 + 66.
constexpr int kRankProbes = 4;
template <int ITEMS>
__global__ void __launch_bounds__(kRankThreads) k_rank_members(const int32_t *__restrict__ hmem, int64_t total,
                                                               int32_t *c, int32_t *__restrict__ rank) {
  constexpr int TILE = kRankThreads * ITEMS;
  static_assert(TILE <= 4096 && (TILE & (TILE - 1)) == 0, "12-bit slots and places");
  __shared__ int32_t key[TILE], cnt[TILE];
  for (int p = threadIdx.x; p < TILE; p += kRankThreads) {
    key[p] = -1;
    cnt[p] = 0;
  }
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * TILE + threadIdx.x;
  uint32_t at[ITEMS];  // slot << 16 | place among the block's members of the node
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const int64_t i = base + r * kRankThreads;
    at[r] = ~0u;
    if (i >= total) continue;
    const int32_t u = hmem[i];
    uint32_t p = ((uint32_t)u * 0x9E3779B1u) >> 20 & (TILE - 1);
    bool found = false;
    for (int k = 0; k < kRankProbes && !found; ++k) {
      int32_t have = *(volatile int32_t *)&key[p];
      if (have == -1) have = atomicCAS(&key[p], -1, u);
      found = have == -1 || have == u;
      if (!found) p = (p + 1) & (TILE - 1);
    }
    if (found)
      at[r] = (p << 16) | (uint32_t)atomicAdd(&cnt[p], 1);
    else
      rank[i] = atomicAdd(&c[u], 1);
  }
  __syncthreads();
  for (int p = threadIdx.x; p < TILE; p += kRankThreads)
    if (key[p] >= 0) cnt[p] = atomicAdd(&c[key[p]], cnt[p]);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r)
    if (at[r] != ~0u) rank[base + r * kRankThreads] = cnt[at[r] >> 16] + (int32_t)(at[r] & 0xFFFFu);
}

// GS lanes per sample: each member u gets j at its place of row u (the order
// within a row is free; every consumer of the rows is order-free).
template <int GS>
__global__ void k_place_members(const int64_t *__restrict__ hoff, const int32_t *__restrict__ hmem, uint64_t m,
                                const int64_t *__restrict__ noff, const int32_t *__restrict__ rank, int32_t *nsamp) {
  const int lane = threadIdx.x & (GS - 1);
  const uint64_t groups = (uint64_t)gridDim.x * blockDim.x / GS;
  for (uint64_t j = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / GS; j < m; j += groups) {
    const int64_t e1 = hoff[j + 1];
    for (int64_t e = hoff[j] + lane; e < e1; e += GS) nsamp[noff[hmem[e]] + rank[e]] = (int32_t)j;
  }
}

// Rows of the samples that hold each node.  The members' places lie in hmemh,
// which build_heavy fills anew afterwards.
void build_incidence(cen_job *job) {
  if (job->inc_m == job->m) return;
  cudaStream_t st = job->st;
  Stats *S = &job->stats;
  const int32_t n = job->g->n;
  const size_t members = (size_t)job->members;
  job->c.ensure(heavy_ctl_at(job) + sizeof(HeavyCtl), st);
  job->noff.ensure(8 * ((size_t)n + 1), st);
  job->nsamp.ensure(4 * (members + 1), st);
  job->hmemh.ensure(4 * (members + 1), st);
  job->heavy_m = ~0ull;
  CEN_CK(cudaMemsetAsync(job->c.p, 0, heavy_ctl_at(job) + sizeof(HeavyCtl), st));
  job->heavy_clear = true;
  if (members)
    launch(S, K_TRANSPOSE, st, [&] {
      const bool wide = members >= kRankWide;
      auto kernel = wide ? k_rank_members<8> : k_rank_members<2>;
      const int tile = kRankThreads * (wide ? 8 : 2);
      kernel<<<(unsigned)((members + tile - 1) / tile), kRankThreads, 0, st>>>(
          job->hmem.as<int32_t>(), job->members, job->c.as<int32_t>(), job->hmemh.as<int32_t>());
    });
  counts_to_offsets(job->c.as<int32_t>(), job->noff.as<int64_t>(), (size_t)n, job->scan_tmp, st, S);
  if (members)
    launch(S, K_TRANSPOSE, st, [&] {
      const bool wide = job->members > kShortMembers * (int64_t)job->m;
      auto kernel = wide ? k_place_members<32> : k_place_members<4>;
      kernel<<<grid_for(job->m * (wide ? 32 : 4), 256), 256, 0, st>>>(
          job->hoff.as<int64_t>(), job->hmem.as<int32_t>(), job->m, job->noff.as<int64_t>(),
          job->hmemh.as<int32_t>(), job->nsamp.as<int32_t>());
    });
  job->inc_m = job->m;
}

// ------------------------------------------------------- heavy nodes
// Counts of the c_u buckets.
__global__ void __launch_bounds__(256) k_heavy_hist(const int32_t *__restrict__ c, int32_t n, HeavyCtl *ctl) {
  __shared__ uint32_t h[kHeavyBuckets];
  for (int i = threadIdx.x; i < kHeavyBuckets; i += 256) h[i] = 0;
  __syncthreads();
  for (int64_t u = (int64_t)blockIdx.x * 256 + threadIdx.x; u < n; u += (int64_t)gridDim.x * 256) {
    const int32_t cu = c[u];
    if (cu > 0) atomicAdd(&h[heavy_bucket((uint32_t)cu)], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kHeavyBuckets; i += 256)
    if (h[i]) atomicAdd(&ctl->hist[i], h[i]);
}

// Lists the nodes with c_u >= tau (tau from the bucket counts, by every block;
// order of arrival) with their c_u, the chunks of their rows, and for every
// node its list entry or -1.  With `all`, entry u is node u and tau is 1.
__global__ void __launch_bounds__(256) k_heavy_list(const int32_t *__restrict__ c, int32_t n, bool all, HeavyCtl *ctl,
                                                    int32_t *list, int32_t *hc, int32_t *idx, uint2 *chunks) {
  __shared__ uint32_t wsum[8];
  __shared__ int s_cut;
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t tau = 1;
  if (!all) {
    // thread i holds buckets from the top: [B - (i+1) P, B - i P)
    constexpr int P = (kHeavyBuckets + 255) / 256;
    const int top = kHeavyBuckets - tid * P;
    uint32_t sum = 0;
    for (int q = 0; q < P; ++q)
      if (top - 1 - q >= 1) sum += ctl->hist[top - 1 - q];
    uint32_t inc = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[tid >> 5] = inc;
    if (tid == 0) s_cut = 1;  // every bucket fits
    __syncthreads();
    for (int w = 0; w < (tid >> 5); ++w) inc += wsum[w];
    if (inc > (uint32_t)kHeavyMax && inc - sum <= (uint32_t)kHeavyMax) {  // the bucket that overflows is in here
      uint32_t run = inc - sum;
      for (int q = 0; q < P && top - 1 - q >= 1; ++q) {
        run += ctl->hist[top - 1 - q];
        if (run > (uint32_t)kHeavyMax) {
          s_cut = top - q;  // the buckets above it
          break;
        }
      }
    }
    __syncthreads();
    tau = s_cut >= kHeavyBuckets ? 0x7fffffffu : heavy_bucket_low(s_cut);
  }
  if (blockIdx.x == 0 && tid == 0) {
    ctl->tau = (int32_t)tau;
    if (all) ctl->count = (uint32_t)n;
  }
  const int64_t span = ((int64_t)n + 31) & ~(int64_t)31;  // whole warps
  for (int64_t u = (int64_t)blockIdx.x * 256 + tid; u < span; u += (int64_t)gridDim.x * 256) {
    const int32_t cu = u < n ? c[u] : 0;
    const bool in = cu > 0 && (uint32_t)cu >= tau;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    int32_t at = -1;
    uint32_t parts = in ? ((uint32_t)cu + kRadeChunk - 1) / kRadeChunk : 0u;
    if (m) {
      uint32_t base = 0, inc = parts;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
      uint32_t cbase = 0;
      if (lane == 0) {
        if (!all) base = atomicAdd(&ctl->count, (uint32_t)__popc(m));
        cbase = atomicAdd(&ctl->nchunks, total);
      }
      base = __shfl_sync(0xffffffffu, base, 0);
      cbase = __shfl_sync(0xffffffffu, cbase, 0);
      if (in) {
        at = all ? (int32_t)u : (int32_t)(base + __popc(m & ((1u << lane) - 1u)));
        for (uint32_t q = 0; q < parts; ++q) chunks[cbase + inc - parts + q] = make_uint2((uint32_t)at, q);
      }
    }
    if (u < n && !all) idx[u] = at;
    if (all && u < n) at = (int32_t)u;
    if (at >= 0) {
      list[at] = (int32_t)u;
      hc[at] = cu;
    }
  }
}

// Members as list entries (-1: not listed), so that a pick does not look them up.
__global__ void __launch_bounds__(256) k_heavy_members(const int32_t *__restrict__ hmem, int64_t total,
                                                       const int32_t *__restrict__ idx, int32_t *out) {
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256)
    out[e] = idx[hmem[e]];
}

void heavy_list_all(const int32_t *c, int32_t n, HeavyCtl *ctl, int32_t *list, int32_t *hc, uint2 *chunks,
                    cudaStream_t st) {
  k_heavy_list<<<grid_for((size_t)n, 256 * 4, sm_count() * 4), 256, 0, st>>>(c, n, true, ctl, list, hc, nullptr, chunks);
}

// Chunks that the rows of `nodes` nodes can have.
static size_t heavy_chunks_most(const cen_job *job, size_t nodes) {
  return nodes + (size_t)job->members / kRadeChunk + 1;
}

// The heavy nodes of the current sample (incidence current), on the job's stream.
void build_heavy(cen_job *job) {
  if (job->heavy_m == job->m) return;
  cudaStream_t st = job->st;
  Stats *S = &job->stats;
  const int32_t n = job->g->n;
  const bool all = n <= kHeavyMax;
  const size_t most = all ? (size_t)n : (size_t)kHeavyMax;
  job->hlist.ensure(4 * most, st);
  job->hc.ensure(4 * most, st);
  job->hidx.ensure(all ? 4 : 4 * (size_t)n, st);
  job->hchunks.ensure(8 * heavy_chunks_most(job, most), st);
  HeavyCtl *ctl = heavy_ctl(job);
  if (!job->heavy_clear) CEN_CK(cudaMemsetAsync(ctl, 0, sizeof(HeavyCtl), st));  // (a call that failed left it)
  job->heavy_clear = false;
  if (!all)
    launch(S, K_TRANSPOSE, st, [&] {
      k_heavy_hist<<<grid_for((size_t)n, 256 * 8, sm_count() * 4), 256, 0, st>>>(job->c.as<int32_t>(), n, ctl);
    });
  launch(S, K_TRANSPOSE, st, [&] {
    k_heavy_list<<<grid_for((size_t)n, 256 * 4, sm_count() * 4), 256, 0, st>>>(
        job->c.as<int32_t>(), n, all, ctl, job->hlist.as<int32_t>(), job->hc.as<int32_t>(), job->hidx.as<int32_t>(),
        job->hchunks.as<uint2>());
  });
  if (!all && job->members) {
    job->hmemh.ensure(4 * (size_t)job->members, st);
    launch(S, K_TRANSPOSE, st, [&] {
      k_heavy_members<<<grid_for((size_t)job->members, 256 * 4), 256, 0, st>>>(
          job->hmem.as<int32_t>(), job->members, job->hidx.as<int32_t>(), job->hmemh.as<int32_t>());
    });
  }
  job->heavy_m = job->m;
}

HeavyView heavy_view(const cen_job *job) {
  return HeavyView{heavy_ctl(job), job->hlist.as<int32_t>(), job->hc.as<int32_t>(),
                   job->hchunks.as<uint2>()};
}

// ---------------------------------------------------------------- greedy
// Control words: key[2] (ping-pong argmax keys), covered count, picks, done.
struct GreedyCtl {
  unsigned long long key[2];
  unsigned long long covered;
  int size;
  int done;
  int short_;  // a pick among the heavy nodes fell below tau: all nodes are needed
  int S[1];    // k entries follow
};

__global__ void k_gain_init(const int32_t *__restrict__ c, int32_t *gain, int32_t n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) gain[i] = c[i];
}

// Lowers the gains of the members of the covered samples, GS lanes a sample.
template <int GS>
__global__ void __launch_bounds__(256) k_gain_drop(const int64_t *__restrict__ hoff, const int32_t *__restrict__ hmem,
                                                   uint64_t m, const uint32_t *__restrict__ covered, int32_t *gain) {
  const int lane = threadIdx.x & (GS - 1);
  const uint64_t groups = (uint64_t)gridDim.x * 256 / GS;
  for (uint64_t j = ((uint64_t)blockIdx.x * 256 + threadIdx.x) / GS; j < m; j += groups) {
    if (!((covered[j >> 5] >> (j & 31)) & 1u)) continue;
    const int64_t e1 = hoff[j + 1];
    for (int64_t e = hoff[j] + lane; e < e1; e += GS) atomicSub(&gain[hmem[e]], 1);
  }
}

// argmax over nodes of key = gain << 32 | (2^32 - 1 - u): the max key has the
// largest gain and, among equal gains, the lowest id.
__global__ void __launch_bounds__(256) k_greedy_argmax(const int32_t *__restrict__ gain, int32_t n, GreedyCtl *ctl,
                                                       int slot) {
  if (ctl->done) return;
  unsigned long long best = 0;
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
    const unsigned long long k = ((unsigned long long)(uint32_t)gain[u] << 32) | (0xFFFFFFFFu - (uint32_t)u);
    best = k > best ? k : best;
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
    best = y > best ? y : best;
  }
  __shared__ unsigned long long wb[8];
  if ((threadIdx.x & 31) == 0) wb[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) best = wb[w] > best ? wb[w] : best;
    if (best) atomicMax(&ctl->key[slot], best);
  }
}

// Warp per incident sample of the pick u*: a still-uncovered sample becomes
// covered and every member's gain drops by one.
__global__ void __launch_bounds__(256) k_greedy_update(const int64_t *__restrict__ noff,
                                                       const int32_t *__restrict__ nsamp,
                                                       const int64_t *__restrict__ hoff,
                                                       const int32_t *__restrict__ hmem, int32_t *gain,
                                                       uint32_t *covered, GreedyCtl *ctl, int slot, int it) {
  if (ctl->done) return;
  const unsigned long long key = ctl->key[slot];
  const uint32_t g = (uint32_t)(key >> 32);
  if (g == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->done = 1;
    return;
  }
  const int32_t u = (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFu));
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->S[it] = u;
    ctl->size = it + 1;
    ctl->covered += g;
    ctl->key[slot ^ 1] = 0;  // reset the other slot for the next argmax
  }
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t r0 = noff[u], r1 = noff[u + 1];
  for (int64_t q = r0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); q < r1; q += nwarps) {
    const int32_t j = nsamp[q];
    const uint32_t mask = 1u << (j & 31);
    if (covered[j >> 5] & mask) continue;  // j occurs once in row u: only this warp can set its bit now
    if (lane == 0) atomicOr(&covered[j >> 5], mask);
    for (int64_t e = hoff[j] + lane; e < hoff[j + 1]; e += 32) atomicSub(&gain[hmem[e]], 1);
  }
}

// All k iterations in one cooperative launch: each iteration is the argmax
// (block maxima, one atomicMax per block), a grid barrier, the update of the
// picked node's samples, and another barrier.  The first ctl->size picks are
// made already.  The picks, ties and counts
// are those of k_greedy_argmax / k_greedy_update.  A cooperative launch runs
// only when every block is resident at once, so the barriers always complete.
__global__ void __launch_bounds__(256) k_greedy_all(const int64_t *__restrict__ noff, const int32_t *__restrict__ nsamp,
                                                    const int64_t *__restrict__ hoff, const int32_t *__restrict__ hmem,
                                                    int32_t *gain, int32_t n, uint32_t *covered, GreedyCtl *ctl,
                                                    int k) {
  cg::grid_group grid = cg::this_grid();
  __shared__ unsigned long long wb[8];
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int it = ctl->size; it < k; ++it) {  // (size is first written behind a grid barrier)
    const int slot = it & 1;
    unsigned long long best = 0;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
      const unsigned long long key = ((unsigned long long)(uint32_t)gain[u] << 32) | (0xFFFFFFFFu - (uint32_t)u);
      best = key > best ? key : best;
    }
    for (int o = 16; o; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, best, o);
      best = y > best ? y : best;
    }
    if (lane == 0) wb[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) best = wb[w] > best ? wb[w] : best;
      if (best) atomicMax(&ctl->key[slot], best);
    }
    grid.sync();
    const unsigned long long key = ((volatile unsigned long long *)ctl->key)[slot];
    const uint32_t g = (uint32_t)(key >> 32);
    if (g == 0) break;  // every block sees the same key: all leave together
    const int32_t u = (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFu));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ctl->S[it] = u;
      ctl->size = it + 1;
      ctl->covered += g;
      ctl->key[slot ^ 1] = 0;
    }
    const int64_t r0 = noff[u], r1 = noff[u + 1];
    for (int64_t q = r0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); q < r1; q += nwarps) {
      const int32_t j = nsamp[q];
      const uint32_t mask = 1u << (j & 31);
      if (covered[j >> 5] & mask) continue;
      if (lane == 0) atomicOr(&covered[j >> 5], mask);
      for (int64_t e = hoff[j] + lane; e < hoff[j + 1]; e += 32) atomicSub(&gain[hmem[e]], 1);
    }
    grid.sync();
  }
}

// All k iterations in one thread-block cluster of C CTAs (16 where the device
// allows clusters that large, else 8), the gains held in the CTAs' shared
// memory: item i (a heavy node's list entry, or with HEAVY = false node i) is
// CTA i % C's.  Per iteration: each CTA takes the largest key of its items (the
// same key as k_greedy_all: largest gain, lowest id), a cluster barrier, every
// CTA reads the others' keys through distributed shared memory and so picks
// the same u*; then a thread per incident sample of u* sets the sample's
// covered bit and, if it was not set, decrements the gains of the sample's
// members in their owners' shared memory; another cluster barrier.  With
// HEAVY = false the first ctl->size picks are made already, and `gains` follow from
// them.  The picks and counts are those of k_greedy_all.  A cluster is launched only when all
// of its CTAs are resident at once, so the barriers always complete.
//
// Over the heavy nodes a CTA of 16 holds at most 1,024 gains (two keys a thread;
// of 8, 2,048), so
// a pick costs its two barriers and the chain of loads of the picked row, some
// 3.2 us: R-MAT 18, m = 65,536, k = 50: 0.21 -> 0.16 ms; directed R-MAT 22, k =
// 100, whose 4.2 million gains no cluster holds: 3.2 -> 0.37 ms against the
// grid form; the rewired grid of 4.2 million nodes, with samples of 36 members:
// 4.0 -> 0.26 ms (1.7 with one lane a sample).
constexpr int kGreedyClusterMax = 16;  // non-portable; 8 is the portable size
// 512 threads: cheaper barriers per pick than 1,024 (measured over all nodes 0.215 vs 0.23 ms per
// R-MAT 18 round with 16 CTAs; 0.24 vs 0.25 ms with 8; over the heavy nodes 16 and 8 CTAs are equal)
constexpr int kGreedyThreads = 512;

template <bool HEAVY>
__global__ void __launch_bounds__(kGreedyThreads, 1)
    k_greedy_cluster(const int32_t *__restrict__ gains, HeavyView H, const int64_t *__restrict__ noff,
                     const int32_t *__restrict__ nsamp, const int64_t *__restrict__ hoff,
                     const int32_t *__restrict__ hmem, int32_t n, uint32_t *covered, GreedyCtl *ctl, int k, int lg) {
  extern __shared__ int64_t s_items[];
  __shared__ uint32_t s_wgain[kGreedyThreads / 32], s_wid[kGreedyThreads / 32];
  // the CTA's best and the cluster's: the node's complement (so that larger wins), its gain, its incidence row
  struct __align__(16) Best {
    uint32_t id, gain;
    int32_t len, pad;
    int64_t r0, pad2;
  };
  __shared__ Best s_best, s_pick;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int C = (int)cl.num_blocks(), lgC = 31 - __clz(C);
  const int32_t items = HEAVY ? (int32_t)H.ctl->count : n;
  const uint32_t tau = HEAVY ? (uint32_t)H.ctl->tau : 1u;
  const int32_t mine = (items - rank + C - 1) >> lgC;  // items rank, rank + C, ...
  const int32_t per = (items + C - 1) >> lgC;
  int64_t *s_row = s_items;                                        // first incidence of an item (HEAVY)
  int32_t *s_gain = (int32_t *)(s_items + (HEAVY ? per : 0));
  int32_t *s_id = s_gain + per, *s_len = s_id + per;               // its node and c_u (HEAVY)
  for (int32_t i = tid; i < mine; i += kGreedyThreads) {
    if (HEAVY) {
      const int32_t u = H.list[i * C + rank], cu = H.c[i * C + rank];
      s_gain[i] = cu;
      s_len[i] = cu;
      s_id[i] = u;
      s_row[i] = noff[u];
    } else {
      s_gain[i] = gains[i * C + rank];
    }
  }
  const int first = HEAVY ? 0 : ctl->size;
  cl.sync();
  // a sample's members are dealt to 2^lg lanes
  const int gl = tid & ((1 << lg) - 1);
  const unsigned gmask = (lg == 5 ? 0xffffffffu : (1u << (1 << lg)) - 1u) << (lane & ~((1 << lg) - 1));
  const int64_t gt = ((int64_t)rank * kGreedyThreads + tid) >> lg;
  const int64_t ngroups = ((int64_t)C * kGreedyThreads) >> lg;
  for (int it = first; it < k; ++it) {
    uint32_t bg = 0, bi = 0;  // the thread's best gain, and the complement of its node
    int32_t bat = 0;
    for (int32_t i = tid; i < mine; i += kGreedyThreads) {
      const uint32_t g = (uint32_t)s_gain[i], id = 0xFFFFFFFFu - (HEAVY ? (uint32_t)s_id[i] : (uint32_t)(i * C + rank));
      if (g > bg || (g == bg && id > bi)) {
        bg = g;
        bi = id;
        bat = i;
      }
    }
    // the warp's best, then (every warp for itself) the CTA's
    uint32_t g = __reduce_max_sync(0xffffffffu, bg);
    uint32_t id = __reduce_max_sync(0xffffffffu, bg == g ? bi : 0u);
    if (lane == 0) {
      s_wgain[wid] = g;
      s_wid[wid] = id;
    }
    __syncthreads();
    const uint32_t wg = lane < kGreedyThreads / 32 ? s_wgain[lane] : 0u;
    const uint32_t wi = lane < kGreedyThreads / 32 ? s_wid[lane] : 0u;
    g = __reduce_max_sync(0xffffffffu, wg);
    id = __reduce_max_sync(0xffffffffu, wg == g ? wi : 0u);
    if (g == 0) {
      if (tid == 0) s_best.gain = 0;
    } else if (bg == g && bi == id) {  // one thread holds it
      const int64_t r = HEAVY ? s_row[bat] : noff[bat * C + rank];
      s_best.gain = g;
      s_best.id = id;
      s_best.r0 = r;
      s_best.len = HEAVY ? s_len[bat] : (int32_t)(noff[bat * C + rank + 1] - r);
    }
    cl.sync();  // every CTA's best is in place
    if (wid == 0) {
      uint4 o = make_uint4(0, 0, 0, 0);
      int64_t r = 0;
      if (lane < C) {
        const Best *from = cl.map_shared_rank(&s_best, lane);
        o = *(const uint4 *)from;
        r = from->r0;
      }
      const uint32_t pg = __reduce_max_sync(0xffffffffu, o.y);
      const uint32_t pi = __reduce_max_sync(0xffffffffu, o.y == pg ? o.x : 0u);
      if (pg == 0 ? lane == 0 : o.y == pg && o.x == pi) {
        s_pick.gain = pg;
        s_pick.id = pi;
        s_pick.len = (int32_t)o.z;
        s_pick.r0 = r;
      }
    }
    __syncthreads();
    g = s_pick.gain;
    if (g < tau) {  // nothing left to cover (tau = 1), or a lighter node may come next
      if (HEAVY && tau > 1 && rank == 0 && tid == 0) ctl->short_ = 1;
      break;  // every CTA holds the same pick: all leave together
    }
    const int64_t r0 = s_pick.r0, r1 = r0 + s_pick.len;
    if (rank == 0 && tid == 0) {
      ctl->S[it] = (int32_t)(0xFFFFFFFFu - s_pick.id);
      ctl->size = it + 1;
      ctl->covered += g;
    }
    for (int64_t q = r0 + gt; q < r1; q += ngroups) {
      const int32_t j = nsamp[q];
      const uint32_t mask = 1u << (j & 31);
      const int64_t e0 = hoff[j], e1 = hoff[j + 1];  // loaded alongside the covered bit
      uint32_t old = 0;
      if (gl == 0) old = atomicOr(&covered[j >> 5], mask);
      if (lg) old = __shfl_sync(gmask, old, 0, 1 << lg);
      if (old & mask) continue;  // covered by an earlier pick
      for (int64_t e = e0 + gl; e < e1; e += 1 << lg) {
        const int32_t i = hmem[e];
        if (!HEAVY || i >= 0) atomicSub(cl.map_shared_rank(s_gain + (i >> lgC), i & (C - 1)), 1);
      }
    }
    cl.sync();  // every gain update has landed before the next argmax
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
}

// Nodes per CTA the cluster form can hold (the rest of the shared memory is
// the kernel's own).
constexpr int64_t kGreedyClusterMaxPer = (227 * 1024 - 2048) / 4;

size_t greedy_result_bytes(int32_t k) { return sizeof(GreedyCtl) + 4 * (size_t)k; }

// The covered bits lie behind the control words and are cleared with them.
static size_t greedy_control_bytes(int32_t k) { return (greedy_result_bytes(k) + 15) & ~(size_t)15; }
static uint32_t *greedy_covered(const cen_job *job, int32_t k) {
  return (uint32_t *)(job->gctl.as<char>() + greedy_control_bytes(k));
}

// Whether a cluster of C CTAs of `kernel` with `smem` bytes can be resident on
// this device (the kernel's shared-memory limit is raised, and clusters over 8
// allowed, once per device).
template <class K>
static bool greedy_cluster_ready(K kernel, int C, size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<int, const void *>, int> attr;  // 1: set, 2: clusters over 8 too
  int dev = 0;
  CEN_CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  int &have = attr[{dev, (const void *)kernel}];
  if (!have) {
    have = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kGreedyClusterMaxPer * 4 + 8)) == cudaSuccess ? 1 : -1;
    cudaGetLastError();
    if (have > 0 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
      have = 2;
    cudaGetLastError();
  }
  if (have < 0 || (C > 8 && have < 2)) return false;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(kGreedyThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  const bool ok = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters >= 1;
  cudaGetLastError();
  return ok;
}

// Enqueues k_greedy_cluster<HEAVY> over `items` gains in the largest cluster
// that holds them (`gains` of all nodes when not HEAVY); false when none does.  Diagnostic: CEN_GREEDY_CLUSTER=8
// keeps the portable cluster size.
template <bool HEAVY>
static bool greedy_cluster(cen_job *job, int32_t k, int64_t items, const int32_t *gains, cudaStream_t run,
                           GreedyCtl *ctl) {
  const char *size_env = getenv("CEN_GREEDY_CLUSTER");
  // the members of a sample as list entries, and lanes for about its mean number of members
  const int32_t *members = (HEAVY && job->g->n > kHeavyMax ? job->hmemh : job->hmem).as<int32_t>();
  int lg = 0;
  while (lg < 5 && (double)((int64_t)2 << lg) * (double)job->m <= (double)job->members) ++lg;
  for (int C : {kGreedyClusterMax, 8}) {
    if (C > 8 && size_env && atoi(size_env) == 8) continue;
    const int64_t per = (items + C - 1) / C;
    const size_t smem = (size_t)per * (HEAVY ? 20 : 4) + 8;
    if (smem > (size_t)kGreedyClusterMaxPer * 4 + 8 || !greedy_cluster_ready(k_greedy_cluster<HEAVY>, C, smem)) continue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kGreedyThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = run;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch(&job->stats, K_GREEDY, run, [&] {
      CEN_CK(cudaLaunchKernelEx(&cfg, k_greedy_cluster<HEAVY>, gains, heavy_view(job),
                                (const int64_t *)job->noff.as<int64_t>(), (const int32_t *)job->nsamp.as<int32_t>(),
                                (const int64_t *)job->hoff.as<int64_t>(), members, job->g->n,
                                greedy_covered(job, k), ctl, (int)k, lg));
    });
    return true;
  }
  return false;
}

// Sizes the greedy workspace for k picks (allocations ordered on the job's
// stream).  The incidence must be current.
void greedy_prepare(cen_job *job, int32_t k) {
  CEN_REQUIRE(k >= 1, CEN_EINVAL, "cen_greedy_cover: k must be >= 1");
  cudaStream_t st = job->st;
  job->gain.ensure(4 * (size_t)job->g->n, st);
  job->gctl.ensure(greedy_control_bytes(k) + 4 * ((job->m + 31) / 32 + 1), st);
}

// Enqueues greedyCover(k) on stream `run` (after greedy_prepare), over the
// heavy nodes or over all; the result reaches hdst (pinned,
// greedy_result_bytes(k)) once `run` has drained.  With made > 0 (over all
// nodes) the control words and covered bits hold that many picks already, and
// their gains are taken from the covered bits.
static void greedy_enqueue_from(cen_job *job, int32_t k, cudaStream_t run, void *hdst, bool heavy, int made) {
  Stats *St = &job->stats;
  const int32_t n = job->g->n;
  const size_t cbytes = greedy_result_bytes(k);
  uint32_t *const cov = greedy_covered(job, k);
  GreedyCtl *ctl = job->gctl.as<GreedyCtl>();
  const int32_t *gains = job->c.as<int32_t>();
  if (made) {
    CEN_CK(cudaMemsetAsync(&ctl->short_, 0, sizeof(ctl->short_), run));
    int32_t *left = job->gain_left.as<int32_t>();
    launch(St, K_GREEDY, run, [&] { k_gain_init<<<grid_for(n, 256), 256, 0, run>>>(gains, left, n); });
    launch(St, K_GREEDY, run, [&] {
      const bool wide = job->members > kShortMembers * (int64_t)job->m;
      auto kernel = wide ? k_gain_drop<32> : k_gain_drop<4>;
      kernel<<<grid_for(job->m * (wide ? 32 : 4), 256), 256, 0, run>>>(job->hoff.as<int64_t>(),
                                                                       job->hmem.as<int32_t>(), job->m, cov, left);
    });
    gains = left;
  } else {
    CEN_CK(cudaMemsetAsync(job->gctl.p, 0, greedy_control_bytes(k) + 4 * ((job->m + 31) / 32 + 1), run));
  }
  // diagnostic: CEN_GREEDY_GRID=1 keeps the cooperative grid form
  const char *grid_env = getenv("CEN_GREEDY_GRID");
  const bool grid_form = grid_env && grid_env[0] == '1';
  const bool done = !grid_form && (heavy ? greedy_cluster<true>(job, k, std::min<int64_t>(n, kHeavyMax), gains, run, ctl)
                                         : greedy_cluster<false>(job, k, n, gains, run, ctl));
  if (done) {
    CEN_CK(cudaMemcpyAsync(hdst, ctl, cbytes, cudaMemcpyDeviceToHost, run));
    return;
  }
  int32_t *const work = made ? job->gain_left.as<int32_t>() : job->gain.as<int32_t>();
  if (!made) launch(St, K_GREEDY, run, [&] { k_gain_init<<<grid_for(n, 256), 256, 0, run>>>(gains, work, n); });
  const int coop = cooperative_grid((const void *)k_greedy_all, 256);
  if (coop > 0) {
    const int64_t *a_noff = job->noff.as<int64_t>();
    const int32_t *a_nsamp = job->nsamp.as<int32_t>();
    const int64_t *a_hoff = job->hoff.as<int64_t>();
    const int32_t *a_hmem = job->hmem.as<int32_t>();
    int32_t *a_gain = work;
    int32_t a_n = n;
    uint32_t *a_cov = cov;
    int a_k = k;
    void *args[] = {&a_noff, &a_nsamp, &a_hoff, &a_hmem, &a_gain, &a_n, &a_cov, &ctl, &a_k};
    launch(St, K_GREEDY, run, [&] {
      CEN_CK(cudaLaunchCooperativeKernel((const void *)k_greedy_all, dim3(coop), dim3(256), args, 0, run));
    });
  } else {
    const int gblocks = grid_for((size_t)n, 256, sm_count() * 4);
    for (int it = made; it < k; ++it) {
      const int slot = it & 1;
      launch(St, K_GREEDY, run, [&] { k_greedy_argmax<<<gblocks, 256, 0, run>>>(work, n, ctl, slot); });
      launch(St, K_GREEDY, run, [&] {
        k_greedy_update<<<sm_count() * 4, 256, 0, run>>>(job->noff.as<int64_t>(), job->nsamp.as<int32_t>(),
                                                   job->hoff.as<int64_t>(), job->hmem.as<int32_t>(),
                                                   work, cov, ctl, slot, it);
      });
    }
  }
  CEN_CK(cudaMemcpyAsync(hdst, ctl, cbytes, cudaMemcpyDeviceToHost, run));
}

// S, |S| and the covered count from the copied result; false when the heavy
// nodes did not decide every pick.
bool greedy_result(const void *h, int32_t *S, int32_t *S_size, uint64_t *covered) {
  const GreedyCtl *hc = (const GreedyCtl *)h;
  if (hc->short_) return false;
  *S_size = hc->size;
  *covered = hc->covered;
  for (int i = 0; i < hc->size; ++i) S[i] = hc->S[i];
  return true;
}

void greedy_enqueue(cen_job *job, int32_t k, cudaStream_t run, void *hdst, bool heavy) {
  greedy_enqueue_from(job, k, run, hdst, heavy, 0);
}

// Goes on over all nodes, on the job's stream, where the heavy ones left the
// copied result h.  Their picks stand: each gain was at least tau, and no other
// node's can be.  A call of as many picks or more goes over all nodes at once
// where they were less than half.  A first round's greedy and AMCERA, the picks made
// again, over all nodes alone, and as it is: ring of 60,000 nodes, 40,000 walks, k =
// 6,000 28.5, 22.0, 19.9 ms; BA n = 200,000, 65,536 walks, k = 3,000 19.2, 11.9, 10.0.
void greedy_over_all(cen_job *job, int32_t k, void *h, int32_t *S, int32_t *S_size, uint64_t *covered) {
  const int made = ((const GreedyCtl *)h)->size;
  if (2 * (int64_t)made < k) job->greedy_all_k = std::min(job->greedy_all_k, k);
  if (made) job->gain_left.ensure(4 * (size_t)job->g->n, job->st);
  greedy_enqueue_from(job, k, job->st, h, false, made);
  CEN_CK(cudaStreamSynchronize(job->st));
  greedy_result(h, S, S_size, covered);
}

// ------------------------------------------- greedyCover one pick at a time
// For a sample split over several GPUs (shards): every shard keeps its own
// gains and covered bits; the caller sums the shards' gains, takes the pick
// (shard_pick, the same key as k_greedy_all: largest gain, lowest id) and
// applies it to every shard.  A shard's newly covered samples are exactly its
// part of the pick's summed gain.

// Warp per incident sample of u, as k_greedy_update; counts the samples it
// newly covers.
__global__ void __launch_bounds__(256) k_shard_apply(const int64_t *__restrict__ noff,
                                                     const int32_t *__restrict__ nsamp,
                                                     const int64_t *__restrict__ hoff,
                                                     const int32_t *__restrict__ hmem, int32_t *gain,
                                                     uint32_t *covered, int32_t u, unsigned long long *newly) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t r0 = noff[u], r1 = noff[u + 1];
  unsigned long long mine = 0;
  for (int64_t q = r0 + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); q < r1; q += nwarps) {
    const int32_t j = nsamp[q];
    const uint32_t mask = 1u << (j & 31);
    if (covered[j >> 5] & mask) continue;  // j occurs once in row u: only this warp can set its bit now
    if (lane == 0) {
      atomicOr(&covered[j >> 5], mask);
      ++mine;
    }
    for (int64_t e = hoff[j] + lane; e < hoff[j + 1]; e += 32) atomicSub(&gain[hmem[e]], 1);
  }
  if (lane == 0 && mine) atomicAdd(newly, mine);
}

void shard_greedy_begin(cen_job *job) {
  build_incidence(job);
  greedy_prepare(job, 1);
  cudaStream_t st = job->st;
  const int32_t n = job->g->n;
  job->covered.ensure(4 * ((job->m + 31) / 32 + 1), st);
  CEN_CK(cudaMemsetAsync(job->covered.p, 0, 4 * ((job->m + 31) / 32 + 1), st));
  launch(&job->stats, K_GREEDY, st,
         [&] { k_gain_init<<<grid_for(n, 256), 256, 0, st>>>(job->c.as<int32_t>(), job->gain.as<int32_t>(), n); });
  CEN_CK(cudaStreamSynchronize(st));
  job->shard_greedy_m = (int64_t)job->m;
}

static void require_shard_greedy(const cen_job *job, const char *what) {
  CEN_REQUIRE(job->shard_greedy_m == (int64_t)job->m, CEN_EINVAL,
              std::string(what) + ": call cen_shard_greedy_begin after the last cen_sample");
}

void shard_gains(const cen_job *job, int32_t *dst) {
  require_shard_greedy(job, "cen_shard_gains");
  CEN_CK(cudaMemcpyAsync(dst, job->gain.p, 4 * (size_t)job->g->n, cudaMemcpyDeviceToDevice, job->st));
  CEN_CK(cudaStreamSynchronize(job->st));
}

void shard_pick(cen_job *job, const int32_t *gains, int32_t *u, int32_t *gain) {
  cudaStream_t st = job->st;
  const int32_t n = job->g->n;
  job->gctl.ensure(greedy_result_bytes(1), st);
  GreedyCtl *ctl = job->gctl.as<GreedyCtl>();
  CEN_CK(cudaMemsetAsync(ctl, 0, sizeof(GreedyCtl), st));
  launch(&job->stats, K_GREEDY, st, [&] {
    k_greedy_argmax<<<grid_for((size_t)n, 256, sm_count() * 4), 256, 0, st>>>(gains, n, ctl, 0);
  });
  unsigned long long *h = (unsigned long long *)host_staging(job, 8);
  CEN_CK(cudaMemcpyAsync(h, &ctl->key[0], 8, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  const unsigned long long key = *h;
  *gain = (int32_t)(uint32_t)(key >> 32);
  *u = key ? (int32_t)(0xFFFFFFFFu - (uint32_t)(key & 0xFFFFFFFFu)) : -1;
}

void shard_apply(cen_job *job, int32_t u, uint64_t *newly) {
  require_shard_greedy(job, "cen_shard_apply");
  CEN_REQUIRE(u >= 0 && u < job->g->n, CEN_EINVAL, "cen_shard_apply: node out of range");
  cudaStream_t st = job->st;
  GreedyCtl *ctl = job->gctl.as<GreedyCtl>();
  CEN_CK(cudaMemsetAsync(&ctl->covered, 0, 8, st));
  launch(&job->stats, K_GREEDY, st, [&] {
    k_shard_apply<<<sm_count() * 4, 256, 0, st>>>(job->noff.as<int64_t>(), job->nsamp.as<int32_t>(),
                                                  job->hoff.as<int64_t>(), job->hmem.as<int32_t>(),
                                                  job->gain.as<int32_t>(), job->covered.as<uint32_t>(), u,
                                                  &ctl->covered);
  });
  unsigned long long *h = (unsigned long long *)host_staging(job, 8);
  CEN_CK(cudaMemcpyAsync(h, &ctl->covered, 8, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  *newly = *h;
}

void greedy_cover(cen_job *job, int32_t k, int32_t *S, int32_t *S_size, uint64_t *covered) {
  CEN_REQUIRE(k >= 1, CEN_EINVAL, "cen_greedy_cover: k must be >= 1");
  Range range("cen_greedy_cover");
  build_incidence(job);
  build_heavy(job);
  greedy_prepare(job, k);
  void *h = host_staging(job, greedy_result_bytes(k));
  greedy_enqueue(job, k, job->st, h, k < job->greedy_all_k);
  CEN_CK(cudaStreamSynchronize(job->st));
  if (!greedy_result(h, S, S_size, covered)) greedy_over_all(job, k, h, S, S_size, covered);
}

}  // namespace cen
