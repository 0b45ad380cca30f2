// AMCERA numerators (Sec. 4.1; Alg. 1 lines computing r_j^u, r_j and the average).
//
// R_q^u = sum over samples j holding u of sigma_{q,j} = 2 P_q^u - c_u, where
// P_q^u counts u's samples whose sign bit q is set.  The sup over |S| <= k of
// sum_{u in S} R_q^u is the sum of the <= k largest positive R_q^u (the
// objective is additive in S), found per row by an exact MSB-first radix
// select; the same select over c_u gives the wimpy-variance numerator.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>

#include "heavy.cuh"

namespace cen {

// ---- R over incidence rows
// A warp takes one chunk (at most kRadeChunk incidences) of one listed node's
// row.  Each lane adds the sign words of its incidences into bit-sliced
// counters (plane b holds bit b of 32 column counts), so that an incidence
// costs a load and a few logic operations for 32 sign vectors instead of a
// ballot for each.  Five butterfly steps add the lanes' counters, bit-sliced
// too, and lane q reads column q.  A node with more than one chunk adds its
// parts into R, which starts at zero.  Bound by the gathered sign rows and, for
// short rows, by the butterfly.  R-MAT 16, m = 262,144, t = 256: 4.6 ms (a warp
// per node of any row length, ballots) -> 0.06; R-MAT 18, m = 65,536, t = 10:
// 0.074 -> 0.018 ms.
template <int NB>
__device__ __forceinline__ void planes_add(uint32_t *p, uint32_t x) {  // one bit per column
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const uint32_t carry = p[b] & x;
    p[b] ^= x;
    x = carry;
  }
}
// Adds NB-plane counters over the warp's lanes; column q's total in lane q.
template <int NB>
__device__ __forceinline__ int32_t planes_total(const uint32_t *in) {
  const int lane = threadIdx.x & 31;
  uint32_t p[NB + 5];
#pragma unroll
  for (int b = 0; b < NB; ++b) p[b] = in[b];
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    uint32_t carry = 0;
#pragma unroll
    for (int b = 0; b < NB + s; ++b) {
      const uint32_t y = __shfl_xor_sync(0xffffffffu, p[b], 1 << s);
      const uint32_t half = p[b] ^ y;
      const uint32_t up = (p[b] & y) | (half & carry);
      p[b] = half ^ carry;
      carry = up;
    }
    p[NB + s] = carry;
  }
  int32_t v = 0;
#pragma unroll
  for (int b = 0; b < NB + 5; ++b) v |= (int32_t)((p[b] >> lane) & 1u) << b;
  return v;
}

constexpr int kRadePlanes = 7;  // a lane's share of a chunk: at most 64 incidences
static_assert(kRadeChunk / 32 < (1 << kRadePlanes), "a lane's counters hold its share of a chunk");

// One chunk's column sums for words w0 .. w0 + W - 1 of the sign rows.
template <int W, int NB, bool VEC>
__device__ __forceinline__ void rade_words(const int32_t *__restrict__ samp, int len, int nw, int w0, int t,
                                           const uint32_t *__restrict__ sign, int32_t *R, int64_t stride, int64_t at,
                                           bool add) {
  const int lane = threadIdx.x & 31;
  uint32_t p[W][NB];
#pragma unroll
  for (int w = 0; w < W; ++w)
#pragma unroll
    for (int b = 0; b < NB; ++b) p[w][b] = 0;
#pragma unroll 2
  for (int i = lane; i < len; i += 32) {
    const uint32_t *row = sign + (int64_t)samp[i] * nw + w0;
    if constexpr (VEC) {
      const uint4 x = *(const uint4 *)row;
      planes_add<NB>(p[0], x.x);
      planes_add<NB>(p[1], x.y);
      planes_add<NB>(p[2], x.z);
      planes_add<NB>(p[3], x.w);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (w0 + w < nw) planes_add<NB>(p[w], row[w]);
    }
  }
#pragma unroll
  for (int w = 0; w < W; ++w) {
    if (w0 + w >= nw) break;
    const int32_t v = 2 * planes_total<NB>(p[w]) - len;
    const int q = 32 * (w0 + w) + lane;
    if (q >= t) continue;
    int32_t *dst = R + (int64_t)q * stride + at;
    if (add)
      atomicAdd(dst, v);
    else
      *dst = v;
  }
}

template <int W, bool VEC>
__global__ void __launch_bounds__(256) k_rade(HeavyView H, int t, int nw, const int64_t *__restrict__ noff,
                                              const int32_t *__restrict__ nsamp, const uint32_t *__restrict__ sign,
                                              int32_t *R, int64_t stride, unsigned long long *units) {
  const uint32_t nwarps = gridDim.x * 8, nchunks = H.ctl->nchunks;
  unsigned long long scanned = 0;
  for (uint32_t ci = blockIdx.x * 8 + (threadIdx.x >> 5); ci < nchunks; ci += nwarps) {
    const uint2 ch = H.chunks[ci];
    const int32_t u = H.list[ch.x], cu = H.c[ch.x];
    const int first = (int)ch.y * kRadeChunk, len = min(kRadeChunk, cu - first);
    const int32_t *samp = nsamp + noff[u] + first;
    const bool add = cu > kRadeChunk;
    for (int w0 = 0; w0 < nw; w0 += W) {
      if (len <= 32)
        rade_words<W, 1, VEC>(samp, len, nw, w0, t, sign, R, stride, ch.x, add);
      else if (len <= 32 * 7)
        rade_words<W, 3, VEC>(samp, len, nw, w0, t, sign, R, stride, ch.x, add);
      else
        rade_words<W, kRadePlanes, VEC>(samp, len, nw, w0, t, sign, R, stride, ch.x, add);
    }
    scanned += (unsigned long long)len;
  }
  __shared__ unsigned long long s_scanned;
  if (threadIdx.x == 0) s_scanned = 0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && scanned) atomicAdd(&s_scanned, scanned);
  __syncthreads();
  if (threadIdx.x == 0 && s_scanned) atomicAdd(units, s_scanned);
}

// Enqueues R (t rows at `stride`, column = list entry) of H's nodes.
static void rade_enqueue(cen_job *job, const HeavyView &H, int32_t *R, int64_t stride, cudaStream_t run) {
  const int t = job->t, nw = job->nw;
  CEN_CK(cudaMemsetAsync(R, 0, 4 * (size_t)stride * t, run));
  unsigned long long *units = (unsigned long long *)(job->stats.d_units + K_RADE);
  const int grid = sm_count() * 8;
  const int64_t *noff = job->noff.as<int64_t>();
  const int32_t *nsamp = job->nsamp.as<int32_t>();
  const uint32_t *sign = job->sign.as<uint32_t>();
  launch(&job->stats, K_RADE, run, [&] {
    if (nw == 1)
      k_rade<1, false><<<grid, 256, 0, run>>>(H, t, nw, noff, nsamp, sign, R, stride, units);
    else if (nw % 4 == 0 && ((uintptr_t)sign & 15) == 0)  // 16-byte sign loads are aligned
      k_rade<4, true><<<grid, 256, 0, run>>>(H, t, nw, noff, nsamp, sign, R, stride, units);
    else
      k_rade<4, false><<<grid, 256, 0, run>>>(H, t, nw, noff, nsamp, sign, R, stride, units);
  });
}

// ------------------------------------------------------------ radix select
// Per row: prefix/mask of the k-th largest positive value found so far, the
// count still to take (krem) and the sum of values already known to be in.
struct SelRow {
  uint32_t prefix, mask;
  int32_t krem;
  int32_t done;
  long long sum;
};

__global__ void k_sel_init(SelRow *rows, int nrows, int32_t k) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += gridDim.x * blockDim.x)
    rows[r] = SelRow{0u, 0u, k, 0, 0ll};
}

// Histogram of digit `shift` over positive values matching the row's prefix.
__global__ void __launch_bounds__(256) k_sel_hist(const int32_t *__restrict__ vals, int64_t n, int nrows, int shift,
                                                  const SelRow *__restrict__ rows, unsigned int *hcnt,
                                                  unsigned long long *hsum) {
  __shared__ unsigned int sc[256];
  __shared__ unsigned long long ss[256];
  const int r = blockIdx.y;
  const SelRow row = rows[r];
  if (row.done) return;
  sc[threadIdx.x] = 0;
  ss[threadIdx.x] = 0;
  __syncthreads();
  const int32_t *v = vals + (int64_t)r * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = v[i];
    if (x > 0 && ((uint32_t)x & row.mask) == row.prefix) {
      const uint32_t d = ((uint32_t)x >> shift) & 255u;
      atomicAdd(&sc[d], 1u);
      atomicAdd(&ss[d], (unsigned long long)x);
    }
  }
  __syncthreads();
  if (sc[threadIdx.x]) {
    atomicAdd(&hcnt[r * 256 + threadIdx.x], sc[threadIdx.x]);
    atomicAdd(&hsum[r * 256 + threadIdx.x], ss[threadIdx.x]);
  }
}

// One block of 256 threads per row, thread i on digit 255 - i: scans of the
// bucket counts and sums from the top digit down give, for each digit, what
// the buckets above it hold.  Whole buckets are taken while their running
// count stays below krem; the first bucket whose running count reaches krem
// is descended into (its digit joins the prefix).  If every matching value
// fits in krem, all are taken.  Clears the row's buckets for the next digit.
__global__ void __launch_bounds__(256) k_sel_step(int nrows, int shift, SelRow *rows, unsigned int *hcnt,
                                                  unsigned long long *hsum) {
  __shared__ long long wc[8], ws[8];
  const int r = blockIdx.x, i = threadIdx.x, lane = i & 31, w = i >> 5;
  if (r >= nrows) return;
  const SelRow row = rows[r];  // every thread reads it before thread 0 may rewrite it
  if (row.done) return;        // the histogram pass skipped the row: its buckets are zero
  const int d = 255 - i;
  const long long c = (long long)hcnt[r * 256 + d];
  const long long sv = (long long)hsum[r * 256 + d];
  long long ci = c, si = sv;  // inclusive scans over digits 255 .. d
  for (int o = 1; o < 32; o <<= 1) {
    const long long yc = __shfl_up_sync(0xffffffffu, ci, o), ys = __shfl_up_sync(0xffffffffu, si, o);
    if (lane >= o) {
      ci += yc;
      si += ys;
    }
  }
  if (lane == 31) {
    wc[w] = ci;
    ws[w] = si;
  }
  __syncthreads();
  long long total = 0, stotal = 0;
  for (int q = 0; q < 8; ++q) {
    if (q < w) {
      ci += wc[q];
      si += ws[q];
    }
    total += wc[q];
    stotal += ws[q];
  }
  hcnt[r * 256 + d] = 0;
  hsum[r * 256 + d] = 0;
  SelRow out = row;
  if (total <= row.krem) {  // every matching value is in
    if (i != 0) return;
    out.sum += stotal;
    out.krem = 0;
    out.done = 1;
  } else {
    const long long ce = ci - c, se = si - sv;  // the buckets above digit d
    if (!(ci >= row.krem && ce < row.krem)) return;  // not the bucket that reaches krem
    out.krem = row.krem - (int32_t)ce;
    out.sum += se;
    out.prefix |= (uint32_t)d << shift;
    out.mask |= 255u << shift;
    if (shift == 0) {  // prefix is now the exact k-th value; krem copies of it remain
      out.sum += (long long)out.krem * (long long)out.prefix;
      out.krem = 0;
      out.done = 1;
    }
  }
  rows[r] = out;
}

// ---- top-k over the heavy nodes
// A block per row with the row's values in registers: the k-th largest
// positive value by bisection, then the sum.  done = 1 when no unlisted node
// (whose values are below tau) could raise the sum: fewer than k positive
// values need every touched node listed (tau = 1), else the k-th must be at
// least tau - 1.  One launch of some 8 us (barriers of the bisection) in place
// of two per digit: R-MAT 18 0.08 -> 0.008 ms; directed R-MAT 22, t = 100, whose
// rows of 4.2 million were read three times: 1.9 -> 0.008 ms.
constexpr int kTopThreads = 1024, kTopPer = kHeavyMax / kTopThreads;
__global__ void __launch_bounds__(kTopThreads) k_heavy_top(HeavyView H, const int32_t *__restrict__ R, int64_t stride,
                                                           int t, int32_t k, SelRow *rows) {
  __shared__ uint32_t s_cnt[2][32];
  __shared__ unsigned long long s_sum[32];
  const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int32_t count = (int32_t)H.ctl->count, tau = H.ctl->tau;
  const int32_t *row = r < t ? R + (int64_t)r * stride : H.c;
  int32_t v[kTopPer];
  uint32_t most = 0, npos = 0;
#pragma unroll
  for (int i = 0; i < kTopPer; ++i) {
    const int at = i * kTopThreads + tid;
    v[i] = at < count ? max(row[at], 0) : 0;
    most = max(most, (uint32_t)v[i]);
    npos += v[i] > 0;
  }
  most = __reduce_max_sync(0xffffffffu, most);
  npos = __reduce_add_sync(0xffffffffu, npos);
  if (lane == 0) {
    s_cnt[0][wid] = most;
    s_cnt[1][wid] = npos;
  }
  __syncthreads();
  most = __reduce_max_sync(0xffffffffu, s_cnt[0][lane]);
  npos = __reduce_add_sync(0xffffffffu, s_cnt[1][lane]);
  uint32_t kth = 0, above = npos;  // values > kth (kth = 0: every positive value is in)
  if (npos >= (uint32_t)k) {
    uint32_t lo = 1, hi = most;  // the largest value that at least k values reach
    int par = 0;
    while (lo < hi) {
      const uint32_t mid = lo + ((hi - lo + 1) >> 1);
      uint32_t c = 0;
#pragma unroll
      for (int i = 0; i < kTopPer; ++i) c += (uint32_t)v[i] >= mid;
      c = __reduce_add_sync(0xffffffffu, c);
      __syncthreads();  // the last turn's counts have been read
      if (lane == 0) s_cnt[par][wid] = c;
      __syncthreads();
      c = __reduce_add_sync(0xffffffffu, s_cnt[par][lane]);
      par ^= 1;
      if (c >= (uint32_t)k)
        lo = mid;
      else
        hi = mid - 1;
    }
    kth = lo;
  }
  unsigned long long sum = 0;
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < kTopPer; ++i)
    if ((uint32_t)v[i] > kth) {
      sum += (unsigned long long)v[i];
      ++c;
    }
  sum = warp_sum(sum);
  c = __reduce_add_sync(0xffffffffu, c);
  __syncthreads();
  if (lane == 0) {
    s_sum[wid] = sum;
    s_cnt[0][wid] = c;
  }
  __syncthreads();
  if (tid == 0) {
    sum = 0;
    above = 0;
    for (int w = 0; w < 32; ++w) {
      sum += s_sum[w];
      above += s_cnt[0][w];
    }
    if (kth) sum += (unsigned long long)(k - (int32_t)above) * kth;
    rows[r].sum = (long long)sum;
    rows[r].done = tau <= 1 || (kth != 0 && (int32_t)kth >= tau - 1);
  }
}

// Enqueues on `run` the sums of the <= k largest positive entries of each of
// `nrows` rows of length n (select state sized beforehand, see mcera_prepare);
// the per-row results reach hdst (pinned, nrows SelRow) once `run` drains.
static void topk_enqueue(cen_job *job, const int32_t *vals, int64_t n, int nrows, int32_t k, cudaStream_t run,
                         SelRow *hdst, int64_t vmax = INT32_MAX) {
  Stats *S = &job->stats;
  SelRow *rows = job->selst.as<SelRow>();
  unsigned int *hcnt = job->selh.as<unsigned int>();
  unsigned long long *hsum = (unsigned long long *)(hcnt + (size_t)nrows * 256);
  CEN_CK(cudaMemsetAsync(job->selh.p, 0, (size_t)nrows * 256 * 12, run));
  launch(S, K_SELECT, run, [&] { k_sel_init<<<grid_for(nrows, 128), 128, 0, run>>>(rows, nrows, k); });
  const int bx = grid_for((size_t)n, 256 * 8, 512);
  // digits above the highest one a value <= vmax can have are 0 for every
  // value, so their passes would only descend into digit 0
  int top = 24;
  while (top > 0 && (vmax >> top) == 0) top -= 8;
  for (int shift = top; shift >= 0; shift -= 8) {
    launch(S, K_SELECT, run, [&] {
      k_sel_hist<<<dim3(bx, nrows), 256, 0, run>>>(vals, n, nrows, shift, rows, hcnt, hsum);
    });
    launch(S, K_SELECT, run, [&] { k_sel_step<<<nrows, 256, 0, run>>>(nrows, shift, rows, hcnt, hsum); });
  }
  CEN_CK(cudaMemcpyAsync(hdst, rows, sizeof(SelRow) * (size_t)nrows, cudaMemcpyDeviceToHost, run));
}

// Host bytes mcera_enqueue copies into: t + 1 select rows, then b_H.
size_t mcera_result_bytes(const cen_job *job) { return sizeof(SelRow) * (size_t)(job->t + 1) + 8; }

// The list that k_rade takes for R over all nodes (column = node): every node
// with its c_u, and the chunks of every row.  The incidence must be current.
static HeavyView all_nodes(cen_job *job, cudaStream_t st) {
  const int32_t n = job->g->n;
  HeavyCtl *ctl = job->hctl_all.as<HeavyCtl>();
  CEN_CK(cudaMemsetAsync(ctl, 0, offsetof(HeavyCtl, hist), st));
  launch(&job->stats, K_RADE, st, [&] {
    heavy_list_all(job->c.as<int32_t>(), n, ctl, job->hlist_all.as<int32_t>(), job->hc_all.as<int32_t>(),
                   job->hchunks_all.as<uint2>(), st);
  });
  return HeavyView{ctl, job->hlist_all.as<int32_t>(), job->hc_all.as<int32_t>(),
                   job->hchunks_all.as<uint2>()};
}

// Sizes the workspace of R over all nodes (allocations ordered on the job's stream).
static void rade_all_prepare(cen_job *job) {
  cudaStream_t st = job->st;
  const size_t n = (size_t)job->g->n;
  job->R.ensure(4 * n * (job->t + 1), st);
  job->hctl_all.ensure(sizeof(HeavyCtl), st);
  job->hlist_all.ensure(4 * n, st);
  job->hc_all.ensure(4 * n, st);
  job->hchunks_all.ensure(8 * (n + (size_t)job->members / kRadeChunk + 1), st);
}

// R over all nodes into job->R (row t: c), on `run`.
void rade_all(cen_job *job, cudaStream_t run) {
  const int32_t n = job->g->n;
  rade_enqueue(job, all_nodes(job, run), job->R.as<int32_t>(), n, run);
  CEN_CK(cudaMemcpyAsync(job->R.as<int32_t>() + (size_t)n * job->t, job->c.p, 4 * (size_t)n, cudaMemcpyDeviceToDevice,
                         run));
  job->rade_all_m = job->m;
}

// Rows q0 .. q0 + rows - 1 of R (zero before) and, where c is not null, c of samples 0 .. m - 1: a warp per
// sample, its lanes the rows.  For cen_job_copy_rade alone, bound by its atomics.
__global__ void __launch_bounds__(256) k_rade_of_prefix(const int64_t *__restrict__ hoff,
                                                        const int32_t *__restrict__ hmem, uint64_t m, int32_t n,
                                                        int q0, int rows, int nw, const uint32_t *__restrict__ sign,
                                                        int32_t *R, int32_t *c) {
  const int lane = threadIdx.x & 31;
  const uint64_t nwarps = (uint64_t)gridDim.x * 8;
  for (uint64_t j = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5); j < m; j += nwarps) {
    const uint32_t *row = sign + (int64_t)j * nw;
    for (int64_t e = hoff[j]; e < hoff[j + 1]; ++e) {
      const int32_t u = hmem[e];
      for (int r = lane; r < rows; r += 32)
        atomicAdd(&R[(int64_t)r * n + u], (row[(q0 + r) >> 5] >> ((q0 + r) & 31)) & 1u ? 1 : -1);
      if (c && lane == 0) atomicAdd(&c[u], 1);
    }
  }
}

// R and c of the sample that the last AMCERA read (rade_m: the first samples of the store, which may have
// grown), to the host.  Where job->R does not hold them they are summed from the store, as many rows at a
// time as kRadeCopyBytes hold, in buffers of the call's own: the job is only read.
constexpr size_t kRadeCopyBytes = (size_t)256 << 20;
void rade_copy(const cen_job *job, int32_t *R, int32_t *c) {
  cudaStream_t st = job->st;
  const size_t n = (size_t)job->g->n;
  const int t = job->t;
  if (job->rade_all_m == job->rade_m) {
    if (R) CEN_CK(cudaMemcpyAsync(R, job->R.p, 4 * n * t, cudaMemcpyDeviceToHost, st));
    if (c) CEN_CK(cudaMemcpyAsync(c, job->R.as<int32_t>() + n * t, 4 * n, cudaMemcpyDeviceToHost, st));
    CEN_CK(cudaStreamSynchronize(st));
    return;
  }
  if (!R && !c) return;
  const int most = R ? (int)std::max<size_t>(1, std::min<size_t>(t, kRadeCopyBytes / (4 * n))) : 0;
  DevBuf buf;
  buf.ensure_exact(4 * n * (most + 1), st);
  int32_t *dc = buf.as<int32_t>() + n * most;
  for (int q0 = 0; q0 < (R ? t : 1); q0 += std::max(1, most)) {
    const int rows = std::min(most, t - q0);
    CEN_CK(cudaMemsetAsync(buf.p, 0, 4 * n * (most + 1), st));
    if (job->rade_m) {
      k_rade_of_prefix<<<grid_for(job->rade_m, 8), 256, 0, st>>>(job->hoff.as<int64_t>(), job->hmem.as<int32_t>(),
                                                                 job->rade_m, job->g->n, q0, rows, job->nw,
                                                                 job->sign.as<uint32_t>(), buf.as<int32_t>(),
                                                                 c && q0 == 0 ? dc : nullptr);
      CEN_CK(cudaGetLastError());
    }
    if (rows) CEN_CK(cudaMemcpyAsync(R + n * q0, buf.p, 4 * n * rows, cudaMemcpyDeviceToHost, st));
    if (c && q0 == 0) CEN_CK(cudaMemcpyAsync(c, dc, 4 * n, cudaMemcpyDeviceToHost, st));
  }
  CEN_CK(cudaStreamSynchronize(st));
}

// Sizes the AMCERA workspace (allocations ordered on the job's stream).  The
// incidence must be current, and the heavy nodes listed.
void mcera_prepare(cen_job *job, int32_t k) {
  CEN_REQUIRE(k >= 1, CEN_EINVAL, "cen_mcera: k must be >= 1");
  cudaStream_t st = job->st;
  const int nrows = job->t + 1;
  job->selst.ensure(sizeof(SelRow) * (size_t)nrows, st);
  if (k < job->rade_all_k) {
    job->Rh.ensure(4 * (size_t)std::min(job->g->n, kHeavyMax) * job->t, st);
    return;
  }
  rade_all_prepare(job);
  job->selh.ensure((size_t)nrows * 256 * (4 + 8), st);
}

// Enqueues the AMCERA of Alg. 1 on stream `run` (after mcera_prepare): every
// Rnum (rows 0 .. t-1) and Wnum (row t, over c_u), over the heavy nodes or over
// all.  Results reach hdst (pinned, mcera_result_bytes) once `run` drains.
void mcera_enqueue(cen_job *job, int32_t k, cudaStream_t run, void *hdst, bool heavy) {
  const int32_t n = job->g->n;
  const int t = job->t;
  SelRow *hrows = (SelRow *)hdst;
  if (heavy) {
    const HeavyView H = heavy_view(job);
    const int64_t stride = std::min(n, kHeavyMax);
    SelRow *rows = job->selst.as<SelRow>();
    rade_enqueue(job, H, job->Rh.as<int32_t>(), stride, run);
    launch(&job->stats, K_SELECT, run, [&] {
      k_heavy_top<<<t + 1, kTopThreads, 0, run>>>(H, job->Rh.as<int32_t>(), stride, t, k, rows);
    });
    CEN_CK(cudaMemcpyAsync(hrows, rows, sizeof(SelRow) * (size_t)(t + 1), cudaMemcpyDeviceToHost, run));
  } else {
    rade_all(job, run);
    // |R_q^u| <= c_u <= m: every value the select ranks is at most m
    topk_enqueue(job, job->R.as<int32_t>(), n, t + 1, k, run, hrows, (int64_t)job->m);
  }
  if (job->m) CEN_CK(cudaMemcpyAsync(hrows + t + 1, job->bmax.p, 4, cudaMemcpyDeviceToHost, run));  // b_H = 0 if m = 0
}

// Rnum[t], Wnum and b_H from the copied result; false when the heavy nodes did
// not decide every row.
bool mcera_result(cen_job *job, int32_t k, const void *h, int64_t *Rnum, int64_t *Wnum, int32_t *b) {
  const SelRow *hrows = (const SelRow *)h;
  const int t = job->t;
  for (int q = 0; q <= t; ++q)
    if (!hrows[q].done) return false;
  for (int q = 0; q < t; ++q) Rnum[q] = hrows[q].sum;
  *Wnum = hrows[t].sum;  // the c_u are positive, so this is the sum of the k largest
  int hb = 0;
  memcpy(&hb, hrows + t + 1, 4);
  *b = job->m ? hb : 0;
  job->rade_valid_k = k;
  job->rade_m = job->m;
  return true;
}

// The AMCERA over all nodes, on the job's stream.
static void mcera_over_all(cen_job *job, int32_t k, void *h, int64_t *Rnum, int64_t *Wnum, int32_t *b) {
  job->rade_all_k = std::min(job->rade_all_k, k);
  mcera_prepare(job, k);
  mcera_enqueue(job, k, job->st, h, false);
  CEN_CK(cudaStreamSynchronize(job->st));
  CEN_REQUIRE(mcera_result(job, k, h, Rnum, Wnum, b), CEN_ECUDA, "cen_mcera: the select left a row open");
}

// The first such call of a job with at most this many nodes and sign words to
// read (members x words) runs the AMCERA ahead of greedyCover on the job's stream:
// there a second stream costs more to make and give back than it hides, and many
// jobs make one call.  First call and release, one stream and two, us: BA n = 2,000,
// 2,423 words 163 and 168, 9,692 161 and 165, 11,992 166 and 172, 28,771 180 and 172,
// 120,130 213 and 192; R-MAT 14, 9,163 words 187 and 177; BA n = 200,000, 3,760 words 194
// and 187.
constexpr uint64_t kAsideWork = (uint64_t)1 << 14;

// greedyCover on the job's stream and the AMCERA on its second stream at the
// same time: the two read the same incidence and write disjoint buffers, so
// the results are those of greedy_cover followed by mcera.
void cover_and_mcera(cen_job *job, int32_t k, int32_t *S, int32_t *S_size, uint64_t *covered, int64_t *Rnum,
                     int64_t *Wnum, int32_t *b) {
  CEN_REQUIRE(k >= 1, CEN_EINVAL, "cen_cover_and_mcera: k must be >= 1");
  Range range("cen_cover_and_mcera");
  build_incidence(job);
  build_heavy(job);
  greedy_prepare(job, k);
  mcera_prepare(job, k);
  const size_t gb = (greedy_result_bytes(k) + 15) & ~(size_t)15;
  char *h = (char *)host_staging(job, gb + mcera_result_bytes(job));
  if (!job->covered_once && !job->aux.st && k < job->greedy_all_k && k < job->rade_all_k &&
      (uint64_t)job->g->n + (uint64_t)job->members * (uint64_t)job->nw <= kAsideWork) {
    job->covered_once = true;
    mcera_enqueue(job, k, job->st, h + gb, true);
    greedy_enqueue(job, k, job->st, h, true);
    CEN_CK(cudaStreamSynchronize(job->st));
    if (!greedy_result(h, S, S_size, covered)) greedy_over_all(job, k, h, S, S_size, covered);
    if (!mcera_result(job, k, h + gb, Rnum, Wnum, b)) mcera_over_all(job, k, h + gb, Rnum, Wnum, b);
    return;
  }
  job->aux.ensure();
  CEN_CK(cudaEventRecord(job->aux.fork, job->st));
  CEN_CK(cudaStreamWaitEvent(job->aux.st, job->aux.fork, 0));
  greedy_enqueue(job, k, job->st, h, k < job->greedy_all_k);
  try {
    mcera_enqueue(job, k, job->aux.st, h + gb, k < job->rade_all_k);
  } catch (...) {  // still join, so that nothing on the job's stream outruns the second stream
    cudaEventRecord(job->aux.join, job->aux.st);
    cudaStreamWaitEvent(job->st, job->aux.join, 0);
    throw;
  }
  CEN_CK(cudaEventRecord(job->aux.join, job->aux.st));
  CEN_CK(cudaStreamWaitEvent(job->st, job->aux.join, 0));
  CEN_CK(cudaStreamSynchronize(job->st));
  if (!greedy_result(h, S, S_size, covered)) greedy_over_all(job, k, h, S, S_size, covered);
  if (!mcera_result(job, k, h + gb, Rnum, Wnum, b)) mcera_over_all(job, k, h + gb, Rnum, Wnum, b);
}

// ----------------------------------------------- AMCERA of a split sample
// A shard's R (rows 0 .. t-1) and c (row t) over its own samples, into a
// caller's device matrix, and its b_H; the caller sums the shards' matrices
// (R and c are sums over samples) and takes shard_topk of the sum.
void shard_rade(cen_job *job, int32_t *R_out, int32_t *b) {
  build_incidence(job);
  rade_all_prepare(job);
  cudaStream_t st = job->st;
  const int32_t n = job->g->n;
  rade_all(job, st);
  CEN_CK(cudaMemcpyAsync(R_out, job->R.p, 4 * (size_t)n * (job->t + 1), cudaMemcpyDeviceToDevice, st));
  int32_t *h = (int32_t *)host_staging(job, 4);
  *h = 0;
  if (job->m) CEN_CK(cudaMemcpyAsync(h, job->bmax.p, 4, cudaMemcpyDeviceToHost, st));
  CEN_CK(cudaStreamSynchronize(st));
  *b = job->m ? *h : 0;
}

// Sums of the <= k largest positive entries of each of nrows rows of length n
// (the job's graph's n) of a device matrix, with the job's select workspace.
void shard_topk(cen_job *job, const int32_t *vals, int32_t nrows, int32_t k, int64_t *out) {
  CEN_REQUIRE(nrows >= 1 && k >= 1, CEN_EINVAL, "cen_shard_topk: need nrows >= 1 and k >= 1");
  cudaStream_t st = job->st;
  job->selst.ensure(sizeof(SelRow) * (size_t)nrows, st);
  job->selh.ensure((size_t)nrows * 256 * (4 + 8), st);
  SelRow *h = (SelRow *)host_staging(job, sizeof(SelRow) * (size_t)nrows);
  topk_enqueue(job, vals, job->g->n, nrows, k, st, h);
  CEN_CK(cudaStreamSynchronize(st));
  for (int r = 0; r < nrows; ++r) out[r] = h[r].sum;
}

void mcera(cen_job *job, int32_t k, int64_t *Rnum, int64_t *Wnum, int32_t *b) {
  CEN_REQUIRE(k >= 1, CEN_EINVAL, "cen_mcera: k must be >= 1");
  Range range("cen_mcera");
  build_incidence(job);
  build_heavy(job);
  mcera_prepare(job, k);
  void *h = host_staging(job, mcera_result_bytes(job));
  mcera_enqueue(job, k, job->st, h, k < job->rade_all_k);
  CEN_CK(cudaStreamSynchronize(job->st));
  if (!mcera_result(job, k, h, Rnum, Wnum, b)) mcera_over_all(job, k, h, Rnum, Wnum, b);
}

}  // namespace cen

// ---------------------------------------------------------------------------
// Allocation-free top-k positive sums (no counterpart in the paper).
//
// Same kernels as the select inside cen_mcera, but the scratch (per-row
// select state and the 256-bucket count/sum histograms) lives in one
// file-scope __device__ array, so a call allocates no device memory.  Every
// call on a device shares that array; calls that overlap on the GPU race.
namespace cen {

constexpr int kNoAllocMaxRows = 128;
struct NoAllocScratch {
  SelRow rows[kNoAllocMaxRows];
  unsigned int hcnt[kNoAllocMaxRows * 256];
  unsigned long long hsum[kNoAllocMaxRows * 256];
};
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int kNoAllocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static void *g_noalloc_addr[kNoAllocMaxDevices] = {};

// Device address of the array on the current device, looked up once per
// device.  The host-side name is only a stand-in for the symbol.
static NoAllocScratch *noalloc_scratch() {
  int dev = -1;
  CEN_CK(cudaGetDevice(&dev));
  CEN_REQUIRE(dev >= 0 && dev < kNoAllocMaxDevices, CEN_EINVAL, "cen_topk_positive_sum_noalloc: device id too large");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess)
      fail(CEN_ECUDA, std::string("cen_topk_positive_sum_noalloc: cudaGetSymbolAddress failed: ") +
                          cudaGetErrorString(e));
    g_noalloc_addr[dev] = p;
  }
  return static_cast<NoAllocScratch *>(g_noalloc_addr[dev]);
}

}  // namespace cen

extern "C" int cen_topk_positive_sum_noalloc(const int32_t *vals, int64_t n, int32_t nrows, int32_t k, int64_t *out,
                                             void *stream) {
  using namespace cen;
  try {
    CEN_REQUIRE(vals && out, CEN_EINVAL, "cen_topk_positive_sum_noalloc: null argument");
    CEN_REQUIRE(nrows >= 1 && nrows <= kNoAllocMaxRows, CEN_EINVAL,
                "cen_topk_positive_sum_noalloc: nrows must be in [1, 128] (size of the static scratch)");
    CEN_REQUIRE(n >= 0 && k >= 1, CEN_EINVAL, "cen_topk_positive_sum_noalloc: need n >= 0 and k >= 1");
    // the select's bucket counts are 32-bit
    CEN_REQUIRE(n <= INT32_MAX, CEN_EINVAL, "cen_topk_positive_sum_noalloc: rows longer than 2^31 - 1 entries");
    cudaStream_t st = (cudaStream_t)stream;
    NoAllocScratch *sc = noalloc_scratch();
    // the histograms must start at zero; the row states are written by k_sel_init
    CEN_CK(cudaMemsetAsync(sc->hcnt, 0, sizeof(sc->hcnt) + sizeof(sc->hsum), st));
    launch(nullptr, K_SELECT, st, [&] { k_sel_init<<<grid_for(nrows, 128), 128, 0, st>>>(sc->rows, nrows, k); });
    const int bx = grid_for((size_t)(n > 0 ? n : 1), 256 * 8, 512);
    for (int shift = 24; shift >= 0; shift -= 8) {
      launch(nullptr, K_SELECT, st, [&] {
        k_sel_hist<<<dim3(bx, nrows), 256, 0, st>>>(vals, n, nrows, shift, sc->rows, sc->hcnt, sc->hsum);
      });
      launch(nullptr, K_SELECT, st,
             [&] { k_sel_step<<<nrows, 256, 0, st>>>(nrows, shift, sc->rows, sc->hcnt, sc->hsum); });
    }
    SelRow h[kNoAllocMaxRows];
    CEN_CK(cudaMemcpyAsync(h, sc->rows, sizeof(SelRow) * (size_t)nrows, cudaMemcpyDeviceToHost, st));
    CEN_CK(cudaStreamSynchronize(st));
    for (int r = 0; r < nrows; ++r) out[r] = h[r].sum;
    return CEN_OK;
  } catch (const Error &e) {
    set_last_error(e.msg);
    return e.code;
  } catch (...) {
    set_last_error("cen_topk_positive_sum_noalloc: unexpected internal error");
    return CEN_ECUDA;
  }
}
