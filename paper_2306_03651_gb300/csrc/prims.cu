// Generic device primitives of libcen: exclusive scans and a stable LSD radix
// sort of (key, value) pairs; plus error and accounting plumbing.
#include <stdio.h>

#include <cstring>
#include <atomic>
#include <map>
#include <memory>
#include <algorithm>
#include <mutex>
#include <vector>

#include "scan.cuh"

namespace cen {

// ------------------------------------------------------------- errors
static thread_local std::string g_last_error;
void set_last_error(const std::string &msg) { g_last_error = msg; }
const std::string &last_error() { return g_last_error; }
[[noreturn]] void fail(int code, const std::string &msg) { throw Error{code, msg}; }

// --------------------------------------------------------- accounting
const char *const kClassNames[K_COUNT] = {"pairs", "target_check", "expand_push", "expand_pull", "level_finalize",
                                          "cone", "cone_sigma", "walk", "append", "sign", "transpose", "greedy",
                                          "rade", "select", "graph", "misc", "bidir", "space"};

Stats::Stats() {
  memset(k, 0, sizeof(k));
  for (int c = 0; c < K_COUNT; ++c) snprintf(k[c].name, sizeof(k[c].name), "%s", kClassNames[c]);
}
Stats::~Stats() {
  for (auto &p : pending) {
    cudaEventDestroy(p.a);
    cudaEventDestroy(p.b);
  }
  for (auto e : pool) cudaEventDestroy(e);
  if (d_units) dev_free(d_units, sizeof(uint64_t) * K_COUNT, nullptr, d_units_al);
}
void Stats::init(cudaStream_t st) {
  if (!d_units) {
    d_units = (uint64_t *)dev_alloc(sizeof(uint64_t) * K_COUNT, st, &d_units_al);
    CEN_CK(cudaMemsetAsync(d_units, 0, sizeof(uint64_t) * K_COUNT, st));
  }
}
cudaEvent_t Stats::ev() {  // caller holds mu
  if (!pool.empty()) {
    cudaEvent_t e = pool.back();
    pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  CEN_CK(cudaEventCreate(&e));
  return e;
}
void Stats::begin(int cls, cudaStream_t st, cudaEvent_t *a, cudaEvent_t *b) {
  std::lock_guard<std::mutex> lock(mu);
  k[cls].launches++;
  if (!timing) return;
  *a = ev();
  *b = ev();
  CEN_CK(cudaEventRecord(*a, st));
}
void Stats::end(int cls, cudaStream_t st, cudaEvent_t a, cudaEvent_t b) {
  if (!a) return;
  std::lock_guard<std::mutex> lock(mu);
  CEN_CK(cudaEventRecord(b, st));
  pending.push_back({cls, a, b});
}
void Stats::resolve() {
  std::lock_guard<std::mutex> lock(mu);
  for (auto &p : pending) {
    float ms = 0.f;
    CEN_CK(cudaEventElapsedTime(&ms, p.a, p.b));
    k[p.cls].ms += ms;
    k[p.cls].timed++;
    pool.push_back(p.a);
    pool.push_back(p.b);
  }
  pending.clear();
}
void Stats::reset(cudaStream_t st) {
  resolve();
  std::lock_guard<std::mutex> lock(mu);
  for (int c = 0; c < CEN_NKCLASS; ++c) {
    k[c].launches = 0;
    k[c].ms = 0;
    k[c].timed = 0;
    k[c].units = 0;
  }
  if (d_units) CEN_CK(cudaMemsetAsync(d_units, 0, sizeof(uint64_t) * K_COUNT, st));
}

// ------------------------------------------------------ fault hook
static std::atomic<long long> g_fail_alloc{0};
void alloc_fault_tick() {
  if (g_fail_alloc.load(std::memory_order_relaxed) <= 0) return;
  if (g_fail_alloc.fetch_sub(1) == 1) fail(CEN_ENOMEM, "device allocation failed (injected by cen_debug_fail_alloc)");
}

// ------------------------------------------------------ memory source
static std::atomic<const Allocator *> g_allocator{nullptr};

void set_allocator(cen_alloc_fn alloc, cen_free_fn free_fn, void *ctx) {
  static std::mutex mu;
  static std::vector<std::unique_ptr<Allocator>> installed;  // kept for the buffers they made
  std::lock_guard<std::mutex> lk(mu);
  if (!alloc) {
    g_allocator.store(nullptr);
    return;
  }
  installed.emplace_back(new Allocator{alloc, free_fn, ctx});
  g_allocator.store(installed.back().get());
}

void *dev_alloc(size_t bytes, cudaStream_t s, const Allocator **al) {
  alloc_fault_tick();
  const Allocator *a = g_allocator.load();
  void *p = nullptr;
  if (a) {
    p = a->alloc(bytes, (void *)s, a->ctx);
    CEN_REQUIRE(p, CEN_ENOMEM, "device allocation of " + std::to_string(bytes) + " bytes failed (installed allocator)");
  } else {
    CEN_CK(cudaMallocAsync(&p, bytes, s));
  }
  *al = a;
  return p;
}

void dev_free(void *p, size_t bytes, cudaStream_t s, const Allocator *al) noexcept {
  if (!p) return;
  if (al) {
    cudaStreamSynchronize(s);  // the allocator may hand p out again at once
    al->free(p, bytes, (void *)s, al->ctx);
  } else {
    cudaFreeAsync(p, s);
  }
}

// ------------------------------------------------------ occupancy
int sm_count() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int dev = 0;
  CEN_CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  int sms = 0;
  CEN_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  cache[dev] = sms > 0 ? sms : 1;
  return cache[dev];
}

int resident_grid(const void *kernel, int block) {
  static std::mutex mu;
  static std::map<std::pair<int, const void *>, int> cache;
  int dev = 0;
  CEN_CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({dev, kernel});
  if (it != cache.end()) return it->second;
  int sms = 0, per = 0;
  CEN_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CEN_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, block, 0));
  const int g = sms * (per > 0 ? per : 1);
  cache[{dev, kernel}] = g;
  return g;
}

void allow_shared(const void *kernel, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void *>, size_t> done;
  int dev = 0;
  CEN_CK(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  size_t &have = done[{dev, kernel}];
  if (have >= bytes) return;
  CEN_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  CEN_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  have = bytes;
}

// -------------------------------------------------------------- scans
template <class T>
static void exclusive_scan(const T *in, T *out, size_t n, T *d_total, DevBuf &tmp, cudaStream_t st, Stats *S) {
  if (n == 0) {
    if (d_total) CEN_CK(cudaMemsetAsync(d_total, 0, sizeof(T), st));
    return;
  }
  device_scan<T>(ScanArray<T, T>{in}, ScanOffsets<T>{out, d_total, n}, n, tmp, st, S);
}

void exclusive_scan_i64(const int64_t *in, int64_t *out, size_t n, int64_t *d_total, DevBuf &tmp, cudaStream_t st,
                        Stats *S) {
  exclusive_scan<int64_t>(in, out, n, d_total, tmp, st, S);
}

void counts_to_offsets(const int32_t *cnt, int64_t *out, size_t n, DevBuf &tmp, cudaStream_t st, Stats *S) {
  if (n == 0) {
    CEN_CK(cudaMemsetAsync(out, 0, sizeof(int64_t), st));
    return;
  }
  device_scan<int64_t>(ScanArray<int64_t, int32_t>{cnt}, ScanOffsets<int64_t>{out, out + n, n}, n, tmp, st, S);
}

// --------------------------------------------------------- radix sort
// Passes of up to kRsMaxBits key bits.  Pass: per-tile digit histograms
// (digit-major), one exclusive scan over them gives every (digit, tile) its
// output base, and the scatter ranks equal digits inside a tile in input order
// (stable), puts the tile in digit order in shared memory and writes it from
// there, so that a digit's pairs leave in runs of consecutive addresses.  Bound
// by shared-memory latency at 32 warps an SM (0.139 ms a scatter of 16.8 million
// pairs, 1.9 TB/s).  Two passes of 10 bits for ids below 2^20 in place of three of
// 8 that scattered straight from registers: 0.59 -> 0.36 ms for those pairs.  Passes
// of 11 bits leave one block an SM: three of 8 are faster for 2^22 ids (the load of
// directed R-MAT 22 5.0 against 6.1 ms).
constexpr int kRsMaxBits = 10;
constexpr int kRsThreads = 512, kRsRounds = 16, kRsTile = kRsThreads * kRsRounds, kRsWarps = kRsThreads / 32;

__global__ void __launch_bounds__(kRsThreads) rs_hist(const uint32_t *__restrict__ keys, size_t n, int shift, int bits,
                                                      uint32_t *hist, int ntiles) {
  __shared__ uint32_t h[1 << kRsMaxBits];
  const int bins = 1 << bits;
  for (int d = threadIdx.x; d < bins; d += kRsThreads) h[d] = 0;
  __syncthreads();
  const size_t base = (size_t)blockIdx.x * kRsTile;
  auto count = [&](uint32_t k) { atomicAdd(&h[(k >> shift) & (uint32_t)(bins - 1)], 1u); };
  if (base + kRsTile <= n && ((uintptr_t)keys & 15) == 0) {
    const uint4 *k4 = (const uint4 *)(keys + base);
    uint4 x[kRsRounds / 4];
#pragma unroll
    for (int r = 0; r < kRsRounds / 4; ++r) x[r] = k4[r * kRsThreads + threadIdx.x];
#pragma unroll
    for (int r = 0; r < kRsRounds / 4; ++r) {
      count(x[r].x);
      count(x[r].y);
      count(x[r].z);
      count(x[r].w);
    }
  } else {
    for (size_t i = base + threadIdx.x; i < n && i < base + kRsTile; i += kRsThreads) count(keys[i]);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += kRsThreads) hist[(size_t)d * ntiles + blockIdx.x] = h[d];
}

// Dynamic shared memory of rs_scatter for 2^bits digits.
static size_t rs_smem(int bits) { return (size_t)kRsTile * 8 + ((size_t)1 << bits) * (2 * kRsWarps + 8); }

__global__ void __launch_bounds__(kRsThreads, 2) rs_scatter(const uint32_t *__restrict__ kin,
                                                         const uint32_t *__restrict__ vin, uint32_t *kout,
                                                         uint32_t *vout, size_t n, int shift, int bits,
                                                         const uint32_t *__restrict__ hist, int ntiles) {
  extern __shared__ uint32_t rs_sh[];
  const int bins = 1 << bits, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t dmask = (uint32_t)(bins - 1);
  uint32_t *sk = rs_sh, *sv = sk + kRsTile;  // the tile in digit order
  uint32_t *local = sv + kRsTile;            // digit -> its first place in the tile
  uint32_t *gbase = local + bins;            // digit -> its first place in the output, less the former
  uint16_t *wcnt = (uint16_t *)(gbase + bins);  // [warp][digit]: counts, then what the warps before it hold
  __shared__ uint32_t wsum[kRsWarps];
  for (int i = tid; i < bins * kRsWarps / 2; i += kRsThreads) ((uint32_t *)wcnt)[i] = 0;
  __syncthreads();
  // a warp's items are consecutive; equal digits of a round are ranked by lane
  const size_t tile = (size_t)blockIdx.x * kRsTile;
  const int tn = (int)(n - tile < (size_t)kRsTile ? n - tile : (size_t)kRsTile);
  uint32_t k[kRsRounds], rank[kRsRounds / 2];  // two 16-bit ranks a word
  uint16_t *mine = wcnt + (size_t)warp * bins;
#pragma unroll
  for (int r = 0; r < kRsRounds; ++r) {
    const int i = (warp * kRsRounds + r) * 32 + lane;
    k[r] = i < tn ? kin[tile + i] : 0xFFFFFFFFu;
  }
#pragma unroll
  for (int r = 0; r < kRsRounds; ++r) {
    const bool on = (warp * kRsRounds + r) * 32 + lane < tn;
    const uint32_t d = on ? (k[r] >> shift) & dmask : 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const unsigned before = peers & ((1u << lane) - 1u);
    uint32_t old = 0;
    if (on && before == 0) {
      old = mine[d];
      mine[d] = (uint16_t)(old + (uint32_t)__popc(peers));
    }
    __syncwarp();
    const uint32_t at = __shfl_sync(0xffffffffu, old, __ffs(peers) - 1) + (uint32_t)__popc(before);
    rank[r / 2] = r & 1 ? rank[r / 2] | (at << 16) : at;
  }
  __syncthreads();
  // each digit's warps in turn, two digits (16 bits each) a word, then the digits
  const int words = bins / 2, P = (words + kRsThreads - 1) / kRsThreads;
  constexpr int kMaxP = (1 << kRsMaxBits) / 2 / kRsThreads > 0 ? (1 << kRsMaxBits) / 2 / kRsThreads : 1;
  uint32_t tot[kMaxP], sum = 0;
#pragma unroll
  for (int q = 0; q < kMaxP; ++q) {
    const int x = tid * P + q;
    uint32_t acc = 0;
    if (q < P && x < words) {
      uint32_t *p = (uint32_t *)wcnt + x;
#pragma unroll 8
      for (int w = 0; w < kRsWarps; ++w) {
        const uint32_t c = p[w * words];
        p[w * words] = acc;
        acc += c;
      }
    }
    tot[q] = acc;
    sum += (acc & 0xFFFFu) + (acc >> 16);
  }
  uint32_t inc = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  uint32_t at = inc - sum;
  for (int w = 0; w < warp; ++w) at += wsum[w];
#pragma unroll
  for (int q = 0; q < kMaxP; ++q) {
    const int x = tid * P + q;
    if (q < P && x < words)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int d = 2 * x + h;
        local[d] = at;
        gbase[d] = hist[(size_t)d * ntiles + blockIdx.x] - at;
        at += h ? tot[q] >> 16 : tot[q] & 0xFFFFu;
      }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRsRounds; ++r) {
    if ((warp * kRsRounds + r) * 32 + lane >= tn) continue;
    const uint32_t d = (k[r] >> shift) & dmask;
    const uint32_t p = local[d] + mine[d] + (r & 1 ? rank[r / 2] >> 16 : rank[r / 2] & 0xFFFFu);
    sk[p] = k[r];
    sv[p] = vin[tile + (warp * kRsRounds + r) * 32 + lane];
  }
  __syncthreads();
  for (int i = tid; i < tn; i += kRsThreads) {
    const uint32_t key = sk[i];
    const uint32_t p = gbase[(key >> shift) & dmask] + (uint32_t)i;
    kout[p] = key;
    vout[p] = sv[i];
  }
}

void radix_sort_pairs(uint32_t *keys, uint32_t *vals, size_t n, int key_bits, DevBuf &k2, DevBuf &v2, DevBuf &hist,
                      DevBuf &tmp, cudaStream_t st, Stats *S) {
  if (n <= 1) return;
  CEN_REQUIRE(n < (1ull << 32), CEN_EINVAL, "radix_sort_pairs: too many elements");
  const int ntiles = (int)((n + kRsTile - 1) / kRsTile);
  const int total_bits = key_bits <= 0 ? 1 : key_bits;  // (a word holds two digits: at least one bit)
  const int passes = (total_bits + kRsMaxBits - 1) / kRsMaxBits, bits = (total_bits + passes - 1) / passes;
  k2.ensure(n * 4, st);
  v2.ensure(n * 4, st);
  hist.ensure((size_t)ntiles * 4 << bits, st);
  allow_shared((const void *)rs_scatter, rs_smem(kRsMaxBits));
  uint32_t *ka = keys, *va = vals, *kb = k2.as<uint32_t>(), *vb = v2.as<uint32_t>();
  for (int p = 0; p < passes; ++p) {
    const int shift = bits * p;
    uint32_t *h = hist.as<uint32_t>();
    launch(S, K_MISC, st, [&] { rs_hist<<<ntiles, kRsThreads, 0, st>>>(ka, n, shift, bits, h, ntiles); });
    exclusive_scan<uint32_t>(h, h, (size_t)ntiles << bits, nullptr, tmp, st, S);
    launch(S, K_MISC, st, [&] {
      rs_scatter<<<ntiles, kRsThreads, rs_smem(bits), st>>>(ka, va, kb, vb, n, shift, bits, h, ntiles);
    });
    std::swap(ka, kb);
    std::swap(va, vb);
  }
  if (ka != keys) {
    CEN_CK(cudaMemcpyAsync(keys, ka, n * 4, cudaMemcpyDeviceToDevice, st));
    CEN_CK(cudaMemcpyAsync(vals, va, n * 4, cudaMemcpyDeviceToDevice, st));
  }
}

}  // namespace cen

extern "C" int cen_debug_fail_alloc(int64_t n) {
  if (n < 0) {
    cen::set_last_error("cen_debug_fail_alloc: n must be >= 0");
    return CEN_EINVAL;
  }
  cen::g_fail_alloc.store(n);
  return CEN_OK;
}

namespace cen {
// Stream-ordered frees return memory to the device's default pool; with the
// release threshold at its maximum the pool keeps it mapped for the next
// allocation instead of handing it back at every synchronisation.  Once per
// device; cen_release_cached trims the pool.
void keep_pool_memory() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t thr = ~0ull;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
  }
  done[dev] = true;
}
}  // namespace cen

namespace cen {
int cooperative_grid(const void *kernel, int block) {
  int dev = 0, coop = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0) != cudaSuccess || per_sm < 1) return 0;
  return sms * std::min(per_sm, 2);
}
}  // namespace cen

namespace cen {
// Pinned host buffers of finished jobs, kept for the next ones: allocating and
// freeing page-locked memory costs far more than a round's small copies.
namespace {
constexpr size_t kPinnedKeep = 16;
struct PinnedPool {
  std::mutex mu;
  std::vector<std::pair<void *, size_t>> idle;
};
PinnedPool &pinned_pool() {
  static PinnedPool *p = new PinnedPool();  // never destroyed: nothing is freed after the runtime unloads
  return *p;
}
}  // namespace

void *pinned_take(size_t bytes, size_t *cap) {
  {
    PinnedPool &pp = pinned_pool();
    std::lock_guard<std::mutex> lk(pp.mu);
    size_t best = pp.idle.size();
    for (size_t i = 0; i < pp.idle.size(); ++i)
      if (pp.idle[i].second >= bytes && (best == pp.idle.size() || pp.idle[i].second < pp.idle[best].second)) best = i;
    if (best < pp.idle.size()) {
      void *p = pp.idle[best].first;
      *cap = pp.idle[best].second;
      pp.idle.erase(pp.idle.begin() + (ptrdiff_t)best);
      return p;
    }
  }
  size_t c = 4096;
  while (c < bytes) c *= 2;
  void *p = nullptr;
  CEN_CK(cudaMallocHost(&p, c));
  *cap = c;
  return p;
}

void pinned_give(void *p, size_t cap) {
  if (!p) return;
  PinnedPool &pp = pinned_pool();
  std::lock_guard<std::mutex> lk(pp.mu);
  pp.idle.emplace_back(p, cap);
  if (pp.idle.size() > kPinnedKeep) {
    cudaFreeHost(pp.idle.front().first);
    pp.idle.erase(pp.idle.begin());
  }
}

void pinned_drop_cached() {
  PinnedPool &pp = pinned_pool();
  std::lock_guard<std::mutex> lk(pp.mu);
  for (auto &e : pp.idle) cudaFreeHost(e.first);
  pp.idle.clear();
}
}  // namespace cen
