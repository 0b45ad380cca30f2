// Device-wide exclusive scans whose items are computed as they are read and
// whose results go where the caller wants them, so that the passes that made
// the items and moved the offsets are part of the scan.
#pragma once

#include "common.cuh"

namespace cen {

constexpr int kScanThreads = 1024, kScanItems = 4, kScanTile = kScanThreads * kScanItems;
// Up to this many tiles a block sums the tiles before its own itself (all
// blocks together read at most 2^21 sums from L2); more are scanned by a
// kernel of one block in between.
constexpr size_t kScanDirect = 2048;

template <class T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *smem_warp, T *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) smem_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T w = (lane < (int)(blockDim.x >> 5)) ? smem_warp[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < (int)(blockDim.x >> 5)) smem_warp[lane] = w;  // inclusive warp totals
  }
  __syncthreads();
  T before = warp ? smem_warp[warp - 1] : T(0);
  *total = smem_warp[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before + x - v;
}

// Items: T in(size_t i).  Results: out(size_t i, T before, T item).
template <class T, class In>
__global__ void __launch_bounds__(kScanThreads) scan_partials(In in, size_t n, T *part) {
  __shared__ T sw[32];
  const size_t base = (size_t)blockIdx.x * kScanTile + (size_t)threadIdx.x * kScanItems;
  T s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < n) s += in(base + i);
  T tot;
  block_exclusive_scan<T>(s, sw, &tot);
  if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads) scan_top(T *part, size_t nparts) {
  __shared__ T sw[32];
  T carry = 0;
  for (size_t base = 0; base < nparts; base += blockDim.x) {
    const size_t i = base + threadIdx.x;
    const T v = i < nparts ? part[i] : T(0);
    T tot;
    const T ex = block_exclusive_scan<T>(v, sw, &tot);
    if (i < nparts) part[i] = carry + ex;
    carry += tot;
  }
}

// `summed`: part holds each tile's start, else each tile's sum.
template <class T, class In, class Out>
__global__ void __launch_bounds__(kScanThreads) scan_emit(In in, Out out, size_t n, const T *part, bool summed) {
  __shared__ T sw[32];
  const size_t base = (size_t)blockIdx.x * kScanTile + (size_t)threadIdx.x * kScanItems;
  T v[kScanItems], s = 0, start = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < n ? in(base + i) : T(0);
    s += v[i];
  }
  if (summed) {
    start = part[blockIdx.x];
  } else if (blockIdx.x) {
    T mine = 0;
    for (unsigned p = threadIdx.x; p < blockIdx.x; p += kScanThreads) mine += part[p];
    block_exclusive_scan<T>(mine, sw, &start);
  }
  T tot;
  T ex = start + block_exclusive_scan<T>(s, sw, &tot);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < n) out(base + i, ex, v[i]);
    ex += v[i];
  }
}

// Exclusive scan of n items (out may write where in reads: an item is read
// before the block that holds it writes, and a block writes its own items'
// results only).  One launch up to a tile, two up to kScanDirect tiles, else
// three.  Small scans are all launches: one of 2,000 counts took widening,
// sums, starts and offsets (four launches, 9 us with the gaps) and takes one
// of 3 us; one of 2^20 counts 13.9 and now 8.6 us.
template <class T, class In, class Out>
void device_scan(In in, Out out, size_t n, DevBuf &tmp, cudaStream_t st, Stats *S, int cls = K_MISC) {
  if (n == 0) return;
  const size_t nparts = (n + kScanTile - 1) / kScanTile;
  tmp.ensure(nparts * sizeof(T), st);
  T *part = tmp.as<T>();
  if (nparts > 1)
    launch(S, cls, st, [&] { scan_partials<T><<<(unsigned)nparts, kScanThreads, 0, st>>>(in, n, part); });
  if (nparts > kScanDirect) launch(S, cls, st, [&] { scan_top<T><<<1, kScanThreads, 0, st>>>(part, nparts); });
  launch(S, cls, st, [&] {
    scan_emit<T><<<(unsigned)nparts, kScanThreads, 0, st>>>(in, out, n, part, nparts > kScanDirect);
  });
}

// Offsets of consecutive runs: out[i] = the items before i; total (may be null) = all of them.
template <class T>
struct ScanOffsets {
  T *out, *total;
  size_t n;
  __device__ void operator()(size_t i, T before, T item) const {
    out[i] = before;
    if (total && i == n - 1) *total = before + item;
  }
};
template <class T, class E>
struct ScanArray {
  const E *p;
  __device__ T operator()(size_t i) const { return (T)p[i]; }
};

}  // namespace cen
