// The heavy nodes of a sample: those in the most samples (included by cover.cu
// and amcera.cu).
//
// greedyCover picks nodes by gain, and a gain is at most the node's c_u;
// R_q^u is at most c_u too.  So both need only the nodes with c_u >= tau as
// long as the smallest gain picked is at least tau and the k-th largest R_q^u
// of every row at least tau - 1: no other node could have been picked, or
// raised a row's sum.  tau is the lowest bound of a c_u bucket that leaves at
// most kHeavyMax nodes (1 when that many nodes or fewer are in a sample at
// all).  Each use checks its condition on the device and reports when it does
// not hold; greedyCover then goes on over all nodes from the picks it has, the
// AMCERA (some 50 us) is repeated over all.  A job's later calls of as large a k go
// over all nodes at once (greedyCover: where less than half of the picks were made).
// Listing costs two passes over c_u (34 us
// for 4.2 million nodes).  Measured over all nodes against the heavy ones: a
// round's greedy and AMCERA on directed R-MAT 22 (t = 100) 3.5 -> 0.4 ms, on the
// rewired grid of 4.2 million nodes 4.4 -> 0.3 ms.
#pragma once
#include "job.cuh"

namespace cen {

constexpr int kHeavyMax = 16384;   // gains of a cluster's shared memory; a block's registers in k_heavy_top
constexpr int kHeavyBuckets = 256 + 23 * 128;  // exact c_u below 256, then 128 steps per power of two
constexpr int kRadeChunk = 2048;   // incidences of one warp in k_rade

struct HeavyCtl {
  int32_t tau;       // c_u of the listed nodes is at least this; 0x7fffffff: too many share one bucket
  uint32_t count;    // listed nodes
  uint32_t nchunks;  // chunks of their incidence rows
  uint32_t pad;
  uint32_t hist[kHeavyBuckets];
};

__device__ __forceinline__ int heavy_bucket(uint32_t c) {
  if (c < 256u) return (int)c;
  const int e = 31 - __clz((int)c);
  return 256 + (e - 8) * 128 + (int)((c >> (e - 7)) & 127u);
}
__device__ __forceinline__ uint32_t heavy_bucket_low(int b) {
  if (b < 256) return (uint32_t)b;
  const int e = 8 + (b - 256) / 128;
  return (1u << e) + ((uint32_t)((b - 256) & 127) << (e - 7));
}

// The list of a job's current sample, or of all its nodes.
struct HeavyView {
  const HeavyCtl *ctl;
  const int32_t *list, *c;  // list entry -> node, its c_u
  const uint2 *chunks;      // (list entry, chunk of its row)
};

// Its control words lie behind the counts c and are cleared with them.
inline size_t heavy_ctl_at(const cen_job *job) { return (4 * (size_t)job->g->n + 15) & ~(size_t)15; }
inline HeavyCtl *heavy_ctl(const cen_job *job) { return (HeavyCtl *)(job->c.as<char>() + heavy_ctl_at(job)); }
HeavyView heavy_view(const cen_job *job);
// The list of all n nodes (entry u = node u) and the chunks of their rows; ctl's head is zero.
void heavy_list_all(const int32_t *c, int32_t n, HeavyCtl *ctl, int32_t *list, int32_t *hc, uint2 *chunks,
                    cudaStream_t st);

}  // namespace cen
