// Searches of the bidirectional sampler that live in shared memory (included
// by bidir.cu).  A CTA searches one sample.  Its node table, ball queues, path
// counts and a log of the shortest-path arcs are all in shared memory, so the
// phases after discovery touch no global memory but the arena:
//
//   - discovery logs every arc from a ball level to the next one (tail and
//     head as table positions) and, on the level that touches the other ball,
//     every crossing arc; arcs out of s and into t are not logged (every
//     level-1 node has exactly one);
//   - the path counts sigma_s are sums along the logged arcs, level by level:
//     up the forward ball, over the crossing arcs, down the backward ball.
//     Backward-ball nodes off every shortest path keep the count 0, so no cone
//     needs to be cut;
//   - a step of the walk picks among the logged arcs into the current node,
//     by the running count over ascending tail ids: the rule, and the draw,
//     of the scan of the node's sorted in-row.
//
// Why: with the tables in global memory a search of an R-MAT 18 pair took 181k
// cycles, 73k of them discovery and 108k the cone, counts and walk, whose few
// hundred arcs cost chains of dependent L2 accesses.  Here it takes 57k, 43k of
// them discovery.  Most of a search's arcs (some 5,000 of 6,500) are in its
// last level, where nothing needs to be claimed once the balls are known to
// touch: such a level is scanned against a filter of the other frontier, one
// shared load and some ten instructions an arc (1.4 ms instead of 4.2 ms for
// 65,536 pairs with table lookups and claims there).
//
// The counts are 32 bits with the wrap detected.  A search that outgrows the
// table, the log, the levels or the counts is handed on before it has written
// anything but the pair (a count that wraps is found before the distance is
// written): its id goes to the launch's output list.
#pragma once

constexpr int32_t kLogMaxNodes = 1 << 24; // entries hold 24-bit node ids
constexpr uint32_t kLogMaxArcs = 1u << 24;  // a level of this many arcs is always handed on
constexpr int kPickBits = 6;              // id digit of a walk step among many candidates

// Whether 2, 3, 5 and 7 are all of h's prime factors.
constexpr bool log_smooth(int h) {
  for (int f : {2, 3, 5, 7})
    while (h % f == 0) h /= f;
  return h == 1;
}

// T threads; H table entries; NQ nodes (both balls); LQ logged arcs; LV levels per side; a level
// of more than ARCS arcs is handed on; CTAS resident CTAs per SM.
template <int T_, int H_, int NQ_, int LQ_, int LV_, int ARCS_, int CTAS_>
struct LogCfg {
  static constexpr int T = T_, H = H_, NQ = NQ_, LQ = LQ_, ARCS = ARCS_, CTAS = CTAS_;
  static constexpr int LV = LV_;  // levels per side
  static constexpr bool WIDE = T_ == 512;
  static constexpr int U = T_ > 128 ? 4 : 1;  // arcs of a lane per turn of the filtered scan
  static constexpr int FLOG = T_ > 256 ? 17 : T_ > 128 ? 16 : 15, FW = 1 << (FLOG - 5);  // bits and words of the frontier filter
  static_assert(4 * FW + 14 * T_ <= 4 * H_, "the filter and the rows share the counts' memory");
  static_assert(ARCS_ < (1 << 24) && T_ <= 1024, "level costs saturate above the limit");
  static_assert(H_ % 4 == 0 && H_ <= 65536 && NQ_ + T_ < H_, "positions take 16 bits and the table never fills");
  static_assert((T_ & (T_ - 1)) == 0, "the row search halves T");
  static_assert(LV <= 62, "a level takes 6 bits of an entry");
};

// The three sizes of shared-memory search.  Measured (R-MAT 18, 65,536 pairs,
// against 5.33 ms with the tables in global memory): small 1.34 ms for all but
// 3% of the searches, wide 0.42 ms for all of those.  The small one is bound by
// instruction issue and the latency of short phases: 10 CTAs of 128 threads per
// SM took 1.38 ms, 9 took 1.44 and 7 (with a table of 2,048 entries) 1.68;
// 64-thread CTAs 1.57.  A level of more than 65,536 arcs goes to a wide CTA: at
// 32,768 the small launch falls to 1.19 ms and the wide one rises to 0.61.
// Nodes and logged arcs: the small one with 700 and 1,100 hands more on (the
// batch's wide launches 2.3 -> 5.8 ms); the wide one with 5,600 and 8,192 left
// a few R-MAT 18 searches to a huge one, 0.10 ms and a host synchronisation;
// the huge one with 14,000 and 19,400 is slower on directed R-MAT 22 (0.25 ->
// 0.38 ms), where one that does not fit either is searched longer in vain.
// Levels: as many as an entry's 6 bits and, in the small one, the memory of 10 CTAs
// hold (with 60, 9 CTAs fit: R-MAT rounds 5% slower).  With 32 a cycle of 150 nodes,
// whose searches have 38 levels of two nodes, took 3.9 ms a round of 3,000 pairs, all
// but the levels' number fitting, against 1.24 in global memory; now 0.69.
using LogSmall = LogCfg<128, 1536, 1100, 1344, 56, 65536, 10>;
using LogWide = LogCfg<512, 7168, 6400, 10000, 62, (1 << 24) - 1, 2>;
using LogHuge = LogCfg<1024, 15360, 12288, 18432, 62, (1 << 24) - 1, 1>;

template <class C>
struct LogSh {
  uint32_t tab[C::H];  // node 24 | side 1 (bit 6) | level + 1 (6 bits); 0: free
  union {
    uint32_t sig[C::H];  // path counts by table position (after discovery)
    struct {             // discovery
      uint32_t filt[C::FW];       // two bits for each node of the other side's frontier
      const int32_t *rbeg[C::T];  // the rows being scanned: first arc,
      uint32_t rend[C::T];        // end among their arcs,
      uint16_t rpos[C::T];        // table position
    } sc;
  };
  uint32_t log[C::LQ];   // scanned node's position << 16 | neighbour's position
  uint16_t q[C::NQ];   // table positions: side 0 from the front, side 1 from the back
  uint32_t cand[32], cval[32];  // walk candidates: position, count
  uint32_t hist[1 << kPickBits];
  int lo[2][C::LV + 1];  // level L of side x: queue entries lo[x][L] .. lo[x][L+1]
  int seg[2][C::LV];     // arcs logged from level L of side x: seg .. sege
  int sege[2][C::LV];
  int32_t path[2 * C::LV];
  uint32_t fc[2];               // arcs out of the two frontiers (saturated)
  int lvl[2];
  int added, nlog, logged, nodes;
  int stop;                     // 1: the balls touched, 2: table or queue full, 4: log full
  int ovf;                      // a path count wrapped
  uint32_t ps, pt;              // table positions of s and t
  uint32_t item[2], skip[2], none;
  uint32_t red[C::T / 32];
  unsigned long long arcs;
};

// The entry tried after entry p for a node: one of eight strides by the node's
// hash, so that runs of entries do not grow into one another as they do when
// every node steps by one (a search fills its table to 0.7 or more before it
// hands on, and a warp waits for its longest probe).  The strides are 1 mod
// 210, so each passes through every entry of a table whose size has no prime
// factor above 7.  65,536 pairs, small CTAs: R-MAT 18 1.41 -> 1.34 ms, directed
// R-MAT 22 1.41 -> 0.93 ms.
template <int H>
__device__ __forceinline__ uint32_t log_next(uint32_t p, uint32_t node) {
  static_assert(H > 1 + 210 * 7 && log_smooth(H), "every stride is below H and prime to it");
  p += 1u + 210u * (((node * 0x9E3779B1u) >> 12) & 7u);
  return p >= (uint32_t)H ? p - (uint32_t)H : p;
}

// One step of the walk: among n entries, val(i) the path count that entry i
// contributes (0: not a candidate) and pos(i) its node's table position, the
// node whose running count over ascending ids first exceeds r; its position,
// or ~0u if there is none.  At most 32 candidates are ranked by id directly;
// more are first narrowed by histograms of the counts over id digits, from the
// top (kPickBits at a time).  Called by one warp.
template <class C, class V, class PF>
__device__ __forceinline__ uint32_t log_pick(LogSh<C> &S, int n, uint32_t r, int32_t nodes, V &&val, PF &&pos) {
  const int lane = threadIdx.x & 31;
  int shift = 32 - __clz(nodes - 1);  // ids whose bits from `shift` up are `top` are still candidates
  uint32_t top = 0;
  for (;;) {
    int cnt = 0;
    for (int b = 0; b < n; b += 32) {
      const int i = b + lane;
      uint32_t v = 0, p = 0;
      if (i < n) {
        v = val(i);
        p = pos(i);
        if (((S.tab[p] >> 8) >> shift) != top) v = 0;
      }
      const unsigned m = __ballot_sync(0xffffffffu, v != 0);
      const int at = cnt + __popc(m & ((1u << lane) - 1u));
      if (v != 0 && at < 32) {
        S.cand[at] = p;
        S.cval[at] = v;
      }
      cnt += __popc(m);
      if (cnt > 32) break;
    }
    __syncwarp();
    if (cnt <= 32 || shift == 0) {
      const uint32_t p = lane < cnt ? S.cand[lane] : 0u;
      const uint32_t v = lane < cnt ? S.cval[lane] : 0u;
      const uint32_t id = S.tab[p] >> 8;
      uint32_t pre = 0;  // counts of the candidates with smaller ids
      for (int k = 0; k < cnt; ++k) {
        const uint32_t ik = __shfl_sync(0xffffffffu, id, k), vk = __shfl_sync(0xffffffffu, v, k);
        if (ik < id) pre += vk;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, v != 0 && pre <= r && r - pre < v);
      __syncwarp();
      return hit ? __shfl_sync(0xffffffffu, p, __ffs(hit) - 1) : ~0u;
    }
    const int w = shift < kPickBits ? shift : kPickBits;
    shift -= w;
    for (int k = lane; k < (1 << kPickBits); k += 32) S.hist[k] = 0;
    __syncwarp();
#pragma unroll 4
    for (int i = lane; i < n; i += 32) {
      const uint32_t v = val(i), id = S.tab[pos(i)] >> 8;
      if (v != 0 && (id >> (shift + w)) == top) atomicAdd(&S.hist[(id >> shift) & ((1u << w) - 1u)], v);
    }
    __syncwarp();
    static_assert(kPickBits == 6, "two buckets per lane");
    const uint32_t h0 = S.hist[2 * lane], h1 = S.hist[2 * lane + 1];
    uint32_t inc = h0 + h1;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    const unsigned over = __ballot_sync(0xffffffffu, inc > r);
    if (!over) return ~0u;
    const int src = __ffs(over) - 1;
    const uint32_t before = __shfl_sync(0xffffffffu, inc - h0 - h1, src);
    const uint32_t b0 = __shfl_sync(0xffffffffu, h0, src);
    const uint32_t second = r - before >= b0 ? 1u : 0u;
    r -= before + (second ? b0 : 0u);
    top = (top << w) | (2u * (uint32_t)src + second);
    __syncwarp();
  }
}

// Searches sample jr; returns false when it is handed on.  S.tab is zero.
// Called by the whole CTA.
template <class C>
__device__ __forceinline__ bool log_search(const BiArgs &A, LogSh<C> &S, uint64_t jr, int QC) {
  constexpr int T = C::T, H = C::H;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint64_t j = A.j0 + jr;
  uint32_t *const sig = S.sig, *const log = S.log;
  // side x's queue entry i
  auto qat = [&](int x, int i) -> uint16_t & { return S.q[x ? C::NQ - 1 - i : i]; };
  if (tid < 32) {
    // Sec. 5: s uniform over V; t uniform over V \ {s} (Sec. 3.1 pairs u != v); lane 0 draws s, lane 1 t
    int32_t draw = 0;
    if (lane < 2)
      draw = (int32_t)uniform_below64(A.key.seed, A.key.id(j), lane ? kPurposeT : kPurposeS, (uint64_t)(A.n - lane));
    const int32_t s = __shfl_sync(0xffffffffu, draw, 0);
    const int32_t tt = __shfl_sync(0xffffffffu, draw, 1);
    const int32_t t = tt + (tt >= s);
    if (lane < 2) {
      const int32_t v = lane ? t : s;
      const int64_t *o = lane ? A.roff : A.off;
      const unsigned long long deg = (unsigned long long)(o[v + 1] - o[v]);
      (lane ? A.pt : A.ps)[j] = v;
      S.fc[lane] = deg > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)deg;
      S.lo[lane][0] = 0;
      S.lo[lane][1] = 1;
      S.lvl[lane] = 0;
    }
    if (lane == 0) {
      const uint32_t p = __umulhi((uint32_t)s * 0x9E3779B1u, (uint32_t)H);
      uint32_t p2 = __umulhi((uint32_t)t * 0x9E3779B1u, (uint32_t)H);
      if (p2 == p) p2 = log_next<H>(p, (uint32_t)t);
      S.tab[p] = ((uint32_t)s << 8) | 1u;
      S.tab[p2] = ((uint32_t)t << 8) | 64u | 1u;
      qat(0, 0) = (uint16_t)p;
      qat(1, 0) = (uint16_t)p2;
      S.ps = p;
      S.pt = p2;
      S.nodes = 2;
      S.added = S.nlog = S.logged = S.stop = S.ovf = 0;
      S.arcs = 0;
    }
  }
  __syncthreads();

  // ---- discovery: grow the cheaper side (on a tie the shallower) until the
  // balls touch; the level that touches is scanned to its end
  int x, L;
  for (;;) {
    const uint32_t c0 = S.fc[0], c1 = S.fc[1];
    x = c0 < c1 || (c0 == c1 && S.lvl[0] <= S.lvl[1]) ? 0 : 1;
    L = S.lvl[x];
    const uint32_t fcost = x ? c1 : c0;
    if (L + 1 >= C::LV || fcost > (uint32_t)C::ARCS) return false;
    const int f0 = S.lo[x][L], f1 = S.lo[x][L + 1], base = S.nodes;
    const int64_t *__restrict__ o = x ? A.roff : A.off;
    const int32_t *__restrict__ c = x ? A.rcol : A.col;
    const uint32_t code = ((uint32_t)x << 6) | (uint32_t)(L + 2);  // side and level + 1 of the next level
    // The arc from position pv to node w (none when w < 0).  Called by a whole warp.
    auto visit = [&](uint32_t pv, int w) {
      const int stop = *(volatile int *)&S.stop;  // nothing more is claimed once it is set
      uint32_t p = __umulhi((uint32_t)w * 0x9E3779B1u, (uint32_t)H), e = 0;
      bool claimed = false;
      if (w >= 0) {
        for (;;) {
          e = *(volatile uint32_t *)&S.tab[p];
          if (e == 0) {
            if (stop) break;
            e = atomicCAS(&S.tab[p], 0u, ((uint32_t)w << 8) | code);
            claimed = e == 0;
            if (claimed) break;
          }
          if ((e >> 8) == (uint32_t)w) break;
          p = log_next<H>(p, (uint32_t)w);
        }
      }
      __syncwarp();
      const bool cross = e != 0 && (int)((e >> 6) & 1u) != x;  // an arc between the balls
      const bool child = claimed || (!stop && e != 0 && (e & 127u) == code);
      if (!__any_sync(0xffffffffu, claimed || cross || (child && L > 0))) return;
      const unsigned below = (1u << lane) - 1u;
      const unsigned cm = __ballot_sync(0xffffffffu, claimed);
      if (cm) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&S.added, __popc(cm));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(cm & below);
        if (claimed) {
          if (base + at < C::NQ && f1 + at < QC)
            qat(x, f1 + at) = (uint16_t)p;
          else
            atomicOr(&S.stop, 2);
        }
      }
      const bool keep = cross || (child && L > 0);
      const unsigned km = __ballot_sync(0xffffffffu, keep);
      if (km) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&S.nlog, __popc(km));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(km & below);
        if (keep) {
          if (at < C::LQ)
            log[at] = (pv << 16) | p;
          else
            atomicOr(&S.stop, 4);
          if (cross && !(stop & 1)) atomicOr(&S.stop, 1);
        }
      }
      __syncwarp();
    };
    // The rows' arcs, each given to f with its row's position.  The rows are taken T at a time.  A scan of their lengths deals the arcs
    // out: each warp gets an equal run of them, its lanes interleaved, and a
    // lane steps from row to row as it goes.  Every lane of a warp makes the
    // same number of turns and the warp comes together after each probe.
    auto scan = [&](auto per_turn, auto &&f) {
    constexpr int U = decltype(per_turn)::value;  // arcs of a lane per turn
    for (int r0 = f0; r0 < f1; r0 += T) {
      uint32_t len = 0;
      if (r0 + tid < f1) {
        const uint32_t pv = qat(x, r0 + tid);
        const uint32_t v = S.tab[pv < (uint32_t)H ? pv : 0u] >> 8;
        int64_t e0 = 0;
        if (v < (uint32_t)A.n) {
          e0 = o[v];
          len = (uint32_t)(o[v + 1] - e0);
        } else {
          atomicExch(&A.ctl->err, CEN_EINVAL);  // cannot happen
        }
        S.sc.rpos[tid] = (uint16_t)pv;
        S.sc.rbeg[tid] = c + e0;
      }
      uint32_t inc = len;
      for (int k = 1; k < 32; k <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, k);
        if (lane >= k) inc += y;
      }
      if (lane == 31) S.red[tid >> 5] = inc;
      __syncthreads();
      uint32_t before = 0, total = 0;
#pragma unroll
      for (int k = 0; k < T / 32; ++k) {
        const uint32_t y = S.red[k];
        before += k < (tid >> 5) ? y : 0u;
        total += y;
      }
      S.sc.rend[tid] = before + inc;
      __syncthreads();
      const uint32_t share = (total + T - 1) / T * 32;  // arcs of each warp
      const uint32_t a0 = (uint32_t)(tid >> 5) * share, a1 = min(total, a0 + share);
      if (a0 < a1) {
        uint32_t a = a0 + lane;
        int row = 0;  // the row of arc a: the first that ends beyond it
        for (int step = T / 2; step; step >>= 1)
          if (S.sc.rend[row + step - 1] <= min(a, a1 - 1)) row += step;
        uint32_t end = S.sc.rend[row];
        const int32_t *at = S.sc.rbeg[row] - (row ? S.sc.rend[row - 1] : 0u);
        uint32_t pv = S.sc.rpos[row];
        auto next = [&](uint32_t &pos) {  // the lane's next arc: its head, or -1
          int w = -1;
          if (a < a1) {
            if (a >= end) {
              uint32_t first;
              do {
                first = end;
                end = S.sc.rend[++row];
              } while (a >= end);
              at = S.sc.rbeg[row] - first;
              pv = S.sc.rpos[row];
            }
            w = at[a];
          }
          pos = pv;
          a += 32;
          return w;
        };
        if constexpr (U == 1) {
          uint32_t p0;
          int w0 = next(p0);
          for (uint32_t b = a0; b < a1; b += 32) {
            uint32_t p1;
            const int w1 = next(p1);  // loaded before the arc at hand is looked up
            f(p0, w0);
            p0 = p1;
            w0 = w1;
          }
        } else {
          for (uint32_t b = a0; b < a1; b += 32 * U) {
            uint32_t ps[U];
            int ws[U];
#pragma unroll
            for (int u = 0; u < U; ++u) ws[u] = next(ps[u]);
            f(ps, ws);
          }
        }
      }
      __syncthreads();
    }
    };
    // A level that probably touches the other ball (the expected number of
    // crossing arcs, were arcs to fall at random, is 1/2 or more) is first
    // scanned for crossing arcs alone: nothing is claimed, and a filter of the
    // other frontier's nodes spares most arcs the table.
    bool met = false;
    if (fcost >= 256 && (float)fcost * (float)(x ? c0 : c1) >= 0.5f * (float)A.nnz) {
      uint4 *f4 = (uint4 *)S.sc.filt;
      for (int i = tid; i < C::FW / 4; i += T) f4[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
      const int L2 = S.lvl[x ^ 1], g1 = S.lo[x ^ 1][L2 + 1];
      for (int i = S.lo[x ^ 1][L2] + tid; i < g1; i += T) {
        const uint32_t h = (S.tab[qat(x ^ 1, i)] >> 8) * 0x9E3779B1u;
        const uint32_t i1 = h >> (32 - C::FLOG), i2 = (h >> 2) & ((1u << C::FLOG) - 1u);
        atomicOr(&S.sc.filt[i1 >> 5], 1u << (i1 & 31u));
        atomicOr(&S.sc.filt[i2 >> 5], 1u << (i2 & 31u));
      }
      scan(std::integral_constant<int, C::U>(), [&](auto ps_, auto ws_) {  // (its first barrier completes the filter)
        uint32_t ps[C::U];
        int ws[C::U];
        if constexpr (C::U == 1) {
          ps[0] = ps_;
          ws[0] = ws_;
        } else {
#pragma unroll
          for (int u = 0; u < C::U; ++u) {
            ps[u] = ps_[u];
            ws[u] = ws_[u];
          }
        }
        unsigned in = 0;
#pragma unroll
        for (int u = 0; u < C::U; ++u) {
          const uint32_t i1 = ((uint32_t)ws[u] * 0x9E3779B1u) >> (32 - C::FLOG);
          if (ws[u] >= 0 && ((S.sc.filt[i1 >> 5] >> (i1 & 31u)) & 1u)) in |= 1u << u;
        }
        if (!__any_sync(0xffffffffu, in != 0)) return;
#pragma unroll
        for (int u = 0; u < C::U; ++u) {
          if (!__any_sync(0xffffffffu, (in >> u) & 1u)) continue;
          const uint32_t h = (uint32_t)ws[u] * 0x9E3779B1u;
          const uint32_t i2 = (h >> 2) & ((1u << C::FLOG) - 1u);
          uint32_t p = __umulhi(h, (uint32_t)H);
          bool cross = false;
          if (((in >> u) & 1u) && ((S.sc.filt[i2 >> 5] >> (i2 & 31u)) & 1u)) {
            for (;;) {
              const uint32_t e = S.tab[p];
              if (e == 0) break;
              if ((e >> 8) == (uint32_t)ws[u]) {
                cross = (int)((e >> 6) & 1u) != x;
                break;
              }
              p = log_next<H>(p, (uint32_t)ws[u]);
            }
          }
          __syncwarp();
          const unsigned km = __ballot_sync(0xffffffffu, cross);
          if (!km) continue;
          int at = 0;
          if (lane == 0) {
            at = atomicAdd(&S.nlog, __popc(km));
            atomicOr(&S.stop, at + __popc(km) > C::LQ ? 5 : 1);
          }
          at = __shfl_sync(0xffffffffu, at, 0) + __popc(km & ((1u << lane) - 1u));
          if (cross && at < C::LQ) log[at] = (ps[u] << 16) | p;
        }
      });
      met = S.stop != 0;
      if (tid == 0) S.arcs += fcost;
      __syncthreads();
    }
    if (!met) scan(std::integral_constant<int, 1>(), visit);
    const int stop = S.stop, nadd = S.added;
    if (tid == 0) {
      if (!met) S.arcs += fcost;
      S.seg[x][L] = S.logged;
      S.sege[x][L] = S.logged = S.nlog;
    }
    if ((stop & ~1) && stop != 3) return false;  // without the whole log, or a level cut short
    if (stop & 1) break;
    if (nadd == 0) break;  // this side's ball is closed: t is unreachable
    // arcs out of the new level
    unsigned long long cost = 0;
    for (int i = tid; i < nadd; i += T) {
      const uint32_t v = S.tab[qat(x, f1 + i)] >> 8;
      cost += (unsigned long long)(o[v + 1] - o[v]);
    }
    // (a thread's share saturates above every limit on a level, so that 32 bits hold the sum)
    const uint32_t c32 = __reduce_add_sync(0xffffffffu, cost > kLogMaxArcs ? kLogMaxArcs : (uint32_t)cost);
    if (lane == 0) S.red[tid >> 5] = min(c32, 4u * kLogMaxArcs);
    __syncthreads();
    if (tid == 0) {
      uint32_t tot = 0;
      for (int w = 0; w < T / 32; ++w) tot += S.red[w];
      S.fc[x] = tot;
      S.lo[x][L + 2] = f1 + nadd;
      S.lvl[x] = L + 1;
      S.nodes = base + nadd;
      S.added = 0;
    }
    __syncthreads();
  }
  const bool met = S.stop & 1;  // (else t is unreachable)
  const int ls = S.lvl[0], lb = S.lvl[1];
  const int d = met ? ls + lb + 1 : -1;
  if (d < 2) {  // adjacent or unreachable: the empty hyper-edge
    if (tid == 0) {
      A.pd[j] = d;
      A.aoff[jr] = -1;
    }
    return true;
  }
  // ---- path counts along the logged arcs
  for (int i = tid; i < H / 4; i += T) ((uint4 *)sig)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if (ls == 0) {
    if (tid == 0) sig[S.ps] = 1;
  } else {
    const int f0 = S.lo[0][1], f1 = S.lo[0][2];
    for (int i = f0 + tid; i < f1; i += T) sig[qat(0, i)] = 1;
  }
  __syncthreads();
  for (int l = 1; l < ls; ++l) {
    const int b = S.sege[0][l];
    for (int i = S.seg[0][l] + tid; i < b; i += T) {
      const uint32_t a = log[i], add = sig[a >> 16];
      const uint32_t old = atomicAdd(&sig[a & 0xFFFFu], add);
      if (old + add < old) S.ovf = 1;
    }
    __syncthreads();
  }
  const int cb = S.seg[x][L], ce = S.sege[x][L];
  for (int i = cb + tid; i < ce; i += T) {
    const uint32_t a = log[i], pv = a >> 16, pw = a & 0xFFFFu;
    if ((int)((S.tab[pw] >> 6) & 1u) == x) continue;  // an arc of the level cut short
    const uint32_t add = sig[x ? pw : pv];
    const uint32_t old = atomicAdd(&sig[x ? pv : pw], add);
    if (old + add < old) S.ovf = 1;
  }
  __syncthreads();
  for (int l = lb - 1; l >= 1; --l) {
    const int b = S.sege[1][l];
    for (int i = S.seg[1][l] + tid; i < b; i += T) {
      const uint32_t a = log[i], add = sig[a & 0xFFFFu];
      if (add) {
        const uint32_t old = atomicAdd(&sig[a >> 16], add);
        if (old + add < old) S.ovf = 1;
      }
    }
    __syncthreads();
  }
  if (lb >= 1) {
    const int f0 = S.lo[1][1], f1 = S.lo[1][2];
    for (int i = f0 + tid; i < f1; i += T) {
      const uint32_t add = sig[qat(1, i)];
      if (add) {
        const uint32_t old = atomicAdd(&sig[S.pt], add);
        if (old + add < old) S.ovf = 1;
      }
    }
    __syncthreads();
  }
  if (S.ovf) return false;  // 2^32 paths or more: 64-bit counts
  // ---- the distance, the members' place, and the backward walk from t (one
  // warp), the forward sampler's rule: at v on distance D draw r below sigma_v
  // and take the in-neighbour on D - 1 (ascending id) whose running count
  // first exceeds r
  if (tid < 32) {
    unsigned long long place = 0;
    if (lane == 0) {
      A.pd[j] = d;
      atomicMax(A.bmax, d - 1);
      place = atomicAdd(&A.ctl->cursor, (unsigned long long)(d - 1));
    }
    // the draw of step i, first attempt, by lane i (later attempts and steps as they come)
    uint32_t x0 = 0;
    if (lane < d - 1) x0 = philox_block(A.key.seed, A.key.id(j), kPurposeWalk0 + (uint32_t)lane, 0).x;
    uint32_t pv = S.pt;
    bool bad = false;
    for (int D = d; D >= 2 && !bad; --D) {
      const int step = d - D;
      const uint32_t B = sig[pv];
      uint32_t r;
      {  // uniform_below64 for a 32-bit bound: its mask keeps low bits of the first word only
        const uint32_t mask = B <= 1 ? 0u : 0xFFFFFFFFu >> __clz((int)(B - 1));
        uint32_t w = step < 32 ? __shfl_sync(0xffffffffu, x0, step)
                               : philox_block(A.key.seed, A.key.id(j), kPurposeWalk0 + (uint32_t)step, 0).x;
        for (uint32_t a = 1; (r = w & mask) >= B; ++a) {
          if (B == 0) break;
          w = philox_block(A.key.seed, A.key.id(j), kPurposeWalk0 + (uint32_t)step, a).x;
        }
      }
      uint32_t pu = ~0u;
      // where the candidates are: a run of the log, or of the queue (from t)
      const bool from_t = D == d && lb >= 1;
      const int b = from_t ? S.lo[1][1] : D > ls + 1 ? S.seg[1][d - D] : D == ls + 1 ? cb : S.seg[0][D - 1];
      const int n = (from_t ? S.lo[1][2] : D > ls + 1 ? S.sege[1][d - D] : D == ls + 1 ? ce : S.sege[0][D - 1]) - b;
      int64_t e0 = 0, e1 = n;
      if (n > 256 && !from_t) {
        const uint32_t v = S.tab[pv] >> 8;
        e0 = A.roff[v];
        e1 = A.roff[v + 1];
      }
      if (e1 - e0 < n / 2) {  // the node's row is shorter than the run: scan it, looking its nodes up
        const uint32_t want = D - 1 <= ls ? (uint32_t)D : 64u | (uint32_t)(d - D + 2);  // side and level + 1
        uint32_t cum = 0;
        for (int64_t base = e0; base < e1 && pu == ~0u; base += 32) {
          uint32_t p = 0, val = 0;
          if (base + lane < e1) {
            const uint32_t u = (uint32_t)A.rcol[base + lane];
            p = __umulhi(u * 0x9E3779B1u, (uint32_t)H);
            for (;;) {
              const uint32_t e = S.tab[p];
              if (e == 0) break;
              if ((e >> 8) == u) {
                if ((e & 127u) == want) val = sig[p];
                break;
              }
              p = log_next<H>(p, u);
            }
          }
          __syncwarp();
          uint32_t pre = val;
          for (int k = 1; k < 32; k <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, pre, k);
            if (lane >= k) pre += y;
          }
          const unsigned hit = __ballot_sync(0xffffffffu, val != 0 && cum + pre > r);
          if (hit) pu = __shfl_sync(0xffffffffu, p, __ffs(hit) - 1);
          cum += __shfl_sync(0xffffffffu, pre, 31);
        }
      } else if (from_t) {  // all of side 1's first level
        pu = log_pick<C>(
            S, n, r, A.n, [&](int i) { return sig[qat(1, b + i)]; }, [&](int i) { return (uint32_t)qat(1, b + i); });
      } else if (D > ls + 1) {  // backward ball: v on its level d - D
        pu = log_pick<C>(
            S, n, r, A.n, [&](int i) { return (log[b + i] >> 16) == pv ? sig[log[b + i] & 0xFFFFu] : 0u; },
            [&](int i) { return log[b + i] & 0xFFFFu; });
      } else if (D == ls + 1) {  // over the crossing arcs
        const int hs = x ? 16 : 0;  // where the head is
        pu = log_pick<C>(
            S, n, r, A.n,
            [&](int i) {
              const uint32_t a = log[b + i];
              return ((a >> hs) & 0xFFFFu) == pv && (int)((S.tab[a & 0xFFFFu] >> 6) & 1u) != x
                         ? sig[(a >> (16 - hs)) & 0xFFFFu]
                         : 0u;
            },
            [&](int i) { return (log[b + i] >> (16 - hs)) & 0xFFFFu; });
      } else {  // forward ball: v on level D
        pu = log_pick<C>(
            S, n, r, A.n, [&](int i) { return (log[b + i] & 0xFFFFu) == pv ? sig[log[b + i] >> 16] : 0u; },
            [&](int i) { return log[b + i] >> 16; });
      }
      bad = pu == ~0u;
      pv = bad ? 0u : pu;
      if (lane == 0) S.path[D - 2] = (int32_t)(S.tab[pv] >> 8);
    }
    place = __shfl_sync(0xffffffffu, place, 0);
    const bool fits = (long long)(place + (unsigned long long)(d - 1)) <= A.arena_cap;
    __syncwarp();
    if (fits && !bad)
      for (int i = lane; i < d - 1; i += 32) A.arena[(long long)place + i] = S.path[i];
    if (lane == 0) {
      A.aoff[jr] = fits && !bad ? (long long)place : -1ll;
      if (!fits) A.dwalk[atomicAdd(&A.ctl->nwalk, 1ull)] = j;
      if (bad) atomicExch(&A.ctl->err, CEN_EINVAL);  // cannot happen with consistent counts
    }
  }
  return true;
}

// Searches of every sample of the launch, or (LIST) of the listed ones.  Once
// most of what was taken has been handed on, the rest follows unsearched.  In the
// wide CTAs it also does where most searches are deep and some were handed on: a
// graph's first call, of which many are left to search, finds out here that they
// are better off in global memory (see kManyDeep), or before it takes up any when
// the small CTAs could finish hardly one, or where most that it hands on have too
// many levels or paths for any size (marked, for the huge CTAs to leave out).  The fewer are handed on, the more must be left
// (first rounds on 1% rewired grids, searched here to the end and not, ms: 500 a side, 10%
// handed on, 3,000 pairs 3.45 and 3.84, 4,500 4.77 and 3.91; 350, 1%, 4,500 pairs 2.96 and
// 3.38, 8,000 4.78 and 4.17).
template <class C, bool LIST>
__global__ void __launch_bounds__(C::T, C::CTAS) k_bidir_log(BiArgs A) {
  extern __shared__ uint4 smem4[];
  LogSh<C> &S = *(LogSh<C> *)smem4;
  const int tid = threadIdx.x;
  const uint32_t count = LIST ? (uint32_t) * (volatile const unsigned long long *)A.list_count : (uint32_t)A.count;
  const int QC = (int)(A.QC < C::NQ ? A.QC : C::NQ);
  unsigned long long arcs = 0;
  if (tid == 0) {
    S.item[0] = (uint32_t)atomicAdd(A.next, 1ull);
    // whether to take up none: many, of which the small CTAs finished one in sixteen at most, those not shallow
    S.none = C::WIDE && LIST && count > kManyLeft * 3 / 2 && 16 * (A.count - count) < count &&
             ld_vol(&A.ctl->cursor) > 8 * (A.count - count);
    S.skip[0] = S.none;
  }
  for (int par = 0;; par ^= 1) {
    __syncthreads();
    const uint32_t i = S.item[par];
    if (i >= count) break;
    uint32_t skip = S.skip[par];
    const uint64_t jr = LIST ? A.list[i] : i;
    if constexpr (C::T > 512) skip |= jr >= kLongId;
    if (!skip)
      for (int p = tid; p < C::H / 4; p += C::T) ((uint4 *)S.tab)[p] = make_uint4(0, 0, 0, 0);
    if (tid == C::T - 32) {  // the next item, fetched while this one is set up
      const uint32_t nx = (uint32_t)atomicAdd(A.next, 1ull);
      const unsigned long long out = ld_vol(A.out_count);
      bool rest = (out > 256 && 2 * out > nx) || (C::WIDE && S.none);
      if (C::WIDE && out && nx + kManyLeft < count) {
        const unsigned long long deep = out + ld_vol(&A.ctl->ndeep), left = count - nx;
        rest |= deep > 256 && 2 * deep > nx && (left > 4096 || left * out > 256ull * nx);
      }
      if (C::WIDE && out) {
        const unsigned long long lng = ld_vol(&A.ctl->nlong);
        rest |= lng > 64 && 2 * lng > nx;
      }
      S.item[par ^ 1] = nx;
      S.skip[par ^ 1] = rest;
    }
    __syncthreads();
    if (skip || !log_search<C>(A, S, jr, QC)) {
      if (tid == 0) {
        uint64_t e = jr;
        if constexpr (C::WIDE)
          if (!skip) {
            atomicAdd(&A.ctl->noutgrown, 1ull);
            if (S.ovf || max(S.lvl[0], S.lvl[1]) + 1 >= C::LV) {
              atomicAdd(&A.ctl->nlong, 1ull);
              e |= kLongId;
            }
          }
        A.out[atomicAdd(A.out_count, 1ull)] = e;
      }
    } else if (tid == 0) {
      arcs += S.arcs;
      if (C::WIDE && S.lvl[0] + S.lvl[1] >= (int)kDeepLevels) atomicAdd(&A.ctl->ndeep, 1ull);
    }
  }
  if (tid == 0 && arcs) atomicAdd(A.units, arcs * 4ull);  // an arc read; its lookup stays in shared memory
}
