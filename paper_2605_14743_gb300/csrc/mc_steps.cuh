// mc_steps.cuh -- Brandes from one source by one warp, by settle steps (Dijkstra with the IN
// and OUT finality criteria), used by both counting paths: source slots in shared memory
// (mc_kernel.cu) or split between shared memory (distances) and device memory (mc_global.cu).
//
// Every step settles, at once, all pending nodes v whose tentative distance d(v) is below
// d_min + m(v) (the "IN" criterion) or below the smallest d(u) + m(u) over the pending nodes u (the
// "OUT" criterion), where m(v) is a lower bound on v's arcs to unsettled nodes: its smallest
// incident length, or its second smallest once the smallest one leads to a settled node (LONG
// form, StepGraph).  Such a distance is final, and no pending node can precede v on a shortest
// path, so every predecessor of a step's nodes was settled in an earlier step: path counts are
// pulled from them in the same arc scan that relaxes the step's other arcs.  Dependencies take
// one reverse scan per arc, by levels (hop depth in the shortest-path graph) or, for short
// lengths, step by step in reverse.  Per-source results do not depend on which warp runs the
// source, and the exact betweenness sum does not depend on the order in which sources finish.
//
// What bounds it: issue and shared-memory latency of 16 source warps per SM.  On ws1000 (per
// source, LONG form against the plain one): 63 settle steps instead of 86, 43 backward groups of
// up to 32 nodes instead of 87, 67 K warp instructions instead of 92 K; 1,000 realizations 92 ms
// instead of 135 ms.
#pragma once
#include "mc_common.cuh"

namespace afc {

// One source slot, wide form (16 bytes per node): dist[n] (u32 | kFlag once settled), sig[n]
// (sigma, then rho in place), ord[n] (settle order; bit 15 marks the first node of a step) and
// plist[n] (the pending nodes: discovered, not yet settled, each once).
//
// Compact form (COMPACT = true, 12 bytes per node): dist[n] and n 8-byte words, word[k] =
// sigma of node k (low 32 bits) | pending-list entry k (16 bits) | settle-order entry k (top
// 16 bits); the separate ord and plist arrays are not used.  The backward pass no longer needs
// sigma of a node once its rho is known, nor the pending list, nor 32-bit distances: when the
// forward pass ends, node v's distance mod 2^16 moves into the pending-list half of word[v],
// and rho(v) (64 bits) takes dist[v] (high half) and the sigma half of word[v] (low half).
// Distances mod 2^16 identify successors exactly when every length is below 2^15 (adjacent
// nodes' distances differ by at most the arc's length), and sigma must stay below 2^32: a
// realization outside either limit runs on wide slots (the routine reports a path count above
// 2^32 - 1 as ovf bit 1 and the caller redoes the realization).
//
// A settled node's dist word also carries its level (the longest hop count of a shortest path
// from the source) above the low `dbits` bits that the distance needs: kFlag | level << dbits |
// distance.  hist: kLevelHist counters in shared memory for slots in the device arena (slots on
// chip count levels in the pending list's place).
struct StepSlot {
  uint32_t *dist;
  uint64_t *sig;
  uint16_t *ord, *plist;
  uint32_t *hist;
};

constexpr uint32_t kLevelHist = 64;

// Bits of the largest distance of a realization: at most n - 1 arcs of at most wmax each (the
// next arc's candidate distance included).
__device__ __forceinline__ uint32_t dist_bits(uint32_t n, uint32_t wmax) {
  const uint64_t most = (uint64_t)n * (uint64_t)wmax;
  return most >= 0x7FFFFFFFull ? 31u : max(1u, 32u - (uint32_t)__clz((uint32_t)most));
}

constexpr uint32_t kOvfWide = 2u;          // ovf bit: a path count does not fit a compact slot
constexpr uint32_t kCompactMaxLen = 32767;  // longest length a compact slot supports

template <bool COMPACT>
__device__ __forceinline__ uint16_t *pend_at(const StepSlot &sl, uint32_t j) {
  if constexpr (COMPACT)
    return reinterpret_cast<uint16_t *>(sl.sig) + 4u * j + 2u;
  else
    return sl.plist + j;
}

template <bool COMPACT>
__device__ __forceinline__ uint16_t *ord_at(const StepSlot &sl, uint32_t k) {
  if constexpr (COMPACT)
    return reinterpret_cast<uint16_t *>(sl.sig) + 4u * k + 3u;
  else
    return sl.ord + k;
}

// sigma(v) during the forward pass (and of a node not yet given its rho in the backward pass)
template <bool COMPACT>
__device__ __forceinline__ uint64_t sig_get(const StepSlot &sl, uint32_t v) {
  if constexpr (COMPACT)
    return (uint64_t)reinterpret_cast<const uint32_t *>(sl.sig)[2u * v];
  else
    return sl.sig[v];
}

template <bool COMPACT>
__device__ __forceinline__ void sig_put(const StepSlot &sl, uint32_t v, uint64_t x) {
  if constexpr (COMPACT)
    reinterpret_cast<uint32_t *>(sl.sig)[2u * v] = (uint32_t)x;
  else
    sl.sig[v] = x;
}

// rho(v) in the backward pass (kIntTag | integer, or the bits of a DT)
template <bool COMPACT>
__device__ __forceinline__ uint64_t rho_get(const StepSlot &sl, uint32_t v) {
  if constexpr (COMPACT)
    return ((uint64_t)sl.dist[v] << 32) | reinterpret_cast<const uint32_t *>(sl.sig)[2u * v];
  else
    return sl.sig[v];
}

template <bool COMPACT>
__device__ __forceinline__ void rho_put(const StepSlot &sl, uint32_t v, uint64_t x) {
  if constexpr (COMPACT) {
    sl.dist[v] = (uint32_t)(x >> 32);
    reinterpret_cast<uint32_t *>(sl.sig)[2u * v] = (uint32_t)x;
  } else {
    sl.sig[v] = x;
  }
}

// Distance of a settled node in the backward pass: exact (wide) or mod 2^16 (compact).
template <bool COMPACT>
__device__ __forceinline__ uint32_t bdist(const StepSlot &sl, uint32_t v, uint32_t dmask) {
  if constexpr (COMPACT)
    return reinterpret_cast<const uint16_t *>(sl.sig)[4u * v + 2u];
  else
    return sl.dist[v] & dmask;
}

// Counter of level l for the level order (level_order): compact slots count in the pending-list
// half of word[l] (a 32-bit add of less than 2^16 leaves the settle-order half above it alone),
// wide slots on chip in the pending list's bytes, arena slots in their shared-memory histogram.
template <bool COMPACT, bool ONCHIP>
__device__ __forceinline__ uint32_t *level_counter(const StepSlot &sl, uint32_t l) {
  if constexpr (COMPACT)
    return reinterpret_cast<uint32_t *>(sl.sig) + 2u * l + 1u;
  else if constexpr (ONCHIP)
    return reinterpret_cast<uint32_t *>(sl.plist) + l;
  else
    return sl.hist + l;
}
template <bool COMPACT>
__device__ __forceinline__ void level_put(uint32_t *c, uint32_t x) {
  if constexpr (COMPACT) *reinterpret_cast<uint16_t *>(c) = (uint16_t)x;
  else *c = x;
}
template <bool COMPACT>
__device__ __forceinline__ uint32_t level_get(const uint32_t *c) {
  return COMPACT ? (uint32_t)*reinterpret_cast<const uint16_t *>(c) : *c;
}

constexpr uint16_t kStepStart = 0x8000u;   // ord entry opens a step (node ids stay below 2^15)

// Rewrites the settle order of a finished forward pass as the order by level (levels 0..lmax,
// each one's first entry marked kStepStart): a counting sort over the settled nodes by one warp.
// Every successor of a node has a larger level, so the backward pass may take whole levels in
// descending order, and there are far fewer levels than settle steps (ws1000: 20 against 85 per
// source, and 43 against 87 groups of up to 32 nodes, so a backward group has twice as many
// lanes at work).  The order inside a level depends on the schedule; no result does.

// Whether a realization fits the LONG form's doubled 16-bit lengths and 31-bit distances.
__host__ __device__ inline bool long_lengths(uint32_t n, uint32_t wmax) {
  return wmax <= kCompactMaxLen && (uint64_t)n * wmax < (1ull << 30);
}

// The graph as the source routine reads it: row offsets (16-bit on chip), packed arcs and the
// per-node length bounds.
//   plain form: arc = neighbour | length << 16; mwt[v] = smallest alive incident length (0xFFFF:
//               no alive arc).
//   LONG form:  distances are kept doubled, with a low bit: arc = neighbour | (2 length + b) << 16
//               with b = 0 when the arc's length is the smallest at its head, and mwt[v] =
//               2 (second smallest incident length) | 2 (smallest) << 16 (65534: no such arc).
//               A pending node whose key has b = 0 was reached over its shortest arc from a
//               settled node, so every arc from an unsettled node to it, and every arc it can
//               still relax, is at least its second smallest: the bounds of the settle criteria
//               use that one (ws1000: 63 steps per source instead of 86).
template <typename RP>
struct StepGraph {
  uint32_t n;
  const RP *rp;
  const uint32_t *arc;
  const uint32_t *mwt;
};

// Fills mwt and, for the LONG form, rewrites the arcs; H.rp is the 32-bit offsets.  All threads
// of the CTA, which must be synchronised before (arcs complete) and is after.
__device__ inline void step_tables(const Realized &H, uint32_t *arc, uint32_t *mwt, bool lng) {
  for (uint32_t v = threadIdx.x; v < H.n; v += blockDim.x) {
    uint32_t m1 = 0xFFFFu, m2 = 0xFFFFu;
    for (uint32_t e = H.rp[v]; e < H.rp[v + 1]; ++e) {
      const uint32_t w = arc[e] >> 16;
      m2 = min(m2, max(m1, w));
      m1 = min(m1, w);
    }
    mwt[v] = lng ? 2u * min(m2, 32767u) | (2u * min(m1, 32767u)) << 16 : m1;
  }
  __syncthreads();
  if (!lng) return;
  for (uint32_t v = threadIdx.x; v < H.n; v += blockDim.x)
    for (uint32_t e = H.rp[v]; e < H.rp[v + 1]; ++e) {
      const uint32_t u = arc[e] & 0xFFFFu, x = 2u * (arc[e] >> 16);
      arc[e] = u | (x + (x == mwt[u] >> 16 ? 0u : 1u)) << 16;
    }
  __syncthreads();
}

// Exclusive prefix of x over the warp's lanes; total = the sum over all lanes.
__device__ __forceinline__ uint32_t warp_excl(uint32_t x, uint32_t &total) {
  const uint32_t lane = lane_id();
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  total = __shfl_sync(kFull, incl, 31);
  return incl - x;
}

// Issue widths of the routine, by where the source slot lives (measured on ws1000 for slots in
// shared memory, on the batched mix's 2,300-3,800-node graphs for slots in the device arena):
// pend: pending-list windows (32 nodes each) loaded together at the start of a step's
// selection; fwd / bwd: arcs of a lane's node whose loads (and relaxations) are issued
// together in the forward / backward pass.
template <bool ONCHIP> struct StepTune;
template <> struct StepTune<true> { static constexpr int pend = 6, fwd = 4, bwd = 2; };
template <> struct StepTune<false> { static constexpr int pend = 8, fwd = 4, bwd = 8; };

// How a source ended: done; failed (a consistency bound was hit: err has the bits); too_wide (a
// path count does not fit a compact slot, nothing was accumulated).
enum class StepResult { done, failed, too_wide };

template <bool COMPACT, bool ONCHIP>
__device__ __forceinline__ void level_order(const StepSlot &sl, uint32_t n, uint32_t lmax,
                                            uint32_t dbits) {
  const uint32_t lane = lane_id();
  auto at = [&](uint32_t l) { return level_counter<COMPACT, ONCHIP>(sl, l); };
  __syncwarp();
  for (uint32_t l = lane; l <= lmax; l += 32) level_put<COMPACT>(at(l), 0u);
  __syncwarp();
  for (uint32_t v = lane; v < n; v += 32) {
    const uint32_t w = sl.dist[v];
    if (w & kFlag) atomicAdd(at((w & kMask) >> dbits), 1u);
  }
  __syncwarp();
  uint32_t base = 0;
  for (uint32_t l0 = 0; l0 <= lmax; l0 += 32) {
    const uint32_t l = l0 + lane;
    uint32_t total;
    const uint32_t x = l <= lmax ? level_get<COMPACT>(at(l)) : 0u;
    const uint32_t off = base + warp_excl(x, total);
    if (l <= lmax) level_put<COMPACT>(at(l), off);
    base += total;
  }
  __syncwarp();
  // A compact slot's counter is one half of a word whose other half takes an order entry: all
  // counters of a group of nodes first, then the entries, the warp together in between.
  constexpr int kGroup = 4;
  for (uint32_t v0 = 0; v0 < n; v0 += 32u * kGroup) {
    uint32_t pos[kGroup];
#pragma unroll
    for (int t = 0; t < kGroup; ++t) {
      const uint32_t v = v0 + 32u * t + lane;
      const uint32_t w = v < n ? sl.dist[v] : 0u;
      pos[t] = w & kFlag ? atomicAdd(at((w & kMask) >> dbits), 1u) & 0xFFFFu : n;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kGroup; ++t)
      if (pos[t] < n) *ord_at<COMPACT>(sl, pos[t]) = (uint16_t)(v0 + 32u * t + lane);
    __syncwarp();
  }
  // a level's counter now holds its end, i.e. the start of the next one (no level is empty)
  for (uint32_t l = lane; l <= lmax; l += 32) {
    const uint32_t start = l ? level_get<COMPACT>(at(l - 1u)) : 0u;
    *ord_at<COMPACT>(sl, start) |= kStepStart;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------------------
// Brandes from source s by one warp (Sec. 3.1 definitions: d_H, sigma_st, ordered-pair
// betweenness).  Forward: settle steps (see the file comment), sigma pulled from the
// predecessors while the step's arcs are relaxed; the next step's bounds d_min and
// min (d + m) come from the pending nodes that stay and from the relaxations (every pending
// node's current distance is one of those values, and no recorded value is below the node's
// current distance), so no separate pass over the pending list is needed.  Backward
// (want_delta): the levels or steps in reverse; rho(v) = (1 + delta(v)) / sigma(v) replaces sigma
// in place, delta(v) =
// sigma(v) * sum over successors w of rho(w) in arc order; unique-path subtrees (sigma = 1
// throughout) stay exact integers.  delta_s(v) for v != s goes to the exact accumulators of
// the CTA scratch (fx_red).  Every lane of the warp must call it; err / ovf collect
// device-error bits and path-count overflow per lane (bit 0: above 2^64 - 1; bit 1, compact
// slots only: above 2^32 - 1, after which the backward pass is skipped).  Compact slots need
// every length below 2^15 (kCompactMaxLen).
// ---------------------------------------------------------------------------------------
template <typename DT, bool COMPACT, bool ONCHIP, bool LONG, typename RP>
__device__ StepResult source_steps(const StepGraph<RP> &H, const StepSlot &sl, uint32_t s,
                                   uint32_t dbits, bool want_delta, const BcAcc &cs,
                                   uint32_t &err, uint32_t &ovf) {
  using Tune = StepTune<ONCHIP>;
  constexpr int kPendCache = Tune::pend, kArcsFwd = Tune::fwd, kArcsBwd = Tune::bwd;
  static_assert(!COMPACT || ONCHIP, "compact slots live in shared memory");
  const uint32_t n = H.n, lane = lane_id();
  const uint32_t dmask = kMask >> (31u - dbits), levmax = kMask >> dbits;
  constexpr uint32_t kKey = LONG ? ~1u : ~0u;   // the distance part of a key
  // the bound of a node with table entry m at key d (see StepGraph)
  auto bound = [](uint32_t m, uint32_t d) {
    return LONG ? ((d & 1u) ? m >> 16 : m & 0xFFFFu) : m;
  };
  uint32_t lmax = 0;   // largest level seen by this lane
  for (uint32_t v = lane; v < n; v += 32) sl.dist[v] = kInf;
  __syncwarp();
  if (lane == 0) {
    sl.dist[s] = 0u;
    sig_put<COMPACT>(sl, s, 1ull);
    *pend_at<COMPACT>(sl, 0) = (uint16_t)s;
  }
  __syncwarp();

  // ---- forward
  uint32_t nord = 0, pc = 1;                   // settled nodes, pending nodes (warp-uniform)
  uint32_t groups = 0;                         // groups of up to 32 nodes, over all steps
  // d_min and min (d + bound) over the pending nodes (the source alone at first)
  uint32_t dmin = 0u, lout = LONG ? 2u : 1u;
  for (uint32_t step = 0;; ++step) {
    if (step > n) { err |= kErrPassLimit; return StepResult::failed; }
    if (pc == 0) break;   // nothing pending: the source's component is done
    // (1) settle every pending v with d(v) < d_min + mw(v) (IN) or d(v) < lout (OUT; the node
    // at d_min always qualifies): append it to ord, flag it settled; the others stay, compacted,
    // and give the next step's bounds together with the relaxations below
    const uint32_t g0 = nord;
    const uint32_t below = lanemask_lt();
    uint32_t kept = 0, ndmin = kInf, nlout = 0xFFFFFFFFu;
    auto place = [&](bool sel, bool keep, uint32_t spos, uint32_t kpos, uint32_t v, uint32_t d,
                     uint32_t m) {
      if (sel) {
        if (spos < n) {
          *ord_at<COMPACT>(sl, spos) = (uint16_t)(v | (spos == g0 ? kStepStart : 0u));
          sl.dist[v] = (d & kKey) | kFlag;
        } else {
          err |= kErrCapacity;
        }
      } else if (keep) {
        *pend_at<COMPACT>(sl, kpos) = (uint16_t)v;
        ndmin = min(ndmin, d & kKey);
        nlout = min(nlout, (d & kKey) + m);
      }
    };
    {
      // a window of 32 entries: its valid lanes are its first ones, so one ballot and two counts
      // give the positions of both kinds (POPC runs at a fraction of the plain integer rate)
      auto window = [&](uint32_t j0, uint32_t v, uint32_t d, uint32_t m) {
        const bool valid = j0 + lane < pc;
        const bool sel = valid && (d < dmin + m || d < lout);
        const uint32_t sm = __ballot_sync(kFull, sel);
        const uint32_t before = (uint32_t)__popc(sm & below), cnt = (uint32_t)__popc(sm);
        place(sel, valid && !sel, nord + before, kept + lane - before, v, d, m);
        nord += cnt;
        kept += min(32u, pc - j0) - cnt;
      };
      // kPendCache windows at a time: every load first, then the decisions, then the stores (to
      // positions below the entries still to be read).  On chip one such round, then window by
      // window (most steps have no more); in the device arena rounds to the end, since a lone
      // window would wait for its loads (n = 3,000 with lengths 1..100: 201 against 242 ms).
      uint32_t j0 = 0;
      do {
        uint32_t cv[kPendCache], cm[kPendCache], cd[kPendCache];
#pragma unroll
        for (int c = 0; c < kPendCache; ++c) {
          const uint32_t j = j0 + (uint32_t)c * 32u + lane;
          cv[c] = j < pc ? (uint32_t)*pend_at<COMPACT>(sl, j) : 0u;
        }
#pragma unroll
        for (int c = 0; c < kPendCache; ++c) {
          const bool valid = j0 + (uint32_t)c * 32u + lane < pc;
          cm[c] = valid ? H.mwt[cv[c]] : 0u;
          cd[c] = valid ? (uint32_t)sl.dist[cv[c]] : 0u;
        }
#pragma unroll
        for (int c = 0; c < kPendCache; ++c) cm[c] = bound(cm[c], cd[c]);
#pragma unroll
        for (int c = 0; c < kPendCache; ++c) {
          if (j0 + (uint32_t)c * 32u >= pc) break;   // warp-uniform
          window(j0 + (uint32_t)c * 32u, cv[c], cd[c], cm[c]);
        }
        j0 += kPendCache * 32u;
      } while (!ONCHIP && j0 < pc);
      if constexpr (ONCHIP)
        for (; j0 < pc; j0 += 32u) {
          uint32_t v = 0, d = 0, m = 0;
          if (j0 + lane < pc) {
            v = *pend_at<COMPACT>(sl, j0 + lane);
            d = sl.dist[v];
            m = bound(H.mwt[v], d);
          }
          window(j0, v, d, m);
        }
    }
    __syncwarp();
    pc = kept;
    // (2) the step's arcs: sigma and the level from the (settled) predecessors and relaxation of
    // the rest; each group of kArcsFwd arcs issues its loads and atomics together.  A member
    // takes one lane, or two (alternate groups of its arcs) when at most 16 members are left,
    // as in three quarters of ws1000's steps: the longest row then costs half the rounds.
    const uint32_t g1 = min(nord, n);
    groups += (g1 - g0 + 31u) >> 5;
    for (uint32_t c0 = g0; c0 < g1; c0 += 32) {
      const uint32_t two = LONG && g1 - c0 <= 16u ? 1u : 0u;   // warp-uniform
      const uint32_t k = c0 + (lane >> two);
      const bool mine = k < g1;
      uint32_t v = 0, dv = 0, e = 0, e1 = 0;
      if (mine) {
        v = *ord_at<COMPACT>(sl, k) & 0x7FFFu;
        dv = sl.dist[v] & kMask;   // its level is not set yet
        e = H.rp[v] + (lane & two) * (uint32_t)kArcsFwd;
        e1 = H.rp[v + 1];
      }
      unsigned long long sg = 0;
      uint32_t top = 0;
      while (__any_sync(kFull, e < e1)) {
        uint32_t pk[kArcsFwd], du[kArcsFwd], old[kArcsFwd];
        unsigned long long x[kArcsFwd];
#pragma unroll
        for (int t = 0; t < kArcsFwd; ++t) pk[t] = e + t < e1 ? H.arc[e + t] : 0u;
#pragma unroll
        for (int t = 0; t < kArcsFwd; ++t) du[t] = e + t < e1 ? sl.dist[pk[t] & 0xFFFFu] : kFlag;
#pragma unroll
        for (int t = 0; t < kArcsFwd; ++t) {
          const uint32_t u = pk[t] & 0xFFFFu, len = pk[t] >> 16;
          // a predecessor: settled in an earlier step
          const bool pred = (du[t] & kFlag) && (((du[t] & dmask) + len) & kKey) == dv && e + t < e1;
          x[t] = pred ? sig_get<COMPACT>(sl, u) : 0ull;
          // the largest predecessor word: its level is the largest one
          if (LONG && pred) top = max(top, du[t]);
          const uint32_t nd = dv + len;
          const bool relax = !(du[t] & kFlag) && nd < du[t];
          old[t] = relax ? atomicMin(&sl.dist[u], nd) : 0u;
          if (relax) {   // a pending node's new distance: the next step's bounds
            ndmin = min(ndmin, nd & kKey);
            nlout = min(nlout, (nd & kKey) + bound(H.mwt[u], nd));
          }
        }
        // discovered now (each node once): onto the pending list
        uint32_t dm[kArcsFwd];
#pragma unroll
        for (int t = 0; t < kArcsFwd; ++t) dm[t] = __ballot_sync(kFull, old[t] == kInf);
#pragma unroll
        for (int t = 0; t < kArcsFwd; ++t) {
          const unsigned long long nx = sg + x[t];
          if (!COMPACT && nx < sg) ovf |= 1u;   // compact addends are below 2^32: no wrap
          sg = nx;
          if ((dm[t] >> lane) & 1u)
            *pend_at<COMPACT>(sl, pc + (uint32_t)__popc(dm[t] & below)) =
                (uint16_t)(pk[t] & 0xFFFFu);
          pc += (uint32_t)__popc(dm[t]);
        }
        e += (uint32_t)kArcsFwd << two;
      }
      if (two) {   // warp-uniform: the pair's halves together
        const unsigned long long other = __shfl_xor_sync(kFull, sg, 1);
        const unsigned long long nx = sg + other;
        if (!COMPACT && nx < sg) ovf |= 1u;
        sg = nx;
        if (LONG) top = max(top, __shfl_xor_sync(kFull, top, 1));
      }
      if (COMPACT && (sg >> 32)) ovf |= kOvfWide;
      if (mine && (lane & two) == 0u) {
        if (v != s) sig_put<COMPACT>(sl, v, sg);
        if constexpr (LONG) {
          const uint32_t lev = top ? ((top & kMask) >> dbits) + 1u : 0u;
          sl.dist[v] = kFlag | (min(lev, levmax) << dbits) | dv;
          lmax = max(lmax, lev);
        }
      }
    }
    dmin = __reduce_min_sync(kFull, ndmin);
    lout = __reduce_min_sync(kFull, nlout);
    __syncwarp();
  }
  if (!want_delta) return StepResult::done;
  lmax = __reduce_max_sync(kFull, lmax);
  // a path count that a compact slot cannot hold: the caller redoes the realization
  if (COMPACT && __any_sync(kFull, ovf & kOvfWide)) return StepResult::too_wide;
  // the order by level where it saves groups of up to 32 nodes in the backward pass (about
  // nord / 32 and half a group per level are left; ordering costs about as much as n / 96
  // groups), unless the levels outgrow the dist word's free bits or the counters (deep graphs
  // with long lengths): otherwise the backward pass takes the settle steps in reverse
  if (LONG && groups > (nord >> 5) + (lmax >> 1) + n / 96u + 1u && lmax <= levmax &&
      lmax < (COMPACT ? n : ONCHIP ? n / 2u : kLevelHist))
    level_order<COMPACT, ONCHIP>(sl, n, lmax, dbits);
  if constexpr (COMPACT) {
    // distances mod 2^16 into the (now empty) pending-list halves; every node the backward
    // pass reads was reached (settled nodes and their neighbours)
    uint16_t *w16 = reinterpret_cast<uint16_t *>(sl.sig);
    for (uint32_t v = lane; v < n; v += 32) w16[4u * v + 2u] = (uint16_t)((sl.dist[v] & dmask) >> (LONG ? 1 : 0));
    __syncwarp();
  }

  // ---- backward: the levels (or settle steps) in reverse, one member per lane
  uint32_t hi = min(nord, n);
  while (hi > 0) {
    // the group holding position hi - 1 starts at the nearest mark at or below it
    uint32_t lo = 0;
    for (int32_t top = (int32_t)hi - 1; top >= 0; top -= 32) {
      const int32_t p = top - (int32_t)lane;
      const bool mark = p >= 0 && (*ord_at<COMPACT>(sl, (uint32_t)p) & kStepStart);
      const uint32_t mm = __ballot_sync(kFull, mark);
      if (mm) {
        lo = (uint32_t)(top - (__ffs(mm) - 1));
        break;
      }
    }
    for (uint32_t c0 = lo; c0 < hi; c0 += 32) {
      const uint32_t k = c0 + lane;
      const bool mine = k < hi;
      uint32_t v = 0, dv = 0, e = 0, e1 = 0;
      uint64_t sg = 0;
      if (mine) {
        v = *ord_at<COMPACT>(sl, k) & 0x7FFFu;
        dv = bdist<COMPACT>(sl, v, dmask);
        e = H.rp[v];
        e1 = H.rp[v + 1];
        sg = sig_get<COMPACT>(sl, v);
      }
      // the successors' rho in arc order: integral ones exactly, the others in DT
      uint32_t acc_i = 0;
      DT acc_f = 0;
      bool any_f = false;
      while (__any_sync(kFull, e < e1)) {
        uint32_t pk[kArcsBwd];
        uint64_t rw[kArcsBwd];
#pragma unroll
        for (int t = 0; t < kArcsBwd; ++t) pk[t] = e + t < e1 ? H.arc[e + t] : 0u;
#pragma unroll
        for (int t = 0; t < kArcsBwd; ++t) {
          const uint32_t w = pk[t] & 0xFFFFu;
          const uint32_t want = dv + (!LONG ? pk[t] >> 16 : COMPACT ? pk[t] >> 17 : (pk[t] >> 16) & ~1u);
          const bool suc = e + t < e1 && bdist<COMPACT>(sl, w, dmask) == (COMPACT ? want & 0xFFFFu : want);
          rw[t] = suc ? rho_get<COMPACT>(sl, w) : kIntTag;   // kIntTag alone adds 0
        }
#pragma unroll
        for (int t = 0; t < kArcsBwd; ++t) {
          if (rw[t] & kIntTag) {
            acc_i += (uint32_t)rw[t];
          } else {
            acc_f += *reinterpret_cast<const DT *>(&rw[t]);
            any_f = true;
          }
        }
        e += kArcsBwd;
      }
      if (mine) {
        if (sg == 1ull && !any_f) {
          // delta(v) = sum of the successors' subtree sizes: exact in integers
          rho_put<COMPACT>(sl, v, kIntTag | (uint64_t)(1u + acc_i));
          if (v != s && acc_i) atomicAdd(&cs.a0[v], (unsigned long long)acc_i);
        } else {
          DT dep, rho;
          if constexpr (COMPACT) dependency<DT, uint32_t>((uint32_t)sg, (DT)acc_i + acc_f, dep, rho);
          else dependency<DT, uint64_t>(sg, (DT)acc_i + acc_f, dep, rho);
          uint64_t bits = 0;
          *reinterpret_cast<DT *>(&bits) = rho;
          rho_put<COMPACT>(sl, v, bits);
          if (v != s) fx_red(cs.a0, cs.a1, cs.a2, v, (double)dep);
        }
      }
    }
    __syncwarp();
    hi = lo;
  }
  return StepResult::done;
}

}  // namespace afc
