// The light-edge index of a graph and the 64-bit keys of the light engine (dj_light.cu).
//
// Most entries of a dense matrix can never matter to a solve: an entry W[u][v] offers v at least
// dist[u] + W[u][v], so once every node holds some path length, only entries of at most (largest
// path length - dist[u]) can still change anything.  On a random graph of n nodes whose rows list
// their K lightest edges up to weight h, the largest distance is about 2 ln(n) / K of h (the
// flooding time of a graph with K / h edges per node and unit of weight), far below h for K = 64.
// So every graph keeps, beside its matrix, each row's up to kLightCap lightest edges and the
// smallest weight it does not list (hmin).  A solve runs on the listed edges, and then
//   dist[u] + hmin[u] > max over v of dist[v]   for every u
// proves that no unlisted entry can improve or tie any node: the answer is exact.  The rows that
// fail the test are relaxed whole from the matrix (see dj_light.cu), so the answer is exact on
// every graph; the test only decides how many rows are read.
//
// Keys.  With every weight >= 1, Algorithm 1's pred[v] is the u of smallest (dist[u], u) among
// those offering dist[v].  Among equal offers the smaller dist[u] is the larger weight, so
//   key(v) = (dist << 32) | ((WF - w) << b) | u,  b = bits(n), WF = 2^(32 - b) - 1
// orders offers exactly that way without knowing dist[u] again.  Every weight fits its field:
// (n - 1) * max weight < 2^31 and n > 2^(b - 1) give max weight <= WF.  The smallest key a node is
// ever offered by final rows is Algorithm 1's (dist, pred), whatever the order of relaxation:
// an offer made from a dist[u] that later shrinks is beaten by the one made from the smaller dist[u].
#pragma once

#include "dj_common.cuh"
#include "dj_internal.h"

namespace dj {

constexpr uint32_t kNoEdge = 0xFFFFFFFFu;  // an unused slot of a row's list (no edge packs to all ones)

__device__ __forceinline__ uint32_t weight_field(uint32_t bits_u) { return 0xFFFFFFFFu >> bits_u; }

// The key u's edge of weight w makes for a dist[u] of du.
__device__ __forceinline__ uint64_t light_key(uint32_t du, uint32_t w, uint32_t u, uint32_t bits_u) {
  return (static_cast<uint64_t>(du + w) << 32) | ((weight_field(bits_u) - w) << bits_u) | u;
}

// The low word of the key that u makes from its listed edge e.
__device__ __forceinline__ uint32_t light_tie(uint32_t e, uint32_t u, uint32_t umask) { return (~e & ~umask) | u; }

// What a solve takes from the index's statistics: its phase window (c times the mean spacing of a
// row's listed weights) and log2 of the lanes that share a row (about the longest list's length).
__device__ __forceinline__ void light_window(const uint32_t* light, float c, uint32_t* delta, int* gshift) {
  const uint4 a = __ldg(reinterpret_cast<const uint4*>(light));
  const uint4 b = __ldg(reinterpret_cast<const uint4*>(light) + 1);
  const float last = static_cast<float>((static_cast<uint64_t>(a.w) << 32) | a.z);
  const float cnt = static_cast<float>((static_cast<uint64_t>(b.y) << 32) | b.x);
  *delta = static_cast<uint32_t>(fminf(1.0e9f, cnt > 0.f ? c * last / cnt : 0.f));
  *gshift = b.z <= 8 ? 3 : b.z <= 16 ? 4 : 5;
}

__device__ __forceinline__ uint32_t light_delta(const uint32_t* light, float c) {
  uint32_t delta;
  int unused;
  light_window(light, c, &delta, &unused);
  return delta;
}

// Per-warp selection of a row's lightest edges.  scan(f, pass) must call f(c0, x) for every group of
// four columns c0 .. c0 + 3 of the row, one group per lane, warp-uniformly often (a lane without a
// group, and columns beyond n, pass INF).  `thr` is the warp's weight threshold, carried from row to
// row: rows of one graph look alike, so one scan is the rule.
//   A scan puts the edges of weight <= thr into buf (kLightBuf words of shared memory) and takes
//   their count and the smallest weight above thr.  Too few (below kLightCap, and more exist) or too
//   many (above kLightBuf): thr moves and the row (in L2 by now) is scanned again; thr is bracketed
//   by [lo, hi], which shrinks with every scan.
// Then the kLightCap smallest packed words (weight, column) go out in ascending order: an entry's
// place is the number of smaller ones.
constexpr int kLightBuf = 384;

struct LightRow {
  uint32_t first;  // smallest weight of the row (INF: no edge)
  uint32_t ties;   // listed edges of that weight (all of them if hmin > first)
  uint32_t cnt;    // listed edges
  uint32_t hmin;   // smallest weight not listed (INF: every edge is listed)
  uint32_t last;   // largest weight listed (0: none)
};

template <class Scan>
__device__ __forceinline__ LightRow light_select(const Scan& scan, uint32_t u, uint32_t bits_u, uint32_t* buf,
                                                 uint32_t* edge, uint32_t& thr) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t wcap = min(weight_field(bits_u), kInf - 1u);  // weights beyond it are never listed
  uint32_t lo = 0, hi = wcap;
  uint32_t cnt = 0, rest = kInf;
  thr = min(thr, wcap);
  for (int pass = 0;; ++pass) {
    cnt = 0;
    rest = kInf;
    const uint32_t t = thr;
    scan(
        [&](uint32_t c0, int4 x) {
          uint32_t w[4] = {static_cast<uint32_t>(x.x), static_cast<uint32_t>(x.y), static_cast<uint32_t>(x.z),
                           static_cast<uint32_t>(x.w)};
          bool h[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (c0 + q == u) w[q] = kInf;  // the diagonal is no edge
            h[q] = w[q] <= t;
            rest = min(rest, h[q] ? kInf : w[q]);
          }
          if (__any_sync(0xffffffffu, h[0] | h[1] | h[2] | h[3])) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t bal = __ballot_sync(0xffffffffu, h[q]);
              const uint32_t at = cnt + __popc(bal & lt);
              if (h[q] && at < static_cast<uint32_t>(kLightBuf)) buf[at] = (w[q] << bits_u) | (c0 + q);
              cnt += __popc(bal);
            }
          }
        },
        pass);
    rest = warp_min_u32(rest);
    if (cnt > static_cast<uint32_t>(kLightBuf)) {  // too many
      if (t == 0) {  // of weight 0: list nothing
        rest = 0;
        cnt = 0;
        break;
      }
      hi = t - 1;
      thr = hi > lo ? lo + (hi - lo) / 2 : hi;
    } else if (cnt < static_cast<uint32_t>(kLightCap) && rest < kInf && t < hi) {  // too few, and more exist
      lo = t + 1;
      // the next weight at least; fast growth while there is no upper bracket
      thr = min(hi, max(hi == wcap ? 2 * t + 1 : lo + (hi - lo) / 2, rest));
    } else {
      break;
    }
    __syncwarp();
  }
  __syncwarp();
  LightRow r;
  uint32_t first = kNoEdge;
  for (uint32_t i = lane; i < cnt; i += 32) first = min(first, buf[i]);
  first = warp_min_u32(first);
  r.first = cnt ? first >> bits_u : rest;
  uint32_t beyond = kNoEdge, ties = 0, last = 0;
  for (uint32_t i = lane; i < cnt; i += 32) {
    const uint32_t e = buf[i];
    uint32_t rank = 0;
    for (uint32_t j = 0; j < cnt; ++j) rank += buf[j] < e ? 1u : 0u;
    if (rank < static_cast<uint32_t>(kLightCap)) {
      edge[rank] = e;
      ties += (e >> bits_u) == r.first ? 1u : 0u;
      last = max(last, e >> bits_u);
    } else {
      beyond = min(beyond, e);
    }
  }
  beyond = warp_min_u32(beyond);
  r.ties = warp_sum_u32(ties);
  r.last = __reduce_max_sync(0xffffffffu, last);
  r.cnt = min(cnt, static_cast<uint32_t>(kLightCap));
  r.hmin = min(rest, beyond == kNoEdge ? kInf : beyond >> bits_u);
  for (uint32_t i = r.cnt + lane; i < static_cast<uint32_t>(kLightCap); i += 32) edge[i] = kNoEdge;
  __syncwarp();  // buf is rewritten by the next row
  return r;
}

}  // namespace dj
