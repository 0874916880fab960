// The light-edge index of a graph and the 64-bit keys of the light engine (dj_light_cta.cu, dj_light_cluster.cu,
// dj_light_grid.cu).
//
// Most entries of a dense matrix can never matter to a solve: an entry W[u][v] offers v at least
// dist[u] + W[u][v], so once every node holds some path length, only entries of at most (largest
// path length - dist[u]) can still change anything.  On a random graph of n nodes whose rows list
// their K lightest edges up to weight h, the largest distance is about 2 ln(n) / K of h (the
// flooding time of a graph with K / h edges per node and unit of weight), far below h for K = 64.
// So every graph keeps, beside its matrix, each row's up to kLightCap lightest edges (kLightWide, if the
// first are too few and these are enough) and the smallest weight it does not list (hmin).  A solve runs on the listed edges, and then
//   dist[u] + hmin[u] > max over v of dist[v]   for every u
// proves that no unlisted entry can improve or tie any node: the answer is exact.  The rows that
// fail the test are relaxed whole from the matrix (see dj_light_grid.cu), so the answer is exact on
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
#include "dj_light_rules.h"

namespace dj {

constexpr uint32_t kNone = kRuleNone;      // no dist, no bound
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

// A guess of the largest dist, from the trial solve's (word kLightGuess): that and 1 / part of it more,
// no guess without one.
__device__ __forceinline__ uint32_t light_guess(const uint32_t* light, uint32_t part) {
  const uint32_t x = __ldg(light + kLightGuess);
  return x == 0 ? kNone : x - 1 + max(1u, (x - 1) / part);
}

// Per-warp selection of a row's lightest edges.  scan(f, pass) must call f(c0, x) for every group of
// four columns c0 .. c0 + 3 of the row (or f(c0, x, step): c0 .. c0 + 3 * step), one group per lane,
// warp-uniformly often (a lane without a group, and columns beyond n, pass INF).  `thr` is the warp's weight threshold, carried from row to
// row: rows of one graph look alike, so one scan is the rule.
//   A scan puts the edges of weight <= thr into buf (kLightBuf words of shared memory) and takes
//   their count and the smallest weight above thr.  Too few (below Cap, and more exist) or too
//   many (above kLightBuf): thr moves and the row (in L2 by now) is scanned again; thr is bracketed
//   by [lo, hi], which shrinks with every scan.  After too many, buf holds a sample of them, and thr
//   goes where the sample says that about Cap + 96 edges lie (light_sample): one scan more instead of up to
//   ten by halving where weights are spread unevenly.
// Then the Cap smallest packed words (weight, column) go out in ascending order, from the kLightCap-th on
// at edge2: an entry's place is the number of smaller ones.
constexpr int kLightBuf = 384;

struct LightRow {
  uint32_t first;  // smallest weight of the row (INF: no edge)
  uint32_t ties;   // listed edges of that weight (all of them if hmin > first)
  uint32_t cnt;    // listed edges
  uint32_t hmin;   // smallest weight not listed (INF: every edge is listed)
  uint32_t last;   // largest weight listed (0: none)
  uint32_t seen;   // edges of weight <= thr
};

// The largest t in [lo, hi] that at most k of the warp's weights x do not exceed (lo if there is none).
template <int N>
__device__ __forceinline__ uint32_t light_sample(const uint32_t (&x)[N], uint32_t k, uint32_t lo, uint32_t hi) {
  while (lo < hi) {
    const uint32_t mid = hi - (hi - lo) / 2;
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) c += x[i] <= mid ? 1u : 0u;
    if (warp_sum_u32(c) <= k)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

template <int Cap, class Scan>
__device__ __forceinline__ LightRow light_select(const Scan& scan, uint32_t u, uint32_t bits_u, uint32_t* buf,
                                                 uint32_t* edge, uint32_t* edge2, uint32_t& thr) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t wcap = min(weight_field(bits_u), kInf - 1u);  // weights beyond it are never listed
  uint32_t lo = 0, hi = wcap;
  uint32_t cnt = 0, rest = kInf, few = 1;  // few: the edges of weight < lo, as scanned
  thr = min(thr, wcap);
  for (int pass = 0;; ++pass) {
    cnt = 0;
    rest = kInf;
    const uint32_t t = thr;
    scan(
        [&](uint32_t c0, int4 x, uint32_t step = 1) {
          uint32_t w[4] = {static_cast<uint32_t>(x.x), static_cast<uint32_t>(x.y), static_cast<uint32_t>(x.z),
                           static_cast<uint32_t>(x.w)};
          bool h[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (c0 + step * q == u) w[q] = kInf;  // the diagonal is no edge
            h[q] = w[q] <= t;
            rest = min(rest, h[q] ? kInf : w[q]);
          }
          if (__any_sync(0xffffffffu, h[0] | h[1] | h[2] | h[3])) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t bal = __ballot_sync(0xffffffffu, h[q]);
              const uint32_t at = cnt + __popc(bal & lt);
              if (h[q] && at < static_cast<uint32_t>(kLightBuf)) buf[at] = (w[q] << bits_u) | (c0 + step * q);
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
      if (hi < lo && few == 0) {  // weights below t: none, of weight t: too many
        rest = t;
        cnt = 0;
        break;
      }
      __syncwarp();
      uint32_t x[kLightBuf / 32];
#pragma unroll
      for (int i = 0; i < kLightBuf / 32; ++i) x[i] = buf[32 * i + lane] >> bits_u;
      thr = hi > lo ? light_sample(x, max(1u, kLightBuf * (Cap + 96u) / cnt), lo, hi) : hi;
    } else if (cnt < static_cast<uint32_t>(Cap) && rest < kInf && t < hi) {  // too few, and more exist
      lo = t + 1;
      few = cnt;
      thr = min(hi, max(min(2 * t + 1, lo + (hi - lo) / 2), rest));  // the next weight at least
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
  r.seen = cnt;
  const uint32_t r_first = r.first;
  uint32_t beyond = kNoEdge, ties = 0, last = 0;
  if (lane < 4 && cnt + lane < static_cast<uint32_t>(kLightBuf)) buf[cnt + lane] = kNoEdge;
  __syncwarp();
  for (uint32_t i0 = lane; i0 - lane < cnt; i0 += 128) {
    // four entries a lane against four of the buffer per 16-byte load
    uint32_t e[4], rank[4] = {0, 0, 0, 0};
#pragma unroll
    for (int r = 0; r < 4; ++r) e[r] = i0 + 32 * r < cnt ? buf[i0 + 32 * r] : kNoEdge;
    for (uint32_t j = 0; j < cnt; j += 4) {
      const uint4 y = *reinterpret_cast<const uint4*>(buf + j);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        rank[r] += (y.x < e[r] ? 1u : 0u) + (y.y < e[r] ? 1u : 0u) + (y.z < e[r] ? 1u : 0u) + (y.w < e[r] ? 1u : 0u);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (e[r] == kNoEdge) continue;
      if (rank[r] < static_cast<uint32_t>(Cap)) {
        if (Cap == kLightCap || rank[r] < static_cast<uint32_t>(kLightCap))
          edge[rank[r]] = e[r];
        else
          edge2[rank[r] - kLightCap] = e[r];
        ties += (e[r] >> bits_u) == r_first ? 1u : 0u;
        last = max(last, e[r] >> bits_u);
      } else {
        beyond = min(beyond, e[r]);
      }
    }
  }
  beyond = warp_min_u32(beyond);
  r.ties = warp_sum_u32(ties);
  r.last = __reduce_max_sync(0xffffffffu, last);
  r.cnt = min(cnt, static_cast<uint32_t>(Cap));
  r.hmin = min(rest, beyond == kNoEdge ? kInf : beyond >> bits_u);
  for (uint32_t i = r.cnt + lane; i < static_cast<uint32_t>(kLightCap); i += 32) edge[i] = kNoEdge;
  if (Cap > kLightCap)
    for (uint32_t i = max(r.cnt, static_cast<uint32_t>(kLightCap)) + lane; i < static_cast<uint32_t>(Cap); i += 32)
      edge2[i - kLightCap] = kNoEdge;
  __syncwarp();  // buf is rewritten by the next row
  return r;
}

// ------------------------------------------------------------------ relaxing rows from shared memory

constexpr int kWarpRows = 64;            // a warp's waiting rows: 31 left over and 32 of the next word

// Shared words that other warps change meanwhile are read through this.
__device__ __forceinline__ uint32_t word_now(const uint32_t* p) { return *const_cast<const volatile uint32_t*>(p); }

// Where a row's edges beyond the first kLightCap lie, counted from where they would follow these (so that
// the first keep their 256 bytes a row, which is all that most graphs use).
__device__ __forceinline__ size_t light_apart(int32_t n) { return (static_cast<size_t>(n) - 1) * kLightCap; }

// The rows of the index: up to `most` edges each, padded.
struct LightListEdges {
  static constexpr bool kApart = true;
  const uint32_t* __restrict__ edge;
  int32_t n;
  uint32_t most;
  __device__ __forceinline__ uint4 load(uint32_t u, uint32_t k0, int sub) const {
    return __ldg(reinterpret_cast<const uint4*>(edge + static_cast<size_t>(u) * kLightCap + k0) + sub);
  }
};

// Relax (with kTies: take the ties of) the listed edges of a warp's rows: get(i) is row i, i < count, as
// (u, dist[u]) or, where there is nothing to do, (u, kNone).  Four lanes share a row and take four edges
// each with one 16-byte load, so a warp's load covers 16 edges of 8 rows in 8 pieces of 64 bytes, and
// 16 rows are in flight.  Edges whose offer exceeds B are dropped; a row goes on to its next 16
// edges only if the heaviest of these was of use.  (A lane per edge, 16 lanes per row, took three times the
// instructions per edge; a lane per row read 32 lines with every load and was bound by the L1.)
template <bool kTies, class Store, class Edges, class Get>
__device__ __forceinline__ void light_rows(const Store& s, const Edges& edges, const Get& get, int count, uint32_t B,
                                           uint32_t bits_u, uint32_t& lmin) {
  const int lane = static_cast<int>(threadIdx.x) & 31, sub = lane & 3;
  const uint32_t umask = (1u << bits_u) - 1u;
  constexpr int R = 2;  // 16-byte loads in flight per lane (4: 395 against 298 us for the batch)
  for (int i0 = 0; i0 < count; i0 += 8 * R) {
    uint32_t u[R], du[R];
    bool on[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = i0 + 8 * r + (lane >> 2);
      const uint2 x = get(min(i, count - 1));
      u[r] = x.x;
      du[r] = x.y;
      on[r] = i < count && x.y != kNone;
    }
    // Where the listed edges beyond kLightCap lie, counted in rows (light_apart).  Carried along, it costs graphs
    // without such edges 1 % (256 solves of n = 8192: 265 us, 267 now; compared and added per step 270).
    uint32_t part = 0;
    for (uint32_t k0 = 0; k0 < edges.most; k0 += 16) {  // most bounds every row
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r)
        x[r] = on[r] ? edges.load(u[r] + part, k0, sub) : make_uint4(kNoEdge, kNoEdge, kNoEdge, kNoEdge);
      uint32_t more = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint32_t e[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
        uint32_t old[4];
        bool use = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t c = du[r] + (e[q] >> bits_u), v = e[q] & umask;
          use = e[q] != kNoEdge && c <= B;
          if (kTies)
            old[q] = use ? s.dist_of(v) : 0u;
          else
            old[q] = use ? s.offer(v, c) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t c = du[r] + (e[q] >> bits_u), v = e[q] & umask;
          if (kTies) {
            if (old[q] == c && e[q] != kNoEdge) s.tie_min(v, light_tie(e[q], u[r], umask));
          } else if (c < old[q]) {
            s.won(v, c);
            lmin = min(lmin, c);
          }
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, use);  // the last of the lane's four edges
        on[r] = (bal >> (lane | 3)) & 1u;
        more |= bal & 0x88888888u;
      }
      if (more == 0) break;
      if (Edges::kApart && k0 == static_cast<uint32_t>(kLightCap) - 16u) part = edges.n - 1;
    }
  }
  __syncwarp();
}

// The same for a piece of row u, of dist du, from the matrix: 16-byte groups [g0, g1) (one warp).
template <bool kTies, class Store>
__device__ __forceinline__ void light_matrix_row(const Store& s, const SolveDesc& d, uint32_t u, uint32_t du, int g0,
                                                 int g1, uint32_t D, uint32_t& lmin) {
  const int lane = static_cast<int>(threadIdx.x) & 31;
  const int32_t* row = d.W + static_cast<int64_t>(u) * d.pitch;
  constexpr int R = 4;
  for (int g = g0 + lane; g < g1; g += 32 * R) {
    int4 x[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
      x[r] = g + 32 * r < g1 ? ld_stream16(row + 4 * (g + 32 * r)) : make_int4(int(kInf), int(kInf), int(kInf), int(kInf));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t w4[4] = {static_cast<uint32_t>(x[r].x), static_cast<uint32_t>(x[r].y),
                              static_cast<uint32_t>(x[r].z), static_cast<uint32_t>(x[r].w)};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t v = 4 * (g + 32 * r) + q, c = du + w4[q];
        if (w4[q] >= kInf || c > D || v == u) continue;
        if (kTies) {
          if (s.dist_of(v) == c) s.tie_min(v, static_cast<uint32_t>(light_key(du, w4[q], u, d.bits_u)));
        } else {
          if (c < s.offer(v, c)) {
            s.won(v, c);
            lmin = min(lmin, c);
          }
        }
      }
    }
  }
  __syncwarp();
}

// Rows relaxed whole are cut into pieces of this many 16-byte groups, which the CTA's warps take in turn
// (one warp per row of 16384 columns took 32 us a row).
constexpr int kRowPiece = 256;
template <class Store>
__device__ __forceinline__ void light_whole_rows(const Store& s, const SolveDesc& d, const uint2* list, int count,
                                                 uint32_t D, uint32_t& lmin) {
  const int nv = static_cast<int>(d.pitch / 4), pieces = (nv + kRowPiece - 1) / kRowPiece;
  for (int it = static_cast<int>(threadIdx.x >> 5); it < count * pieces; it += static_cast<int>(blockDim.x >> 5)) {
    const uint2 x = list[it / pieces];
    const int g0 = (it % pieces) * kRowPiece;
    light_matrix_row<false>(s, d, x.x, x.y, g0, min(nv, g0 + kRowPiece), D, lmin);
  }
}
// Their ties: row(word, bit) is the row of a bit of whole[word] with its dist.
template <class Store, class Row>
__device__ __forceinline__ void light_whole_ties(const Store& s, const SolveDesc& d, const uint32_t* whole, int words,
                                                 const Row& row, uint32_t B) {
  const int nv = static_cast<int>(d.pitch / 4);
  uint32_t unused = 0;
  for (int w = 0; w < words; ++w)
    for (uint32_t todo = whole[w]; todo; todo &= todo - 1) {
      const uint2 x = row(w, __ffs(todo) - 1);
      for (int g0 = static_cast<int>(threadIdx.x >> 5) * kRowPiece; g0 < nv;
           g0 += static_cast<int>(blockDim.x >> 5) * kRowPiece)
        light_matrix_row<true>(s, d, x.x, x.y, g0, min(nv, g0 + kRowPiece), B, unused);
    }
}

}  // namespace dj
