// Graph construction: edge list (or dense matrix) -> device adjacency matrix.
//
// Section III of the paper: the input is an edge list that each program
// writes into an n x n adjacency matrix (not timed); Section III-A: the -w
// flag fills a directed graph, otherwise undirected.  Here the matrix is
// built directly in HBM: a vectorised INF fill with a zero diagonal, a scatter
// of the edges with atomicMin (so a repeated pair keeps its smallest weight,
// independent of order), and one pass computing each row's smallest finite
// off-diagonal weight (minout) and each column's (minin), both used by the
// phase-batched solve to prove nodes final.  Rows are
// padded to a multiple of 32 int32 (128 bytes) with INF, the device analogue
// of the paper's INF padding of Section III-B.
#include <algorithm>
#include <cstring>
#include <string>

#include "dj_common.cuh"
#include "dj_internal.h"
#include "dj_light.cuh"
#include "dj_light_rules.h"

namespace dj {

__global__ void k_fill(int32_t* __restrict__ W, int64_t pitch, int32_t n) {
  const int64_t nv = static_cast<int64_t>(n) * pitch / 4;
  int4* W4 = reinterpret_cast<int4*>(W);
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < nv;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t e = i * 4;
    const int64_t r = e / pitch;
    const int64_t c = e - r * pitch;
    int4 v = make_int4(int(kInf), int(kInf), int(kInf), int(kInf));
    if (r >= c && r < c + 4) (&v.x)[r - c] = 0;
    W4[i] = v;
  }
}

// Scatter edges [0, m) (edge 0 is number `first` of the caller's list) into the matrix, checking each:
// node ids in [0, n), weights in [0, INF).  A bad edge is not written; check[0..1] (64 bits, zero before)
// becomes the largest ~number, so the first bad edge, and check[2] the largest weight of an edge that is
// no self-loop.  src, dst and w may be the caller's own pageable arrays where the device can read host
// memory (see dj_load_edges); then the loads are what takes the time, so each thread has kScatterEdges
// edges in flight.
constexpr int kScatterEdges = 4;
__global__ void __launch_bounds__(256) k_scatter(int32_t* __restrict__ W, int64_t pitch, int32_t n,
                                                 const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                 const int32_t* __restrict__ w, int64_t m, int64_t first, int directed,
                                                 uint32_t* check) {
  const int64_t step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  int32_t wmax = 0;
  int64_t bad = -1;
  for (int64_t e0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e0 < m; e0 += kScatterEdges * step) {
    int32_t u[kScatterEdges], v[kScatterEdges], x[kScatterEdges];
#pragma unroll
    for (int k = 0; k < kScatterEdges; ++k) {
      const int64_t e = e0 + k * step;
      u[k] = e < m ? src[e] : 0;
      v[k] = e < m ? dst[e] : 0;  // beyond the list: a self-loop
      x[k] = e < m ? w[e] : 0;
    }
#pragma unroll
    for (int k = 0; k < kScatterEdges; ++k) {
      if (static_cast<uint32_t>(u[k]) >= static_cast<uint32_t>(n) || static_cast<uint32_t>(v[k]) >= static_cast<uint32_t>(n) ||
          static_cast<uint32_t>(x[k]) >= kInf) {
        if (bad < 0) bad = first + e0 + k * step;  // ascending within a thread
        continue;
      }
      if (u[k] == v[k]) continue;  // self-loops ignored: the diagonal stays 0
      wmax = max(wmax, x[k]);
      atomicMin(W + static_cast<int64_t>(u[k]) * pitch + v[k], x[k]);
      if (!directed) atomicMin(W + static_cast<int64_t>(v[k]) * pitch + u[k], x[k]);
    }
  }
  if (bad >= 0) atomicMax(reinterpret_cast<unsigned long long*>(check), ~static_cast<unsigned long long>(bad));
  wmax = __reduce_max_sync(0xffffffffu, wmax);
  if ((threadIdx.x & 31) == 0 && wmax > 0) atomicMax(check + 2, static_cast<uint32_t>(wmax));
}

// Copy a dense matrix with row stride ld into the padded layout (padding columns INF), checking every
// entry lies in [0, INF]; bad entries set flags[0].  A block per row at a time, in 16-byte pieces where A
// allows them (vec): n = 16384 (1 GiB read, 1 GiB written) was bound by a 64-bit division per entry.
__global__ void __launch_bounds__(256) k_copy_dense(int32_t* __restrict__ W, int64_t pitch, const int32_t* __restrict__ A,
                                                    int64_t ld, int32_t n, int vec, uint32_t* flags) {
  uint32_t sign = 0;  // the entries' top bits
  for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
    const int32_t* a = A + r * ld;
    int32_t* d = W + r * pitch;
    int c0 = 0;
    if (vec) {
      const int nq = n / 4;
      for (int q = threadIdx.x; q < nq; q += 256) {
        const int4 x = reinterpret_cast<const int4*>(a)[q];
        sign |= static_cast<uint32_t>(x.x | x.y | x.z | x.w);
        reinterpret_cast<int4*>(d)[q] = x;
      }
      c0 = 4 * nq;
    }
    for (int c = c0 + static_cast<int>(threadIdx.x); c < pitch; c += 256) {
      const int32_t x = c < n ? a[c] : static_cast<int32_t>(kInf);
      sign |= static_cast<uint32_t>(x);
      d[c] = x;
    }
  }
  if (sign >> 31) atomicOr(flags, 1u);
}

// One warp per row: minout[u] = min finite W[u][v], v != u; plus the global
// finite min / max and the number of finite entries (stats[0] = min,
// stats[1] = max, stats[2..3] = count as a 64-bit word).
__global__ void k_rowmin(const int32_t* __restrict__ W, int64_t pitch, int32_t n, int32_t* __restrict__ minout,
                         uint32_t* stats) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  uint32_t gmin = kInf, gmax = 0;
  unsigned long long cnt = 0;
  for (int64_t u = warp; u < n; u += nwarps) {
    const int32_t* row = W + u * pitch;
    uint32_t mn = kInf, mx = 0;
    for (int64_t v = lane; v < n; v += 32) {
      const uint32_t x = static_cast<uint32_t>(row[v]);
      if (v != u && x < kInf) {
        mn = min(mn, x);
        mx = max(mx, x);
        ++cnt;
      }
    }
    mn = warp_min_u32(mn);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) minout[u] = static_cast<int32_t>(mn);
    gmin = min(gmin, mn);
    gmax = max(gmax, mx);
  }
  if (stats) {
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (lane == 0) {
      atomicMin(stats, gmin);
      atomicMax(stats + 1, gmax);
      atomicAdd(reinterpret_cast<unsigned long long*>(stats + 2), cnt);
    }
  }
}

// One warp per row: the row's light-edge list (dj_light.cuh) and, from it, what the other engines
// keep of a row: minout[u], with `ties` (a symmetric matrix, whose column u is row u and whose minin is
// minout) column u's tie sources as k_tiesrc lists them, and the statistics of the index.
constexpr int kTieSourceCap = 32;
struct LightOut {
  uint32_t* light;  // the index (stats, hmin, edges)
  int32_t* minout;
  int32_t* tsrc;  // nullptr: not symmetric
  int32_t* tcnt;
  int32_t cap;
  uint32_t bits_u;
  int32_t n;
  float deg;      // edges per row and largest weight if known (deg 0: not; wmax 0: word 14 of the index),
  uint32_t wmax;  // for each warp's first threshold (first_threshold)
  float first;    // uploads: the first threshold itself
};
struct LightSums {
  unsigned long long last = 0, cnt = 0;
  unsigned long long seen = 0, thr = 0;  // rows with cut lists: edges up to their thresholds, and these
  uint32_t cut = 0;
  uint32_t hmin = 0xFFFFFFFFu, most = 0, trial = 0;
};

// The first threshold of light_select, in the middle of its window of counts: an upload takes the mean of those
// that served the loaded matrix, an edge list's load goes by deg edges per row, as if the weights were uniform up to
// the largest (word 14), and a matrix's load takes the weight that about `want` edges of the warp's first row do not
// exceed, by the row's first 512 columns.  A warp has only a few rows, so a bad guess costs scans: 8192 rows of 4096
// edges took 265 us from 0 and take 98, against 125 us for the row minima and tie sources this pass replaces.
__device__ __forceinline__ uint32_t first_threshold(const LightOut& o, const int32_t* row, uint32_t u, float want) {
  if (!row) return static_cast<uint32_t>(o.first);
  if (o.deg > 0.f) {
    const float wmax = static_cast<float>(o.wmax ? o.wmax : o.light[14]);
    return static_cast<uint32_t>(fminf(2.0e9f, o.deg <= want ? wmax : wmax * want / o.deg));
  }
  const int c1 = min(o.n, 512);
  uint32_t x[16], most = 0, cnt = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int c = 32 * i + (static_cast<int>(threadIdx.x) & 31);
    x[i] = c < c1 && static_cast<uint32_t>(c) != u ? static_cast<uint32_t>(row[c]) : kInf;
    if (x[i] < kInf) {
      most = max(most, x[i]);
      ++cnt;
    }
  }
  const uint32_t k = static_cast<uint32_t>(want * static_cast<float>(c1) / static_cast<float>(o.n));
  if (warp_sum_u32(cnt) <= k) return kInf;
  return light_sample(x, k, 0, __reduce_max_sync(0xffffffffu, most));
}

template <int Cap, class Scan>
__device__ __forceinline__ void light_row(const LightOut& o, const Scan& scan, uint32_t u, uint32_t* buf,
                                          uint32_t& thr, LightSums& sums) {
  const int lane = threadIdx.x & 31;
  uint32_t* hmin = o.light + kLightStats;
  uint32_t* edge = hmin + light_pad(o.n) + static_cast<size_t>(u) * kLightCap;
  const LightRow r = light_select<Cap>(scan, u, o.bits_u, buf, edge, edge + kLightCap + light_apart(o.n), thr);
  if (lane == 0) {
    o.minout[u] = static_cast<int32_t>(r.first);
    if (o.tsrc) o.minout[o.n + u] = static_cast<int32_t>(r.first);  // minin: the same
    hmin[u] = r.hmin;
    // a list that misses some edges of the smallest weight counts as too many to list
    if (o.tsrc) o.tcnt[u] = r.first >= kInf ? 0 : static_cast<int32_t>(r.hmin > r.first ? r.ties : max(r.ties, o.cap + 1u));
  }
  if (o.tsrc && lane < o.cap && static_cast<uint32_t>(lane) < r.ties)
    o.tsrc[static_cast<int64_t>(u) * o.cap + lane] = static_cast<int32_t>(edge[lane] & ((1u << o.bits_u) - 1u));
  if (r.hmin < kInf && r.seen > 0) {
    sums.seen += r.seen;
    sums.thr += thr;
    ++sums.cut;
  }
  sums.last += r.last;
  sums.cnt += r.cnt;
  sums.hmin = min(sums.hmin, r.hmin);
  sums.most = max(sums.most, r.cnt);
  sums.trial = max(sums.trial, light_trial_word(u, r.cnt, r.first < kInf, static_cast<uint32_t>(o.n)));
}

// Every warp's sums into the index: the block's first, then one reduction per word and block (one per warp to the
// same few words took 15 us for 8192 rows).
struct LightBlockSums {
  unsigned long long add[5];  // last, cnt, seen, thr, finite entries
  uint32_t top[5];            // ~hmin, most, trial, ~finite min, finite max
  uint32_t cut;
};
__device__ __forceinline__ void light_sums_out(const LightOut& o, const LightSums& s, bool stats = false,
                                               uint32_t gmin = 0, uint32_t gmax = 0, unsigned long long entries = 0) {
  __shared__ LightBlockSums t;
  const int tid = static_cast<int>(threadIdx.x);
  __syncthreads();
  if (tid < 5) {
    t.add[tid] = 0;
    t.top[tid] = 0;
  }
  if (tid == 0) t.cut = 0;
  __syncthreads();
  if ((tid & 31) == 0) {
    const unsigned long long add[5] = {s.last, s.cnt, s.seen, s.thr, entries};
    const uint32_t top[5] = {s.hmin < kInf ? ~s.hmin : 0u, s.most, s.trial, ~gmin, gmax};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      atomicAdd(&t.add[i], add[i]);
      atomicMax(&t.top[i], top[i]);
    }
    atomicAdd(&t.cut, s.cut);
  }
  __syncthreads();
  constexpr int kAdd[5] = {2, 4, kLightSeen, kLightSeen + 2, 10}, kTop[5] = {0, 6, 7, 8, 9};
  if (tid < (stats ? 5 : 4)) atomicAdd(reinterpret_cast<unsigned long long*>(o.light + kAdd[tid]), t.add[tid]);
  if (tid < (stats ? 5 : 3) && t.top[tid]) atomicMax(o.light + kTop[tid], t.top[tid]);
  if (tid == 0 && t.cut) atomicAdd(o.light + kLightSeen + 4, t.cut);
}

// The rows of the resident matrix; with `stats` also the finite min / max and the number of finite
// entries (the index's words 8..11).
template <int Cap>
__global__ void __launch_bounds__(256) k_light_rows(const int32_t* __restrict__ W, int64_t pitch, const LightOut o,
                                                    bool stats) {
  __shared__ __align__(16) uint32_t s_buf[8][kLightBuf];
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  const int64_t nq = pitch / 4;
  uint32_t thr = warp < o.n ? first_threshold(o, W + warp * pitch, static_cast<uint32_t>(warp), 2.25f * Cap) : 0u, gmin = kInf, gmax = 0;
  unsigned long long cnt = 0;
  LightSums sums;
  for (int64_t u = warp; u < o.n; u += nwarps) {
    const int32_t* row = W + u * pitch;
    uint32_t mx = 0, c = 0;
    auto scan = [&](const auto& f, int pass) {
      for (int64_t q0 = 0; q0 < nq; q0 += 4 * 32) {
        int4 x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int64_t q = q0 + 32 * r + lane;
          x[r] = q < nq ? __ldg(reinterpret_cast<const int4*>(row) + q)
                        : make_int4(int(kInf), int(kInf), int(kInf), int(kInf));
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const uint32_t c0 = static_cast<uint32_t>(4 * (q0 + 32 * r + lane));
          if (pass == 0 && stats) {
            const uint32_t w4[4] = {static_cast<uint32_t>(x[r].x), static_cast<uint32_t>(x[r].y),
                                    static_cast<uint32_t>(x[r].z), static_cast<uint32_t>(x[r].w)};
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (w4[k] < kInf && c0 + k != u) {
                mx = max(mx, w4[k]);
                ++c;
              }
          }
          f(c0, x[r]);
        }
      }
    };
    light_row<Cap>(o, scan, static_cast<uint32_t>(u), s_buf[threadIdx.x >> 5], thr, sums);
    if (lane == 0) gmin = min(gmin, static_cast<uint32_t>(o.minout[u]));
    gmax = max(gmax, mx);
    cnt += c;
  }
  for (int k = 16; k > 0; k >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, k);
  light_sums_out(o, sums, stats, gmin, __reduce_max_sync(0xffffffffu, gmax), cnt);
}

// Upload from pinned host memory (device-accessible through unified addressing): each warp copies one
// row at a time from `src` (row stride ld) into the graph's row and selects its light edges on the
// way (k_light_rows), so the matrix crosses the host link once and is not read from HBM again.  With
// `vec` (ld a multiple of 4, src 16-byte aligned) the row moves in 16-byte pieces, four in flight per
// lane, otherwise in 4-byte pieces, eight in flight (sixteen: n = 6001 796 us, not 773).  Padding columns are left
// as they are (INF).
__global__ void __launch_bounds__(256) k_upload_rows(const int32_t* __restrict__ src, int64_t ld,
                                                     int32_t* __restrict__ W, int64_t pitch, const LightOut o,
                                                     int vec) {
  __shared__ __align__(16) uint32_t s_buf[8][kLightBuf];
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  const int4 none = make_int4(int(kInf), int(kInf), int(kInf), int(kInf));
  uint32_t thr = first_threshold(o, nullptr, 0, 0.f);
  LightSums sums;
  for (int64_t u = warp; u < o.n; u += nwarps) {
    const int32_t* s = src + u * ld;
    int32_t* d = W + u * pitch;
    auto scan = [&](const auto& f, int pass) {
      if (!vec && pass == 0) {
        for (int64_t b = 0; b < o.n; b += 2 * 128) {
          int4 x[2];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int64_t c = b + 128 * r + lane;
            x[r].x = c < o.n ? s[c] : none.x;
            x[r].y = c + 32 < o.n ? s[c + 32] : none.x;
            x[r].z = c + 64 < o.n ? s[c + 64] : none.x;
            x[r].w = c + 96 < o.n ? s[c + 96] : none.x;
          }
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int64_t c = b + 128 * r + lane;
            if (c < o.n) d[c] = x[r].x;
            if (c + 32 < o.n) d[c + 32] = x[r].y;
            if (c + 64 < o.n) d[c + 64] = x[r].z;
            if (c + 96 < o.n) d[c + 96] = x[r].w;
            if (b + 128 * r < o.n) f(static_cast<uint32_t>(c), x[r], 32u);
          }
        }
        __syncwarp();  // later scans read the row as every lane wrote it
        return;
      }
      const bool copy = vec && pass == 0;
      const int4* from = reinterpret_cast<const int4*>(copy ? s : d);
      const int64_t nq = copy ? o.n / 4 : pitch / 4;
      for (int64_t q0 = 0; q0 < nq; q0 += 4 * 32) {
        int4 x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int64_t q = q0 + 32 * r + lane;
          x[r] = q < nq ? from[q] : none;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int64_t q = q0 + 32 * r + lane;
          if (copy && q < nq) reinterpret_cast<int4*>(d)[q] = x[r];
          f(static_cast<uint32_t>(4 * q), x[r]);
        }
      }
      if (copy) {
        const int64_t c0 = 4 * nq;  // the last n mod 4 entries
        int4 x = none;
        if (lane == 0) {
          if (c0 < o.n) d[c0] = x.x = s[c0];
          if (c0 + 1 < o.n) d[c0 + 1] = x.y = s[c0 + 1];
          if (c0 + 2 < o.n) d[c0 + 2] = x.z = s[c0 + 2];
        }
        if (c0 < o.n) f(static_cast<uint32_t>(c0 + 4 * lane), x);
        __syncwarp();  // later scans read the row as every lane wrote it
      }
    };
    light_row<kLightCap>(o, scan, static_cast<uint32_t>(u), s_buf[threadIdx.x >> 5], thr, sums);
  }
  light_sums_out(o, sums);
}

// The rows' kInLists smallest weights with their columns (what k_outlist gives), from the index: a
// thread per row.  A row whose index list is shorter than that and misses edges lists nothing, which
// keeps the static minimum as its bound.
__global__ void k_index_lists(const uint32_t* __restrict__ light, int32_t n, uint32_t bits_u,
                              uint2* __restrict__ outlist, uint32_t* __restrict__ outrest) {
  const int64_t u = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (u >= n) return;
  const uint32_t* hmin = light + kLightStats;
  const uint32_t* edge = hmin + light_pad(n) + u * kLightCap;
  uint32_t e[kInLists + 1];
#pragma unroll
  for (int i = 0; i <= kInLists; ++i) e[i] = edge[i];
  const bool missing = hmin[u] < kInf;
  const bool use = !missing || e[kInLists - 1] != kNoEdge;
#pragma unroll
  for (int i = 0; i < kInLists; ++i)
    outlist[u * kInLists + i] =
        use && e[i] != kNoEdge ? make_uint2(e[i] >> bits_u, e[i] & ((1u << bits_u) - 1u)) : make_uint2(kInf, 0xFFFFFFFFu);
  outrest[u] = use && (e[kInLists] != kNoEdge || missing) ? e[kInLists - 1] >> bits_u : kInf;
}

// minin[v] = min finite W[u][v], u != v.  A block covers 256 columns x kColRows
// rows (coalesced row reads), keeps a per-column minimum in registers and
// folds it into minin with one atomicMin per column.  minin starts at INF.
constexpr int kColRows = 256;
__global__ void k_colmin(const int32_t* __restrict__ W, int64_t pitch, int32_t n, int32_t* __restrict__ minin) {
  const int64_t v = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * kColRows;
  if (v >= n) return;
  uint32_t mn = kInf;
  const int64_t r1 = min(static_cast<int64_t>(n), r0 + kColRows);
  for (int64_t u = r0; u < r1; ++u) {
    const uint32_t x = static_cast<uint32_t>(W[u * pitch + v]);
    if (u != v) mn = min(mn, x);
  }
  if (mn < kInf) atomicMin(minin + v, static_cast<int32_t>(mn));
}

// Tie sources: for every column v, the rows u != v with W[u][v] == minin[v],
// up to cap per column; tcnt[v] counts them all (starts at 0).  A column whose
// stored dist equals m + minin[v] can only be tied by one of these rows.  A
// block covers 256 columns x kColRows rows like k_colmin: each thread keeps
// its column's minin in a register and reads the rows coalesced.
__global__ void k_tiesrc(const int32_t* __restrict__ W, int64_t pitch, int32_t n, const int32_t* __restrict__ minin,
                         int32_t* __restrict__ tsrc, int32_t* __restrict__ tcnt, int32_t cap) {
  const int64_t v = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * kColRows;
  if (v >= n) return;
  const int32_t mv = minin[v];
  if (static_cast<uint32_t>(mv) >= kInf) return;  // no finite weight into v
  const int64_t r1 = min(static_cast<int64_t>(n), r0 + kColRows);
#pragma unroll 8
  for (int64_t u = r0; u < r1; ++u) {
    if (W[u * pitch + v] == mv && u != v) {
      const int32_t pos = atomicAdd(tcnt + v, 1);
      if (pos < cap) tsrc[v * cap + pos] = static_cast<int32_t>(u);
    }
  }
}

// In-lists: for every column v the kInLists smallest finite off-diagonal weights W[u][v] with
// their rows u, ascending by (weight, row), and a lower bound on every other in-weight (the
// kInLists-th weight when the column has more in-edges, INF otherwise).  A block takes 32 columns, a
// thread per column in each of its 8 warps, which read rows 8 at a time (128 contiguous bytes each) and
// merge their lists at the end; a thread per column alone left too few loads in flight (n = 32768,
// 4 GiB: 2.99 ms, now 0.94).
__global__ void __launch_bounds__(256) k_inlist(const int32_t* __restrict__ W, int64_t pitch, int32_t n,
                                                uint2* __restrict__ inlist, uint32_t* __restrict__ inrest) {
  constexpr int kWarps = 8;
  __shared__ uint64_t s_key[kWarps][kInLists][32];
  __shared__ uint32_t s_cnt[kWarps][32];
  const int lane = static_cast<int>(threadIdx.x) & 31, warp = static_cast<int>(threadIdx.x) >> 5;
  const int64_t v = static_cast<int64_t>(blockIdx.x) * 32 + lane;  // < pitch: padding columns are INF
  uint64_t k[kInLists];
#pragma unroll
  for (int i = 0; i < kInLists; ++i) k[i] = ~0ull;
  uint32_t cnt = 0;
  auto insert = [&](uint64_t key) {  // into the sorted list
#pragma unroll
    for (int i = 0; i < kInLists; ++i)
      if (key < k[i]) {
        const uint64_t t = k[i];
        k[i] = key;
        key = t;
      }
  };
  const int32_t* col = W + v;
  for (int64_t u0 = 8 * warp; u0 < n; u0 += 8 * kWarps) {
    uint32_t w8[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) w8[r] = u0 + r < n ? static_cast<uint32_t>(__ldg(col + (u0 + r) * pitch)) : kInf;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int64_t u = u0 + r;
      if (w8[r] >= kInf || u == v) continue;
      ++cnt;
      insert((static_cast<uint64_t>(w8[r]) << 32) | static_cast<uint32_t>(u));
    }
  }
#pragma unroll
  for (int i = 0; i < kInLists; ++i) s_key[warp][i][lane] = k[i];
  s_cnt[warp][lane] = cnt;
  __syncthreads();
  if (warp != 0 || v >= n) return;
  for (int g = 1; g < kWarps; ++g) {
    cnt += s_cnt[g][lane];
#pragma unroll
    for (int i = 0; i < kInLists; ++i) insert(s_key[g][i][lane]);
  }
#pragma unroll
  for (int i = 0; i < kInLists; ++i)
    inlist[v * kInLists + i] = k[i] == ~0ull ? make_uint2(kInf, 0xFFFFFFFFu)
                                             : make_uint2(static_cast<uint32_t>(k[i] >> 32), static_cast<uint32_t>(k[i]));
  inrest[v] = cnt > static_cast<uint32_t>(kInLists) ? static_cast<uint32_t>(k[kInLists - 1] >> 32) : kInf;
}

// Out-lists: for every row u the kInLists smallest finite off-diagonal weights W[u][v] with their
// columns, ascending by (weight, column), and the lower bound on the others (as k_inlist).  One
// warp per row: each lane keeps the smallest of its columns, then the warp takes the list's
// entries one by one as the minimum of the lanes' heads.
__global__ void k_outlist(const int32_t* __restrict__ W, int64_t pitch, int32_t n, uint2* __restrict__ outlist,
                          uint32_t* __restrict__ outrest) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t u = warp; u < n; u += nwarps) {
    const int32_t* row = W + u * pitch;
    uint64_t k[kInLists];
#pragma unroll
    for (int i = 0; i < kInLists; ++i) k[i] = ~0ull;
    uint32_t cnt = 0;
    for (int64_t v = lane; v < n; v += 32) {
      const uint32_t w = static_cast<uint32_t>(__ldg(row + v));
      if (w >= kInf || v == u) continue;
      ++cnt;
      uint64_t key = (static_cast<uint64_t>(w) << 32) | static_cast<uint32_t>(v);
#pragma unroll
      for (int i = 0; i < kInLists; ++i)
        if (key < k[i]) {
          const uint64_t t = k[i];
          k[i] = key;
          key = t;
        }
    }
    cnt = warp_sum_u32(cnt);
    uint64_t out[kInLists];
#pragma unroll
    for (int i = 0; i < kInLists; ++i) {  // the warp's i-th smallest: the minimum of the lanes' heads
      const uint64_t mn = warp_min_u64(k[0]);
      out[i] = mn;
      if (k[0] == mn && mn != ~0ull) {  // keys are distinct (the column is in the key): one lane pops
#pragma unroll
        for (int j = 0; j + 1 < kInLists; ++j) k[j] = k[j + 1];
        k[kInLists - 1] = ~0ull;
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < kInLists; ++i)
        outlist[u * kInLists + i] = out[i] == ~0ull ? make_uint2(kInf, 0xFFFFFFFFu)
                                                    : make_uint2(static_cast<uint32_t>(out[i] >> 32),
                                                                 static_cast<uint32_t>(out[i]));
      outrest[u] = cnt > static_cast<uint32_t>(kInLists) ? static_cast<uint32_t>(out[kInLists - 1] >> 32) : kInf;
    }
  }
}

__global__ void k_fill_i32(int32_t* __restrict__ p, int64_t count, int32_t value) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    p[i] = value;
}

// Columns [n, pitch) of every row hold INF.
__global__ void k_pad_cols(int32_t* __restrict__ W, int64_t pitch, int32_t n) {
  const int64_t padw = pitch - n;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < padw * n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t r = i / padw;
    W[r * pitch + n + (i - r * padw)] = static_cast<int32_t>(kInf);
  }
}

// flags[0] |= 1 if any of the n x n entries is negative.
__global__ void __launch_bounds__(256) k_check_nonneg(const int32_t* __restrict__ W, int64_t pitch, int32_t n,
                                                      uint32_t* flags) {
  uint32_t sign = 0;
  for (int64_t r = blockIdx.x; r < n; r += gridDim.x)
    for (int c = threadIdx.x; c < n; c += 256) sign |= static_cast<uint32_t>(W[r * pitch + c]);
  if (sign >> 31) atomicOr(flags, 1u);
}

}  // namespace dj

using namespace dj;

static int grid_for(int64_t work, int threads = 256) {
  int64_t b = (work + threads - 1) / threads;
  return static_cast<int>(std::min<int64_t>(std::max<int64_t>(b, 1), 152 * 32));
}

// One allocation for the matrix, the minima, the tie sources and the light-edge index (a cudaMalloc
// each cost as much as building a small graph).
static int alloc_graph(int32_t n, int directed, dj_graph** out) {
  auto* g = new dj_graph();
  g->n = n;
  g->pitch = (n + 31) / 32 * 32;
  g->directed = directed ? 1 : 0;
  cudaGetDevice(&g->device);
  auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t mbytes = static_cast<size_t>(n) * g->pitch * sizeof(int32_t);
  const size_t min_bytes = 2 * static_cast<size_t>(n) * sizeof(int32_t);
  const size_t tie_bytes = static_cast<size_t>(n) * (kTieSourceCap + 1) * sizeof(int32_t);
  const size_t base = up(mbytes) + up(min_bytes) + up(tie_bytes);
  g->light_bytes = light_index_bytes(n);
  if (cudaMalloc(&g->block, base + g->light_bytes) != cudaSuccess) {
    cudaGetLastError();
    g->light_bytes = 0;  // no room for the index: the graph is solved from the matrix alone
    if (cudaMalloc(&g->block, base) != cudaSuccess) {
      cudaGetLastError();
      delete g;
      return set_error(DJ_ENOMEM, "cudaMalloc of the adjacency matrix failed (" + std::to_string(mbytes) + " bytes)");
    }
  }
  auto* p = static_cast<uint8_t*>(g->block);
  g->W = reinterpret_cast<int32_t*>(p);
  g->minout = reinterpret_cast<int32_t*>(p + up(mbytes));
  g->minin = g->minout + n;
  g->tsrc = reinterpret_cast<int32_t*>(p + up(mbytes) + up(min_bytes));
  g->tcap = kTieSourceCap;
  g->tcnt = g->tsrc + static_cast<size_t>(n) * kTieSourceCap;
  if (g->light_bytes) g->light = reinterpret_cast<uint32_t*>(p + base);
  g->bytes = mbytes + min_bytes + tie_bytes + g->light_bytes;
  *out = g;
  return DJ_OK;
}

static void launch_inlists(dj_graph* g, cudaStream_t st) {
  if (g->light) {
    k_index_lists<<<static_cast<unsigned>((g->n + 255) / 256), 256, 0, st>>>(
        g->light, g->n, host_bits_for(static_cast<uint32_t>(g->n)), g->outlist, g->outrest);
    if (g->outlist == g->inlist) return;  // symmetric: a node's in-edges are its out-edges
    k_inlist<<<static_cast<unsigned>((g->n + 31) / 32), 256, 0, st>>>(g->W, g->pitch, g->n, g->inlist, g->inrest);
    return;
  }
  k_inlist<<<static_cast<unsigned>((g->n + 31) / 32), 256, 0, st>>>(g->W, g->pitch, g->n, g->inlist, g->inrest);
  if (g->outlist != g->inlist)
    k_outlist<<<grid_for(static_cast<int64_t>(g->n) * 32), 256, 0, st>>>(g->W, g->pitch, g->n, g->outlist, g->outrest);
}

static LightOut light_out(const dj_graph* g) {
  return LightOut{g->light, g->minout, g->directed ? nullptr : g->tsrc, g->tcnt, g->tcap,
                  host_bits_for(static_cast<uint32_t>(g->n)), g->n, g->light_deg,
                  static_cast<uint32_t>(g->wmax), g->light_first};
}

// Row minima (with the index, on a symmetric matrix the tie sources too; unless `have_rows`: the upload kernel took
// them), column minima, tie sources and, for graphs that keep them, the in- and out-lists.
static void launch_minima(dj_graph* g, uint32_t* stats, cudaStream_t st, bool have_rows = false) {
  const bool rows_done = have_rows || g->light;
  if (!have_rows && g->light) {
    k_light_rows<kLightCap><<<grid_for(static_cast<int64_t>(g->n) * 32), 256, 0, st>>>(g->W, g->pitch, light_out(g), stats != nullptr);
  } else if (!have_rows) {
    k_rowmin<<<grid_for(static_cast<int64_t>(g->n) * 32), 256, 0, st>>>(g->W, g->pitch, g->n, g->minout, stats);
  }
  if (!(rows_done && !g->directed)) {  // symmetric: the rows gave minin and the tie sources
    if (!g->directed) {
      cudaMemcpyAsync(g->minin, g->minout, static_cast<size_t>(g->n) * sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
    } else {
      k_fill_i32<<<grid_for(g->n), 256, 0, st>>>(g->minin, g->n, static_cast<int32_t>(kInf));
      dim3 grid(static_cast<unsigned>((g->n + 255) / 256), static_cast<unsigned>((g->n + kColRows - 1) / kColRows));
      k_colmin<<<grid, 256, 0, st>>>(g->W, g->pitch, g->n, g->minin);
    }
    cudaMemsetAsync(g->tcnt, 0, static_cast<size_t>(g->n) * sizeof(int32_t), st);
    dim3 tgrid(static_cast<unsigned>((g->n + 255) / 256), static_cast<unsigned>((g->n + kColRows - 1) / kColRows));
    k_tiesrc<<<tgrid, 256, 0, st>>>(g->W, g->pitch, g->n, g->minin, g->tsrc, g->tcnt, g->tcap);
  }
  if (g->inlist) launch_inlists(g, st);
}

// The trial solve on the index, and the index's leading words on their way to the host.
static bool launch_trial(dj_graph* g, uint32_t* idx, cudaStream_t st) {
  const bool tried = launch_light_trial(g, kTrialFirst, g->light + 1, st) == DJ_OK;
  clear_error();  // it cannot run here: the other engines
  cudaMemcpyAsync(idx, g->light, kLightHost * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  return tried;
}

// Whether a graph with cut lists is one whose solves hardly need a row whole, by its trial (idx) and, where
// that leaves it open, by further ones: side by side, a CTA each, where the state fits one (n = 4099 and 8192
// 78 and 96 us, n = 6001 on lists of 128 133; one over every SM takes 34-52), else one after another.
static int cut_lists_serve(dj_graph* g, const uint32_t* idx, cudaStream_t st, bool* good) {
  const int verdict = light_trial_verdict(idx[1], idx[kLightGuess], idx[kLightRisky]);
  *good = verdict == kTrialAll;
  if (verdict != kTrialAsk) return DJ_OK;
  uint32_t* more = g->light + kLightMore;
  cudaMemsetAsync(more, 0, kMoreTrials * sizeof(uint32_t), st);
  bool tried = true;
  if (g->directed) {  // for the grid form: one more
    tried = launch_light_trial(g, kTrialFar, more, st) == DJ_OK;
  } else if (light_cta_fits(g->n)) {
    LightPlan plan;
    tried = plan_light(g->n, kMoreTrials, kJobsTrial, &plan) == DJ_OK &&
            run_light_trials(plan, make_desc(g, 0, nullptr, nullptr, 0), g->light, st) == DJ_OK;
  } else {
    for (int i = 0; i < 6; ++i)  // the farthest node, the farthest from that, and four places
      tried = tried && launch_light_trial(g, i < 2 ? kTrialFar : static_cast<int32_t>(static_cast<int64_t>(g->n) * (2 * i - 3) / 8),
                                          more + i, st) == DJ_OK;
  }
  clear_error();
  static_assert(kLightMore + kMoreTrials == kLightError, "one copy takes both");
  uint32_t rows[kMoreTrials + 1] = {0};  // and the error bits
  cudaMemcpyAsync(rows, more, sizeof(rows), cudaMemcpyDeviceToHost, st);
  const cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_error(e, "trial solves");
  *good = tried && rows[kMoreTrials] == 0 && *std::max_element(rows, rows + kMoreTrials) <= kTrialMoreRows;
  return DJ_OK;
}

// Whether lists of kLightWide edges would hold every edge that matters: the source's row needs the most of
// them, those of weight up to the largest dist (the trial's).  Their number is estimated from the lists, from the
// edges up to the thresholds (a list cut among equal weights misses some of those), and as if the weights were uniform
// between the smallest and the largest, whichever is most.
static double sum_at(const uint32_t* words) { return words[0] + 4294967296.0 * words[1]; }
static bool wide_suffices(const dj_graph* g, const uint32_t* idx) {
  if (idx[kLightGuess] == 0) return false;
  const double D = idx[kLightGuess] - 1.0;
  const double listed = sum_at(idx + 4), last = sum_at(idx + 2);  // edges per unit of weight, in the lists
  const double seen = sum_at(idx + kLightSeen), thr = sum_at(idx + kLightSeen + 2);  // and up to the thresholds
  const double uniform = g->light_deg * (D - g->wmin + 1.0) / (static_cast<double>(g->wmax) - g->wmin + 1.0);
  return std::max({last > 0 ? listed / last * D : 0.0, thr > 0 ? seen / thr * D : 0.0, uniform}) <= 1.1 * kLightWide;
}

// Row and column minima, index, global weight range, then the overflow rule (n-1) * wmax < INT32_MAX.
// The index's leading words are zero before, but for the edge list's check (words 12..14), whose
// verdict *list gets (nullptr: there was no list).
//
// Whether solves take the light engine is decided here, by a trial solve: one more kernel in front of
// the wait, the only one unless that leaves it open or longer lists are worth a try.
static int finish_graph(dj_graph* g, cudaStream_t st, uint32_t* list) {
  uint32_t* stats = g->light ? g->light + 8 : nullptr;
  uint32_t idx[kLightHost] = {0};
  cudaError_t e = cudaSuccess;
  if (!g->light) {
    e = cudaMallocAsync(&stats, 4 * sizeof(uint32_t), st);
    if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync(stats)");
    uint32_t init[4] = {kInf, 0, 0, 0};
    cudaMemcpyAsync(stats, init, sizeof(init), cudaMemcpyHostToDevice, st);
  }
  launch_minima(g, stats, st);
  bool tried = false;
  if (g->light) {
    tried = launch_trial(g, idx, st);
  } else {
    cudaMemcpyAsync(idx + 8, stats, 4 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(stats, st);
  }
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_error(e, "building the row minima");
  if (list && g->light) std::memcpy(list, idx + 12, 3 * sizeof(uint32_t));
  g->wmin = static_cast<int32_t>(g->light ? ~idx[8] : idx[8]);
  g->wmax = static_cast<int32_t>(idx[9]);
  g->entries = static_cast<uint64_t>(idx[10]) | (static_cast<uint64_t>(idx[11]) << 32);
  g->light_deg = static_cast<float>(static_cast<double>(g->entries) / g->n);
  if (g->n > 1 && static_cast<int64_t>(g->n - 1) * g->wmax >= static_cast<int64_t>(DJ_INF))
    return set_error(DJ_EOVERFLOW, "(n-1) * max weight >= INT32_MAX: path lengths could overflow int32");
  // Taken at once if every row's list is complete, else if trial solves relaxed next to no row whole:
  // where many are needed (nearly equal weights, distances long against what the lists reach, parts that
  // a source cannot reach) the other engines stream the matrix better (n = 8192, p = 0.5, weights 1..10: 410
  // rows whole, 112 us; grid engine 37).  One CTA or cluster relaxes many whole rows slowly (4500 in 7 ms,
  // the grid form in 0.2), so these forms are for complete lists and symmetric matrices.  Where the first
  // trial does not settle it for every source (light_trial_verdict), more are made.  A graph whose
  // trial did not reach every node that something leads to is left to the other engines: two parts of 4000
  // nodes, p = 0.3, took a CTA 15.3 ms a solve, the cluster engine 0.7.
  // Lists of kLightWide edges are built instead (one more pass and its trials) where these look enough: n = 6001,
  // p = 0.05, weights 1..10 needs 288 rows whole with 64 edges listed, none with 128, and takes 14.6 us a
  // solve (the streaming grid engine 51) for a load of 0.69 ms instead of 0.45 (before the index: 1.60).
  bool good = false;
  uint32_t guess = idx[kLightGuess];  // 0: lists of 64 hold every edge, or the trial missed some node
  tried = tried && g->wmin >= 1;
  bool complete = tried && ~idx[0] >= kInf;
  if (tried && !complete)
    if (int rc = cut_lists_serve(g, idx, st, &good)) return rc;
  if (tried && !complete && !good && wide_suffices(g, idx)) {
    cudaMemsetAsync(g->light, 0, 8 * sizeof(uint32_t), st);
    cudaMemsetAsync(g->light + kLightGuess, 0, 9 * sizeof(uint32_t), st);  // to kLightRisky
    k_light_rows<kLightWide><<<grid_for(static_cast<int64_t>(g->n) * 32), 256, 0, st>>>(g->W, g->pitch, light_out(g),
                                                                                        false);
    tried = launch_trial(g, idx, st);
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_error(e, "building the longer lists");
    g->light_wide = true;
    complete = tried && ~idx[0] >= kInf;  // (then there was no trial on the longer ones)
    if (idx[kLightGuess]) guess = idx[kLightGuess];
    if (tried && !complete)
      if (int rc = cut_lists_serve(g, idx, st, &good)) return rc;
  }
  // an upload's first threshold: the mean of those that served this matrix (the new one is likely of its kind)
  const uint32_t cut = idx[kLightSeen + 4];
  g->light_first = cut ? static_cast<float>(sum_at(idx + kLightSeen + 2) / cut + 0.5) : ~idx[0] >= kInf ? 2.0e9f : 0.f;
  g->light_ok = complete || good;
  g->light_few = g->light_ok && light_few(g->n, guess, g->wmin);
  g->light_cta = g->light_ok && (complete || !g->directed);
  // graphs that are not dense keep in-lists for the grid engine's dynamic IN bound
  const uint64_t nn = static_cast<uint64_t>(g->n) * static_cast<uint64_t>(g->n);
  if (g->entries * 32 < nn && g->wmin >= 1 && !g->inlist) {
    const size_t lb = static_cast<size_t>(g->n) * kInLists * sizeof(uint2), rb = static_cast<size_t>(g->n) * 4;
    const int lists = g->directed ? 2 : 1;  // a symmetric matrix's out-lists are its in-lists
    uint8_t* buf = nullptr;
    // [in-lists][out-lists][in rests][out rests]: the 8-byte entries first, at multiples of 32 n bytes
    if (cudaMalloc(&buf, lists * (lb + rb)) == cudaSuccess) {
      g->inlist = reinterpret_cast<uint2*>(buf);
      g->outlist = lists == 2 ? reinterpret_cast<uint2*>(buf + lb) : g->inlist;
      g->inrest = reinterpret_cast<uint32_t*>(buf + lists * lb);
      g->outrest = lists == 2 ? reinterpret_cast<uint32_t*>(buf + 2 * lb + rb) : g->inrest;
      g->bytes += lists * (lb + rb);
      launch_inlists(g, st);
      e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return cuda_error(e, "building the in-lists");
    } else {
      cudaGetLastError();  // no room: the static IN bound only
    }
  }
  return DJ_OK;
}

// The status of edge e of the caller's list (the message names it).
static int edge_status(int64_t e, int32_t n, const int32_t* src, const int32_t* dst, const int32_t* w) {
  if (src[e] < 0 || src[e] >= n || dst[e] < 0 || dst[e] >= n)
    return set_error(DJ_EINVAL, "edge " + std::to_string(e) + " has a node id outside [0, n)");
  if (w[e] < 0 || w[e] == DJ_INF)
    return set_error(DJ_EINVAL, "edge " + std::to_string(e) + " has a weight outside [0, INT32_MAX)");
  return DJ_OK;
}

// (n - 1) * wmax must stay below INT32_MAX: path lengths are int32.
static int weight_status(int32_t n, int64_t wmax) {
  if (n > 1 && static_cast<int64_t>(n - 1) * wmax >= static_cast<int64_t>(DJ_INF))
    return set_error(DJ_EOVERFLOW, "(n-1) * max weight >= INT32_MAX: path lengths could overflow int32");
  return DJ_OK;
}

// The whole list checked on the host: only where the device cannot (no device, no memory), so that a
// bad list is reported as such there too.
static int list_status(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, const int32_t* w) {
  int64_t wmax = 0;
  for (int64_t e = 0; e < m; ++e) {
    if (int rc = edge_status(e, n, src, dst, w)) return rc;
    if (src[e] != dst[e]) wmax = std::max<int64_t>(wmax, w[e]);
  }
  return weight_status(n, wmax);
}

extern "C" int dj_load_edges(int32_t n, int64_t m, const int32_t* src, const int32_t* dst, const int32_t* w,
                             int directed, uint64_t stream, dj_graph** out) {
  clear_error();
  if (!out) return set_error(DJ_EINVAL, "out is NULL");
  *out = nullptr;
  if (n < 1) return set_error(DJ_EINVAL, "n must be >= 1");
  if (m < 0) return set_error(DJ_EINVAL, "m must be >= 0");
  if (m > 0 && (!src || !dst || !w)) return set_error(DJ_EINVAL, "edge arrays are NULL");
  DevCtx* ctx = nullptr;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  dj_graph* g = nullptr;
  uint32_t res[3] = {0, 0, 0};
  int rc = get_ctx(&ctx);
  if (rc == DJ_OK) rc = alloc_graph(n, directed, &g);
  if (rc != DJ_OK) {
    const std::string why = dj_last_error();
    if (int lrc = list_status(n, m, src, dst, w)) return lrc;
    return set_error(rc, why);
  }
  // the list's check words lie in the index (read with its statistics), or without one in the tie
  // sources' place, which is filled later
  uint32_t* check = g->light ? g->light + 12 : reinterpret_cast<uint32_t*>(g->tsrc);
  if (g->light) cudaMemsetAsync(g->light, 0, kLightStats * sizeof(uint32_t), st);
  g->light_deg = static_cast<float>(static_cast<double>(directed ? m : 2 * m) / n);
  k_fill<<<grid_for(static_cast<int64_t>(n) * g->pitch / 4), 256, 0, st>>>(g->W, g->pitch, n);
  if (m > 0) {
    cudaError_t e = cudaSuccess;
    if (!g->light) e = cudaMemsetAsync(check, 0, 16, st);
    if (e == cudaSuccess && ctx->pageable && edges_in_place(src, dst, w)) {
      // the device reads the caller's arrays over the host link itself (coherent host memory): one pass,
      // no staging copies, no host loop, no wait of its own.  Loading 67 M edges (805 MB) into n = 16384:
      // 5.4 ms, against 86 ms with a host check and pageable copies, most of it the host's two walks over
      // the list; 2.5 M edges into n = 4099: 0.45 against 3.6 ms; 1491 edges into n = 100: 0.07 against 0.31.
      // Arrays that are not 4-byte aligned go through the copies below, which take any address.
      k_scatter<<<grid_for((m + kScatterEdges - 1) / kScatterEdges), 256, 0, st>>>(g->W, g->pitch, n, src, dst, w, m, 0,
                                                                                   directed, check);
    } else if (e == cudaSuccess) {
      const int64_t chunk = std::min<int64_t>(m, int64_t(1) << 24);  // 16 Mi edges (192 MiB) per stage
      int32_t* stage = nullptr;
      e = cudaMallocAsync(&stage, static_cast<size_t>(chunk) * 3 * sizeof(int32_t), st);
      for (int64_t off = 0; e == cudaSuccess && off < m; off += chunk) {
        const int64_t c = std::min(chunk, m - off);
        cudaMemcpyAsync(stage, src + off, c * sizeof(int32_t), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(stage + chunk, dst + off, c * sizeof(int32_t), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(stage + 2 * chunk, w + off, c * sizeof(int32_t), cudaMemcpyHostToDevice, st);
        k_scatter<<<grid_for((c + kScatterEdges - 1) / kScatterEdges), 256, 0, st>>>(
            g->W, g->pitch, n, stage, stage + chunk, stage + 2 * chunk, c, off, directed, check);
        // the host arrays may be pageable: finish this stage before reusing the buffer
        e = cudaStreamSynchronize(st);
      }
      if (stage) cudaFreeAsync(stage, st);
    }
    if (e == cudaSuccess && !g->light) {
      e = cudaMemcpyAsync(res, check, 3 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (e != cudaSuccess) rc = cuda_error(e, "scattering edges");
  }
  // a bad list's first bad edge is reported before anything the built matrix shows
  const int frc = rc == DJ_OK ? finish_graph(g, st, res) : rc;  // the edge arrays are the caller's again
  const std::string fwhy = dj_last_error();
  if (const uint64_t bad = static_cast<uint64_t>(res[0]) | (static_cast<uint64_t>(res[1]) << 32)) {
    rc = edge_status(static_cast<int64_t>(~bad), n, src, dst, w);
    if (rc == DJ_OK) rc = set_error(DJ_EINVAL, "the edge list changed while it was read");
  } else if (frc != DJ_OK) {
    rc = set_error(frc, fwhy);
  } else {
    rc = weight_status(n, res[2]);
  }
  if (rc != DJ_OK) {
    const std::string why = dj_last_error();
    dj_graph_free(g);
    return set_error(rc, why);
  }
  *out = g;
  return DJ_OK;
}

static int copy_dense_in(dj_graph* g, const int32_t* W, int64_t ld, int w_on_device, cudaStream_t st) {
  const int32_t n = g->n;
  uint32_t* flags = nullptr;
  cudaError_t e = cudaMallocAsync(&flags, sizeof(uint32_t), st);
  if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync(flags)");
  cudaMemsetAsync(flags, 0, sizeof(uint32_t), st);
  if (w_on_device) {
    const int vec = ld % 4 == 0 && reinterpret_cast<uintptr_t>(W) % 16 == 0;
    k_copy_dense<<<std::min(n, 152 * 16), 256, 0, st>>>(g->W, g->pitch, W, ld, n, vec, flags);
  } else {
    e = cudaMemcpy2DAsync(g->W, static_cast<size_t>(g->pitch) * sizeof(int32_t), W,
                          static_cast<size_t>(ld) * sizeof(int32_t), static_cast<size_t>(n) * sizeof(int32_t),
                          static_cast<size_t>(n), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpy2DAsync(host matrix)");
    k_check_nonneg<<<std::min(n, 152 * 16), 256, 0, st>>>(g->W, g->pitch, n, flags);
    if (g->pitch > n) k_pad_cols<<<grid_for(static_cast<int64_t>(g->pitch - n) * n), 256, 0, st>>>(g->W, g->pitch, n);
  }
  uint32_t bad = 0;
  cudaMemcpyAsync(&bad, flags, sizeof(bad), cudaMemcpyDeviceToHost, st);
  cudaFreeAsync(flags, st);
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_error(e, "copying the dense matrix");
  if (bad) return set_error(DJ_EINVAL, "matrix holds a negative entry");
  return DJ_OK;
}

extern "C" int dj_load_dense(int32_t n, const int32_t* W, int64_t ld, int w_on_device, uint64_t stream,
                             dj_graph** out) {
  clear_error();
  if (!out) return set_error(DJ_EINVAL, "out is NULL");
  *out = nullptr;
  if (n < 1 || !W || ld < n) return set_error(DJ_EINVAL, "need n >= 1, W != NULL and ld >= n");
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  dj_graph* g = nullptr;
  if (int rc = alloc_graph(n, 1, &g)) return rc;
  if (int rc = copy_dense_in(g, W, ld, w_on_device, st)) {
    dj_graph_free(g);
    return rc;
  }
  if (g->light) cudaMemsetAsync(g->light, 0, kLightStats * sizeof(uint32_t), st);
  if (int rc = finish_graph(g, st, nullptr)) {
    dj_graph_free(g);
    return rc;
  }
  *out = g;
  return DJ_OK;
}

extern "C" int dj_graph_upload(dj_graph* g, const int32_t* W, int64_t ld, uint64_t stream) {
  clear_error();
  if (int rc = require_dense(g)) return rc;
  if (!g || !W || ld < g->n) return set_error(DJ_EINVAL, "need g, W != NULL and ld >= n");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e;
  // The index is rebuilt below whichever way the matrix comes: its statistics start anew, above all the
  // length of the longest list, which captured solves read (past it lie edges of the old matrix).  The
  // trial's largest dist (kLightGuess) stays: it only bounds offers at first.
  if (g->light) cudaMemsetAsync(g->light, 0, 12 * sizeof(uint32_t), st);
  // pinned host memory the device can address: one kernel copies the rows and takes their minima
  cudaPointerAttributes pa;
  const cudaError_t pe = cudaPointerGetAttributes(&pa, W);
  if (pe != cudaSuccess) cudaGetLastError();  // clear that query's own status only
  const bool zero_copy = g->light && pe == cudaSuccess && pa.type == cudaMemoryTypeHost &&
                         pa.devicePointer != nullptr && in_place(pa.devicePointer);  // else the copies: any address
  if (zero_copy) {
    const int32_t* src = static_cast<const int32_t*>(pa.devicePointer);
    const int vec = (ld % 4 == 0 && reinterpret_cast<uintptr_t>(src) % 16 == 0) ? 1 : 0;
    // two blocks an SM keep the host link busy; with a warp for every row all would select their edges at the end,
    // when nothing is left to copy (n = 8192, weights 1..10: 1358 us, 1323 so; n = 6001, unaligned: 792 and 773)
    const int blocks = std::min((g->n + 7) / 8, 152 * 2);
    k_upload_rows<<<blocks, 256, 0, st>>>(src, ld, g->W, g->pitch, light_out(g), vec);
    e = cudaGetLastError();
  } else if (ld == g->n && g->n == g->pitch) {  // no padding columns on either side: one contiguous copy
    e = cudaMemcpyAsync(g->W, W, static_cast<size_t>(g->n) * g->pitch * sizeof(int32_t), cudaMemcpyHostToDevice, st);
  } else {
    e = cudaMemcpy2DAsync(g->W, static_cast<size_t>(g->pitch) * sizeof(int32_t), W,
                          static_cast<size_t>(ld) * sizeof(int32_t), static_cast<size_t>(g->n) * sizeof(int32_t),
                          static_cast<size_t>(g->n), cudaMemcpyHostToDevice, st);
  }
  if (e != cudaSuccess) return cuda_error(e, "host-to-device matrix copy (upload)");
  g->upload_pending = 1;
  // The index follows the matrix (a captured solve may be replayed on it), but it was tried on the
  // loaded one: nothing tells here, without a wait, whether it suits the new one.
  g->light_ok = g->light_cta = g->light_few = g->light_wide = false;
  launch_minima(g, nullptr, st, zero_copy);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "row minima");
  return DJ_OK;
}

extern "C" int dj_graph_download(const dj_graph* g, int32_t* W, int64_t ld, uint64_t stream) {
  clear_error();
  if (int rc = require_dense(g)) return rc;
  if (!g || !W || ld < g->n) return set_error(DJ_EINVAL, "need g, W != NULL and ld >= n");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpy2DAsync(W, static_cast<size_t>(ld) * sizeof(int32_t), g->W,
                                    static_cast<size_t>(g->pitch) * sizeof(int32_t), static_cast<size_t>(g->n) * sizeof(int32_t),
                                    static_cast<size_t>(g->n), cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_error(e, "cudaMemcpy2DAsync(download)");
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_error(e, "download");
  return DJ_OK;
}

extern "C" int dj_graph_get_info(const dj_graph* g, dj_graph_info* info) {
  clear_error();
  if (!g || !info) return set_error(DJ_EINVAL, "NULL argument");
  info->n = g->n;
  info->pitch = g->pitch;
  info->directed = g->directed;
  info->min_weight = g->wmin;
  info->max_weight = g->wmax;
  info->device = g->device;
  info->matrix = g->W;
  info->minout = g->minout;
  info->minin = g->minin;
  info->bytes = g->bytes;
  info->entries = g->entries;
  info->format = g->format;
  return DJ_OK;
}

extern "C" int dj_graph_free(dj_graph* g) {
  clear_error();
  if (!g) return DJ_OK;
  cudaFree(g->block);   // dense: matrix, minima, tie sources and index; compressed rows: the minima
  cudaFree(g->inlist);  // inrest shares this allocation
  cudaFree(g->row_ptr);
  cudaFree(g->edge);
  cudaFree(g->tiled);
  delete g;
  return DJ_OK;
}

namespace dj {
int require_dense(const dj_graph* g) {
  if (g && g->format != DJ_FORMAT_DENSE)
    return set_error(DJ_EUNSUPPORTED, "this call needs the dense matrix; the graph was loaded in compressed-row form");
  return DJ_OK;
}
}  // namespace dj
