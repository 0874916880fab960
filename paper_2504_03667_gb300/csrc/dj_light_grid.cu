// Light engine, grid form: one solve of Algorithm 1 over every SM, for graphs whose every weight is
// >= 1, from the light-edge index (dj_light.cuh) or from compressed rows.
//
// Keys only ever shrink, towards the smallest offer any node makes from its final dist, so rows may
// be relaxed in any order; the order only decides how much is relaxed twice.  The solve works in
// phases: the nodes whose dist changed since their row was last relaxed are dirty; a phase relaxes
// the dirty nodes of dist <= m + delta (m: the smallest dirty dist, delta: a few times the mean
// spacing of a row's listed weights, so a row has a few edges that stay inside the window).  A row is
// read up to the first edge whose offer exceeds a bound: D, the largest dist of any node (all ones until
// every node something leads to is reached), or the guess of D that the graph's trial solve left, if
// that is less.  When nothing is dirty and D is above the guess, the guess is raised and every row
// relaxed once more.  Then the index's test (hmin) either proves the answer complete or names the rows to
// relax whole from the matrix:
//   pending = { u : dist[u] + hmin[u] <= D, not yet relaxed whole }, and
//   those with dist[u] < min over pending of (dist + hmin) are final -- a shorter path would use an
//   unlisted edge of a pending row -- so each row is read from the matrix at most once (light_below also
//   sees to it that every round takes the row that gives the minimum).
//
// What bounds it: latency.  A phase is one grid barrier (which also carries m and D) and a chain of
// three L2 round trips (own keys, edges, targets' keys) around a few hundred KB of list reads.
#include <algorithm>
#include <string>

#include "dj_common.cuh"
#include "dj_internal.h"
#include "dj_jobs.cuh"
#include "dj_light.cuh"

namespace dj {

namespace {
constexpr int kLightGridThreads = 512;
constexpr int kLightRows = 4;  // rows in flight per lane group
// delta in units of the listed weights' mean spacing: a wider window means fewer phases and more
// rows relaxed twice (directed n = 32768, 8 edges per node: 90 us with 3, 81 with 8).
constexpr float kGridDelta = 8.0f;
}  // namespace

struct LightGridParams {
  const int32_t* W;           // dense graphs: the matrix (rows relaxed whole)
  const uint32_t* light;      // dense graphs: the index (dj_light.cuh); compressed rows: nullptr
  const int64_t* row_ptr;     // compressed rows: n + 1 offsets into edge
  const uint32_t* edge;       // packed edges, ascending within a row
  const int32_t* minin;
  int32_t* dist_out;
  int32_t* pred_out;
  uint32_t* ctl;              // workspace control words (zero when a launch starts)
  unsigned long long* gkey;   // n keys
  uint32_t* words;            // per-device words: [0] error bits, [1] phases
  uint32_t* heavy;            // trial: rows relaxed whole are counted here
  SolveMark mark;
  uint32_t* guess;            // the first trial: the index's kLightGuess
  int64_t pitch;
  int64_t timeout_ns;
  int32_t n;
  int32_t swcap;
  int32_t source;             // trial: or kTrialFirst, kTrialFar
  uint32_t bits_u;
  uint32_t delta;     // compressed rows (dense graphs: from the index's statistics, light_window)
  int32_t gshift;     // the same: log2 of the lanes that share a row
  int32_t skip_cta;
  int32_t trial;      // nothing is written (light_needs_trial)
};

// Control words: an abort flag and an exit counter at the grid engine's places, and three barrier
// slots of 16 bytes used in turn.  A slot holds the arrivals and, as maxima over the CTAs, ~lmin and
// the largest dist; one 16-byte acquire load returns all three together.  CTA 0 zeroes a slot once
// the next barrier has passed (everyone has read it by then) and before it arrives at the one after
// (so the zero precedes the slot's next use).
constexpr int kLgAbort = 5, kLgExit = 12, kLgSlots = 16;

__device__ __forceinline__ uint4 ld_acquire_gpu_16(const uint32_t* p) {
  uint64_t lo, hi;
  asm volatile("{\n\t.reg .b128 t;\n\tld.acquire.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(lo), "=l"(hi)
               : "l"(p)
               : "memory");
  return make_uint4(static_cast<uint32_t>(lo), static_cast<uint32_t>(lo >> 32), static_cast<uint32_t>(hi),
                    static_cast<uint32_t>(hi >> 32));
}
__device__ __forceinline__ void red_max_relaxed_gpu(uint32_t* p, uint32_t v) {
  asm volatile("red.relaxed.gpu.global.max.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

struct LgShared {
  uint32_t lmin[32], dmax[32];
  uint32_t m, D, ok, cnt, big;
};

// Grid barrier number `nbar` (0, 1, ...): combines lmin (minimum) and dmax (maximum) over the grid.
// Bounded like grid_barrier.  Every thread gets m and D; false: the launch is being aborted.
__device__ __forceinline__ bool light_barrier(const LightGridParams& p, LgShared& sh, uint32_t nbar, uint32_t lmin,
                                              uint32_t dmax, uint32_t* m, uint32_t* D) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  lmin = warp_min_u32(lmin);
  dmax = __reduce_max_sync(0xffffffffu, dmax);
  if (lane == 0) {
    sh.lmin[warp] = lmin;
    sh.dmax[warp] = dmax;
  }
  __syncthreads();
  if (warp == 0) {
    lmin = warp_min_u32(lane < nw ? sh.lmin[lane] : kNone);
    dmax = __reduce_max_sync(0xffffffffu, lane < nw ? sh.dmax[lane] : 0u);
    if (lane == 0) {
      uint32_t* slot = p.ctl + kLgSlots + 4 * (nbar % 3);
      if (lmin != kNone) red_max_relaxed_gpu(slot + 1, ~lmin);
      red_max_relaxed_gpu(slot + 2, dmax);
      red_add_release_gpu(slot, 1u);
      uint32_t ok = 1;
      uint4 x = ld_acquire_gpu_16(slot);
      if (x.x != gridDim.x) {
        const uint64_t t0 = global_ns();
        uint32_t spins = 0;
        while ((x = ld_acquire_gpu_16(slot)).x != gridDim.x) {
          if ((++spins & 63u) == 0) {
            if (ld_relaxed_gpu(p.ctl + kLgAbort)) {
              ok = 0;
              break;
            }
            if (static_cast<int64_t>(global_ns() - t0) > p.timeout_ns) {
              atomicOr(p.words, kErrTimeout);
              atomicExch(p.ctl + kLgAbort, 1u);
              ok = 0;
              break;
            }
          }
        }
      }
      if (blockIdx.x == 0 && ok && nbar > 0) {
        uint32_t* old = p.ctl + kLgSlots + 4 * ((nbar - 1) % 3);
        old[0] = 0;
        old[1] = 0;
        old[2] = 0;
      }
      sh.m = ~x.y;
      sh.D = x.z;
      sh.ok = ok;
      sh.cnt = 0;
      sh.big = 0;
    }
  }
  __syncthreads();
  *m = sh.m;
  *D = sh.D;
  return sh.ok != 0;
}

// Offer a key to v in global memory: read first (most offers lose), then a reduction.
__device__ __forceinline__ void light_offer_global(unsigned long long* gkey, uint32_t v, uint64_t key, uint64_t old,
                                                   uint32_t& lmin) {
  if (key < old) {
    atomicMin(gkey + v, static_cast<unsigned long long>(key));
    const uint32_t c = static_cast<uint32_t>(key >> 32);
    if (c < static_cast<uint32_t>(old >> 32)) lmin = min(lmin, c);
  }
}

template <bool CSR>
__device__ __forceinline__ void light_grid_solve(const LightGridParams& p, uint8_t* smem, LgShared& sh) {
  const int G = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
  const int tid = static_cast<int>(threadIdx.x), T0 = kLightGridThreads;
  const int c0 = static_cast<int>(static_cast<int64_t>(b) * p.n / G);
  const int sw = static_cast<int>(static_cast<int64_t>(b + 1) * p.n / G) - c0;
  uint8_t* q = smem;
  int64_t* start = reinterpret_cast<int64_t*>(q);
  if (CSR) q += static_cast<size_t>(p.swcap) * 8;
  uint2* list = reinterpret_cast<uint2*>(q);  // (slice index, dist) of the phase's rows; long rows from the end
  q += static_cast<size_t>(p.swcap) * 8;
  uint32_t* rdist = reinterpret_cast<uint32_t*>(q);  // dist at which the row was last relaxed
  q += static_cast<size_t>(p.swcap) * 4;
  uint32_t* aux = reinterpret_cast<uint32_t*>(q);  // compressed rows: the row's length; dense: its hmin
  q += static_cast<size_t>(p.swcap) * 4;
  uint8_t* flags = q;  // 1: something leads to the node, 2: its row was relaxed whole

  const uint32_t bits_u = p.bits_u, umask = (1u << bits_u) - 1u;
  const uint32_t* hmin = CSR ? nullptr : p.light + kLightStats;
  const uint32_t hmin_min = CSR ? kInf : ~__ldg(p.light);
  const uint32_t most = CSR ? 0u : __ldg(p.light + 6);  // edges in the longest list
  uint32_t delta = p.delta;
  int gshift = p.gshift;
  if (!CSR) light_window(p.light, kGridDelta, &delta, &gshift);
  // a trial is of use to graphs whose solves may take this engine: some list cut, no weight of 0
  if (!CSR && p.trial && !light_needs_trial(hmin_min, ~__ldg(p.light + 8))) return;
  const int source = p.source >= 0            ? p.source
                     : p.source == kTrialFirst ? static_cast<int>(light_trial_source(__ldcg(p.light + 7), p.n))
                                               : static_cast<int>(__ldcg(p.light + kLightFar));
  // offers above the guessed largest dist are dropped at first (see below); the trial makes the guess
  uint32_t guess = CSR || p.trial || hmin_min >= kInf ? kNone : light_guess(p.light, 8);
  for (int j = tid; j < sw; j += T0) {
    const int v = c0 + j;
    p.gkey[v] = v == source ? 0ull : ~0ull;
    rdist[j] = v == source ? 0u : kInf;
    flags[j] = static_cast<uint32_t>(__ldg(p.minin + v)) < kInf ? 1 : 0;
    if (CSR) {
      const int64_t s0 = p.row_ptr[v];
      start[j] = s0;
      aux[j] = static_cast<uint32_t>(p.row_ptr[v + 1] - s0);
    } else {
      aux[j] = __ldg(hmin + v);
    }
  }
  __syncthreads();
  // the source's listed edges that land in this slice (every CTA reads the list)
  uint32_t lmin = kNone;
  {
    const int64_t s0 = CSR ? p.row_ptr[source] : static_cast<int64_t>(source) * kLightCap;
    const int64_t len = CSR ? p.row_ptr[source + 1] - s0 : most;
    for (int64_t i = tid; i < len; i += T0) {
      const uint32_t e = __ldg(p.edge + s0 + i + (!CSR && i >= kLightCap ? light_apart(p.n) : 0));
      if (e == kNoEdge) break;
      const uint32_t v = e & umask;
      if (v - static_cast<uint32_t>(c0) >= static_cast<uint32_t>(sw) || static_cast<int>(v) == source) continue;
      const uint64_t key = light_key(0u, e >> bits_u, static_cast<uint32_t>(source), bits_u);
      p.gkey[v] = key;  // one edge per target
      lmin = min(lmin, e >> bits_u);
    }
  }
  uint32_t nbar = 0, m, D;
  if (b == p.skip_cta) return;  // testing: this CTA never arrives
  if (!light_barrier(p, sh, nbar++, lmin, kNone, &m, &D)) return;

  const int gsz = 1 << gshift;
  const int gl = tid & (gsz - 1), gid = tid >> gshift, ng = T0 >> gshift;
  const uint32_t longrow = CSR ? static_cast<uint32_t>(gsz) * 16u : kNone;
  const int last = (tid & 31) | (gsz - 1);  // last lane of this lane's group; lasts: of every group
  const uint32_t lasts = gshift == 2 ? 0x88888888u : gshift == 3 ? 0x80808080u : gshift == 4 ? 0x80008000u : 0x80000000u;
  uint32_t phases = 0;
  bool again = false;  // this phase relaxes every reached row, whatever its dist
  int raised = 0;
  for (;;) {
    lmin = kNone;
    uint32_t dmax = 0;
    if (m != kNone) {
      const uint32_t T = again ? kNone : m + delta;
      const uint32_t B = min(D, guess);
      again = false;
      for (int j = tid; j < sw; j += T0) {
        const uint32_t d = static_cast<uint32_t>(__ldcg(p.gkey + c0 + j) >> 32);
        if (d < kInf)
          dmax = max(dmax, d);
        else if (flags[j] & 1)
          dmax = kNone;  // not reached yet, and something leads to it
        if (d < rdist[j]) {
          if (d <= T) {
            rdist[j] = d;
            if (CSR && aux[j] > longrow)
              list[p.swcap - 1 - static_cast<int>(atomicAdd(&sh.big, 1u))] = make_uint2(static_cast<uint32_t>(j), d);
            else
              list[atomicAdd(&sh.cnt, 1u)] = make_uint2(static_cast<uint32_t>(j), d);
          } else {
            lmin = min(lmin, d);
          }
        }
      }
      __syncthreads();
      const int cnt = static_cast<int>(sh.cnt);
      for (int i0 = 0; i0 < cnt; i0 += ng * kLightRows) {
        uint32_t u[kLightRows], du[kLightRows], len[kLightRows];
        const uint32_t* row[kLightRows];
        bool on[kLightRows];
#pragma unroll
        for (int r = 0; r < kLightRows; ++r) {
          const int i = i0 + r * ng + gid;
          on[r] = i < cnt;
          const uint2 x = on[r] ? list[i] : make_uint2(0u, 0u);
          u[r] = static_cast<uint32_t>(c0) + x.x;
          du[r] = x.y;
          row[r] = CSR ? p.edge + start[x.x] : p.edge + static_cast<size_t>(u[r]) * kLightCap;
          len[r] = CSR ? aux[x.x] : most;
        }
        for (uint32_t k = gl;; k += gsz) {
          uint32_t e[kLightRows], more = 0;
          uint64_t old[kLightRows];
          bool use[kLightRows];
#pragma unroll
          for (int r = 0; r < kLightRows; ++r) {
            if (!CSR && k - gl == kLightCap) row[r] += light_apart(p.n);
            e[r] = on[r] && k < len[r] ? __ldg(row[r] + k) : kNoEdge;
          }
#pragma unroll
          for (int r = 0; r < kLightRows; ++r) {
            use[r] = e[r] != kNoEdge && du[r] + (e[r] >> bits_u) <= B;
            old[r] = use[r] ? __ldcg(p.gkey + (e[r] & umask)) : 0ull;
            // sorted: a row goes on only if it has more and its group's last lane still had a use for its edge
            const uint32_t bal = __ballot_sync(0xffffffffu, use[r] && k - gl + gsz < len[r]);
            on[r] = (bal >> last) & 1u;
            more |= bal & lasts;
          }
#pragma unroll
          for (int r = 0; r < kLightRows; ++r)
            if (use[r])
              light_offer_global(p.gkey, e[r] & umask, light_key(du[r], e[r] >> bits_u, u[r], bits_u), old[r], lmin);
          if (more == 0) break;
        }
      }
      if (CSR) {  // long rows: the whole block takes one after another
        const int nbig = static_cast<int>(sh.big);
        for (int i = 0; i < nbig; ++i) {
          const uint2 x = list[p.swcap - 1 - i];
          const uint32_t u = static_cast<uint32_t>(c0) + x.x;
          const uint32_t* row = p.edge + start[x.x];
          for (uint32_t k = tid; k < aux[x.x]; k += T0) {
            const uint32_t e = __ldg(row + k);
            if (x.y + (e >> bits_u) > B) break;
            light_offer_global(p.gkey, e & umask, light_key(x.y, e >> bits_u, u, bits_u), __ldcg(p.gkey + (e & umask)),
                               lmin);
          }
        }
      }
      if (!light_barrier(p, sh, nbar++, lmin, dmax, &m, &D)) return;
      ++phases;
      if (p.trial && phases > kTrialPhases) {
        if (b == 0 && tid == 0) atomicAdd(p.heavy, kTrialManyRows);
        break;
      }
      continue;
    }
    // nothing is dirty anywhere; with complete lists (no bound was set) that is all
    if (CSR || hmin_min >= kInf) break;
    if (D > guess) {  // the bound was too low: every row once more, up to D or, with nodes unreached, a higher guess
      guess = D != kNone ? D : ++raised < 4 ? guess + guess / 4 + 1 : kNone;
      for (int j = tid; j < sw; j += T0)
        if (rdist[j] < kInf) rdist[j] = kNone;
      again = true;
      m = 0;
      continue;
    }
    // the index proves the answer, or some rows are relaxed whole
    if (hmin_min > D) break;
    const uint32_t Dx = D;
    uint32_t hb = kNone;
    for (int j = tid; j < sw; j += T0) {
      if ((flags[j] & 2) || rdist[j] >= kInf) continue;  // rdist is the dist of every reached node now
      hb = min(hb, light_pending(rdist[j], aux[j], Dx));
    }
    if (!light_barrier(p, sh, nbar++, hb, 0u, &m, &D)) return;
    hb = m;
    D = Dx;
    if (hb == kNone) break;
    hb = light_below(hb, hmin_min);
    for (int j = tid; j < sw; j += T0) {
      if ((flags[j] & 2) || rdist[j] >= hb || light_pending(rdist[j], aux[j], Dx) == kNone) continue;
      list[atomicAdd(&sh.cnt, 1u)] = make_uint2(static_cast<uint32_t>(j), rdist[j]);
      flags[j] |= 2;
    }
    __syncthreads();
    const int cnt = static_cast<int>(sh.cnt);
    if (p.trial) {  // enough is known once these are too many; every CTA reads the same count between two barriers
      if (tid == 0 && cnt) atomicAdd(p.heavy, static_cast<uint32_t>(cnt));
      uint32_t unused;
      if (!light_barrier(p, sh, nbar++, kNone, 0u, &m, &unused)) return;
      if (__ldcg(p.heavy) > (p.guess ? kTrialManyRows : kTrialMoreRows)) break;
    }
    const int nv = static_cast<int>(p.pitch / 4);
    for (int i = 0; i < cnt; ++i) {
      const uint2 x = list[i];
      const uint32_t u = static_cast<uint32_t>(c0) + x.x;
      const int32_t* row = p.W + static_cast<int64_t>(u) * p.pitch;
      for (int g0 = tid; g0 < nv; g0 += 8 * T0) {
        int4 y[8];
#pragma unroll
        for (int r = 0; r < 8; ++r)
          y[r] = g0 + r * T0 < nv ? ld_stream16(row + 4 * static_cast<int64_t>(g0 + r * T0))
                                  : make_int4(int(kInf), int(kInf), int(kInf), int(kInf));
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const uint32_t w4[4] = {static_cast<uint32_t>(y[r].x), static_cast<uint32_t>(y[r].y),
                                  static_cast<uint32_t>(y[r].z), static_cast<uint32_t>(y[r].w)};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t v = static_cast<uint32_t>(4 * (g0 + r * T0) + c);
            if (w4[c] < kInf && x.y + w4[c] <= Dx && v != u)
              light_offer_global(p.gkey, v, light_key(x.y, w4[c], u, bits_u), __ldcg(p.gkey + v), lmin);
          }
        }
      }
    }
    // every row that was dirty has been relaxed, so the slice's dists (and D) only change through these rows
    if (!light_barrier(p, sh, nbar++, lmin, Dx, &m, &D)) return;
    ++phases;
  }
  if (p.trial) {
    uint64_t far = 0;
    for (int j = tid; j < sw; j += T0)
      if (rdist[j] < kInf) far = max(far, (static_cast<uint64_t>(rdist[j]) << 32) | static_cast<uint32_t>(c0 + j));
    const uint32_t hi = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(far >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(far >> 32) == hi ? static_cast<uint32_t>(far) : 0u);
    if ((tid & 31) == 0)
      atomicMax(reinterpret_cast<unsigned long long*>(const_cast<uint32_t*>(p.light) + kLightFar),
                (static_cast<unsigned long long>(hi) << 32) | lo);
    if (p.guess && D < kInf) {
      if (b == 0 && tid == 0) p.guess[0] = D + 1;
      uint32_t risky = 0;
      for (int j = tid; j < sw; j += T0) risky += light_risky(rdist[j], aux[j], D) ? 1u : 0u;
      risky = warp_sum_u32(risky);
      if ((tid & 31) == 0 && risky) atomicAdd(const_cast<uint32_t*>(p.light) + kLightRisky, risky);
    }
    return;
  }
  for (int j = tid; j < sw; j += T0) {
    const uint64_t k = __ldcg(p.gkey + c0 + j);
    const uint32_t d = static_cast<uint32_t>(k >> 32);
    const bool reached = d < kInf;
    p.dist_out[c0 + j] = static_cast<int32_t>(reached ? d : kInf);
    p.pred_out[c0 + j] = reached && c0 + j != source ? static_cast<int32_t>(static_cast<uint32_t>(k) & umask) : -1;
  }
  if (b == 0 && tid == 0) p.words[1] = phases;
}

template <bool CSR>
__global__ void __launch_bounds__(kLightGridThreads, 1) k_light_grid(const LightGridParams p) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ LgShared sh;
  if (threadIdx.x == 0) {
    sh.cnt = 0;
    sh.big = 0;
  }
  pdl_launch_dependents();
  pdl_wait();
  light_grid_solve<CSR>(p, smem, sh);
  // the last CTA to leave puts the control words back to zero for the next launch on the stream
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(p.ctl + kLgExit, 1u) == gridDim.x - 1) {
      __threadfence();
      p.ctl[kLgAbort] = 0;
      p.ctl[kLgExit] = 0;
      for (int i = 0; i < 12; ++i) p.ctl[kLgSlots + i] = 0;
      mark_done(p.mark);
    }
  }
}

}  // namespace dj

// ============================================================ host

namespace dj {

// heavy: the launch is a trial.
static int run_light_grid(const dj_graph* g, int32_t source, int32_t* dist, int32_t* pred, const dj_solve_opts& o,
                          uint32_t* heavy, const SolveMark& mark, cudaStream_t st) {
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  if (!ctx->coop) return set_error(DJ_EUNSUPPORTED, "device lacks cooperative launch");
  const bool csr = g->format == DJ_FORMAT_CSR;
  const int G = std::max(1, std::min(ctx->num_sms, static_cast<int>((g->n + 31) / 32)));
  const int swcap = static_cast<int>((static_cast<int64_t>(g->n) + G - 1) / G);
  const size_t smem = static_cast<size_t>(swcap) * ((csr ? 8 : 0) + 8 + 4 + 4 + 1) + 16;
  void* fn = csr ? reinterpret_cast<void*>(&k_light_grid<true>) : reinterpret_cast<void*>(&k_light_grid<false>);
  if (int rc = prepare_function(ctx, fn, smem, false)) return rc;
  int occ = 0;
  if (int rc = function_occupancy(ctx, fn, kLightGridThreads, smem, &occ)) return rc;
  if (occ < 1) return set_error(DJ_EUNSUPPORTED, "light engine cannot be resident");
  const size_t ctl_bytes = 256, ws_bytes = ctl_bytes + static_cast<size_t>(g->n) * 8;
  uint8_t* ws = nullptr;
  cudaError_t e = cudaSuccess;
  if (int rc = stream_workspace(ctx, st, ws_bytes, ctl_bytes, &ws)) return rc;
  const bool own_ws = ws == nullptr;
  if (own_ws) {
    e = cudaMallocAsync(&ws, ws_bytes, st);
    if (e != cudaSuccess) return cuda_error(e, "cudaMallocAsync(light workspace)");
    cudaMemsetAsync(ws, 0, ctl_bytes, st);
  }
  LightGridParams p;
  p.W = g->W;
  p.light = g->light;
  p.row_ptr = g->row_ptr;
  p.edge = csr ? g->edge : g->light + kLightStats + light_pad(g->n);
  p.minin = g->minin;
  p.dist_out = dist;
  p.pred_out = pred;
  p.ctl = reinterpret_cast<uint32_t*>(ws);
  p.gkey = reinterpret_cast<unsigned long long*>(ws + ctl_bytes);
  p.words = heavy ? g->light + kLightError : ctx->words;  // a trial that ran out of time is no caller's error
  p.heavy = heavy;
  p.mark = mark;
  p.guess = heavy && source == kTrialFirst ? g->light + kLightGuess : nullptr;
  p.pitch = g->pitch;
  p.timeout_ns = o.timeout_ns > 0 ? o.timeout_ns : 2000000000LL;
  p.n = g->n;
  p.swcap = swcap;
  p.source = source;
  p.bits_u = host_bits_for(static_cast<uint32_t>(g->n));
  p.delta = static_cast<uint32_t>(std::min(1.0e9f, kGridDelta * g->light_spacing));
  p.gshift = g->light_gshift;
  p.trial = heavy ? 1 : 0;
  p.skip_cta = o.debug_skip_cta;
  void* args[] = {&p};
  e = launch_cooperative(fn, G, kLightGridThreads, args, smem, st, true);
  if (own_ws) cudaFreeAsync(ws, st);
  if (e != cudaSuccess) return cuda_error(e, "cooperative launch (light engine)");
  return DJ_OK;
}

int launch_light_grid(const dj_graph* g, int32_t source, int32_t* dist, int32_t* pred, const dj_solve_opts& o,
                      const SolveMark& mark, cudaStream_t st) {
  return run_light_grid(g, source, dist, pred, o, nullptr, mark, st);
}

int launch_light_trial(const dj_graph* g, int32_t source, uint32_t* heavy, cudaStream_t st) {
  dj_solve_opts o;
  dj_solve_opts_init(&o);
  return run_light_grid(g, source, nullptr, nullptr, o, heavy, SolveMark(), st);
}

}  // namespace dj
