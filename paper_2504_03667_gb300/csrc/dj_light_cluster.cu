// Light engine, cluster form: one solve on one thread-block cluster of C CTAs, its state spread over
// their shared memory, for graphs whose every weight is >= 1 (dense with an index, or compressed rows).
// The algorithm is the CTA form's (dj_light_cta.cu); an offer goes to the owner of its node by a
// distributed-shared-memory atomic, and the phases are separated by cluster barriers.
//
// Why: a phase of the grid form costs about 2.9 us, a grid barrier and three L2 round trips one after
// another; here it is a cluster barrier, one L2 round trip for the edges and one to shared memory
// elsewhere in the cluster.  And a solve leaves most SMs free, so back-to-back solves on a stream run
// side by side (a programmatic dependent launch, as the cluster engine's single solves).
//
// Words of 32 nodes are dealt out in turn: word w = v / 32 lies in rank w mod C, there at w / C, so any
// graph fills every CTA evenly.
#include <algorithm>
#include <string>
#include <type_traits>

#include "dj_common.cuh"
#include "dj_internal.h"
#include "dj_jobs.cuh"
#include "dj_light.cuh"

namespace dj {

namespace {
constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
// delta in units of the listed weights' mean spacing (directed n = 32768, 8 edges per node: 142 us with 5,
// 156 with 8, 198 with 15, whose rows are relaxed too often)
constexpr float kClDelta = 5.0f;
}  // namespace

struct LightClusterParams {
  SolveDesc d;
  const int64_t* row_ptr;  // compressed rows: n + 1 offsets into edge
  const uint32_t* edge;
  const int32_t* minin;
  uint32_t* phases_out;
  SolveMark mark;
  uint32_t delta;          // compressed rows (dense: from the index)
  int32_t cshift;          // log2 C
  int32_t lw;              // words per CTA
};

// Addresses (shared::cluster, of this CTA's arrays; mapa turns them into another rank's).
struct LightClusterStore {
  uint32_t dist, tie, dirty;
  int cshift;
  __device__ __forceinline__ uint32_t rank_of(uint32_t v) const { return (v >> 5) & ((1u << cshift) - 1u); }
  __device__ __forceinline__ uint32_t word_of(uint32_t v) const { return v >> (5 + cshift); }
  __device__ __forceinline__ uint32_t at(uint32_t base, uint32_t rank, uint32_t index) const {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(base + 4u * index), "r"(rank));
    return a;
  }
  __device__ __forceinline__ uint32_t slot(uint32_t base, uint32_t v) const {
    return at(base, rank_of(v), (word_of(v) << 5) | (v & 31u));
  }
  __device__ __forceinline__ uint32_t offer(uint32_t v, uint32_t c) const {
    uint32_t old;
    asm volatile("atom.relaxed.cluster.shared::cluster.min.u32 %0, [%1], %2;"
                 : "=r"(old)
                 : "r"(slot(dist, v)), "r"(c)
                 : "memory");
    return old;
  }
  // The offer's atomic has returned, so the dist is in place before its bit can be seen.
  __device__ __forceinline__ void won(uint32_t v, uint32_t) const {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(at(dirty, rank_of(v), word_of(v))),
                 "r"(1u << (v & 31u))
                 : "memory");
  }
  __device__ __forceinline__ uint32_t dist_of(uint32_t v) const { return ld_dsmem_u32(slot(dist, v)); }
  __device__ __forceinline__ void tie_min(uint32_t v, uint32_t t) const { red_min(slot(tie, v), t); }
  static __device__ __forceinline__ void red_min(uint32_t addr, uint32_t x) {
    asm volatile("red.relaxed.cluster.shared::cluster.min.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
  }
  static __device__ __forceinline__ void red_max(uint32_t addr, uint32_t x) {
    asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
  }
};

// Compressed rows: row u of this CTA starts at start[] and has len[] edges (slots as the store's).
struct LightCsrEdges {
  static constexpr bool kApart = false;
  static constexpr int32_t n = 0;
  const uint32_t* __restrict__ edge;
  const int64_t* start;  // shared
  const uint32_t* len;   // shared
  int cshift;
  uint32_t most;
  __device__ __forceinline__ uint4 load(uint32_t u, uint32_t k0, int sub) const {
    const uint32_t i = ((u >> (5 + cshift)) << 5) | (u & 31u);
    const uint32_t n = len[i];
    const uint32_t* p = edge + start[i] + k0;
    uint32_t x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = k0 + 4 * q + sub < n ? __ldg(p + 4 * q + sub) : kNoEdge;
    return make_uint4(x[0], x[1], x[2], x[3]);
  }
};

template <bool CSR>
__global__ void __launch_bounds__(kClThreads, 1) k_light_cluster(const LightClusterParams p) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint2 s_rows[kClWarps][kWarpRows];
  __shared__ uint32_t s_m[3], s_D, s_bound, s_cnt, s_end;
  const uint32_t rank = cluster_rank(), C = 1u << p.cshift;
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  uint2* rows = s_rows[warp];
  const int LW = p.lw;
  int64_t* start = reinterpret_cast<int64_t*>(smem);
  uint32_t* dist = reinterpret_cast<uint32_t*>(smem + (CSR ? static_cast<size_t>(LW) * 256 : 0));
  uint32_t* tie = dist + LW * 32;
  uint32_t* dirty = tie + LW * 32;
  uint32_t* whole = dirty + LW;
  uint32_t* len = whole + LW;
  const LightClusterStore s{smem_u32(dist), smem_u32(tie), smem_u32(dirty), p.cshift};
  pdl_launch_dependents();
  // the graph is read at once: no kernel ahead on the stream writes it (an upload takes a graph off this engine)

  const SolveDesc& d = p.d;
  const int n = d.n;
  const uint32_t bits_u = d.bits_u, umask = (1u << bits_u) - 1u;
  const uint32_t* hmin = CSR ? nullptr : d.light + kLightStats;
  const uint32_t hmin_min = CSR ? kInf : ~__ldg(d.light);  // >= INF: every row's list is complete
  const uint32_t most = CSR ? kNone : __ldg(d.light + 6);  // edges in the longest list
  const uint32_t delta = CSR ? p.delta : light_delta(d.light, kClDelta);
  uint32_t B = hmin_min < kInf ? light_guess(d.light, 8) : kNone;
  auto global_word = [&](int lw) { return (lw << p.cshift) + static_cast<int>(rank); };

  for (int lw = warp; lw < LW; lw += kClWarps) {
    const int v = 32 * global_word(lw) + lane, i = 32 * lw + lane;
    dist[i] = v == d.source ? 0u : kNone;
    tie[i] = kNone;
    if (CSR) {
      const int64_t a = v < n ? p.row_ptr[v] : 0;
      start[i] = a;
      len[i] = v < n ? static_cast<uint32_t>(p.row_ptr[v + 1] - a) : 0u;
    }
    if (lane == 0) {
      dirty[lw] = global_word(lw) == (d.source >> 5) ? 1u << (d.source & 31) : 0u;
      whole[lw] = 0;
    }
  }
  if (tid == 0) {
    s_m[0] = 0;
    s_m[1] = kNone;
  }
  cluster_sync_all();  // every rank's state is there before anyone offers

  auto run_rows = [&](auto ties, const auto& get, int count, uint32_t& lmin) {
    if constexpr (CSR)
      light_rows<decltype(ties)::value>(s, LightCsrEdges{p.edge, start, len, p.cshift, most}, get, count, B, bits_u, lmin);
    else
      light_rows<decltype(ties)::value>(s, LightListEdges{hmin + light_pad(n), n, most}, get, count, B, bits_u, lmin);
  };
  uint32_t phase = 0, cur = 0;  // cur = phase % 3: the slot of this phase's m, the smallest dirty dist
  int raised = 0;
  bool any_whole = false;
  for (;; ++phase) {
    const uint32_t m = s_m[cur];  // every rank has the same
    const uint32_t nxt = cur == 2 ? 0 : cur + 1;
    if (tid == 0) s_m[nxt == 2 ? 0 : nxt + 1] = kNone;  // the slot after the next: read a phase ago, written in the next
    uint32_t lmin = kNone;
    int cnt = 0;  // rows waiting in this warp's list
    auto relax = [&](int have) {
      __syncwarp();
      run_rows(std::false_type{}, [rows](int i) { return rows[i]; }, have, lmin);
    };
    auto add = [&](uint32_t take, int lw, uint32_t dv) {  // the nodes `take` of word lw, dv: this lane's dist
      if ((take >> lane) & 1u)
        rows[cnt + __popc(take & lt)] = make_uint2(static_cast<uint32_t>(32 * global_word(lw) + lane), dv);
      cnt += __popc(take);
      if (cnt >= 32) {
        relax(32);
        cnt -= 32;
        if (lane < cnt) rows[lane] = rows[32 + lane];
      }
      __syncwarp();
    };
    if (m != kNone) {
      const uint32_t T = m + delta;
      for (int base = 0; base < LW; base += 32 * kClWarps) {
        const int mine = base + warp + kClWarps * lane;  // a word per lane; dirty words are taken 4 at a time
        uint32_t todo = __ballot_sync(0xffffffffu, mine < LW && word_now(dirty + mine) != 0);
        while (todo) {
          constexpr int kWords = 4;
          int lw[kWords];
#pragma unroll
          for (int j = 0; j < kWords; ++j) {
            lw[j] = todo ? base + warp + kClWarps * (__ffs(todo) - 1) : -1;
            todo &= todo - 1;
          }
          // the masks go before the dists are read: a dist lowered before is seen here, one lowered
          // later sets its bit again
          uint32_t bits = 0;
#pragma unroll
          for (int j = 0; j < kWords; ++j)
            if (lane == j && lw[j] >= 0) bits = atomicExch(dirty + lw[j], 0u);
          __syncwarp();
          uint32_t dv[kWords];
#pragma unroll
          for (int j = 0; j < kWords; ++j) dv[j] = lw[j] >= 0 ? word_now(dist + 32 * lw[j] + lane) : kNone;
#pragma unroll
          for (int j = 0; j < kWords; ++j) {
            if (lw[j] < 0) break;
            const uint32_t b = __shfl_sync(0xffffffffu, bits, j);
            const uint32_t take = __ballot_sync(0xffffffffu, ((b >> lane) & 1u) && dv[j] <= T);
            const uint32_t keep = b & ~take;
            if (keep) {
              if ((keep >> lane) & 1u) lmin = min(lmin, dv[j]);
              if (lane == 0) atomicOr(dirty + lw[j], keep);
            }
            add(take, lw[j], dv[j]);
          }
        }
      }
      if (cnt > 0) relax(cnt);
    } else {
      // nothing is dirty; with complete lists (B is kNone then) that is all
      if (hmin_min >= kInf) break;
      if (tid == 0) {
        s_D = 0;
        s_bound = kNone;
        s_cnt = 0;
        s_end = kClWarps * kWarpRows;
      }
      cluster_sync_all();
      uint32_t D = 0;
      for (int lw = warp; lw < LW; lw += kClWarps) {
        const int v = 32 * global_word(lw) + lane;
        const uint32_t dv = dist[32 * lw + lane];
        if (dv != kNone)
          D = max(D, dv);
        else if (v < n && static_cast<uint32_t>(__ldg(p.minin + v)) < kInf)
          D = kNone;  // not reached yet, and something leads to it
      }
      D = __reduce_max_sync(0xffffffffu, D);
      if (lane < static_cast<int>(C)) LightClusterStore::red_max(s.at(smem_u32(&s_D), lane, 0), D);
      __syncwarp();
      cluster_sync_all();
      D = s_D;
      if (D > B) {  // the bound was too low: every row once more, up to D or, with nodes unreached, a higher guess
        B = D != kNone ? D : ++raised < 4 ? B + B / 4 + 1 : kNone;
        for (int lw = warp; lw < LW; lw += kClWarps) {
          const uint32_t dv = word_now(dist + 32 * lw + lane);
          add(__ballot_sync(0xffffffffu, dv != kNone), lw, dv);
        }
        if (cnt > 0) relax(cnt);
      } else {
        // the index proves the answer, or some rows are relaxed whole, in pieces by all warps
        if (hmin_min > D) break;
        B = D;
        auto pending = [&](int lw, uint32_t dv) {  // dist + hmin of this lane's node if its row is pending
          if (dv == kNone || ((whole[lw] >> lane) & 1u)) return kNone;
          return light_pending(dv, __ldg(hmin + 32 * global_word(lw) + lane), D);
        };
        uint32_t hb = kNone;  // the smallest dist + hmin of the pending rows
        for (int lw = warp; lw < LW; lw += kClWarps) hb = min(hb, pending(lw, dist[32 * lw + lane]));
        hb = warp_min_u32(hb);
        if (lane < static_cast<int>(C) && hb != kNone) LightClusterStore::red_min(s.at(smem_u32(&s_bound), lane, 0), hb);
        __syncwarp();
        cluster_sync_all();
        hb = s_bound;
        if (hb == kNone) break;
        // the final ones (light_below): relaxed whole, as many as the list holds now
        hb = light_below(hb, hmin_min);
        for (int lw = warp; lw < LW; lw += kClWarps) {
          const uint32_t dv = dist[32 * lw + lane];
          const bool go = dv < hb && pending(lw, dv) != kNone;
          const uint32_t todo = __ballot_sync(0xffffffffu, go);
          if (todo == 0) continue;
          uint32_t pos = 0;
          if (lane == 0) pos = atomicAdd(&s_cnt, static_cast<uint32_t>(__popc(todo)));
          pos = __shfl_sync(0xffffffffu, pos, 0);
          if (pos + __popc(todo) > kClWarps * kWarpRows) {
            if (lane == 0) atomicMin(&s_end, pos);
            continue;
          }
          if (go) s_rows[0][pos + __popc(todo & lt)] = make_uint2(static_cast<uint32_t>(32 * global_word(lw) + lane), dv);
          if (lane == 0) whole[lw] |= todo;
        }
        cluster_sync_all();  // the lists are complete, and every rank has taken its own before dists change
        any_whole = true;
        light_whole_rows(s, d, s_rows[0], static_cast<int>(min(s_cnt, s_end)), D, lmin);
      }
    }
    lmin = warp_min_u32(lmin);
    if (lane < static_cast<int>(C) && lmin != kNone) LightClusterStore::red_min(s.at(smem_u32(&s_m[nxt]), lane, 0), lmin);
    __syncwarp();
    cluster_sync_all();
    cur = nxt;
  }
  // the dists are final: the best offer of each node's dist.  Only listed edges, and rows relaxed whole,
  // can make one.
  for (int lw = warp; lw < LW; lw += kClWarps) {
    uint32_t unused = 0;
    const int v0 = 32 * global_word(lw);
    const uint32_t dv = dist[32 * lw + lane];
    run_rows(std::true_type{}, [v0, dv](int i) { return make_uint2(v0 + i, __shfl_sync(0xffffffffu, dv, i)); }, 32, unused);
  }
  if (any_whole)
    light_whole_ties(
        s, d, whole, LW,
        [&](int lw, int i) { return make_uint2(static_cast<uint32_t>(32 * global_word(lw) + i), dist[32 * lw + i]); }, B);
  cluster_sync_all();  // every offer has arrived; nobody touches another CTA's memory from here on
  pdl_wait();          // results reach memory in stream order
  if (rank == 0 && tid == 0) mark_done(p.mark);  // before them: it goes to host memory
  for (int lw = warp; lw < LW; lw += kClWarps) {
    const int v = 32 * global_word(lw) + lane;
    if (v >= n) continue;
    const uint32_t dv = dist[32 * lw + lane];
    d.dist[v] = static_cast<int32_t>(dv == kNone ? kInf : dv);
    d.pred[v] = dv == kNone || v == d.source ? -1 : static_cast<int32_t>(tie[32 * lw + lane] & umask);
  }
  if (rank == 0 && tid == 0 && p.phases_out) *p.phases_out = phase;
}

// ============================================================ host

static int light_cluster_words(int32_t n, int C) { return ((n + 31) / 32 + C - 1) / C; }
static size_t light_cluster_smem(int32_t n, int C, bool csr) {
  return static_cast<size_t>(light_cluster_words(n, C)) * (csr ? 256 + 128 + 264 : 264);
}

bool light_cluster_fits(int32_t n, int C, bool csr) {
  DevCtx* ctx = nullptr;
  if (get_ctx(&ctx) != DJ_OK) return false;
  return ctx->cluster_launch && light_cluster_smem(n, C, csr) + 10 * 1024 <= static_cast<size_t>(ctx->max_smem_optin);
}

int prepare_light_cluster(bool csr, int C) {
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  return prepare_function(ctx, csr ? reinterpret_cast<void*>(&k_light_cluster<true>) : reinterpret_cast<void*>(&k_light_cluster<false>),
                          0, C > 8);
}

int run_light_cluster(const dj_graph* g, int C, const SolveDesc& desc, uint32_t* phases_out, const SolveMark& mark,
                      cudaStream_t st) {
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  const bool csr = g->format == DJ_FORMAT_CSR;
  void* fn = csr ? reinterpret_cast<void*>(&k_light_cluster<true>) : reinterpret_cast<void*>(&k_light_cluster<false>);
  const size_t smem = light_cluster_smem(g->n, C, csr);
  if (int rc = prepare_function(ctx, fn, smem, C > 8)) return rc;
  LightClusterParams p;
  p.d = desc;
  p.row_ptr = g->row_ptr;
  p.edge = g->edge;
  p.minin = g->minin;
  p.phases_out = phases_out;
  p.mark = mark;
  p.delta = static_cast<uint32_t>(std::min(1.0e9f, kClDelta * g->light_spacing));
  p.cshift = 0;
  while ((1 << p.cshift) < C) ++p.cshift;
  p.lw = light_cluster_words(g->n, C);
  void* args[] = {&p};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(C));
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(C);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
  if (e != cudaSuccess) {  // not accepted here: the ordinary launch gives the same results
    cudaGetLastError();
    cfg.numAttrs = 1;
    e = cudaLaunchKernelExC(&cfg, fn, args);
  }
  if (e != cudaSuccess) return cuda_error(e, "launch (light engine, cluster form)");
  return DJ_OK;
}

}  // namespace dj
