// Light engine, CTA form: one CTA per solve with its state in shared memory (n up to about 26000),
// for batches and small single solves on graphs whose every weight is >= 1.  The algorithm is the
// grid form's (dj_light_grid.cu) without any communication between CTAs.
#include <algorithm>
#include <string>

#include "dj_common.cuh"
#include "dj_internal.h"
#include "dj_jobs.cuh"
#include "dj_light.cuh"

namespace dj {

namespace {
// delta in units of the listed weights' mean spacing: 19 phases instead of 25 with 1, and 4 % more rows
constexpr float kCtaDelta = 3.0f;
}  // namespace

struct LightCtaParams {
  int32_t npad;     // node slots (largest graph of the launch, rounded up to 64)
};

// Shared memory of a solve (dynamic).  A word of 32 nodes has a mask of dirty ones and a lower bound on
// their dists.
struct LightCta {
  uint32_t* dist;   // kNone: not reached
  uint32_t* tie;    // low word of the key (dj_light.cuh) of the best offer, found last
  uint32_t* dirty;
  uint32_t* wmin;
  uint32_t* whole;  // rows relaxed whole

  // An offer of dist c to v (light_rows); a shorter one makes v dirty.  32-bit shared atomics cost what a
  // load costs (2.5 cycles a warp, against 9.4 for a 64-bit compare-and-swap and 4.6 for a 64-bit load),
  // so dists are settled alone and the ties, which need them final anyway, in one pass at the end.
  __device__ __forceinline__ uint32_t offer(uint32_t v, uint32_t c) const { return atomicMin(dist + v, c); }
  __device__ __forceinline__ void won(uint32_t v, uint32_t c) const {
    atomicOr(dirty + (v >> 5), 1u << (v & 31u));
    atomicMin(wmin + (v >> 5), c);
  }
  __device__ __forceinline__ uint32_t dist_of(uint32_t v) const { return dist[v]; }
  __device__ __forceinline__ void tie_min(uint32_t v, uint32_t t) const { atomicMin(tie + v, t); }
};

// One phase has one block-wide barrier.  Each warp owns every (THREADS / 32)-th word of 32 nodes: it
// takes the dirty nodes of its words whose dist lies in the window, gathers them in its own list and
// relaxes their rows 32 at a time, while other warps may already make more of them dirty -- those go
// along if their word is still to come, else in a later phase.
//
// Rows are first relaxed up to a bound B on the offers: somewhat above the largest dist of the graph's
// trial solve (light_guess), which holds for most sources.  When nothing is dirty the true
// largest dist D is taken; if it is above B every row is relaxed once more up to D.  Dropping offers
// above the largest dist leaves 13 of the 64 listed edges per row for n = 8192, p = 0.05; waiting for D
// to be known first left 37.
template <int THREADS, int PER_SM, class Jobs>
__global__ void __launch_bounds__(THREADS, PER_SM)
    k_light_cta(const LightCtaParams p, const Jobs jobs) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint2 s_rows[THREADS / 32][kWarpRows];
  __shared__ uint32_t s_job, s_bound, s_cnt, s_end, s_m[3];
  LightCta s;
  s.dist = reinterpret_cast<uint32_t*>(smem);
  s.tie = s.dist + p.npad;
  s.dirty = s.tie + p.npad;
  s.wmin = s.dirty + p.npad / 32;
  s.whole = s.wmin + p.npad / 32;
  constexpr int NW = THREADS / 32;
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  uint2* rows = s_rows[warp];
  pdl_launch_dependents();

  for (uint32_t iter = 0;; ++iter) {
    __syncthreads();  // the previous solve's reads of shared memory are done
    if (tid == 0) {
      uint32_t j = 0;
      s_job = jobs.fetch(&j, iter) ? j : kNone;
      if (s_job == kNone) jobs.leave(gridDim.x);
    }
    __syncthreads();
    const uint32_t job = s_job;
    if (job == kNone) return;
    const SolveDesc d = jobs.desc(job);
    if (!jobs.early()) pdl_wait();  // the kernel before may still be writing the graph
    const int n = d.n, nwords = (n + 31) / 32;
    const uint32_t bits_u = d.bits_u, umask = (1u << bits_u) - 1u;
    const uint32_t* hmin = d.light + kLightStats;
    const uint32_t hmin_min = ~__ldg(d.light);  // >= INF: every row's list is complete
    const LightListEdges edges{hmin + light_pad(n), n, __ldg(d.light + 6)};
    const uint32_t delta = light_delta(d.light, kCtaDelta);
    // a wide margin in batches: one takes as long as its slowest solve, one whose bound was too low (256 sources of
    // n = 8192: 296 us with an eighth, 285 with a quarter, 261 with 3/8)
    uint32_t B = hmin_min < kInf ? light_guess(d.light, Jobs::kGuessPart) : kNone;

    for (int wi = warp; wi < nwords; wi += NW) {
      const int v = 32 * wi + lane;
      s.dist[v] = v == d.source ? 0u : kNone;
      s.tie[v] = kNone;
      if (lane == 0) {
        const bool src = wi == (d.source >> 5);
        s.whole[wi] = 0;
        s.dirty[wi] = src ? 1u << (d.source & 31) : 0u;
        s.wmin[wi] = src ? 0u : kNone;
      }
    }
    if (tid == 0) {
      s_m[0] = 0;
      s_m[1] = kNone;
    }
    __syncthreads();
    uint32_t phase = 0, cur = 0;  // cur = phase % 3: the slot of this phase's m, the smallest dirty dist
    int raised = 0;
    bool any_whole = false;
    uint32_t nwhole = 0;  // trial: rows relaxed whole
    for (;; ++phase) {
      const uint32_t m = s_m[cur];
      const uint32_t nxt = cur == 2 ? 0 : cur + 1;
      if (tid == 0) s_m[nxt == 2 ? 0 : nxt + 1] = kNone;  // the slot after the next: everyone has read it a phase ago
      uint32_t lmin = kNone;
      int cnt = 0;  // rows waiting in this warp's list
      auto relax = [&](int have) {
        __syncwarp();
        light_rows<false>(s, edges, [rows](int i) { return rows[i]; }, have, B, bits_u, lmin);
      };
      auto add = [&](uint32_t take, int wi, uint32_t dv) {  // the nodes `take` of word wi, dv: this lane's dist
        if ((take >> lane) & 1u) rows[cnt + __popc(take & lt)] = make_uint2(static_cast<uint32_t>(32 * wi + lane), dv);
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
        for (int base = 0; base < nwords; base += 32 * NW) {
          const int mine = base + warp + NW * lane;  // a word per lane; needed words are taken 4 at a time
          const uint32_t wm = mine < nwords ? word_now(s.wmin + mine) : kNone;
          const bool need = wm != kNone && wm <= T;
          if (!need) lmin = min(lmin, wm);
          uint32_t todo = __ballot_sync(0xffffffffu, need);
          while (todo) {
            constexpr int kWords = 4;
            int wi[kWords];
#pragma unroll
            for (int j = 0; j < kWords; ++j) {
              wi[j] = todo ? base + warp + NW * (__ffs(todo) - 1) : -1;
              todo &= todo - 1;
            }
            // the masks go before the dists are read: a dist lowered before is seen here, one lowered
            // later sets its bit again
            uint32_t bits = 0;
#pragma unroll
            for (int j = 0; j < kWords; ++j)
              if (lane == j && wi[j] >= 0) {
                atomicExch(s.wmin + wi[j], kNone);
                bits = atomicExch(s.dirty + wi[j], 0u);
              }
            __syncwarp();
            uint32_t dv[kWords];
#pragma unroll
            for (int j = 0; j < kWords; ++j) dv[j] = wi[j] >= 0 ? word_now(s.dist + 32 * wi[j] + lane) : kNone;
#pragma unroll
            for (int j = 0; j < kWords; ++j) {
              if (wi[j] < 0) break;
              const uint32_t b = __shfl_sync(0xffffffffu, bits, j);
              const uint32_t take = __ballot_sync(0xffffffffu, ((b >> lane) & 1u) && dv[j] <= T);
              const uint32_t keep = b & ~take;
              if (keep) {
                const uint32_t low = warp_min_u32((keep >> lane) & 1u ? dv[j] : kNone);
                lmin = min(lmin, low);
                if (lane == 0) {
                  atomicOr(s.dirty + wi[j], keep);
                  atomicMin(s.wmin + wi[j], low);
                }
              }
              add(take, wi[j], dv[j]);
            }
          }
        }
        if (cnt > 0) relax(cnt);
      } else {
        // nothing is dirty; with complete lists (B is kNone then) that is all
        if (hmin_min >= kInf) break;
        if (tid == 0) s_bound = 0;
        __syncthreads();
        uint32_t D = 0;
        for (int v = tid; v < n; v += THREADS) {
          const uint32_t dv = word_now(s.dist + v);
          if (dv < kInf)
            D = max(D, dv);
          else if (static_cast<uint32_t>(__ldg(d.minout + n + v)) < kInf)
            D = kNone;  // not reached yet, and something leads to it
        }
        D = __reduce_max_sync(0xffffffffu, D);
        if (lane == 0) atomicMax(&s_bound, D);
        __syncthreads();
        D = s_bound;
        if (D > B) {  // the bound was too low: every row once more, up to D or, with nodes unreached, a higher guess
          B = D != kNone ? D : ++raised < 4 ? B + B / 4 + 1 : kNone;
          for (int wi = warp; wi < nwords; wi += NW) {
            const uint32_t dv = word_now(s.dist + 32 * wi + lane);
            add(__ballot_sync(0xffffffffu, dv < kInf), wi, dv);
          }
          if (cnt > 0) relax(cnt);
        } else {
          // the index proves the answer, or some rows are relaxed whole, in pieces by all warps
          if (hmin_min > D) break;
          B = D;
          __syncthreads();  // everyone has read s_bound
          if (tid == 0) {
            s_bound = kNone;  // the smallest dist + hmin of the pending rows
            s_cnt = 0;
            s_end = NW * kWarpRows;
          }
          __syncthreads();
          auto pending = [&](int wi, uint32_t dv) {  // dist + hmin of this lane's node if its row is pending
            if (dv == kNone || ((s.whole[wi] >> lane) & 1u)) return kNone;
            return light_pending(dv, __ldg(hmin + 32 * wi + lane), D);
          };
          uint32_t hb = kNone;
          for (int wi = warp; wi < nwords; wi += NW) hb = min(hb, pending(wi, s.dist[32 * wi + lane]));
          hb = warp_min_u32(hb);
          if (lane == 0 && hb != kNone) atomicMin(&s_bound, hb);
          __syncthreads();
          hb = s_bound;
          if (hb == kNone) break;
          // the final ones (light_below): relaxed whole, as many as the list holds now
          hb = light_below(hb, hmin_min);
          for (int wi = warp; wi < nwords; wi += NW) {
            const uint32_t dv = s.dist[32 * wi + lane];
            const bool go = dv < hb && pending(wi, dv) != kNone;
            const uint32_t todo = __ballot_sync(0xffffffffu, go);
            if (todo == 0) continue;
            uint32_t pos = 0;
            if (lane == 0) pos = atomicAdd(&s_cnt, static_cast<uint32_t>(__popc(todo)));
            pos = __shfl_sync(0xffffffffu, pos, 0);
            if (pos + __popc(todo) > NW * kWarpRows) {
              if (lane == 0) atomicMin(&s_end, pos);
              continue;
            }
            if (go) s_rows[0][pos + __popc(todo & lt)] = make_uint2(static_cast<uint32_t>(32 * wi + lane), dv);
            if (lane == 0) s.whole[wi] |= todo;
          }
          __syncthreads();
          any_whole = true;
          const int count = static_cast<int>(min(s_cnt, s_end));
          if (Jobs::kTrial && (nwhole += static_cast<uint32_t>(count)) > kTrialMoreRows) break;  // it has its answer
          light_whole_rows(s, d, s_rows[0], count, D, lmin);
        }
      }
      lmin = warp_min_u32(lmin);
      if (lane == 0 && lmin != kNone) atomicMin(&s_m[nxt], lmin);
      __syncthreads();
      cur = nxt;
    }
    if constexpr (Jobs::kTrial) {
      if (tid == 0) *jobs.whole(job) = nwhole;
      continue;
    }
    // the dists are final: the best offer of each node's dist.  Only listed edges, and rows relaxed
    // whole, can make one.
    for (int wi = warp; wi < nwords; wi += NW) {
      uint32_t unused = 0;
      const uint32_t dv = s.dist[32 * wi + lane];
      light_rows<true>(
          s, edges, [wi, dv](int i) { return make_uint2(32 * wi + i, __shfl_sync(0xffffffffu, dv, i)); }, 32, B,
          bits_u, unused);
    }
    if (any_whole)
      light_whole_ties(
          s, d, s.whole, nwords,
          [&s](int w, int i) { return make_uint2(static_cast<uint32_t>(32 * w + i), s.dist[32 * w + i]); }, B);
    __syncthreads();
    jobs.before_write();  // results reach memory in stream order
    for (int v = tid; v < n; v += THREADS) {
      const uint32_t dv = s.dist[v];
      d.dist[v] = static_cast<int32_t>(dv == kNone ? kInf : dv);
      d.pred[v] = dv == kNone || v == d.source ? -1 : static_cast<int32_t>(s.tie[v] & umask);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence_system();  // the outputs are visible system-wide before completion is reported
      jobs.complete(job, phase);
    }
  }
}

}  // namespace dj

// ============================================================ host

namespace dj {

namespace {


constexpr size_t kLightCtaStatic = 10 * 1024;  // static shared memory (512 threads: 8.1 KB) and the system's

size_t light_cta_smem(int32_t n) {
  const size_t np = static_cast<size_t>(light_pad(n));
  return np * 8 + np / 32 * 12;
}

}  // namespace

bool light_cta_fits(int32_t n) {
  DevCtx* ctx = nullptr;
  if (get_ctx(&ctx) != DJ_OK) return false;
  return light_cta_smem(n) + kLightCtaStatic <= static_cast<size_t>(ctx->max_smem_optin);
}

// CTAs of 512 threads, one per SM; two per SM in batches with more solves than SMs where shared memory
// allows (256 sources of n = 8192: 298 us, 354 with one; 48 graphs, which have an SM each, 112 with the
// registers of one, 129 with those of two).  The server's persistent CTAs have 192 threads, one per SM:
// other kernels must find room beside them for as long as the server runs (two CTAs of 512 threads fill
// every register of an SM, and a caller's own kernels waited until the server left); 192 leave 47 of an SM's 64 K
// registers, 256 leave 41.  (The load's trial solves, 54 K, fit beside neither: loading a graph with cut lists
// waits until the server's kernel has left, as it did beside the cluster engine's.)  Its rate is the host's (1500
// waiting requests: 3.4 ms with 192 threads, 3.3 with 256, 3.1 with 512).
int plan_light(int32_t max_n, int32_t k, int kind, LightPlan* plan) {
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  plan->smem = light_cta_smem(max_n);
  plan->npad = light_pad(max_n);
  plan->threads = kind == kJobsServe ? 192 : 512;
  const bool two = kind == kJobsBatch && k > ctx->num_sms &&
                   2 * (plan->smem + kLightCtaStatic) <= static_cast<size_t>(ctx->max_smem_optin);
  plan->fn = kind == kJobsServe    ? reinterpret_cast<void*>(&k_light_cta<192, 1, ServeJobs>)
             : kind == kJobsSingle ? reinterpret_cast<void*>(&k_light_cta<512, 1, SingleJob>)
             : kind == kJobsPlainSingle ? reinterpret_cast<void*>(&k_light_cta<512, 1, PlainSingleJob>)
             : kind == kJobsTrial  ? reinterpret_cast<void*>(&k_light_cta<512, 1, LightTrialJobs>)
             : two                 ? reinterpret_cast<void*>(&k_light_cta<512, 2, BatchJobs>)
                                   : reinterpret_cast<void*>(&k_light_cta<512, 1, BatchJobs>);
  if (int rc = prepare_function(ctx, plan->fn, plan->smem, false)) return rc;
  plan->ctas = kind == kJobsSingle || kind == kJobsPlainSingle ? 1 : kind == kJobsTrial ? kMoreTrials : ctx->num_sms * (two ? 2 : 1);
  if (kind == kJobsBatch) plan->ctas = std::max(1, std::min(plan->ctas, static_cast<int>(k)));
  return DJ_OK;
}

static int launch_light(const LightPlan& plan, void** args, cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(plan.ctas));
  cfg.blockDim = dim3(static_cast<unsigned>(plan.threads));
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaError_t e = cudaLaunchKernelExC(&cfg, plan.fn, args);
  if (e != cudaSuccess && pdl) {  // not accepted here: the ordinary launch gives the same results
    cudaGetLastError();
    cfg.numAttrs = 0;
    e = cudaLaunchKernelExC(&cfg, plan.fn, args);
  }
  if (e != cudaSuccess) return cuda_error(e, "launch (light engine)");
  return DJ_OK;
}

int run_light_batch(const LightPlan& plan, const SolveDesc* descs_dev, int32_t k, uint32_t* queue, bool zero_queue,
                    cudaStream_t st) {
  if (zero_queue) {
    cudaError_t e = cudaMemsetAsync(queue, 0, 2 * sizeof(uint32_t), st);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync(queue)");
  }
  LightCtaParams p{plan.npad};
  BatchJobs jobs;
  jobs.descs = descs_dev;
  jobs.queue = queue;
  jobs.k = k;
  void* args[] = {&p, &jobs};
  return launch_light(plan, args, st, false);
}

int run_light_single(const LightPlan& plan, const SolveDesc& d, uint32_t* phases_out, const SolveMark& mark,
                     cudaStream_t st) {
  LightCtaParams p{plan.npad};
  SingleJob job;
  job.d = d;
  job.phases_out = phases_out;
  job.early_ok = 1;  // no kernel ahead on the stream writes the graph: an upload takes it off this engine
  job.mark = mark;  // beyond the plain job, which the plan's kernel may take
  void* args[] = {&p, &job};
  return launch_light(plan, args, st, true);
}

int run_light_trials(const LightPlan& plan, const SolveDesc& d, uint32_t* light, cudaStream_t st) {
  LightCtaParams p{plan.npad};
  LightTrialJobs jobs;
  jobs.d = d;
  jobs.light = light;
  void* args[] = {&p, &jobs};
  return launch_light(plan, args, st, false);
}

int run_light_serve(const LightPlan& plan, const ServeRing& r, cudaStream_t st) {
  LightCtaParams p{plan.npad};
  ServeJobs jobs;
  jobs.ring = r.ring;
  jobs.tail = r.tail;
  jobs.stop = r.stop;
  jobs.done = r.done;
  jobs.head = r.head;
  jobs.cap_mask = r.cap_mask;
  jobs.idle_ns = r.idle_ns;
  void* args[] = {&p, &jobs};
  return launch_light(plan, args, st, false);
}

}  // namespace dj
