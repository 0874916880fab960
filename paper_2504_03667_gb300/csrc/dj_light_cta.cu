// Light engine, CTA form: one CTA per solve with the keys in shared memory (n up to about 22000),
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
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr int kLightRows = 4;  // rows in flight per lane group
// delta in units of the listed weights' mean spacing (narrower than the grid form's: a phase costs
// little here)
constexpr float kCtaDelta = 1.0f;
}  // namespace

struct LightCtaParams {
  uint32_t* heavy;  // optional: rows relaxed whole are counted here
  int32_t npad;     // key slots (largest graph of the launch, rounded up to 64)
};

// Offer w's key to v in shared memory; a shorter dist makes v dirty and lowers lmin.
__device__ __forceinline__ void light_offer(unsigned long long* keys, uint32_t* dirty, uint32_t v, uint64_t key,
                                            uint32_t& lmin) {
  if (key < keys[v]) {
    const uint64_t old = atomicMin(keys + v, static_cast<unsigned long long>(key));
    const uint32_t c = static_cast<uint32_t>(key >> 32);
    if (c < static_cast<uint32_t>(old >> 32)) {
      atomicOr(dirty + (v >> 5), 1u << (v & 31u));
      lmin = min(lmin, c);
    }
  }
}

template <int THREADS, class Jobs>
__global__ void __launch_bounds__(THREADS) k_light_cta(const LightCtaParams p, const Jobs jobs) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_job, s_cnt, s_m[2], s_D;
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem);
  uint16_t* list = reinterpret_cast<uint16_t*>(smem + static_cast<size_t>(p.npad) * 8);
  uint32_t* dirty = reinterpret_cast<uint32_t*>(smem + static_cast<size_t>(p.npad) * 10);
  uint32_t* hdone = dirty + p.npad / 32;
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31;
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
    const uint32_t* edge = hmin + light_pad(n);
    const uint32_t hmin_min = ~__ldg(d.light);  // >= INF: every row's list is complete
    uint32_t delta;
    int gshift;
    light_window(d.light, kCtaDelta, &delta, &gshift);
    const int gl = tid & ((1 << gshift) - 1), gid = tid >> gshift, ng = THREADS >> gshift, gsz = 1 << gshift;

    for (int v = tid; v < n; v += THREADS) keys[v] = ~0ull;
    for (int i = tid; i < nwords; i += THREADS) {
      dirty[i] = 0;
      hdone[i] = 0;
    }
    __syncthreads();
    if (tid == 0) {
      keys[d.source] = 0;
      dirty[d.source >> 5] = 1u << (d.source & 31);
      s_m[0] = 0;
      s_cnt = 0;
      s_D = 0;
    }
    __syncthreads();
    uint32_t phase = 0;
    uint32_t D = kNone;
    for (;;) {
      const uint32_t m = s_m[phase & 1];
      uint32_t lmin = kNone;
      if (m != kNone) {
        // the dirty nodes within the window, into list (a warp per word of 32 nodes, a lane per node)
        const uint32_t T = m + delta;
        for (int wi = tid >> 5; wi < nwords; wi += THREADS / 32) {
          const uint32_t bits = dirty[wi];
          if (bits == 0) continue;
          const int v = 32 * wi + lane;
          const bool on = (bits >> lane) & 1u;
          const uint32_t dv = on ? static_cast<uint32_t>(keys[v] >> 32) : kNone;
          const bool take = on && dv <= T;
          if (on && !take) lmin = min(lmin, dv);
          const uint32_t bal = __ballot_sync(0xffffffffu, take);
          if (bal == 0) continue;
          uint32_t pos = 0;
          if (lane == 0) {
            pos = atomicAdd(&s_cnt, static_cast<uint32_t>(__popc(bal)));
            dirty[wi] = bits & ~bal;
          }
          pos = __shfl_sync(0xffffffffu, pos, 0);
          if (take) list[pos + __popc(bal & ((1u << lane) - 1u))] = static_cast<uint16_t>(v);
        }
        // D: no offer beyond the largest dist can matter (complete lists are short: not worth it)
        if (hmin_min < kInf) {
          uint32_t mx = 0;
          for (int v = tid; v < n; v += THREADS) {
            const uint32_t dv = static_cast<uint32_t>(keys[v] >> 32);
            if (dv < kInf)
              mx = max(mx, dv);
            else if (static_cast<uint32_t>(__ldg(d.minout + n + v)) < kInf)
              mx = kNone;  // not reached yet, and something leads to it
          }
          mx = __reduce_max_sync(0xffffffffu, mx);
          if (lane == 0) atomicMax(&s_D, mx);
        }
        if (tid == 0) s_m[(phase + 1) & 1] = kNone;
        __syncthreads();
        const int cnt = static_cast<int>(s_cnt);
        if (hmin_min < kInf) D = s_D;
        for (int i0 = gid; i0 < cnt; i0 += ng * kLightRows) {
          uint32_t u[kLightRows], du[kLightRows];
          const uint32_t* row[kLightRows];
          bool on[kLightRows];
#pragma unroll
          for (int r = 0; r < kLightRows; ++r) {
            const int i = i0 + r * ng;
            on[r] = i < cnt;
            u[r] = on[r] ? list[i] : 0u;
            row[r] = edge + static_cast<size_t>(u[r]) * kLightCap;
          }
#pragma unroll
          for (int r = 0; r < kLightRows; ++r) du[r] = static_cast<uint32_t>(keys[u[r]] >> 32);
          for (int k = gl; k < kLightCap; k += gsz) {
            uint32_t e[kLightRows];
#pragma unroll
            for (int r = 0; r < kLightRows; ++r) e[r] = on[r] ? __ldg(row[r] + k) : kNoEdge;
            bool any = false;
#pragma unroll
            for (int r = 0; r < kLightRows; ++r) {
              const uint32_t w = e[r] >> bits_u;
              on[r] = e[r] != kNoEdge && du[r] + w <= D;  // sorted: what follows is heavier
              any |= on[r];
              if (on[r]) light_offer(keys, dirty, e[r] & umask, light_key(du[r], w, u[r], bits_u), lmin);
            }
            if (!any) break;
          }
        }
      } else {
        // nothing is dirty: the index proves the answer, or some rows are relaxed whole
        if (hmin_min > D || hmin_min >= kInf) break;
        if (tid == 0) {
          s_cnt = 0;
          s_job = kNone;  // here: the smallest dist + hmin of the pending rows
          s_m[(phase + 1) & 1] = kNone;
        }
        __syncthreads();
        uint32_t hb = kNone;
        for (int v = tid; v < n; v += THREADS) {
          const uint32_t dv = static_cast<uint32_t>(keys[v] >> 32);
          if (dv >= kInf || ((hdone[v >> 5] >> (v & 31)) & 1u)) continue;
          const uint32_t x = dv + __ldg(hmin + v);
          if (x <= D && x < kInf) hb = min(hb, x);
        }
        hb = warp_min_u32(hb);
        if (lane == 0 && hb != kNone) atomicMin(&s_job, hb);
        __syncthreads();
        hb = s_job;
        if (hb == kNone) break;
        for (int v = tid; v < n; v += THREADS) {
          const uint32_t dv = static_cast<uint32_t>(keys[v] >> 32);
          if (dv >= hb || ((hdone[v >> 5] >> (v & 31)) & 1u)) continue;
          const uint32_t x = dv + __ldg(hmin + v);
          if (x > D || x >= kInf) continue;
          list[atomicAdd(&s_cnt, 1u)] = static_cast<uint16_t>(v);
          atomicOr(hdone + (v >> 5), 1u << (v & 31));
        }
        __syncthreads();
        const int cnt = static_cast<int>(s_cnt);
        if (p.heavy && tid == 0) atomicAdd(p.heavy, static_cast<uint32_t>(cnt));
        const int nv = static_cast<int>(d.pitch / 4);
        for (int i = 0; i < cnt; ++i) {
          const uint32_t u = list[i];
          const uint32_t du = static_cast<uint32_t>(keys[u] >> 32);
          const int4* row = reinterpret_cast<const int4*>(d.W + static_cast<int64_t>(u) * d.pitch);
          for (int g = tid; g < nv; g += THREADS) {
            const int4 x = __ldg(row + g);
            const uint32_t w4[4] = {static_cast<uint32_t>(x.x), static_cast<uint32_t>(x.y), static_cast<uint32_t>(x.z),
                                    static_cast<uint32_t>(x.w)};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t v = 4 * g + q;
              if (w4[q] < kInf && du + w4[q] <= D && v != u)
                light_offer(keys, dirty, v, light_key(du, w4[q], u, bits_u), lmin);
            }
          }
        }
      }
      lmin = warp_min_u32(lmin);
      if (lane == 0 && lmin != kNone) atomicMin(&s_m[(phase + 1) & 1], lmin);
      __syncthreads();
      if (tid == 0) {  // for the next phase's scan; ordered before it by the barrier below
        s_cnt = 0;
        s_D = 0;
      }
      __syncthreads();
      ++phase;
    }
    jobs.before_write();  // results reach memory in stream order
    for (int v = tid; v < n; v += THREADS) {
      const uint64_t k = keys[v];
      const uint32_t dv = static_cast<uint32_t>(k >> 32);
      const bool reached = dv < kInf;
      d.dist[v] = static_cast<int32_t>(reached ? dv : kInf);
      d.pred[v] = reached && v != d.source ? static_cast<int32_t>(static_cast<uint32_t>(k) & umask) : -1;
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


int light_smem_nodes(int32_t n) { return light_pad(n); }
size_t light_cta_smem(int32_t n) {
  const size_t np = static_cast<size_t>(light_smem_nodes(n));
  return np * 10 + np / 32 * 8;
}

template <int THREADS>
void* light_cta_kernel(int kind) {
  if (kind == kJobsServe) return reinterpret_cast<void*>(&k_light_cta<THREADS, ServeJobs>);
  if (kind == kJobsSingle) return reinterpret_cast<void*>(&k_light_cta<THREADS, SingleJob>);
  return reinterpret_cast<void*>(&k_light_cta<THREADS, BatchJobs>);
}

}  // namespace

bool light_cta_fits(int32_t n) {
  DevCtx* ctx = nullptr;
  if (get_ctx(&ctx) != DJ_OK) return false;
  return light_cta_smem(n) + 1024 <= static_cast<size_t>(ctx->max_smem_optin);
}

int plan_light(int32_t max_n, int32_t k, int kind, LightPlan* plan) {
  DevCtx* ctx = nullptr;
  if (int rc = get_ctx(&ctx)) return rc;
  plan->smem = light_cta_smem(max_n);
  plan->npad = light_smem_nodes(max_n);
  // two or more CTAs per SM where shared memory allows, else one large one
  const bool large = plan->smem > static_cast<size_t>(ctx->max_smem_optin) / 2 - 2048;
  plan->threads = large || (kind == kJobsSingle && max_n >= 2048) ? 1024 : 512;
  plan->fn = plan->threads == 1024 ? light_cta_kernel<1024>(kind) : light_cta_kernel<512>(kind);
  if (int rc = prepare_function(ctx, plan->fn, plan->smem, false)) return rc;
  plan->ctas = 1;
  if (kind != kJobsSingle) {
    int occ = 0;
    if (int rc = function_occupancy(ctx, plan->fn, plan->threads, plan->smem, &occ)) return rc;
    if (occ < 1) return set_error(DJ_EUNSUPPORTED, "light engine cannot be resident");
    plan->ctas = ctx->num_sms * occ;
    if (kind == kJobsBatch) plan->ctas = std::max(1, std::min(plan->ctas, static_cast<int>(k)));
  }
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
  LightCtaParams p{nullptr, plan.npad};
  BatchJobs jobs;
  jobs.descs = descs_dev;
  jobs.queue = queue;
  jobs.k = k;
  void* args[] = {&p, &jobs};
  return launch_light(plan, args, st, false);
}

int run_light_single(const LightPlan& plan, const SolveDesc& d, uint32_t* phases_out, uint32_t* heavy, bool early,
                     cudaStream_t st) {
  LightCtaParams p{heavy, plan.npad};
  SingleJob job;
  job.d = d;
  job.phases_out = phases_out;
  job.early_ok = early ? 1 : 0;
  void* args[] = {&p, &job};
  return launch_light(plan, args, st, true);
}

int run_light_serve(const LightPlan& plan, const ServeRing& r, cudaStream_t st) {
  LightCtaParams p{nullptr, plan.npad};
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
