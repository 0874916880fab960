// Where a persistent solve kernel (cluster engine, light engine) gets its solves: a device table
// (batches), one descriptor in the kernel's parameters (single solves) or the serving ring.
#pragma once

#include "dj_common.cuh"
#include "dj_internal.h"

namespace dj {

// A single solve's last write (SolveMark): the host looks whether it has ended, nothing else hangs on it.
__device__ __forceinline__ void mark_done(const SolveMark& m) {
  if (m.done) *const_cast<volatile uint32_t*>(m.done) = m.seq;
}

// fetch() and complete() run on thread 0 of cluster rank 0 (of the CTA in the light engine) only.
struct BatchJobs {
  const SolveDesc* descs;
  uint32_t* queue;  // [0] next solve index, [1] exit count: both zero when a launch starts
  int32_t k;
  __device__ bool fetch(uint32_t* job, uint32_t) const {
    *job = atomicAdd(queue, 1u);
    return *job < static_cast<uint32_t>(k);
  }
  __device__ SolveDesc desc(uint32_t job) const { return descs[job]; }
  __device__ void complete(uint32_t, uint32_t) const {}
  static constexpr uint32_t kGuessPart = 3;  // light engine: the margin of its bound (light_guess)
  static constexpr bool kTrial = false;      // light engine: nothing is written, whole rows are counted
  static constexpr bool kTrace = false;
  __device__ bool early() const { return true; }  // launched the ordinary way: nothing to wait for
  __device__ void before_write() const {}
  // once per worker (a cluster, or a CTA of the light engine), by its first thread, after its last
  // fetch: the last of `workers` to leave zeroes the queue for the next launch (the stream starts it
  // only after this one has ended)
  __device__ void leave(uint32_t workers) const {
    __threadfence();
    if (atomicAdd(queue + 1, 1u) == workers - 1) {
      __threadfence();
      queue[0] = 0u;
      queue[1] = 0u;
    }
  }
};

// One solve whose descriptor travels in the kernel's parameters: no table,
// queue or memset on the device.  Launched as a single cluster; its rank 0
// records the phase count in the per-device word.  It is launched as a
// programmatic dependent of the kernel before it on the stream: it starts
// while that kernel is still running (every CTA lets its own dependents start
// at once), solves from the graph, which no kernel writes meanwhile (unless
// `early_ok` is 0, after an upload: then it waits first), and waits for its
// predecessor to complete only before it writes dist, pred and the phase
// count.  So results reach memory in stream order, and back-to-back solves of
// small graphs overlap on the GPU's idle SMs.
struct PlainSingleJob {
  SolveDesc d;
  uint32_t* phases_out;
  int32_t early_ok;
  __device__ bool fetch(uint32_t* job, uint32_t iter) const {
    *job = 0;
    return iter == 0 && cluster_id_x() == 0;
  }
  __device__ SolveDesc desc(uint32_t) const { return d; }
  __device__ void complete(uint32_t, uint32_t phases) const {
    if (phases_out) *phases_out = phases;
  }
  static constexpr uint32_t kGuessPart = 8;
  static constexpr bool kTrial = false;
  static constexpr bool kTrace = true;  // the per-phase timeline is compiled into this kernel only
  __device__ bool early() const { return early_ok != 0; }
  __device__ void before_write() const { pdl_wait(); }
  __device__ void leave(uint32_t) const {}
};

// The same with a mark for the next solve's choice of form.  (A job of its own: the light engine's CTA form took
// 36.7 us instead of 34.4 for n = 1024 alone with the mark compiled in, used or not.)
struct SingleJob : PlainSingleJob {
  SolveMark mark;
  __device__ void complete(uint32_t job, uint32_t phases) const {
    PlainSingleJob::complete(job, phases);
    mark_done(mark);
  }
};

// Serving: requests arrive in a ring of descriptors in mapped pinned host
// memory.  The host publishes request r by writing ring[r % cap] and then
// tail = r + 1 (release); a cluster claims r by advancing the device-side head
// with a CAS, and reports completion with done[r % cap] = r + 1 (release,
// system scope).  Waiting for work is bounded: after idle_ns without a
// request, or once the host sets *stop, fetch() returns false and the kernel
// exits (the host relaunches it when requests come again).
struct ServeJobs {
  const SolveDesc* ring;  // mapped host memory, cap entries
  const uint32_t* tail;   // mapped host memory
  const uint32_t* stop;   // mapped host memory
  uint32_t* done;         // mapped host memory, cap entries
  uint32_t* head;         // device memory
  uint32_t cap_mask;
  int64_t idle_ns;
  __device__ bool fetch(uint32_t* job, uint32_t) const {
    uint64_t t0 = global_ns();
    for (;;) {
      if (ld_acquire_sys(stop)) return false;
      const uint32_t h = ld_relaxed_gpu(head);
      const uint32_t t = ld_acquire_sys(tail);
      if (static_cast<int32_t>(t - h) > 0) {
        if (atomicCAS(head, h, h + 1) == h) {
          *job = h;
          return true;
        }
        continue;
      }
      if (static_cast<int64_t>(global_ns() - t0) > idle_ns) return false;
      __nanosleep(256);
    }
  }
  __device__ SolveDesc desc(uint32_t job) const {
    const SolveDesc* src = ring + (job & cap_mask);
    SolveDesc d;
    const uint4* s4 = reinterpret_cast<const uint4*>(src);
    uint4* d4 = reinterpret_cast<uint4*>(&d);
#pragma unroll
    for (int i = 0; i < static_cast<int>(sizeof(SolveDesc) / 16); ++i) d4[i] = __ldcv(s4 + i);
    return d;
  }
  __device__ void complete(uint32_t job, uint32_t) const {
    __threadfence_system();
    st_release_sys(done + (job & cap_mask), job + 1);
  }
  static constexpr uint32_t kGuessPart = 8;
  static constexpr bool kTrial = false;
  static constexpr bool kTrace = false;
  __device__ bool early() const { return true; }
  __device__ void before_write() const {}
  __device__ void leave(uint32_t) const {}
};

// Light engine: a CTA each for kMoreTrials trial solves of one graph, the first from the farthest node of
// the trial before, the others from places spread over the ids.
struct LightTrialJobs {
  SolveDesc d;  // without outputs
  uint32_t* light;
  __device__ bool fetch(uint32_t* job, uint32_t iter) const {
    *job = blockIdx.x;
    return iter == 0;
  }
  __device__ SolveDesc desc(uint32_t job) const {
    SolveDesc x = d;
    x.source = job == 0 ? static_cast<int32_t>(__ldcg(light + kLightFar))
                        : static_cast<int32_t>(static_cast<int64_t>(d.n) * (2 * job - 1) / (2 * kMoreTrials - 2));
    return x;
  }
  __device__ void complete(uint32_t, uint32_t) const {}
  __device__ uint32_t* whole(uint32_t job) const { return light + kLightMore + job; }
  static constexpr uint32_t kGuessPart = 8;
  static constexpr bool kTrial = true;
  static constexpr bool kTrace = false;
  __device__ bool early() const { return true; }  // launched the ordinary way: nothing to wait for
  __device__ void before_write() const {}
  __device__ void leave(uint32_t) const {}
};

}  // namespace dj
