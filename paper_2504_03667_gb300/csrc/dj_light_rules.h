// The rules by which the light engine takes rows and graphs are loaded, in plain C++ (some for host and
// device), so that a host-only test can run them.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DJ_RULE __host__ __device__ __forceinline__
#else
#define DJ_RULE inline
#endif

namespace dj {

constexpr uint32_t kRuleInf = 0x7FFFFFFFu;   // the paper's infinity
constexpr uint32_t kRuleNone = 0xFFFFFFFFu;  // no dist

// What a reached row's unlisted edges offer at least, if that can still matter to a solve whose largest
// dist is D; kRuleNone otherwise.
DJ_RULE uint32_t light_pending(uint32_t dist, uint32_t hmin, uint32_t D) {
  if (dist == kRuleNone) return kRuleNone;
  const uint32_t x = dist + hmin;  // both below 2^31
  return x <= D && x < kRuleInf ? x : kRuleNone;
}

// Pending rows of dist below this are relaxed whole now, hb being the least that a pending row offers: a path
// shorter than dist would have to use an unlisted edge of a pending row, which offers no less than hb, so every
// dist up to hb is final.  Where each unlisted weight is at least 1 the row that gives hb lies below it; with
// unlisted weights of 0 it may lie at hb itself (rows below hb alone were none then, and the solve never ended).
// Rows at hb wait otherwise: most need not be relaxed once those below are (n = 8192, p = 0.5, weights 1..10: twice
// as many, and the trial at load 0.2 ms longer).
DJ_RULE uint32_t light_below(uint32_t hb, uint32_t hmin_min) { return hmin_min == 0 ? hb + 1 : hb; }

// Whether a graph's trial solve is run: some list is cut, and no weight is 0 (its solves take the other
// engines then, and its lists may hold nothing but a few of a row's edges of weight 0).
DJ_RULE bool light_needs_trial(uint32_t hmin_min, uint32_t wmin) { return hmin_min < kRuleInf && wmin > 0; }

// The first trial's source: a row with edges, of those with the most edges listed, n / 2 if it is one of
// them (a node that leads nowhere, or into a small part of the graph, says nothing about the others).  The
// rows' words are combined by maximum; n is below 2^24 (the matrix has n^2 entries).
DJ_RULE uint32_t light_trial_word(uint32_t u, uint32_t listed, bool has_edges, uint32_t n) {
  const uint32_t back = (u + n - n / 2 - 1) % n;  // n - 1 for u = n / 2
  return ((has_edges ? listed + 1 : 0u) << 24) | back;
}
DJ_RULE uint32_t light_trial_source(uint32_t word, uint32_t n) { return ((word & 0xFFFFFFu) + n / 2 + 1) % n; }

// Whether a row may have to be relaxed whole for some source s of a symmetric matrix, by the trial from t with the
// largest dist D: s's largest dist is at most D + d(t, s), and the row is pending only if d(s, u) + hmin does not
// exceed that, where d(s, u) >= |d(t, s) - d(t, u)|; so only if hmin <= D + d(t, u).
DJ_RULE bool light_risky(uint32_t dist, uint32_t hmin, uint32_t D) {
  return dist < kRuleInf && hmin < kRuleInf && hmin <= D + dist;
}

// What the first trial says about a graph with cut lists.  kTrialNo: no.  kTrialAll: few rows are ever
// relaxed whole, whatever the source (on a directed matrix the bound is none, but a good sign, and only the grid
// form is at stake).  kTrialAsk: other sources have to be tried (a structured graph's, or one of few distinct
// weights, may need many rows where this one needed none).
enum { kTrialNo, kTrialAll, kTrialAsk };
constexpr uint32_t kTrialRows = 4;         // whole rows the first trial may need
constexpr uint32_t kTrialMoreRows = 16;    // and each further one: seldom sources may need a few (n = 4096, p = 0.1, weights
                                           // 1..10: 126 us a solve in a batch, the streaming cluster engine 511)
constexpr uint32_t kTrialRisky = 32;       // rows at risk: one CTA reads as many in 50 us (n = 8192), and hardly ever must
constexpr uint32_t kTrialManyRows = 1024;  // the first trial stops beyond: its D, on which the longer lists hang, is settled
constexpr uint32_t kTrialPhases = 64;      // and here: dists reach far beyond the lists (a phase is an eighth of them)
inline int light_trial_verdict(uint32_t rows, uint32_t guess, uint32_t risky) {
  if (guess == 0 || rows > kTrialRows) return kTrialNo;  // guess 0: not every node that has an in-edge was reached
  return risky <= kTrialRisky ? kTrialAll : kTrialAsk;
}

// Whether a graph of less than kLightClusterMinN nodes whose lists of 64 edges are cut is one of few phases: its largest dist
// is at most three times its smallest weight, so the streaming engines need about three phases.  Single solves
// that run behind others then stay on the cluster engine: captured alone, n = 550, p = 0.7, weights 1..10 takes
// 35 us there and 50 on the light engine's CTA form, n = 1024 51 and 53; with a largest dist of 4 n = 1300,
// p = 0.3 already takes 70 and 59.  So do batches if every graph is such and has less than kFewBatchMinN nodes
// (16 solves, us: n = 300 39 and 47, n = 550 55 and 57, n = 700, p = 0.1 66 and 56, n = 1024 90 and 60).
constexpr int kLightClusterMinN = 2048, kFewBatchMinN = 600;
inline bool light_few(int32_t n, uint32_t guess, int32_t wmin) {
  return guess != 0 && n < kLightClusterMinN && static_cast<int64_t>(guess) - 1 <= 3 * static_cast<int64_t>(wmin);
}

// Whether the device may read a caller's host array in place: 4-byte loads fault on other addresses.
inline bool in_place(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }
inline bool edges_in_place(const void* src, const void* dst, const void* w) {
  return in_place(src) && in_place(dst) && in_place(w);
}

}  // namespace dj
