// Internal interface of the Monte-Carlo statistics pass, shared by the two per-use checks: a check
// launches each of its statistics passes into a slot of block partials as soon as the pass's inputs
// are queued; at its end one kernel sums the slots, and eight numbers per slot come to the host behind one
// synchronisation.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace bsp {

constexpr int kStatBlocks = 592;     // 4 per SM
constexpr int kStatFields = 8;       // err2, ref2, se2, z2, z, max|z|, count(|z|>3), unused
constexpr size_t kStatSlotDoubles = (size_t)kStatBlocks * kStatFields;
constexpr size_t kStatSlotBytes = kStatSlotDoubles * sizeof(double);   // a multiple of 256

// Launches the pass over n elements into one slot; *blocks_out = blocks whose partials the slot holds.
int mc_stats_launch(const float* g_ref, const float* g, const float* S2, int64_t n, int K, int fresh,
                    const bsp_verdict_rule_t* rule, double* partials, cudaStream_t st, int* blocks_out);
// Sums each of `count` consecutive slots over its blocks (in a fixed order) into out[slot][kStatFields].
constexpr int kMaxPendingStats = 12;      // slots of a workspace; the last one takes the sums of the others
struct StatBlocks { int n[kMaxPendingStats]; };
int mc_stats_sum_slots(const double* slots, const StatBlocks& blocks, int count, double* out, cudaStream_t st);
// Sums `blocks` records of partial statistics in order and fills the result of the use; the
// verdict follows `rule` (NULL: the default thresholds, see default_rule()).
void mc_stats_finish(const double* host, int blocks, int64_t n, int K, int fresh, const bsp_verdict_rule_t* rule,
                     bsp_use_result_t* result);
const bsp_verdict_rule_t* default_rule();
// A rule is usable when its thresholds are ordered: hold <= fail for both statistics, nothing negative.
bool rule_valid(const bsp_verdict_rule_t* rule);

struct PendingStats {
  bsp_use_result_t* result[kMaxPendingStats];
  int blocks[kMaxPendingStats], K[kMaxPendingStats], fresh[kMaxPendingStats];
  int64_t n[kMaxPendingStats];
  int count = 0;
  double* slots = nullptr;           // device: kMaxPendingStats slots of kStatSlotDoubles
  cudaStream_t st = nullptr;
  const bsp_verdict_rule_t* rule = nullptr;

  // A fresh read whose every draw equals the reference (a gradient that does not read the saved
  // tensor): all sums are zero, no pass needed.
  void add_exact_fresh(int64_t n_, int K_, bsp_use_result_t* r) { mc_stats_finish(nullptr, 0, n_, K_, 1, rule, r); }
  int add(const float* g_ref, const float* g, const float* S2, int64_t n_, int K_, int fresh_, bsp_use_result_t* r) {
    if (!fresh_ && g == g_ref) {
      // a read that is the reference itself: its error is exactly zero, no pass needed
      mc_stats_finish(nullptr, 0, n_, K_, 0, rule, r);
      return BSP_OK;
    }
    if (count >= kMaxPendingStats - 1) return BSP_ERR_ARG;
    const int slot = count++;
    result[slot] = r; n[slot] = n_; K[slot] = K_; fresh[slot] = fresh_;
    return mc_stats_launch(g_ref, g, S2, n_, K_, fresh_, rule, slots + (size_t)slot * kStatSlotDoubles, st, &blocks[slot]);
  }
  // One small copy, one synchronisation.  The stream is idle when this returns.  (The slots themselves are 38 KB
  // each: copying and summing them here took 21 us of the smallest check.)
  int flush() {
    double host[kMaxPendingStats * kStatFields];
    if (count > 0) {
      StatBlocks nb;
      for (int i = 0; i < count; ++i) nb.n[i] = blocks[i];
      double* sums = slots + (size_t)(kMaxPendingStats - 1) * kStatSlotDoubles;
      const int rc = mc_stats_sum_slots(slots, nb, count, sums, st);
      if (rc != BSP_OK) return rc;
      const size_t bytes = (size_t)count * kStatFields * sizeof(double);
      BSP_CHECK_CUDA(cudaMemcpyAsync(host, sums, bytes, cudaMemcpyDeviceToHost, st));
      count_d2h(bytes);
    }
    BSP_CHECK_CUDA(cudaStreamSynchronize(st));
    for (int i = 0; i < count; ++i)
      mc_stats_finish(host + (size_t)i * kStatFields, 1, n[i], K[i], fresh[i], rule, result[i]);
    count = 0;
    return BSP_OK;
  }
};

}  // namespace bsp
