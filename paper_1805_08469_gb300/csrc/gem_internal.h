// Internal declarations of the GEM commit library (not installed, not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <vector>

#include "../../include/gem.h"

namespace gem {

// Commits carried by one launch of the batched commit kernel.  They travel in the
// kernel's parameter block (6.4 KB and a header), so a launch needs no device-side
// descriptor; longer batches are split into several launches, in order.
constexpr int kMaxBatchPerLaunch = 200;

// Row stride of m and s (and length of theta): P rounded up to 32 floats = 128 bytes.
constexpr size_t kStrideAlign = 32;

// Host-gradient staging for gem_commit_batch_host: two halves of kStageChunk slots.
constexpr int kStageChunk = 8;

// How a launch scales each commit.
enum RuleKind : int {
  kRuleGem = 0,     // pi from energy matching with the proxy |m_w| (Algorithm 1)
  kRuleScaled = 1,  // the same with the proxy energy_scale |m_w| (App. B, high-energy proxies)
  kRuleFixed = 2,   // pi[k] given per commit; m_w untouched (DOWNPOUR, adaptive staleness)
  kRuleMomentum = 3,  // the proxy itself: theta += (m_w <- mu m_w + dtheta); no factor
};

// L2 policy of a store.
enum L2Hint : uint8_t { kL2Normal = 0, kL2Keep = 1, kL2Stream = 2 };

// How a commit of a launch reads and leaves its worker's m_w and s_w (one word, so that the
// kernel reads it with one load).
//   - slot_out >= 0 (rules with a moment): the worker commits again later in the launch and
//     its lanes stay in that shared-memory slot instead of going to global memory; its next
//     commit takes them from the slot of the same number, slot_in.
//   - slot_in or slot_out < 0: from or to global memory.
//   - keep_s (rules that do not read s_w): 0 skips the store of s_w when the worker commits
//     again in the launch (nothing reads it before that).
//   - l2: policy of the commit's stores of m_w and s_w to global memory (launches of more than
//     kSmallBatch commits, rules with a moment): kL2Keep when a later commit of the launch
//     reads them back from global memory, kL2Stream at the worker's last commit of the launch.
struct CommitCtl {
  uint32_t bits;
  CommitCtl() = default;
  __host__ __device__ CommitCtl(int in, int out, bool keep_s, int l2)
      : bits(uint32_t(uint8_t(in)) | uint32_t(uint8_t(out)) << 8 | uint32_t(keep_s) << 16 | uint32_t(l2) << 24) {}
  __host__ __device__ int slot_in() const { return int8_t(bits); }
  __host__ __device__ int slot_out() const { return int8_t(bits >> 8); }
  __host__ __device__ bool keep_s() const { return (bits >> 16 & 1u) != 0; }
  __host__ __device__ int l2() const { return int(bits >> 24); }
  __host__ __device__ void set_slot_in(int v) { bits = (bits & ~0xFFu) | uint8_t(v); }
  __host__ __device__ void set_slot_out(int v) { bits = (bits & ~0xFF00u) | uint32_t(uint8_t(v)) << 8; }
};

// One commit of a launch (read by the kernel through one address).
struct Commit {
  const float* grad;     // its gradient, P floats
  long long row;         // byte offset of its worker's row in m and s
  float* pi_out;         // receives its scaling factors, P floats, or null
  CommitCtl ctl;
  float pi;              // kRuleFixed: its scaling factor
};

// Arguments of one launch of the fused commit kernel, for up to KCAP commits.  Launches of
// at most kSmallBatch commits (the segments of the simulators) and single commits pass a
// shorter form: the kernel parameters then take about 1 KB or 100 bytes instead of 6.5 KB.
template <int KCAP>
struct BatchArgsT {
  float* theta;                            // [stride]
  float* m;                                // [n][stride]
  float* s;                                // [n][stride]
  size_t P;
  float eta, mu, eps;
  int K;                                   // commits in this launch, 1..KCAP
  int rule;                                // RuleKind
  float energy_scale;                      // kRuleScaled: factor on |m_w|
  int record_pi;                           // 1: a commit's pi_out, when not null, receives its factors
  Commit commit[KCAP];
  // Factor counts of a recording launch (null: none).  For every commit k with pi_out
  // set and every segment s = [pi_seg[s], pi_seg[s + 1]) of the coordinates, the number of
  // recorded factors whose sign bit is set (below +0 in the total order of the medians) is
  // added to pi_counts[2 (k pi_nseg + s)] and the number equal to +0 to the word after it.
  unsigned* pi_counts;
  const long long* pi_seg;                 // device array [pi_nseg + 1], non-decreasing
  int pi_nseg;
  int lane_rows;                           // dynamic shared memory: rows of a 16-byte lane per thread
  int grads_on_host;                       // 1: the gradients lie in page-locked host memory
  int grads_through_l1;                    // 1: the copies of the gradients are cached in L1
};
using BatchArgs = BatchArgsT<kMaxBatchPerLaunch>;
constexpr int kSmallBatch = 32;

// Shared-memory slots of the commit kernel (a worker's m_w and s_w lanes, 32 bytes per
// thread and slot), and the commits whose copies a thread has in flight (rules with a moment):
// 3 stages and 8 slots of a 128-thread block take 50 KB, four blocks per SM.  Measured at
// P = 25M, n = 100 (us per 100 commits): 4 stages and 6 slots 5,170, 2 and 5 (six blocks)
// 5,346, 4 and 12 (three blocks) 5,159, 2 and 9 5,737; at P = 1.2M, n = 20: 189, 191, 232, 208,
// against 190.
#ifndef GEM_COMMIT_SLOTS
#define GEM_COMMIT_SLOTS 8
#endif
constexpr int kCommitSlots = GEM_COMMIT_SLOTS;
#ifndef GEM_COMMIT_DEPTH
#define GEM_COMMIT_DEPTH 3
#endif
constexpr int kCommitDepth = GEM_COMMIT_DEPTH;

// Fill the ctl of a launch's commits from the workers of its a.K commits.
void plan_slots(BatchArgs& a, const int* worker);

// Launch the fused commit kernel for a.K commits on `stream`.
cudaError_t launch_commit_batch(const BatchArgs& a, int sm_count, cudaStream_t stream);

// Shared-memory words a recording launch may use for its factor counts (2 per commit and
// segment); callers split their commits so that K * pi_nseg * 2 stays within it.
constexpr int kMaxCountWords = 4096;

}  // namespace gem

struct gem_ctx {
  int device = 0;
  int sm_count = 0;
  size_t P = 0;
  size_t stride = 0;
  int n = 0;
  float eta = 0.f, mu = 0.f, eps = 0.f;
  float* theta = nullptr;
  float* m = nullptr;
  float* s = nullptr;
  cudaStream_t stream = nullptr;
  uint64_t launches = 0;
  bool broken = false;
  // commit rule (gem_set_mode) and the commit clock the staleness is counted on
  int mode = GEM_MODE_GEM;
  float kappa = 1.f;
  int64_t clock = 0;           // commits issued since gem_set_theta
  std::vector<int64_t> last;   // [n] clock value of worker w's last commit, -1 before its first
  // scratch of the pi median select: histograms and per-problem state, grown on demand
  void* select_scratch = nullptr;
  size_t select_bytes = 0;
  // staging of host gradients (gem_commit_batch_host), allocated on first use
  float* stage = nullptr;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t stage_filled[2] = {nullptr, nullptr};
  cudaEvent_t stage_free[2] = {nullptr, nullptr};
};

namespace gem {

// Launch commits [0, K) of the handle in order, in chunks of kMaxBatchPerLaunch, with the
// handle's commit rule; advances the commit clock and counts the launches.  The arguments
// must have been checked.
// With pi_counts set (K * pi_nseg * 2 <= kMaxCountWords, one launch), the recording launch
// also adds the factor counts of every commit and segment to pi_counts (see BatchArgsT).
// grads_on_host: the gradients are read from page-locked host memory.
cudaError_t commit_ordered(gem_ctx* h, const int* order, const float* const* grads, int K,
                           float* const* pi_out = nullptr, unsigned* pi_counts = nullptr,
                           const long long* pi_seg = nullptr, int pi_nseg = 0, bool grads_on_host = false);

// Segments per median call and commits per select launch.
constexpr int kMaxPiSegments = 64;
constexpr int kMaxPiBatch = 200;

// Exact lower and upper medians of each segment of each of K scaling-factor rows
// (segments seg[0..nseg] shared by all rows), written to lo/hi [K][nseg] on the handle's
// stream.  Uses the handle's select scratch (grown on demand).  Arguments checked by the
// caller.
cudaError_t pi_median_ordered(gem_ctx* h, const float* const* pi, int K, const int64_t* seg,
                              int nseg, float* lo, float* hi);

// Commits [0, K) in order with every factor recorded in pi[k] (all set), then the lower and
// upper medians of each row and segment as pi_median_ordered.  The recording launches also
// count each row's factors below and equal to +0 per segment, so a middle element that lies
// in the run of zeros is known before any selection pass, and a row and segment whose two
// middle elements both lie there is never read again.  Arguments checked by the caller.
cudaError_t commit_pi_median_ordered(gem_ctx* h, const int* order, const float* const* grads,
                                     int K, float* const* pi, const int64_t* seg, int nseg,
                                     float* lo, float* hi);

}  // namespace gem
