// Shared by every translation unit of the verification step: workspace structures, kernel
// parameters, and the entry through which the host reaches the fused context kernel's
// compile-time variants.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "lantern.h"
#include "lantern_device.cuh"

namespace lantern {

#define LANTERN_CONTEXT_KERNEL_REVISION 34   // bump on every change to the fused context kernel

constexpr int MAX_N = 1024;

struct Counters {               // first 256 bytes of the workspace, zeroed per call by the plan kernel
  int work_next;                // dynamic part of the work counter
  int n_bonus;                  // next tokens taken from a context's own target
  int n_evaluated;              // contexts the fused pass evaluated
  int n_skipped;                // contexts it left out because the walk cannot reach them
  int n_tested;                 // drafted nodes it tested
  int status_or;                // OR of every sequence's status bits
  int abort;                    // a bounded wait ran out somewhere: no further work is handed out
  int n_slow_topk;              // rows whose top-k threshold needed the slow exact search
};

struct Record {                 // a context's walk word (see walk_word below), 16 bytes apart
  unsigned long long word, unused;
};

struct ChildInfo {              // one drafted node, stored in the order its parent context tries it
  int node;                     // node index within the sequence
  int token;                    // x~
  float r;                      // its acceptance uniform
  int span;                     // the contexts behind the node, in pre-order: (first position << 16) | count
};

struct WorkItem {               // one context with children: everything its CTA needs, in one 32-byte load
  int item;                     // b * R + c  (row index of the context); -1 = none
  int cbase;                    // index of its first child in the ChildInfo array
  int nchild_node0;             // (number of children << 16) | first child's node index
  int span0;                    // first child's ChildInfo::span
  int tok0;                     // first child's token and uniform, inlined
  float r0;
  float u_final;                // the sequence's uniform for the final draw
  int mark;                     // index of the context's own entry in the array of dead marks
};

struct GroupItem {              // the same, as a producer hands it to its consumer group through shared memory
  int item, cbase, nchild, node0, tok0, span0;
  float r0, u_final;
};

struct VerifyParams {
  const void* target;
  const void* draft;
  const int32_t* tokens;
  const int32_t* parents;
  const int32_t* nbr;
  const float* uniforms;
  int32_t* out_len;
  int32_t* out_tok;
  int32_t* out_path;
  int32_t* out_status;
  float* out_qa;
  float* out_px;
  int32_t* out_m;
  // workspace pieces
  Counters* counters;
  WorkItem* work;               // [N, B]: slot r * B + b holds the r-th context with children of sequence b in
                                //         breadth-first order (by depth, then by index); item = -1 where there is none
  int32_t* leaves;              // [N, B]: slot r * B + b holds the r-th context without children of sequence b, (its place in
                                //         pre-order << 16) | its number, -1 where there is none; null: not listed (see verify.cu)
  unsigned char* dead;          // [B, R], a sequence's contexts in pre-order: 1 once the walk is known not to reach one
  ChildInfo* children;          // [B, N]
  Record* records;              // [B, R]
  int B, N, R, V, k;
  float cfg_scale, T, delta;
  int divergence;               // LANTERN_DIV_TVD or LANTERN_DIV_JSD: what delta bounds
  int top_k;                    // logit filter; 0 = off
  // l / T without a division (divide_by_T): each as a pair of equal fp32 values
  uint64_t T_neg, T_inv, T_inv_hi, T_inv_lo;   // -T, the reciprocal rounded to nearest; rounded towards zero, and what that leaves
  int T_fast;                   // 0: T is so large or so small that a division is done after all
  uint32_t T_least;             // 2 bits(|l|) - 1 of the smallest |l| whose quotient is always a division's
  uint32_t wait_tries;          // limit of every bounded mbarrier wait, in tries
  int32_t* block_words;         // one word per block of the plan kernel: see plan_word
  int withhold_item;            // self-test only: the copies of this context are never issued (-1 = none)
};

constexpr int kNone = 0x7fffffff;
// A residual whose total weight is at most this fraction of the current target's mass defines no
// distribution to draw from (the single-precision residual pass resolves totals to a few 1e-7 of that
// mass): the walk stops there and the next token comes from the context's own target.
constexpr double kDegenerate = 1e-5;

// The walk over the contexts of a sequence (verify_context.cuh): one word per
// context, exchanged by whoever decides the context and by the walk when it gets there.
//   bits 0..1 state; walk waiting: bits 8..15 status so far, bits 16..31 drafts accepted so far;
//   decided: bits 8..15 status, bits 16..31 accepted node + 1 (0 = none), bits 32..63 replacement token
// A context without children starts as kWalkLeaf: the bonus draw is made by the walk when it gets there, or ahead of time by a
// producer that has put kWalkPending in the place of kWalkLeaf first (compare-and-swap); its decided word carries kWalkDrawn.
enum : unsigned { kWalkPending = 0, kWalkWaiting = 1, kWalkDecided = 2, kWalkLeaf = 3, kWalkDrawn = 4 };
__device__ __forceinline__ unsigned long long walk_word(unsigned state, unsigned status, unsigned count, int token = 0) {
  return state | (status << 8) | (static_cast<unsigned long long>(count) << 16) |
         (static_cast<unsigned long long>(static_cast<unsigned>(token)) << 32);
}

constexpr int PLAN_SEQS = 4;    // sequences per block of the plan kernel

// A block of the plan kernel sums up its sequences in one word: the largest number of contexts with children in one of them, the
// largest number of contexts without, and all fault bits.
__device__ __forceinline__ int plan_word(int ranks, int leaves, int faults) { return faults << 22 | leaves << 11 | ranks; }
// The plan's summary, by a whole warp: slots in the occupied parts of the work list and of the list of leaves, and the fault bits
// of all sequences.
struct PlanSummary {
  int slots, leaf_slots, faults;
};
template <bool LEAVES>   // they are listed
__device__ __forceinline__ PlanSummary plan_summary(const VerifyParams& P, int lane) {
  int ranks = P.N > 0 ? 0 : 1, leaves = 0, bits = 0;
  const int blocks = (P.B + PLAN_SEQS - 1) / PLAN_SEQS;
#pragma unroll 4
  for (int i = lane; i < blocks; i += 32) {
    const int w = P.block_words[i];
    ranks = max(ranks, w & 0x7ff);
    leaves = max(leaves, w >> 11 & 0x7ff);
    bits |= w >> 22;
  }
  return {__reduce_max_sync(kFull, ranks) * P.B, LEAVES ? __reduce_max_sync(kFull, leaves) * P.B : 0, static_cast<int>(__reduce_or_sync(kFull, bits))};
}
// The same without the fault bits: a chain has a context with a child for every draft, and one leaf.
template <bool LEAVES>
__device__ __forceinline__ PlanSummary plan_extent(const VerifyParams& P, int lane) {
  if (!P.parents) return {(P.N > 0 ? P.N : 1) * P.B, LEAVES ? P.B : 0, 0};
  return plan_summary<LEAVES>(P, lane);
}

__device__ __forceinline__ float sum8(const float* v) {
  return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
}


// ---- host side ----
// Launch that lets the kernel be put in place while the one before it in the stream still runs (it waits for it by
// grid_dependency_wait before it touches anything).
template <class K>
static inline cudaError_t launch_dependent(K kernel, int grid, int threads, size_t smem, cudaStream_t st, const VerifyParams& P) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, P);
}

// Launch of the fused context kernel (verify_context.cuh).  Its variants -- temperature 1 compiled
// out or not (TONE), TVD or JSD bound, top-k thresholds applied or not, greedy decoding -- are compiled in separate
// translation units (verify_context_v*.cu) so that they build in parallel; this function picks one.
// `items` = upper bound of the contexts with children in the call, `sms` = SMs of the device.
cudaError_t launch_context_kernel(const VerifyParams& P, bool bf16, bool uncond, bool tone, bool jsd, bool topk,
                                  bool greedy, long long items, int sms, cudaStream_t st);

}  // namespace lantern
