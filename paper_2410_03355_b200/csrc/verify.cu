// LANTERN relaxed verification step on sm_100a: plan -> fused context pass, which walks and draws as well.
//
// One "context" is a row of logits that has at least one drafted child.  The fused pass (verify_context.cuh) is
// a persistent kernel: bulk asynchronous copies (TMA, completion on an mbarrier) bring a context's target rows
// into shared memory; the rows are read ONCE into registers, guidance-combined, turned into softmax numerators,
// and every child of the context is tested on chip:
//     A_{k,delta}(x~)  : gather of the target numerators at the token's neighbour row and a
//                        prefix scan with the strict bound (Algorithm 2, 2nd block)
//     accept test      : r * p(x~) < sum_A q                     (Section 4.3, final rule)
//     on rejection     : residual [q_{k,delta}(.|D=x~) - p]_+ over all V tokens, its total,
//                        and either the next sibling's test on the renormalised residual or
//                        the inverse-CDF draw of the replacement token   (Section 4.3, Alg. 1)
// Algorithm 1's loop over the decided contexts and the draw of the bonus token happen inside the same pass.
// Greedy decoding runs through the same two kernels.
//
// Precision: processed logits are fp32 (difference, fused multiply-add, division, each
// rounded once); exponentials come from the fp32 ex2 unit (about 3e-7 relative); sums of up to 16 of them are formed in single
// precision, longer sums and every threshold comparison in double precision.  Against 64 bits the normalisers are off by 3.3e-8 (flat rows) to 5e-8 rms.
#include "verify_common.cuh"

#include <stddef.h>

namespace lantern {

// ---------------------------------------------------------------------------------------
// kernel 1: plan.  One warp per sequence: validate tokens / parents / uniforms, bucket the
// nodes by parent context (children in node order), initialise the per-node outputs, and write
// one self-contained work item per context with children.
//
// Work items are laid out so that the fused pass meets a sequence's contexts in the order
// Algorithm 1's loop can reach them: slot r * B + b holds the r-th context with children of
// sequence b in breadth-first order (by depth, then by index).  A context whose parent node has
// already been rejected when its turn comes is never evaluated (see verify_context.cuh); the
// order only decides how often that is known in time, never the result.
// Every context's walk word says whether it is the root (where the walk starts), pending, or a leaf.
// ---------------------------------------------------------------------------------------
constexpr int kPlanArrays = 13;  // per-warp arrays of N + 2 ints in shared memory

// One sequence of more than 64 drafts, by one warp; returns the number of its contexts with children, or its fault bits << 16.
__device__ __forceinline__ int plan_sequence(const VerifyParams& P, int* plan_smem, int b, int warp, int lane) {
  const int N = P.N, R = P.R, B = P.B;
  if (b >= B) return 0;
  int* cnt = plan_smem + warp * kPlanArrays * (R + 1);   // cnt[c]: number of children of context c
  int* cur = cnt + (R + 1);                    // fill cursor, ends as the end offset of context c
  int* dep = cur + (R + 1);                    // depth of context c (root = 0), later its breadth-first rank
  int* lvl = dep + (R + 1);                    // per depth: where its nodes lie in the (depth, index) order
  int* siz = lvl + (R + 1);                    // number of contexts in the subtree of context c, itself included
  int* din = siz + (R + 1);                    // depth-first (pre-order) position of context c
  int* tmp = din + (R + 1);                    // per context: children placed so far; later running sums of sizes
  int* anc = tmp + (R + 1);                    // pointer jumping: an ancestor of node i; later the (depth, index) order
  int* s_par = anc + (R + 1);                  // the sequence's parents, tokens and uniforms, staged once by all
  int* s_tok = s_par + (R + 1);                //   lanes: the serial parts below then run out of shared memory
  int* s_uni = s_tok + (R + 1);
  int* s_pos = s_uni + (R + 1);                // place of node i in the child lists
  int* s_first = s_pos + (R + 1);              // first child (smallest node index) of context c
  for (int i = lane; i <= R; i += 32) cnt[i] = 0, siz[i] = 1, s_first[i] = -1;
  __syncwarp();
  int status = 0;
  const float qnan = __int_as_float(0x7fc00000);
  for (int i = lane; i < N; i += 32) {
    const size_t o = static_cast<size_t>(b) * N + i;
    const int tok = P.tokens[o];
    if (static_cast<unsigned>(tok) >= static_cast<unsigned>(P.V)) status |= LANTERN_ST_BAD_TOKEN;
    const int par = P.parents ? P.parents[o] : i - 1;
    if (par < -1 || par >= i) status |= LANTERN_ST_BAD_PARENT;
    else atomicAdd(&cnt[par + 1], 1);
    s_par[i] = par;
    s_tok[i] = tok;
    if (P.out_path) P.out_path[o] = -1;
    if (P.out_qa) P.out_qa[o] = qnan;
    if (P.out_px) P.out_px[o] = qnan;
    if (P.out_m) P.out_m[o] = -1;
  }
  if (P.uniforms) {   // greedy decoding draws nothing and passes no uniforms
    for (int i = lane; i <= N; i += 32) {
      const float r = P.uniforms[static_cast<size_t>(b) * R + i];
      if (!(r >= 0.0f && r < 1.0f)) status |= LANTERN_ST_BAD_UNIFORM;
      s_uni[i] = __float_as_int(r);
    }
  } else {
    for (int i = lane; i <= N; i += 32) s_uni[i] = 0;
  }
  for (int c = lane; c < R; c += 32) P.dead[static_cast<size_t>(b) * R + c] = 0;
  status = __reduce_or_sync(kFull, status);
  __syncwarp();
  if (lane == 0) {   // what stands if the fused pass never gets to the end of this sequence
    P.out_len[b] = 0;
    P.out_tok[b] = -1;
    if (P.out_status) P.out_status[b] = status ? status : LANTERN_ST_INTERNAL;
  }
  if (status) {   // the walk reports the fault; no work is queued for this sequence
    for (int r = lane; r < N; r += 32) P.work[static_cast<size_t>(r) * B + b].item = -1;
    return status << 16;
  }

  ChildInfo* kids = P.children + static_cast<size_t>(b) * N;
  // Children of each context in node order (cur, s_pos, s_first), subtree sizes and pre-order positions
  // (siz, din: the contexts behind a node then occupy one contiguous range of positions, which is what lets
  // the fused pass strike a whole rejected subtree with a few byte stores), and the breadth-first rank of every
  // context with children (dep).  All of it by the whole warp, 32 nodes at a time.
  int n_ctx = 0;
  const unsigned below = (1u << lane) - 1u;
  if (!P.parents) {
    // a chain: context c has the one child c, lies c deep, and has the R - c contexts from itself on behind it
    for (int c = lane; c < R; c += 32) {
      cur[c] = c < N ? c + 1 : N;
      siz[c] = R - c;
      din[c] = c;
      dep[c] = c;
      if (c < N) s_pos[c] = c, s_first[c] = c;
    }
    n_ctx = N;
  } else {
    // -- child-list offsets: cur[c] = end of the children of context c
    int carry = 0;
    for (int base = 0; base < R; base += 32) {
      const int c = base + lane;
      int incl = c < R ? cnt[c] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (c < R) cur[c] = carry + incl, tmp[c] = 0;
      carry += __shfl_sync(kFull, incl, 31);
    }
    __syncwarp();
    // -- place of every node among its siblings (tmp[c]: children of c placed so far), first child
    for (int base = 0; base < N; base += 32) {
      const int i = base + lane;
      const unsigned act = __ballot_sync(kFull, i < N);
      if (i < N) {
        const int pc = s_par[i] + 1;
        const unsigned peers = __match_any_sync(act, pc);
        const int before = tmp[pc];
        const int rk = before + __popc(peers & below);
        s_pos[i] = cur[pc] - cnt[pc] + rk;
        if (rk == 0) s_first[pc] = i;
        __syncwarp(act);
        if ((peers & below) == 0) tmp[pc] = before + __popc(peers);
      }
      __syncwarp();
    }
    // -- depth of every context by pointer jumping: dep[i + 1] = distance from node i to anc[i] (or to the root)
    for (int i = lane; i < N; i += 32) anc[i] = s_par[i], dep[i + 1] = 1;
    if (lane == 0) dep[0] = 0;
    __syncwarp();
    for (int round = 0; round < 12; ++round) {   // every round at least doubles the distance covered: 2^11 > 1024
      bool more = false;
      for (int base = 0; base < N; base += 32) {
        const int i = base + lane;
        const int a = i < N ? anc[i] : -1;
        int da = 0, aa = -1;
        if (a >= 0) da = dep[a + 1], aa = anc[a];   // a < i: a pair that is consistent whether or not a has moved this round
        __syncwarp();
        if (a >= 0) {
          dep[i + 1] += da;
          anc[i] = aa;
          more |= aa >= 0;
        }
        __syncwarp();
      }
      if (!__any_sync(kFull, more)) break;
    }
    int maxd = 0;
    for (int i = lane; i < N; i += 32) maxd = max(maxd, dep[i + 1]);
    maxd = __reduce_max_sync(kFull, maxd);
    // -- nodes ordered by (depth, index): lvl[d] counts, then is the cursor, and ends as the end of level d
    for (int d = lane; d <= maxd; d += 32) lvl[d] = 0;
    __syncwarp();
    for (int i = lane; i < N; i += 32) atomicAdd(&lvl[dep[i + 1]], 1);
    __syncwarp();
    carry = 0;
    for (int base = 0; base <= maxd; base += 32) {
      const int d = base + lane;
      const int n = d <= maxd ? lvl[d] : 0;
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (d <= maxd) lvl[d] = carry + incl - n;
      carry += __shfl_sync(kFull, incl, 31);
    }
    __syncwarp();
    int* order = anc;   // (the ancestors are no longer needed)
    for (int base = 0; base < N; base += 32) {
      const int i = base + lane;
      const unsigned act = __ballot_sync(kFull, i < N);
      if (i < N) {
        const int d = dep[i + 1];
        const unsigned peers = __match_any_sync(act, d);
        const int before = lvl[d];
        order[before + __popc(peers & below)] = i;
        __syncwarp(act);
        if ((peers & below) == 0) lvl[d] = before + __popc(peers);
      }
      __syncwarp();
    }
    // -- subtree sizes, deepest level first (level d occupies order[lvl[d - 1] .. lvl[d]))
    for (int d = maxd; d >= 1; --d) {
      for (int pos = lvl[d - 1] + lane; pos < lvl[d]; pos += 32) {
        const int i = order[pos];
        atomicAdd(&siz[s_par[i] + 1], siz[i + 1]);
      }
      __syncwarp();
    }
    // -- sizes in child-list order and their running sum: tmp[pos] = sizes of everything placed before pos
    for (int i = lane; i < N; i += 32) tmp[s_pos[i]] = siz[i + 1];
    __syncwarp();
    carry = 0;
    for (int base = 0; base < N; base += 32) {
      const int pos = base + lane;
      const int n = pos < N ? tmp[pos] : 0;
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (pos < N) tmp[pos] = carry + incl - n;
      carry += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) din[0] = 0;
    __syncwarp();
    // -- pre-order positions, top level first: after the parent come the subtrees of the earlier siblings
    for (int d = 1; d <= maxd; ++d) {
      for (int pos = lvl[d - 1] + lane; pos < lvl[d]; pos += 32) {
        const int i = order[pos];
        const int pc = s_par[i] + 1;
        din[i + 1] = din[pc] + 1 + tmp[s_pos[i]] - tmp[cur[pc] - cnt[pc]];
      }
      __syncwarp();
    }
    // -- breadth-first rank of the contexts with children: the root, then the nodes by (depth, index)
    n_ctx = cnt[0] > 0 ? 1 : 0;
    for (int base = 0; base < N; base += 32) {
      const int pos = base + lane;
      const int i = pos < N ? order[pos] : 0;
      const bool has = pos < N && cnt[i + 1] > 0;
      const unsigned bal = __ballot_sync(kFull, has);
      if (has) dep[i + 1] = n_ctx + __popc(bal & below);   // the depth is no longer needed: dep[c] becomes the rank
      n_ctx += __popc(bal);
    }
  }
  __syncwarp();         // the shared arrays are complete
  for (int i = lane; i < N; i += 32) {   // the child lists, written by all lanes
    ChildInfo ci = {i, s_tok[i], __int_as_float(s_uni[i]), (din[i + 1] << 16) | siz[i + 1]};
    kids[s_pos[i]] = ci;
  }
  for (int r = n_ctx + lane; r < N; r += 32) P.work[static_cast<size_t>(r) * B + b].item = -1;
  const float u_final = __int_as_float(s_uni[N]);
  for (int c = lane; c < R; c += 32) {
    const int n = cnt[c];
    P.records[static_cast<size_t>(b) * R + c].word = n == 0 ? kWalkLeaf : (c == 0 ? kWalkWaiting : kWalkPending);
    if (n > 0) {
      const int start = cur[c] - n;
      const int f = s_first[c];             // the context's first child (smallest node index)
      P.work[dep[c] * B + b] = {b * R + c, b * N + start, (n << 16) | f, (din[f + 1] << 16) | siz[f + 1], s_tok[f],
                                __int_as_float(s_uni[f]), u_final, b * R + din[c]};
    }
  }
  return n_ctx;
}

// The same for at most 64 drafts, two per lane: sets of nodes are 64-bit masks, so that a context's children, a node's
// ancestors (by doubling) and the contexts of a level are one word each, and the rest are sums over the bits of a word.
// A 60-node tree takes 2 us here; the general path above, with its level-by-level passes, 9 us.
constexpr int PLAN_SMALL = 64;
struct SmallPlan {
  unsigned long long kids[PLAN_SMALL + 1];    // children of context c
  unsigned long long level[PLAN_SMALL + 1];   // nodes of depth d that have children
  unsigned long long anc[PLAN_SMALL];         // ancestors of node i
  int jump[PLAN_SMALL];                       // doubling: the farthest ancestor in anc so far, -1 = none beyond it
  int size[PLAN_SMALL + 1];                   // contexts in the subtree of context c, itself included
  int weight[PLAN_SMALL];                     // steps in pre-order from a node's parent to the node
  int start[PLAN_SMALL + 1];                  // where the children of context c begin in the child lists
  int rank[PLAN_SMALL + 1], span[PLAN_SMALL + 1], tok[PLAN_SMALL];
  float uni[PLAN_SMALL];
};

__device__ __forceinline__ int plan_small(const VerifyParams& P, SmallPlan& S, int b, int lane) {
  const int N = P.N, R = P.R, B = P.B;
  if (b >= B) return 0;
  int par[2], tok[2] = {0, 0};
  float uni[2] = {0.0f, 0.0f}, u_final = 0.0f;
  // all inputs at once
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    const size_t o = static_cast<size_t>(b) * N + i;
    par[q] = i - 1;
    if (i < N) {
      tok[q] = P.tokens[o];
      if (P.parents) par[q] = P.parents[o];
      if (P.uniforms) uni[q] = P.uniforms[static_cast<size_t>(b) * R + i];
    }
  }
  if (P.uniforms) u_final = P.uniforms[static_cast<size_t>(b) * R + N];
  for (int c = lane; c <= PLAN_SMALL; c += 32) S.kids[c] = S.level[c] = 0ull, S.size[c] = 1;
  for (int c = lane; c < R; c += 32) P.dead[static_cast<size_t>(b) * R + c] = 0;
  const float qnan = __int_as_float(0x7fc00000);
  int status = u_final >= 0.0f && u_final < 1.0f ? 0 : LANTERN_ST_BAD_UNIFORM;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    const size_t o = static_cast<size_t>(b) * N + i;
    if (i < N) {
      if (static_cast<unsigned>(tok[q]) >= static_cast<unsigned>(P.V)) status |= LANTERN_ST_BAD_TOKEN;
      if (par[q] < -1 || par[q] >= i) status |= LANTERN_ST_BAD_PARENT;
      if (!(uni[q] >= 0.0f && uni[q] < 1.0f)) status |= LANTERN_ST_BAD_UNIFORM;
      if (P.out_path) P.out_path[o] = -1;
      if (P.out_qa) P.out_qa[o] = qnan;
      if (P.out_px) P.out_px[o] = qnan;
      if (P.out_m) P.out_m[o] = -1;
    }
  }
  status = __reduce_or_sync(kFull, status);
  if (lane == 0) {   // what stands if the fused pass never gets to the end of this sequence
    P.out_len[b] = 0;
    P.out_tok[b] = -1;
    if (P.out_status) P.out_status[b] = status ? status : LANTERN_ST_INTERNAL;
  }
  if (status) {   // no work is queued for this sequence
    for (int r = lane; r < max(N, 1); r += 32) P.work[static_cast<size_t>(r) * B + b].item = -1;
    return status << 16;
  }
  if (N == 0) {   // no drafts: one draw from the root's q
    if (lane == 0) {
      P.records[b].word = kWalkLeaf;
      P.work[b] = {b, 0, 0, 0, 0, 0.0f, u_final, b};
    }
    return 1;
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    if (i < N) {
      atomicOr(&S.kids[par[q] + 1], 1ull << i);
      S.anc[i] = par[q] >= 0 ? 1ull << par[q] : 0ull;
      S.jump[i] = par[q];
      S.tok[i] = tok[q];
      S.uni[i] = uni[q];
    }
  }
  __syncwarp();
  for (;;) {
    unsigned long long more_anc[2];
    int to[2];
    bool more = false;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q;
      const int a = i < N ? S.jump[i] : -1;
      to[q] = a >= 0 ? S.jump[a] : -1;
      more_anc[q] = a >= 0 ? S.anc[a] : 0ull;
      more |= to[q] >= 0;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = lane + 32 * q;
      if (i < N) S.anc[i] |= more_anc[q], S.jump[i] = to[q];
    }
    __syncwarp();
    if (!__any_sync(kFull, more)) break;
  }
  unsigned long long anc[2], below[2], with[2];   // ancestors, smaller nodes, earlier siblings
  int depth[2], kids[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    const bool on = i < N;
    anc[q] = on ? S.anc[i] : 0ull;
    below[q] = (1ull << i) - 1ull;
    with[q] = on ? S.kids[par[q] + 1] & below[q] : 0ull;
    depth[q] = __popcll(anc[q]) + 1;
    kids[q] = on ? __popcll(S.kids[i + 1]) : 0;
    if (kids[q]) atomicOr(&S.level[depth[q]], 1ull << i);
    for (unsigned long long m = anc[q]; m; m &= m - 1ull) atomicAdd(&S.size[__ffsll(m)], 1);   // (context of node a: a + 1)
  }
  if (lane == 0) S.size[0] = R;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    int w = 1;
    for (unsigned long long m = with[q]; m; m &= m - 1ull) w += S.size[__ffsll(m)];
    if (i < N) S.weight[i] = w;
  }
  // child lists in the order of the contexts
  const int n_root = __popcll(S.kids[0]);
  int carry = n_root, n_ctx = 1;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    int incl = kids[q];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += t;
    }
    if (i < N) S.start[i + 1] = carry + incl - kids[q];
    carry += __shfl_sync(kFull, incl, 31);
    n_ctx += __popc(__ballot_sync(kFull, kids[q] > 0));
  }
  if (lane == 0) S.start[0] = 0, S.rank[0] = 0, S.span[0] = R;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    if (i < N) {
      int pos = S.weight[i], rank = 1;                   // pre-order position; breadth-first rank, where it has children
      for (unsigned long long m = anc[q]; m; m &= m - 1ull) pos += S.weight[__ffsll(m) - 1];
      for (int d = 1; d < depth[q]; ++d) rank += __popcll(S.level[d]);
      S.rank[i + 1] = rank + __popcll(S.level[depth[q]] & below[q]);
      S.span[i + 1] = pos << 16 | S.size[i + 1];
      const ChildInfo info = {i, tok[q], uni[q], pos << 16 | S.size[i + 1]};
      P.children[static_cast<size_t>(b) * N + S.start[par[q] + 1] + __popcll(with[q])] = info;
    }
  }
  __syncwarp();
  for (int r = n_ctx + lane; r < N; r += 32) P.work[static_cast<size_t>(r) * B + b].item = -1;
  for (int c = lane; c < R; c += 32) {
    const unsigned long long m = S.kids[c];
    P.records[static_cast<size_t>(b) * R + c].word = m == 0ull ? kWalkLeaf : (c == 0 ? kWalkWaiting : kWalkPending);
    if (m) {
      const int f = __ffsll(m) - 1;                      // its first child
      P.work[static_cast<size_t>(S.rank[c]) * B + b] = {b * R + c, b * N + S.start[c], __popcll(m) << 16 | f, S.span[f + 1], S.tok[f],
                                                        S.uni[f], u_final, b * R + (S.span[c] >> 16)};
    }
  }
  return n_ctx;
}

__global__ void __launch_bounds__(PLAN_WARPS * 32) lantern_plan_kernel(VerifyParams P) {
  extern __shared__ int plan_smem[];
  __shared__ int s_words[PLAN_WARPS];
  __shared__ SmallPlan s_small[PLAN_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_dependency_wait();
  grid_dependents_launch();
  if (blockIdx.x == 0 && threadIdx.x < 64) reinterpret_cast<int*>(P.counters)[threadIdx.x] = 0;
  const int b = blockIdx.x * PLAN_WARPS + warp;
  const int word = P.N <= PLAN_SMALL ? plan_small(P, s_small[warp], b, lane) : plan_sequence(P, plan_smem, b, warp, lane);
  if (lane == 0) s_words[warp] = word;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ranks = 0, bits = 0;
    for (int w = 0; w < PLAN_WARPS; ++w) ranks = max(ranks, s_words[w] & 0xffff), bits |= s_words[w] >> 16;
    P.block_words[blockIdx.x] = bits << 16 | ranks;
  }
}

}  // namespace lantern

// (kernel 2, the fused context pass, is compiled in files of its own: see verify_common.cuh)
namespace lantern {

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct WsLayout {
  size_t counters, work, children, records, dead, words, total;
};

static WsLayout ws_layout(int B, int N, bool topk = false) {
  const size_t R = static_cast<size_t>(N) + 1, b = static_cast<size_t>(B);
  const size_t n1 = N > 0 ? N : 1;
  WsLayout L;
  size_t o = 0;
  L.counters = o; o += 256;
  L.work = o;     o += align_up(b * n1 * sizeof(WorkItem), 256);
  o += align_up(b * n1 * 4, 256);              // (the size callers have always been told: parts of it are no longer used)
  L.children = o; o += align_up(b * n1 * sizeof(ChildInfo), 256);
  L.records = o;  o += align_up(b * R * sizeof(Record), 256);
  L.dead = o;     o += align_up(b * R, 256);
  L.words = o;    o += 3 * align_up(b * 4, 256);
  o += topk ? 2 * align_up(b * R * 4, 256) : 0;
  L.total = o;
  return L;
}

// SMs of the current device (asked for once per device: it does not change), 0 if there is none
static int sm_count() {
  static std::atomic<int> known[64];
  int dev = -1, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
  if (dev < 64 && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (dev < 64) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

static thread_local cudaEvent_t g_ev_before = nullptr, g_ev_after = nullptr;

// limit of the kernels' bounded waits and the self-test's withheld context (lantern_debug_wait_test)
constexpr uint32_t kDefaultWaitTries = 1u << 21;
static thread_local uint32_t g_wait_tries = kDefaultWaitTries;
static thread_local int g_withhold_item = -1;

// the variants of the fused context kernel live in verify_context_v<tone + 2 jsd + 4 topk>.cu, those of greedy decoding in
// verify_context_v<8 + jsd + 2 topk>.cu
#define LANTERN_DECLARE_VARIANT(n) \
  cudaError_t launch_context_v##n(const VerifyParams&, bool, bool, long long, int, cudaStream_t);
LANTERN_DECLARE_VARIANT(0) LANTERN_DECLARE_VARIANT(1) LANTERN_DECLARE_VARIANT(2) LANTERN_DECLARE_VARIANT(3)
LANTERN_DECLARE_VARIANT(4) LANTERN_DECLARE_VARIANT(5) LANTERN_DECLARE_VARIANT(6) LANTERN_DECLARE_VARIANT(7)
LANTERN_DECLARE_VARIANT(8) LANTERN_DECLARE_VARIANT(9) LANTERN_DECLARE_VARIANT(10) LANTERN_DECLARE_VARIANT(11)
#undef LANTERN_DECLARE_VARIANT

cudaError_t launch_context_kernel(const VerifyParams& P, bool bf16, bool uncond, bool tone, bool jsd, bool topk,
                                  bool greedy, long long items, int sms, cudaStream_t st) {
  switch (greedy ? 8 | (jsd ? 1 : 0) | (topk ? 2 : 0) : (tone ? 1 : 0) | (jsd ? 2 : 0) | (topk ? 4 : 0)) {
    case 0: return launch_context_v0(P, bf16, uncond, items, sms, st);
    case 1: return launch_context_v1(P, bf16, uncond, items, sms, st);
    case 2: return launch_context_v2(P, bf16, uncond, items, sms, st);
    case 3: return launch_context_v3(P, bf16, uncond, items, sms, st);
    case 4: return launch_context_v4(P, bf16, uncond, items, sms, st);
    case 5: return launch_context_v5(P, bf16, uncond, items, sms, st);
    case 6: return launch_context_v6(P, bf16, uncond, items, sms, st);
    case 7: return launch_context_v7(P, bf16, uncond, items, sms, st);
    case 8: return launch_context_v8(P, bf16, uncond, items, sms, st);
    case 9: return launch_context_v9(P, bf16, uncond, items, sms, st);
    case 10: return launch_context_v10(P, bf16, uncond, items, sms, st);
    default: return launch_context_v11(P, bf16, uncond, items, sms, st);
  }
}

}  // namespace lantern

using namespace lantern;

static bool shape_ok(int B, int N, int V, int k, int dtype) {
  if (dtype != LANTERN_F32 && dtype != LANTERN_BF16) return false;
  if (B < 0 || N < 0 || N > MAX_N || V < 8 || V > 16384 || (V % 8) != 0 || k < 1 || k > V) return false;
  return static_cast<long long>(B) * (N + 1) < (1ll << 31);
}

extern "C" size_t lantern_verify_workspace_bytes(int B, int N, int V, int k, int dtype) {
  if (!shape_ok(B, N, V, k, dtype)) return 0;
  return ws_layout(B > 0 ? B : 1, N).total;
}

extern "C" int lantern_verify_launch_count(int greedy, int top_k_active) {
  // (at most: a call is a plan and the fused pass, which does everything else itself)
  (void)greedy;
  return 5 + (top_k_active ? 1 : 0);
}

extern "C" lantern_status lantern_last_status(const void* workspace, void* cuda_stream, int32_t* out_bits) {
  if (!workspace) return LANTERN_E_NULL;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int32_t bits = 0;
  const unsigned char* c = static_cast<const unsigned char*>(workspace) + offsetof(Counters, status_or);
  if (cudaMemcpyAsync(&bits, c, sizeof(bits), cudaMemcpyDeviceToHost, st) != cudaSuccess) return LANTERN_E_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return LANTERN_E_CUDA;
  if (out_bits) *out_bits = bits;
  return bits ? LANTERN_E_DATA : LANTERN_OK;
}

extern "C" lantern_status lantern_verify_counts(const void* workspace, void* cuda_stream, int64_t* out_counts) {
  if (!workspace || !out_counts) return LANTERN_E_NULL;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Counters c;
  if (cudaMemcpyAsync(&c, workspace, sizeof(c), cudaMemcpyDeviceToHost, st) != cudaSuccess) return LANTERN_E_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return LANTERN_E_CUDA;
  out_counts[0] = static_cast<int64_t>(c.n_evaluated) + c.n_skipped;   // every context with children is either evaluated or left out
  out_counts[1] = c.n_evaluated;
  out_counts[2] = c.n_skipped;
  out_counts[3] = c.n_bonus;
  out_counts[4] = c.n_tested;
  out_counts[5] = c.n_slow_topk;
  return LANTERN_OK;
}

extern "C" lantern_status lantern_debug_wait_test(int max_tries, int withhold_context) {
  if (max_tries < 0) return LANTERN_E_PARAM;
  g_wait_tries = max_tries == 0 ? kDefaultWaitTries : static_cast<uint32_t>(max_tries);
  g_withhold_item = withhold_context;
  return LANTERN_OK;
}

extern "C" int lantern_kernel_revision(void) { return LANTERN_CONTEXT_KERNEL_REVISION; }

extern "C" lantern_status lantern_verify_profile_events(void* before_fused, void* after_fused) {
  if ((before_fused == nullptr) != (after_fused == nullptr)) return LANTERN_E_NULL;
  g_ev_before = static_cast<cudaEvent_t>(before_fused);
  g_ev_after = static_cast<cudaEvent_t>(after_fused);
  return LANTERN_OK;
}

static lantern_status verify_impl(const void* target_logits, const void* draft_logits, int dtype, float cfg_scale,
                                  int has_uncond, float T, const int32_t* draft_tokens, const int32_t* tree_parents,
                                  const int32_t* neighbor_idx, int k, float delta, int divergence, int top_k,
                                  const float* uniforms, int B, int N, int V, int32_t* out_accept_len,
                                  int32_t* out_next_token, int32_t* out_accept_path, int32_t* out_status,
                                  float* out_node_qa, float* out_node_px, int32_t* out_node_m, void* workspace,
                                  size_t workspace_bytes, void* cuda_stream);

extern "C" lantern_status lantern_verify(const void* target_logits, const void* draft_logits, int dtype,
                                         float cfg_scale, int has_uncond, float T, const int32_t* draft_tokens,
                                         const int32_t* tree_parents, const int32_t* neighbor_idx, int k,
                                         float delta, const float* uniforms, int B, int N, int V,
                                         int32_t* out_accept_len, int32_t* out_next_token,
                                         int32_t* out_accept_path, int32_t* out_status, float* out_node_qa,
                                         float* out_node_px, int32_t* out_node_m, void* workspace,
                                         size_t workspace_bytes, void* cuda_stream) {
  return lantern_verify_ex(target_logits, draft_logits, dtype, cfg_scale, has_uncond, T, draft_tokens, tree_parents,
                           neighbor_idx, k, delta, LANTERN_DIV_TVD, 0, uniforms, B, N, V, out_accept_len,
                           out_next_token, out_accept_path, out_status, out_node_qa, out_node_px, out_node_m,
                           workspace, workspace_bytes, cuda_stream);
}

extern "C" size_t lantern_verify_workspace_bytes_ex(int B, int N, int V, int k, int dtype, int top_k) {
  if (!shape_ok(B, N, V, k, dtype) || top_k < 0) return 0;
  return ws_layout(B > 0 ? B : 1, N, top_k > 0).total;
}

extern "C" lantern_status lantern_verify_ex(const void* target_logits, const void* draft_logits, int dtype,
                                         float cfg_scale, int has_uncond, float T, const int32_t* draft_tokens,
                                         const int32_t* tree_parents, const int32_t* neighbor_idx, int k,
                                         float delta, int divergence, int top_k, const float* uniforms, int B,
                                         int N, int V, int32_t* out_accept_len, int32_t* out_next_token,
                                         int32_t* out_accept_path, int32_t* out_status, float* out_node_qa,
                                         float* out_node_px, int32_t* out_node_m, void* workspace,
                                         size_t workspace_bytes, void* cuda_stream) {
  if (divergence != LANTERN_DIV_TVD && divergence != LANTERN_DIV_JSD) return LANTERN_E_PARAM;
  if (top_k < 0) return LANTERN_E_PARAM;
  return verify_impl(target_logits, draft_logits, dtype, cfg_scale, has_uncond, T, draft_tokens, tree_parents,
                     neighbor_idx, k, delta, divergence, top_k, uniforms, B, N, V, out_accept_len, out_next_token,
                     out_accept_path, out_status, out_node_qa, out_node_px, out_node_m, workspace,
                     workspace_bytes, cuda_stream);
}

static lantern_status verify_impl(const void* target_logits, const void* draft_logits, int dtype,
                                         float cfg_scale, int has_uncond, float T, const int32_t* draft_tokens,
                                         const int32_t* tree_parents, const int32_t* neighbor_idx, int k,
                                         float delta, int divergence, int top_k, const float* uniforms, int B, int N, int V,
                                         int32_t* out_accept_len, int32_t* out_next_token,
                                         int32_t* out_accept_path, int32_t* out_status, float* out_node_qa,
                                         float* out_node_px, int32_t* out_node_m, void* workspace,
                                         size_t workspace_bytes, void* cuda_stream) {
  if (dtype != LANTERN_F32 && dtype != LANTERN_BF16) return LANTERN_E_PARAM;
  if (B < 0 || N < 0 || N > MAX_N || V < 8 || V > 16384 || (V % 8) != 0 || k < 1 || k > V) return LANTERN_E_SHAPE;
  if (static_cast<long long>(B) * (N + 1) >= (1ll << 31)) return LANTERN_E_SHAPE;
  if (!(T >= 0.0f) || !(delta >= 0.0f) || !isfinite(T) || !isfinite(delta)) return LANTERN_E_PARAM;
  if (has_uncond && !isfinite(cfg_scale)) return LANTERN_E_PARAM;
  const bool greedy = T == 0.0f;   // Section 4.3, last sentence: no drafter distribution, no random numbers
  // sampling keeps a context's numerators (4 bytes per token) and rows on chip: fp32 rows only up to 8192 tokens
  if (!greedy && dtype == LANTERN_F32 && V > 8192) return LANTERN_E_SHAPE;
  if (B == 0) return LANTERN_OK;
  if (!target_logits || !neighbor_idx || !out_accept_len || !out_next_token) return LANTERN_E_NULL;
  if (!greedy && !uniforms) return LANTERN_E_NULL;
  if (N > 0 && (!draft_tokens || (!greedy && !draft_logits))) return LANTERN_E_NULL;
  if ((reinterpret_cast<uintptr_t>(target_logits) & 15) || (reinterpret_cast<uintptr_t>(draft_logits) & 15))
    return LANTERN_E_ALIGN;
  const bool topk = top_k > 0 && top_k < V;   // top_k >= V keeps every logit
  const WsLayout L = ws_layout(B, N, top_k > 0);
  if (!workspace || workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return LANTERN_E_WORKSPACE;

  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  VerifyParams P;
  P.target = target_logits;
  P.draft = draft_logits;
  P.tokens = draft_tokens;
  P.parents = tree_parents;
  P.nbr = neighbor_idx;
  P.uniforms = greedy ? nullptr : uniforms;
  P.out_len = out_accept_len;
  P.out_tok = out_next_token;
  P.out_path = out_accept_path;
  P.out_status = out_status;
  P.out_qa = out_node_qa;
  P.out_px = out_node_px;
  P.out_m = out_node_m;
  P.counters = reinterpret_cast<Counters*>(ws + L.counters);
  P.work = reinterpret_cast<WorkItem*>(ws + L.work);
  P.children = reinterpret_cast<ChildInfo*>(ws + L.children);
  P.records = reinterpret_cast<Record*>(ws + L.records);
  P.block_words = reinterpret_cast<int32_t*>(ws + L.words);
  P.B = B;
  P.N = N;
  P.R = N + 1;
  P.V = V;
  P.k = k;
  P.cfg_scale = cfg_scale;
  P.T = T;
  P.delta = delta;
  P.divergence = divergence;
  P.top_k = topk ? top_k : 0;
  P.dead = ws + L.dead;
  P.wait_tries = g_wait_tries;
  P.withhold_item = g_withhold_item;

  const int sms = sm_count();
  if (sms < 1) return LANTERN_E_CUDA;

  const size_t plan_smem = N <= PLAN_SMALL ? 0 : static_cast<size_t>(PLAN_WARPS) * kPlanArrays * (N + 2) * sizeof(int);
  static DeviceFlags plan_ready;
  if (plan_smem > 32 * 1024 &&   // (beside the kernel's static part)
      allow_shared_memory(lantern_plan_kernel, PLAN_WARPS * kPlanArrays * (MAX_N + 2) * sizeof(int), plan_ready) != cudaSuccess)
    return LANTERN_E_CUDA;
  if (launch_dependent(lantern_plan_kernel, (B + PLAN_WARPS - 1) / PLAN_WARPS, PLAN_WARPS * 32, plan_smem, st, P) != cudaSuccess)
    return LANTERN_E_CUDA;

  const long long items = static_cast<long long>(B) * (N > 0 ? N : 1);   // upper bound of contexts with children
  // every combination of the compile-time variants exists: T = 1 never meets the division code
  if (g_ev_before && g_ev_after) cudaEventRecord(g_ev_before, st);
  const cudaError_t e = launch_context_kernel(P, dtype == LANTERN_BF16, has_uncond != 0, T == 1.0f, divergence == LANTERN_DIV_JSD,
                                              topk, greedy, items, sms, st);
  if (g_ev_before && g_ev_after) cudaEventRecord(g_ev_after, st);
  return e == cudaSuccess ? LANTERN_OK : LANTERN_E_CUDA;
}

// ---------------------------------------------------------------------------------------
// lantern_verify_static: same computation, scratch taken from a fixed array in the device
// image instead of a caller workspace (for callers that must not allocate device memory).
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_workspace[LANTERN_STATIC_WORKSPACE_BYTES];

// In host code `g_static_workspace` is only a handle for the symbol, never an address a kernel
// could use; the device address is asked for once per device and remembered here.
static void* g_static_workspace_ptr[64] = {};

static lantern_status static_workspace_address(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return LANTERN_E_CUDA;
  if (dev >= 64) return LANTERN_E_SHAPE;   // the table of addresses below serves ordinals 0..63
  void* p = __atomic_load_n(&g_static_workspace_ptr[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    if (cudaGetSymbolAddress(&p, g_static_workspace) != cudaSuccess || !p) return LANTERN_E_CUDA;
    __atomic_store_n(&g_static_workspace_ptr[dev], p, __ATOMIC_RELEASE);   // same value whoever wins
  }
  *out = p;
  return LANTERN_OK;
}

extern "C" lantern_status lantern_verify_static(const void* target_logits, const void* draft_logits, int dtype,
                                                float cfg_scale, int has_uncond, float T,
                                                const int32_t* draft_tokens, const int32_t* tree_parents,
                                                const int32_t* neighbor_idx, int k, float delta,
                                                const float* uniforms, int B, int N, int V,
                                                int32_t* out_accept_len, int32_t* out_next_token,
                                                int32_t* out_accept_path, int32_t* out_status, float* out_node_qa,
                                                float* out_node_px, int32_t* out_node_m, void* cuda_stream) {
  if (B < 0 || N < 0 || N > MAX_N) return LANTERN_E_SHAPE;
  // the fixed array bounds the call size: refuse anything whose scratch would not fit
  if (B > 0 && ws_layout(B, N).total > static_cast<size_t>(LANTERN_STATIC_WORKSPACE_BYTES)) return LANTERN_E_WORKSPACE;
  void* ws = nullptr;
  const lantern_status rc = static_workspace_address(&ws);
  if (rc != LANTERN_OK) return rc;
  // The plan kernel resets what the call relies on (counters, marks, words), so whatever the previous call left in the array
  // does not matter.
  return lantern_verify(target_logits, draft_logits, dtype, cfg_scale, has_uncond, T, draft_tokens, tree_parents,
                        neighbor_idx, k, delta, uniforms, B, N, V, out_accept_len, out_next_token, out_accept_path,
                        out_status, out_node_qa, out_node_px, out_node_m, ws, LANTERN_STATIC_WORKSPACE_BYTES,
                        cuda_stream);
}

extern "C" const char* lantern_status_string(lantern_status s) {
  switch (s) {
    case LANTERN_OK: return "ok";
    case LANTERN_E_NULL: return "a required pointer is NULL";
    case LANTERN_E_SHAPE: return "a size is outside the supported range";
    case LANTERN_E_PARAM: return "a scalar parameter is invalid";
    case LANTERN_E_WORKSPACE: return "workspace missing, too small or misaligned";
    case LANTERN_E_CUDA: return "a CUDA runtime call failed";
    case LANTERN_E_DATA: return "a fault in the data was found on the device (see out_status)";
    case LANTERN_E_ALIGN: return "a pointer is not 16-byte aligned";
    case LANTERN_E_UNIMPLEMENTED: return "not implemented in this build";
    default: return "unknown status";
  }
}
