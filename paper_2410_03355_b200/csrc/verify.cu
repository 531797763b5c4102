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
#include <string.h>

namespace lantern {

// ---------------------------------------------------------------------------------------
// kernel 1: plan.  One warp per sequence, two for a tree of at most 64 drafts: validate tokens / parents / uniforms, bucket the
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

// A tree of more than 64 drafts, by one warp; returns its plan_word.
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
    const int par = P.parents[o];
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
    for (int r = lane; r < N; r += 32) {
      P.work[static_cast<size_t>(r) * B + b].item = -1;
      if (P.leaves) P.leaves[static_cast<size_t>(r) * B + b] = -1;
    }
    return plan_word(0, 0, status);
  }

  ChildInfo* kids = P.children + static_cast<size_t>(b) * N;
  // Children of each context in node order (cur, s_pos, s_first), subtree sizes and pre-order positions
  // (siz, din: the contexts behind a node then occupy one contiguous range of positions, which is what lets
  // the fused pass strike a whole rejected subtree with a few byte stores), and the breadth-first rank of every
  // context with children (dep).  All of it by the whole warp, 32 nodes at a time.
  int n_ctx = 0;
  const unsigned below = (1u << lane) - 1u;
  {
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
  if (P.leaves) {   // the contexts without children, by number
    int n = 0;
    for (int base = 0; base < R; base += 32) {
      const int c = base + lane;
      const bool leaf = c < R && cnt[c] == 0;
      const unsigned bal = __ballot_sync(kFull, leaf);
      if (leaf) P.leaves[static_cast<size_t>(n + __popc(bal & below)) * B + b] = din[c] << 16 | c;
      n += __popc(bal);
    }
    for (int r = n + lane; r < N; r += 32) P.leaves[static_cast<size_t>(r) * B + b] = -1;
  }
  return plan_word(n_ctx, R - n_ctx, 0);
}

// The faults of one draft's inputs, and what stands in its outputs until the fused pass has tested it.
__device__ __forceinline__ int plan_node(const VerifyParams& P, int b, int i, int& tok, float& uni) {
  const size_t o = static_cast<size_t>(b) * P.N + i;
  tok = P.tokens[o];
  uni = P.uniforms ? P.uniforms[static_cast<size_t>(b) * P.R + i] : 0.0f;   // (greedy decoding draws nothing and passes no uniforms)
  const float qnan = __int_as_float(0x7fc00000);
  if (P.out_path) P.out_path[o] = -1;
  if (P.out_qa) P.out_qa[o] = qnan;
  if (P.out_px) P.out_px[o] = qnan;
  if (P.out_m) P.out_m[o] = -1;
  return (static_cast<unsigned>(tok) < static_cast<unsigned>(P.V) ? 0 : LANTERN_ST_BAD_TOKEN) | (uni >= 0.0f && uni < 1.0f ? 0 : LANTERN_ST_BAD_UNIFORM);
}
__device__ __forceinline__ float plan_final(const VerifyParams& P, int b, int& status) {
  const float u = P.uniforms ? P.uniforms[static_cast<size_t>(b) * P.R + P.N] : 0.0f;
  if (!(u >= 0.0f && u < 1.0f)) status |= LANTERN_ST_BAD_UNIFORM;
  return u;
}
// what stands for the sequence if the fused pass never gets to its end
__device__ __forceinline__ void plan_outcome(const VerifyParams& P, int b, int status) {
  P.out_len[b] = 0;
  P.out_tok[b] = -1;
  if (P.out_status) P.out_status[b] = status ? status : LANTERN_ST_INTERNAL;
}
// no work is queued for a sequence with a fault
__device__ __forceinline__ int plan_fault(const VerifyParams& P, int b, int from, int stride, int status) {
  for (int r = from; r < max(P.N, 1); r += stride) {
    P.work[static_cast<size_t>(r) * P.B + b].item = -1;
    if (P.leaves) P.leaves[static_cast<size_t>(r) * P.B + b] = -1;
  }
  return plan_word(0, 0, status);
}

// A chain, by one warp: context c has the one child c, lies c deep, and has the R - c contexts from itself on behind it.  Nothing has to be
// worked out, so that the time is that of the loads and the stores (8192 chains of 7: 4.8 us through the code for trees).
__device__ __forceinline__ int plan_chain(const VerifyParams& P, int b, int lane) {
  const int N = P.N, R = P.R, B = P.B;
  if (b >= B) return 0;
  int status = 0, tok = 0, first_tok = 0;
  float uni = 0.0f, first_uni = 0.0f;
  const float u_final = plan_final(P, b, status);
  for (int c = lane; c < R; c += 32) {
    if (c < N) status |= plan_node(P, b, c, tok, uni);
    if (c == lane) first_tok = tok, first_uni = uni;
    P.dead[static_cast<size_t>(b) * R + c] = 0;
  }
  status = __reduce_or_sync(kFull, status);
  if (lane == 0) plan_outcome(P, b, status);
  if (status) return plan_fault(P, b, lane, 32, status);
  for (int c = lane; c < R; c += 32) {
    tok = first_tok, uni = first_uni;
    if (c != lane && c < N) {   // (from the second 32 on: read again)
      tok = P.tokens[static_cast<size_t>(b) * N + c];
      uni = P.uniforms ? P.uniforms[static_cast<size_t>(b) * R + c] : 0.0f;
    }
    const int span = (c + 1) << 16 | (N - c);
    P.records[static_cast<size_t>(b) * R + c].word = c == N ? kWalkLeaf : (c == 0 ? kWalkWaiting : kWalkPending);
    if (c < N) {
      P.children[static_cast<size_t>(b) * N + c] = {c, tok, uni, span};
      P.work[static_cast<size_t>(c) * B + b] = {b * R + c, b * N + c, 1 << 16 | c, span, tok, uni, u_final, b * R + c};
    } else if (N == 0) {        // no drafts: one draw from the root's q
      P.work[b] = {b * R, 0, 0, 0, 0, 0.0f, u_final, b * R};
    }
    if (P.leaves && c < N) P.leaves[static_cast<size_t>(c) * B + b] = c == 0 ? N << 16 | N : -1;
  }
  return N > 0 ? plan_word(N, 1, 0) : plan_word(1, 0, 0);
}

// A tree of at most 64 drafts, by two warps, a draft per thread: sets of nodes are 64-bit masks, and what else is needed is summed up on
// the way from a node to the root (paths are short where a tree is wide).  By one warp with two drafts per lane, and the ancestors by
// doubling, a 60-node tree took 6.4 us here, of which 1 us is the inputs' way.
constexpr int PLAN_SMALL = 64;
struct alignas(8) SmallPlan {
  unsigned kids[PLAN_SMALL + 1][2];    // children of context c
  unsigned level[PLAN_SMALL + 1][2];   // nodes of depth d that have children
  unsigned parents[2];                 // nodes that have children
  int size[PLAN_SMALL + 1];            // contexts behind context c
  int par[PLAN_SMALL], weight[PLAN_SMALL];   // parent; steps in pre-order from the parent to the node
  int start[PLAN_SMALL + 1];           // where the children of context c begin in the child lists
  int rank[PLAN_SMALL + 1], span[PLAN_SMALL + 1], tok[PLAN_SMALL];
  float uni[PLAN_SMALL];
  int status, placed;
};

__device__ __forceinline__ int plan_small(const VerifyParams& P, SmallPlan& S, int b, int seq, int t) {
  const int N = P.N, R = P.R, B = P.B;
  if (b >= B) return 0;
  auto sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + seq) : "memory"); };
  auto kids_of = [&](int c) { return *reinterpret_cast<const unsigned long long*>(S.kids[c]); };
  auto level_at = [&](int d) { return *reinterpret_cast<const unsigned long long*>(S.level[d]); };
  const bool on = t < N;
  int status = 0, par = -1, tok = 0;
  float uni = 0.0f;
  if (on) {
    par = P.parents[static_cast<size_t>(b) * N + t];
    status = plan_node(P, b, t, tok, uni);
    if (par < -1 || par >= t) status |= LANTERN_ST_BAD_PARENT;
  }
  const float u_final = plan_final(P, b, status);
  for (int c = t; c < R; c += 64) {
    P.dead[static_cast<size_t>(b) * R + c] = 0;
    S.kids[c][0] = S.kids[c][1] = S.level[c][0] = S.level[c][1] = 0u, S.size[c] = 0;
  }
  if (t == 0) S.status = 0;
  if (on) S.par[t] = par, S.tok[t] = tok, S.uni[t] = uni;
  sync();
  if (status) atomicOr(&S.status, status);
  sync();
  status = S.status;
  if (t == 0) plan_outcome(P, b, status);
  if (status) return plan_fault(P, b, t, 64, status);
  // up to the root: depth, and every ancestor counts the node
  int depth = 1;
  if (on) {
    atomicOr(&S.kids[par + 1][t >> 5], 1u << (t & 31));
    for (int a = par; a >= 0; a = S.par[a]) {
      atomicAdd(&S.size[a + 1], 1);
      ++depth;
    }
  }
  if (t == 0) S.size[0] = N;
  sync();
  const unsigned long long below = (1ull << t) - 1ull, with = on ? kids_of(par + 1) & below : 0ull;   // earlier siblings
  if (t == 0) S.placed = __popcll(kids_of(0));
  int weight = 1, n_kids = 0;
  if (on) {
    for (unsigned long long m = with; m; m &= m - 1ull) weight += S.size[__ffsll(m)] + 1;   // (context of node a: a + 1)
    S.weight[t] = weight;
    n_kids = __popcll(kids_of(t + 1));
    if (n_kids) atomicOr(&S.level[depth][t >> 5], 1u << (t & 31));
  }
  {
    const unsigned some = __ballot_sync(kFull, n_kids > 0);
    if ((t & 31) == 0) S.parents[t >> 5] = some;
  }
  sync();
  if (t == 0) S.start[0] = 0, S.rank[0] = 0, S.span[0] = R;
  if (on) {
    if (n_kids) S.start[t + 1] = atomicAdd(&S.placed, n_kids);
    // pre-order position; breadth-first rank, where it has children
    int pos = weight, rank = 1 + __popcll(level_at(depth) & below), d = depth;
    for (int a = par; a >= 0; a = S.par[a]) pos += S.weight[a], rank += __popcll(level_at(--d));
    S.rank[t + 1] = rank;
    S.span[t + 1] = pos << 16 | (S.size[t + 1] + 1);
  }
  sync();
  if (on) P.children[static_cast<size_t>(b) * N + S.start[par + 1] + __popcll(with)] = {t, tok, uni, S.span[t + 1]};
  // contexts with children (by rank) and without (by number)
  const unsigned long long has_kids = *reinterpret_cast<const unsigned long long*>(S.parents);
  const int n_ctx = 1 + __popcll(has_kids), n_leaf = R - n_ctx;
  for (int c = t; c < R; c += 64) {
    const unsigned long long m = kids_of(c);
    P.records[static_cast<size_t>(b) * R + c].word = m == 0ull ? kWalkLeaf : (c == 0 ? kWalkWaiting : kWalkPending);
    if (m) {
      const int f = __ffsll(m) - 1;       // its first child
      P.work[static_cast<size_t>(S.rank[c]) * B + b] = {b * R + c, b * N + S.start[c], __popcll(m) << 16 | f, S.span[f + 1], S.tok[f],
                                                        S.uni[f], u_final, b * R + (S.span[c] >> 16)};
    } else if (P.leaves) {
      const int r = (c - 1) - __popcll(has_kids & ((1ull << (c - 1)) - 1ull));
      P.leaves[static_cast<size_t>(r) * B + b] = S.span[c] >> 16 << 16 | c;
    }
  }
  for (int r = n_ctx + t; r < N; r += 64) P.work[static_cast<size_t>(r) * B + b].item = -1;
  if (P.leaves)
    for (int r = n_leaf + t; r < N; r += 64) P.leaves[static_cast<size_t>(r) * B + b] = -1;
  return plan_word(n_ctx, n_leaf, 0);
}

// threads of the plan kernel per sequence
static inline __host__ __device__ int plan_threads(const VerifyParams& P) { return P.parents && P.N > 0 && P.N <= PLAN_SMALL ? 64 : 32; }

__global__ void __launch_bounds__(PLAN_SEQS * 64) lantern_plan_kernel(VerifyParams P) {
  extern __shared__ int plan_smem[];
  __shared__ int s_words[PLAN_SEQS];
  __shared__ SmallPlan s_small[PLAN_SEQS];
  const int per = plan_threads(P), seq = threadIdx.x / per, t = threadIdx.x % per;
  grid_dependency_wait();
  grid_dependents_launch();
  if (blockIdx.x == 0 && threadIdx.x < 64) reinterpret_cast<int*>(P.counters)[threadIdx.x] = 0;
  const int b = blockIdx.x * PLAN_SEQS + seq;
  const int word = !P.parents || P.N == 0 ? plan_chain(P, b, t)
                                          : (per == 64 ? plan_small(P, s_small[seq], b, seq, t) : plan_sequence(P, plan_smem, b, seq, t));
  if (t == 0) s_words[seq] = word;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ranks = 0, leaves = 0, bits = 0;
    for (int w = 0; w < PLAN_SEQS; ++w) {
      ranks = max(ranks, s_words[w] & 0x7ff);
      leaves = max(leaves, s_words[w] >> 11 & 0x7ff);
      bits |= s_words[w] >> 22;
    }
    P.block_words[blockIdx.x] = plan_word(ranks, leaves, bits);
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
  size_t counters, work, leaves, children, records, dead, words, total;
};

static WsLayout ws_layout(int B, int N, bool topk = false) {
  const size_t R = static_cast<size_t>(N) + 1, b = static_cast<size_t>(B);
  const size_t n1 = N > 0 ? N : 1;
  WsLayout L;
  size_t o = 0;
  L.counters = o; o += 256;
  L.work = o;     o += align_up(b * n1 * sizeof(WorkItem), 256);
  L.leaves = o;   o += align_up(b * n1 * 4, 256);
  L.children = o; o += align_up(b * n1 * sizeof(ChildInfo), 256);
  L.records = o;  o += align_up(b * R * sizeof(Record), 256);
  L.dead = o;     o += align_up(b * R, 256);
  L.words = o;    o += 3 * align_up(b * 4, 256);   // (the size callers have always been told: parts of it are no longer used)
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

// what divide_by_T (verify_context.cuh) goes by
static void set_divisor(VerifyParams& P, float T) {
  const double inv = 1.0 / static_cast<double>(T);
  auto pair = [](float f) {
    uint32_t w;
    memcpy(&w, &f, 4);
    return static_cast<uint64_t>(w) << 32 | w;
  };
  P.T_fast = T >= 0x1p-100f && T <= 0x1p100f;
  const float least = fmaxf(0x1p-100f, T * 0x1p-125f);
  uint32_t bits;
  memcpy(&bits, &least, 4);
  P.T_least = 2u * bits - 1u;
  P.T_neg = pair(-T);
  const float y = P.T_fast ? static_cast<float>(inv) : 1.0f;
  const float hi = static_cast<double>(y) > inv ? nextafterf(y, 0.0f) : y;
  const float lo = P.T_fast ? static_cast<float>(inv - static_cast<double>(hi)) : 0.0f;
  P.T_inv = pair(y);
  P.T_inv_hi = pair(hi);
  P.T_inv_lo = pair(lo > 0.0f ? lo : 0x1p-126f);   // (a power of two leaves nothing; the product with -inf has to be -inf)
}

// Does a call list its leaves, so that bonus draws are made ahead of the walk?  A draw ahead takes a group that would stand idle, and saves the walk
// a dependent step at its end; where there is no such group it delays the contexts.  So calls of few contexts do, up to four per SM where the paths
// are long enough to hide the draws, us per call without | with: 74 chains of 7 drafts 36.2 | 32.9, one tree of 60 20.2 | 17.6, five 28.0 | 25.5, nine
// 29.9 | 28.2, but 16 of them (seven contexts per SM) 37.4 | 39.2.  Paths of one draft are not where a group has its SM for itself (25 chains
// 15.2 | 17.1, 290 24.1 | 27.4), and rows of at most 8192 tokens, three groups to an SM, up to four drafts until every group has a context (one
// chain of one draft 13.5 | 11.3, of 3 drafts 111 chains 17.6 | 16.0, 148 17.9 | 20.4; of one draft 200 15.6 | 15.4, 290 16.2 | 19.6).
static bool leaves_pay(const VerifyParams& P, int sms) {
  const long long contexts = static_cast<long long>(P.B) * P.R;
  if (P.V > 8192) return P.N > 1 && contexts <= 4ll * sms;
  return P.N > 0 && contexts <= (P.N > 4 ? 4ll : 3ll) * sms;
}

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

  const int sms = sm_count();
  if (sms < 1) return LANTERN_E_CUDA;
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
  set_divisor(P, T);
  P.divergence = divergence;
  P.top_k = topk ? top_k : 0;
  P.dead = ws + L.dead;
  P.leaves = leaves_pay(P, sms) ? reinterpret_cast<int32_t*>(ws + L.leaves) : nullptr;
  P.wait_tries = g_wait_tries;
  P.withhold_item = g_withhold_item;


  const size_t plan_smem = !tree_parents || N <= PLAN_SMALL ? 0 : static_cast<size_t>(PLAN_SEQS) * kPlanArrays * (N + 2) * sizeof(int);
  static DeviceFlags plan_ready;
  if (plan_smem > 32 * 1024 &&   // (beside the kernel's static part)
      allow_shared_memory(lantern_plan_kernel, PLAN_SEQS * kPlanArrays * (MAX_N + 2) * sizeof(int), plan_ready) != cudaSuccess)
    return LANTERN_E_CUDA;
  if (launch_dependent(lantern_plan_kernel, (B + PLAN_SEQS - 1) / PLAN_SEQS, PLAN_SEQS * plan_threads(P), plan_smem, st, P) != cudaSuccess)
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
