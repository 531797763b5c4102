// Fused context pass of the LANTERN verification step.
//
// Persistent kernel, one CTA per SM.  The CTA holds one or more independent consumer groups, each
// working on its own context in its own staging area of shared memory, and one producer warp per group
// that hands out contexts, issues the bulk asynchronous copies (TMA, completion on an mbarrier, no
// multicast) of a context's target rows, and walks the decided contexts (see below).  The groups
// drift apart in phase, so the latency-bound deciding part of one context overlaps the issue-bound
// streaming parts of the others.
//
// Three shapes (CtxNarrow, CtxPair, CtxWide below): three groups of eight warps per SM where there are sequences enough
// to fill the GPU, two or one of sixteen warps where there are not.
//
// The area of a group holds the two target rows only (64 KB at V = 16384, bf16): the drafter row, of
// which the common case needs nothing but its maximum, its sum and one entry, is read straight from
// global memory (it was asked into L2 one context ahead) into registers while the target rows are
// still being copied.
//
// Streaming part (per thread, on its own tokens): guidance combine, the maximum of a slice of at most
// 16 tokens, numerators 2^(z log2 e - n) through the hardware ex2 unit with the slice's own integer
// shift n = ceil(max * log2 e), partial sums -- no cross-thread step at all.  The numerators E
// are stored over the context's own raw target rows (every thread overwrites only bytes that it alone has
// read) and stay in the units of their slice; the shifts are tabulated, and because they are integers
// a numerator comes to common units by an exact power of two.  One group barrier then publishes E,
// the table and the per-warp maxima and sums.  Sums over many numerators average the ex2 unit's ~1e-7
// rounding out; the two single probabilities that decide a position, q(x~) and p(x~), are noted by a thread each
// and formed by every thread in double precision (with the logit filter by one warp).
//
// Deciding part, per child (Section 4.3 / Algorithm 2, second block): gather of the neighbour
// row's numerators, double-precision scan against the strict bound (the per-warp totals tell every warp
// which warp the bound falls into; only that one looks for the slot), accept test; on rejection
// the residual [q_{k,delta}(.|D = x~) - p]_+ in one register pass (the drafter logits are read
// again, normally from L2), its total, and either the inverse-CDF draw or the write-back for the
// next sibling.
//
// Which contexts are evaluated.  Algorithm 1 stops at the first rejection, so a context behind a
// rejected node is never tested by the method.  Work items come in breadth-first order per sequence
// (see the plan kernel); when a context has been decided, its producer marks the contexts behind every
// child that was not accepted as dead (a sequence's contexts are numbered in pre-order for this, so that a
// subtree is one contiguous range of marks), and a producer that meets a dead context leaves it out.  A context whose
// parent is still undecided when its turn comes is evaluated anyway: with few sequences per call that keeps every SM
// busy (all contexts of a tree run side by side), with many sequences it is rare, and the walk reads only results on the
// accepted path either way, so the outcome never depends on what was speculated.
//
// The walk (Algorithm 1's loop) needs no pass of its own.  Every context has a word that two parties exchange, each
// once: the producer whose group has decided the context, and the walk when it gets there (from the root, which starts
// as "walk waiting").  Whichever comes second goes on: along the accepted child, to the next word.  So a sequence
// is walked by whoever completes the next piece of its path, nobody waits, and where the walk ends on
// a context without children (or on one whose residual had no weight) the draw from that context's q
// is the next thing the same group does.  Two things save the walk time: a word that it has found decided by reading it, with others, is
// followed without an exchange; and in calls of few contexts (FEW) a producer may claim a context without children ahead of the walk,
// by compare-and-swap, so that its draw is a context like any other.
#pragma once

#include "verify_common.cuh"

namespace lantern {

// GT = threads of one consumer group (8 warps or more), NGRP = groups per CTA, AREAS = staging areas per group,
// CTAS = CTAs per SM.
template <int GT_, int NGRP_, int AREAS_, int CTAS_>
struct CtxShape {
  static constexpr int GT = GT_, NGRP = NGRP_, AREAS = AREAS_, CTAS = CTAS_;
  static constexpr int THREADS = NGRP * (GT + 32);
};
using CtxNarrow = CtxShape<256, 3, 1, 1>;   // 27 warps of 72 registers
using CtxPair = CtxShape<512, 1, 1, 2>;     // 2 * 17 warps of 56 registers
using CtxWide = CtxShape<512, 1, 2, 1>;     // 17 warps
using CtxSingle = CtxShape<512, 1, 1, 1>;   // for areas of 128 KB: greedy decoding on long fp32 rows with guidance
// Which shape.  A context is a chain of dependent steps; sixteen warps get through it in two thirds of the time eight
// need, but three contexts per SM hide one another's latencies.  With few sequences per call the path through each
// is what takes the time (and fewer contexts in flight mean fewer evaluated for nothing), with many the throughput.
// V = 16384, us per call narrow / pair / wide: 8 trees 50 / 46 / 44, 128 trees 116 / 100 / 98, 300 trees 155 / 147 / 138,
// 900 trees 254 / 243 / 270, 1500 trees 334 / 327 / 398; chains of 7: 200 sequences 82 / 69 / 71, 500 113 / 112 / 134,
// 1024 172 / 181 / 233, 8192 981 / 1152 / 1450.  Rows of 8192 tokens and less give sixteen warps too little to do
// (128 trees of 8192 tokens 78 / 78 / 88).
static inline int ctx_shape(const VerifyParams& P, int sms) {   // 0 = narrow, 1 = pair, 2 = wide
  if (P.V <= 8192) return 0;
  if (P.B <= (P.parents ? 2 : 1) * sms) return 2;
  return P.B <= (P.parents ? 10 : 3) * sms ? 1 : 0;
}

// bytes of one staging area: 4 bytes per token for the numerators, which replace the raw target rows
static inline __host__ __device__ size_t ctx_area_bytes(int V, bool bf16, bool uncond) {
  return (static_cast<size_t>(V) * ((bf16 || !uncond) ? 4 : 8) + 127) & ~static_cast<size_t>(127);
}
// Thread t of a group owns, for chunk c, the eight consecutive tokens [(c*GT + t)*8, +8), i.e. 16-byte
// group g = c*GT + t of a bf16 row.  E is laid over the context's own raw target rows: with bf16 logits
// the low four numerators of g replace g's bytes in row slot 0 and the high four replace g's bytes in
// row slot 1; with fp32 logits the eight numerators replace g's own 32 bytes of row slot 0.
// Float index of token x inside the staging area:
template <bool BF16>
__device__ __forceinline__ int ephys(int x, int row_floats) {
  if (BF16) return ((x >> 2) & 1) * row_floats + ((x >> 3) << 2) + (x & 3);
  return x;
}

// 2^(z log2 e) = y * 2^n for one value, n an integer, to about 1.5e-7: the exponent is formed in double precision,
// its fraction split into an fp32 head for the ex2 unit and a tail that is applied to first order.
struct Exp2Split {
  double y, n;
};
__device__ __forceinline__ Exp2Split exp2_split(float z) {
  Exp2Split r = {0.0, 0.0};
  if (z > -1.0e30f) {   // (-inf stays zero)
    const double x = static_cast<double>(z) * 1.4426950408889634074;
    r.n = rint(x);
    const double f = x - r.n;
    const float fh = static_cast<float>(f);
    const float fl = static_cast<float>(f - static_cast<double>(fh));
    const float y = ex2_approx(fh);
    r.y = static_cast<double>(__fmaf_rn(y, fl * 0.693147182464599609375f, y));
  }
  return r;
}
// 2^d for an integer d <= 0 held in a float, 0 below -126: exact, three instructions, no conversion
__device__ __forceinline__ float exp2_int(float d) {
  return __int_as_float(__float_as_int(fmaxf(d, -127.0f) + 12583039.0f) << 23);   // 1.5 * 2^23 + 127
}
// a power of two as a double, without a conversion (of 0: 2^-127, which is as good where it scales a sum down)
__device__ __forceinline__ double pow2_double(float f) { return __hiloint2double((__float_as_int(f) >> 3) + (896 << 20), 0); }
// 2^d for an integer d held in a double, 0 far below the range of what it is compared with (the conversion saturates)
__device__ __forceinline__ double exp2_int_d(double d) {
  const int e = min(__double2int_rn(d), 1000);
  return e <= -1000 ? 0.0 : __hiloint2double((1023 + e) << 20, 0);
}

constexpr int TOPK_LIST = 2080; // values inside the bracket of a threshold search, at most
constexpr int TOPK_BINS = 128;  // bins of its sample
constexpr int TOPK_FINE = 256;  // bins of the bracket
constexpr int TOPK_TINY = 32;   // values of the wanted bin that a warp ranks

struct CtxResult {              // what a group hands back to its producer
  int accepted;                 // accepted child, -1 if there is none
  int token;                    // token drawn, -1 if none
  int status;
};

// scratch of the top-k threshold search (verify_context_topk.cuh)
template <int GW, bool TOPK>
struct GroupTopk {};
template <int GW>
struct GroupTopk<GW, true> {
  alignas(16) int hist[TOPK_BINS];   // the sample, by value; zero between searches
  float range[GW][2];           // per warp: smallest and largest finite value of the sample
  int count[GW][2];             // per warp: values above the bracket, values inside it
  int fine[TOPK_FINE];          // the listed values, by value; zero between searches
  float tiny[TOPK_TINY];        // the values of the wanted bin
  int listed[3], picked[3];     // entries of the list and of tiny, by search (mod 3)
  float threshold;
};

template <int GW, bool TOPK>
struct alignas(16) GroupShared {
  alignas(16) double wz[GW][2]; // per-warp sums of numerators (target, drafter), in the warp's units
  double wt[64];                // per-(chunk, warp) totals for scans and block sums
  // q(x~), p(x~) of the next child to test, not yet in common units, of context i in single[i & 1]: the first threads may note the next
  // context's before the last ones have read the current one's
  Exp2Split single[2][2];
  double tested[2];             // (TOPK) the numerators of the tested token, common units
  double cut_sum;               // moved mass of A where the bound fell into a warp's slots
  double jsd_mass[2];           // the JSD bound as a mass, common units, by scan round (mod 2)
  double hist[32];              // drafter/target scale ratio of each earlier rejection round of this context
  alignas(8) float wn[GW][2];   // the warps' units: their largest shifts
  // shift of every (slice, thread), and from entry 1024 on, with four slices per thread, their sums; before that the list of a
  // threshold search
  float slice[TOPK ? TOPK_LIST : (GW == 8 ? 2048 : 1024)];
  int cut_m;                    // |A| - 1 that goes with cut_sum
  int badslot[3];               // first neighbour slot with an entry outside [0, V), by scan round (mod 3)
  int tok;
  int fail;                     // a bounded wait for the target rows ran out (sticky)
  GroupItem work[2];            // descriptor of context i in work[i & 1]: the next one is published while the current one runs
  CtxResult result[2];          // result of context i in result[i & 1]
  GroupTopk<GW, TOPK> tk;
};

}  // namespace lantern
#include "verify_context_topk.cuh"
namespace lantern {

// one row of a context into one row slot of a staging area, in bulk copies of at most 16 KB
__device__ __forceinline__ void ctx_issue_row(unsigned char* dst, const unsigned char* src, int rowbytes, uint64_t* bar) {
  for (int off = 0; off < rowbytes; off += 16384) {
    const int n = min(16384, rowbytes - off);
    bulk_load(dst + off, src + off, static_cast<uint32_t>(n), bar);
  }
}
// the target rows of a context (conditional, and unconditional if there is one), into row slots 0 and 1
template <bool UNC>
__device__ __forceinline__ void ctx_issue_target(const VerifyParams& P, int item, unsigned char* stage, int rowbytes,
                                                 uint64_t* bar) {
  mbar_expect_tx(bar, static_cast<uint32_t>((UNC ? 2 : 1) * rowbytes));
  const size_t row_off = static_cast<size_t>(item) * rowbytes;
  const unsigned char* t = static_cast<const unsigned char*>(P.target) + row_off;
  ctx_issue_row(stage, t, rowbytes, bar);
  if (UNC) ctx_issue_row(stage + rowbytes, t + static_cast<size_t>(P.B) * P.R * rowbytes, rowbytes, bar);
}

// Ask L2 for rows of a context ahead of time: the drafter row, which the group reads itself, always; the target rows
// where a bulk copy is issued long before its context's turn (two staging areas) -- with one area the copy starts as soon as
// rows that are on their way to the same SM have arrived, and prefetching them as well measured slower (8192 chains
// 1.056 against 1.028 ms; with two areas 128 trees 98 against 103 us the other way round).
template <bool UNC, bool DRAFTER, bool TARGET>
__device__ __forceinline__ void ctx_prefetch_rows(const VerifyParams& P, int item, int rowbytes) {
  const size_t row_off = static_cast<size_t>(item) * rowbytes;
  const unsigned char* d = static_cast<const unsigned char*>(P.draft) + row_off;
  if (DRAFTER && P.draft) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d), "r"(rowbytes) : "memory");
  if (TARGET) {
    const unsigned char* t = static_cast<const unsigned char*>(P.target) + row_off;
    const size_t branch = static_cast<size_t>(P.B) * P.R * rowbytes;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(t), "r"(rowbytes) : "memory");
    if (UNC) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(t + branch), "r"(rowbytes) : "memory");
  }
}

// One logit of a row in global memory, as it lies there, and the same widened to fp32.  The load is issued early and used late, by
// a few threads under a condition: widened there and then, those threads would wait for it inside the condition.
template <bool BF16>
__device__ __forceinline__ uint32_t ctx_raw_logit(const void* base, size_t elem) {
  uint32_t w;
  if (BF16) asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(w) : "l"(static_cast<const unsigned short*>(base) + elem));
  else asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(w) : "l"(static_cast<const float*>(base) + elem));
  return w;
}
template <bool BF16>
__device__ __forceinline__ float ctx_widen(uint32_t w) { return __uint_as_float(BF16 ? w << 16 : w); }

// eight raw logits of one 16-byte group (bf16) or 32 bytes (fp32) of a row in global memory
template <bool BF16>
struct Raw8 {
  uint4 a, b;   // b: second half of an fp32 group
};
template <bool BF16>
__device__ __forceinline__ Raw8<BF16> load_raw8(const unsigned char* row, int g) {
  Raw8<BF16> d;
  if (BF16) {
    d.a = ld_stream(row + static_cast<size_t>(g) * 16);
  } else {
    d.a = ld_stream(row + static_cast<size_t>(g) * 32);
    d.b = ld_stream(row + static_cast<size_t>(g) * 32 + 16);
  }
  return d;
}
// the same as four packed pairs of fp32 values
template <bool BF16>
__device__ __forceinline__ void raw8_pairs(const Raw8<BF16>& d, uint64_t (&o)[4]) {
  if (BF16) {
    const uint32_t w[4] = {d.a.x, d.a.y, d.a.z, d.a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
  } else {
    o[0] = pack2(__uint_as_float(d.a.x), __uint_as_float(d.a.y));
    o[1] = pack2(__uint_as_float(d.a.z), __uint_as_float(d.a.w));
    o[2] = pack2(__uint_as_float(d.b.x), __uint_as_float(d.b.y));
    o[3] = pack2(__uint_as_float(d.b.z), __uint_as_float(d.b.w));
  }
}
// four pairs of 16-byte (bf16) or 32-byte group g of a staged row
template <bool BF16>
__device__ __forceinline__ void staged_pairs(const unsigned char* row, int g, uint64_t (&o)[4]) {
  Raw8<BF16> d;
  if (BF16) {
    d.a = *reinterpret_cast<const uint4*>(row + g * 16);
  } else {
    d.a = *reinterpret_cast<const uint4*>(row + g * 32);
    d.b = *reinterpret_cast<const uint4*>(row + g * 32 + 16);
  }
  raw8_pairs<BF16>(d, o);
}
// maximum of eight raw logits and m (bf16: two running maxima, one per half word)
template <bool BF16>
__device__ __forceinline__ uint32_t raw8_max(const Raw8<BF16>& d, uint32_t m) {
  if (BF16) return bf16x2_max(bf16x2_max(bf16x2_max(d.a.x, d.a.y), bf16x2_max(d.a.z, d.a.w)), m);
  const float v = max3(max3(__uint_as_float(d.a.x), __uint_as_float(d.a.y), __uint_as_float(m)),
                       max3(__uint_as_float(d.a.z), __uint_as_float(d.a.w), __uint_as_float(d.b.x)),
                       max3(__uint_as_float(d.b.y), __uint_as_float(d.b.z), __uint_as_float(d.b.w)));
  return __float_as_uint(v);
}

// totals over the warp of two per-thread values: lanes 0..15 end with the first, lanes 16..31 with the second
__device__ __forceinline__ double warp_pair_sum(double a, double b, int lane) {
  const bool up = lane & 16;
  double z = (up ? b : a) + __shfl_xor_sync(kFull, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(kFull, z, o);
  return z;
}

// Totals over the warp of N per-thread values at once: every exchange halves the values a lane still carries, so
// N values cost N - 1 exchanges plus the rest of the butterfly instead of 5 N.  Lane l ends with the total of
// value l / (32 / N).
template <int N>
__device__ __forceinline__ double warp_transposed_sum(const float (&v)[N], int lane) {
  double d[N];
  int o = 16;
  if constexpr (N > 1) {
    const bool up = lane & 16;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float send = up ? v[i] : v[i + N / 2], keep = up ? v[i + N / 2] : v[i];
      d[i] = static_cast<double>(keep) + static_cast<double>(__shfl_xor_sync(kFull, send, 16));
    }
    o = 8;
#pragma unroll
    for (int n = N / 2; n > 1; n >>= 1) {
      const bool u = lane & o;
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const double send = u ? d[i] : d[i + n / 2], keep = u ? d[i + n / 2] : d[i];
        d[i] = keep + __shfl_xor_sync(kFull, send, o);
      }
      o >>= 1;
    }
  } else {
    d[0] = static_cast<double>(v[0]);
  }
#pragma unroll
  for (; o > 0; o >>= 1) d[0] += __shfl_xor_sync(kFull, d[0], o);
  return d[0];
}

// Four pairs of logits divided by the temperature, each quotient rounded once (IEEE division).  With y_hi + y_lo = 1 / T to 47 bits,
// q = fl(l y_hi + fl(l y_lo)) is off by hardly more than half a unit in the last place, so that the remainder r = l - q T is exact, and
// fl(q + r y) with y = fl(1 / T) is the correctly rounded quotient (Markstein, IBM J. Res. Dev. 34(1), 1990): four packed operations a
// pair where a division takes some ten instructions a value.  Where q is -inf (a masked token: l = -inf, or so low that the quotient
// overflows) the remainder is no number or +inf; its bound keeps the quotient -inf, as it should be (y_lo > 0), and a NaN a NaN.  (Where
// q is +inf the row is reported, be it as +inf or as a NaN.)  For 2^-100 <= T <= 2^100, others are divided by.  Exact where remainder and
// quotient are clear of the subnormal numbers, |l| >= 2^-100 and |l / T| >= 2^-125, or l = 0; below, the quotient can be off by a unit in
// the last place.  Numerators do not see that: 2^(z log2 e - n) is 2^-n for any |z| < 2^-100.  The threshold of the logit filter does, which
// has to be the very value of the tokens it is compared with (that of the tested one is a division's): with the filter a thread looks for such
// logits, in its part of the drafter row once, in the target row as it is processed, and divides where it has any (1024 chains at T = 0.9
// with the filter: 723 us by divisions, 588 without a look, 603 with it, 622 with one at every use of the drafter row).
static __device__ __noinline__ uint64_t divide_pair(uint64_t v, float T) {
  float lo, hi;
  unpack2(v, lo, hi);
  return pack2(__fdiv_rn(lo, T), __fdiv_rn(hi, T));
}
__device__ __forceinline__ void divide_by_T(const VerifyParams& P, uint64_t (&z)[4], bool fast) {
  if (fast) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint64_t q = fma2(z[i], P.T_inv_hi, mul2(z[i], P.T_inv_lo));
      float lo, hi;
      unpack2(fma2(P.T_neg, q, z[i]), lo, hi);
      z[i] = fma2(pack2(fminf(lo, 3.402823466e38f), fminf(hi, 3.402823466e38f)), P.T_inv, q);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) z[i] = divide_pair(z[i], P.T);
  }
}
// the smallest of `least` and eight raw logits' magnitudes, each as 2 bits(|l|) - 1: zero is the largest.  (From the words as they lie there: with
// the values widened first, which the sweeps widen again, the same call took 717 us.)
template <bool BF16>
__device__ __forceinline__ uint32_t least_magnitude(const Raw8<BF16>& d, uint32_t least) {
  const uint32_t w[8] = {d.a.x, d.a.y, d.a.z, d.a.w, BF16 ? 0u : d.b.x, BF16 ? 0u : d.b.y, BF16 ? 0u : d.b.z, BF16 ? 0u : d.b.w};
#pragma unroll
  for (int i = 0; i < (BF16 ? 4 : 8); ++i)
    least = BF16 ? min(least, min((w[i] << 17) - 1u, ((w[i] >> 16) << 17) - 1u)) : min(least, 2u * w[i] - 1u);
  return least;
}
// are there four pairs of logits whose quotients divide_by_T forms without a division?
__device__ __forceinline__ bool quotients_fast(const VerifyParams& P, const uint64_t (&z)[4]) {
  uint32_t least = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float lo, hi;
    unpack2(z[i], lo, hi);
    least = min(least, min(2u * __float_as_uint(lo) - 1u, 2u * __float_as_uint(hi) - 1u));
  }
  return least >= P.T_least;
}

// one bit per token of a thread
template <int CH>
using StruckMask = typename std::conditional<(CH > 4), uint64_t, uint32_t>::type;

// Exchange of a walk word.  The word carries everything its receiver needs and what the two sides store besides does
// not depend on order, so no fence is paid for (with acquire and release the producers became the bottleneck: 1.12
// instead of 1.07 ms on 8192 chains).
__device__ __forceinline__ unsigned long long walk_exchange(Record* rec, unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.relaxed.gpu.global.exch.b64 %0, [%1], %2;" : "=l"(old) : "l"(&rec->word), "l"(v) : "memory");
  return old;
}

// A walk that has fallen behind the deciding of its contexts pays a round trip to L2 per step.  After this many steps in one go it
// reads the words of 32 contexts at once, from the next one on, and follows those that lead on to the next: a chain's contexts do.
// (29 chains of 443 drafts of 6664 fp32 logits 217 us per call, 1069 without it; 2 of 1024 drafts 73 and 722.  Paths of a few
// contexts never get there.)
// With the logit filter, where contexts take three times as long to decide, sequences of at most 64 contexts have all their words read at
// once after three steps, and what was decided is followed without further round trips (1024 chains of 7 drafts 459 us per call, 467 to 473
// without it; other variants lose by it: 2048 chains in greedy decoding 145.6 us without and 146.4 with it, 1000 trees 159.5 and 162.4).
constexpr int kWalkAlone = 6, kWalkFilter = 3;
__device__ __forceinline__ unsigned long long walk_look(const Record* rec) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(&rec->word) : "memory");
  return w;
}

// CH = 8-token chunks per thread (1, 2, 4 or 8); the target's numerators come in slices of CP chunks.
// TONE = the temperature is exactly 1 (the paper's sampling setting): no division is compiled in.
// JSD selects the Section 5.3.2 bound at compile time, so that the default path carries none of its code.
// GREEDY = greedy decoding (Section 4.3, last sentence; TONE is set then): no drafter distribution, no random numbers; x~ is
// accepted iff sum_A q >= max_x q(x) (it is an arg max of q_{k,delta}(.|D = x~): the maximum over A's own members can never
// exceed the sum), children are tried against the same q, and wherever the walk stops the token is arg max q.
// TOPK = the logit filter is on (Appendix B.2): processed logits below the top_k-th largest of their row count as -inf.
// FEW = a call of few contexts, whose leaves are listed (P.leaves): producers make bonus draws ahead of the walk.  At compile time, because
// what they need for it costs the producers of large calls 1 to 5 per cent, also where it is stepped over (greedy decoding of 2048
// chains of 7 drafts 146.4 us per call, 151.0 with one kernel for both; of 8192 tokens and 8 drafts 114.7 and 120.4; sampling, 8192 chains 952
// and 973, 1600 trees of 8192 tokens 252 and 262).
template <class SHAPE, int CH, bool BF16, bool UNC, bool TONE, bool JSD, bool TOPK, bool GREEDY, bool FEW>
__global__ void __launch_bounds__(SHAPE::THREADS, SHAPE::CTAS) lantern_context_kernel(VerifyParams P) {
  constexpr int GT = SHAPE::GT, GW = GT / 32, NGRP = SHAPE::NGRP, AREAS = SHAPE::AREAS;
  constexpr int LOG_GT = GT == 512 ? 9 : 8;
  static_assert((1 << LOG_GT) == GT, "256 or 512 threads per group");
  constexpr int SLOTS = 1024 / GT;            // neighbour slots per thread and scan round
  constexpr int CP = CH > 2 ? 2 : CH;         // chunks per slice
  constexpr int NP = CH / CP;                 // slices per thread
  constexpr int LOG_CP = CP == 2 ? 1 : 0;
  constexpr int AHEAD = BF16 ? (CH < 4 ? CH : 4) : (CH < 2 ? CH : 2);   // drafter groups in flight in a residual pass
  // Few registers hold this thread's part of the drafter row, or there are registers enough: it is kept for the residual passes
  // (which else read it again, a round trip to L2 per rejection).
  constexpr bool HOLD = CH * (BF16 ? 4 : 8) <= 8 || (GT == 512 && SHAPE::CTAS == 1);
  static_assert(NP * GT <= 1024 && CH * GW <= 64 && TOPK_LIST >= 2048, "tables of slices and blocks");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ GroupShared<GW, TOPK> SG[NGRP];
  // Per group: next context published / the next context may be chosen / context i finished (by i mod 2: the producer may
  // look for context i - 1 when context i has been finished too); per area: rows landed
  __shared__ __align__(8) uint64_t bar_item[NGRP], bar_next[NGRP], bar_done[NGRP][2], bar_rows[NGRP][AREAS];

  const int tid = threadIdx.x, lane = tid & 31;
  const int V = P.V, N = P.N, R = P.R, k = P.k;
  const int rowbytes = V * (BF16 ? 2 : 4);
  const int area_bytes = static_cast<int>(ctx_area_bytes(V, BF16, UNC));
  const float L2E = 1.44269502162933349609375f;   // fl32(log2 e)
  const float ninf = __int_as_float(0xff800000);

  if (tid == 0) {
    for (int g = 0; g < NGRP; ++g) {
      mbar_init(&bar_item[g], 1);
      mbar_init(&bar_next[g], GW);
      mbar_init(&bar_done[g][0], GW);
      mbar_init(&bar_done[g][1], GW);
      for (int a = 0; a < AREAS; ++a) mbar_init(&bar_rows[g][a], 1);
      SG[g].fail = 0;
      SG[g].badslot[0] = SG[g].badslot[1] = SG[g].badslot[2] = kNone;
      if constexpr (TOPK) {
        for (int q = 0; q < 3; ++q) SG[g].tk.listed[q] = SG[g].tk.picked[q] = 0;
      }
    }
    fence_mbar_init();
    fence_proxy_async();
  }
  if constexpr (TOPK) {
    for (int q = tid; q < NGRP * TOPK_FINE; q += SHAPE::THREADS) SG[q / TOPK_FINE].tk.fine[q % TOPK_FINE] = 0;
    for (int q = tid; q < NGRP * TOPK_BINS; q += SHAPE::THREADS) SG[q / TOPK_BINS].tk.hist[q % TOPK_BINS] = 0;
  }
  __syncthreads();
  // The plan, and whatever made the inputs.  This kernel may be in place while the plan still writes: what the plan writes is read by
  // ordinary loads, which stay behind this wait.  Logits and neighbour rows are read through the read-only path: they are
  // complete before any CTA of this kernel starts, because every CTA of the plan lets it start only after a wait of its own.
  // Before that: rows that some group begins with whatever the plan says, those of the first roots, are asked into L2 while it runs, a
  // sequence per group.  (All rows of a small call, of which every group gets a few at most, were too much: 74 chains of 7 drafts 33.7
  // us per call, 37.0 with them; no row at all: 500 chains 105.6 instead of 104.3.)
  if (lane == 0 && tid >= NGRP * GT) {
    const int me = ((tid - NGRP * GT) >> 5) * gridDim.x + blockIdx.x;
    if (me < P.B) ctx_prefetch_rows<UNC, !GREEDY, true>(P, me * R, rowbytes);
  }
  grid_dependency_wait();

  // ======================= producer warps =======================
  // One warp per consumer group hands out work, keeps that group's copies going and walks.  Its 32 lanes look
  // at up to 32 consecutive work slots at a time (a batch: the first one dealt statically, later ones
  // from a global counter, in sizes that shrink towards the end of the list so that the groups finish
  // together), drop the empty and the dead ones, and feed the rest to the group one by one, each by the lane that looked at it:
  // the context is chosen, and published, when the group has streamed the one before (so that it can go on to
  // the next drafter row without asking), and its target rows are copied as soon as a staging area is free.  The
  // next batch is loaded while the current one is being worked on, so that no round trip to the work list is
  // on the critical path.
  if (tid >= NGRP * GT) {
    const int grp = (tid - NGRP * GT) >> 5;
    GroupShared<GW, TOPK>& S = SG[grp];
    const int G = gridDim.x * NGRP;              // producers in the grid
    const int me = grp * gridDim.x + blockIdx.x; // few contexts: one to an SM before any SM gets a second one
    const uint32_t tries = P.wait_tries;
    // Slots per batch.  Few live contexts per batch (two; one towards the end of the list, so that the groups
    // finish together): a batch is worked through in order, and the longer that takes the more of its
    // contexts meet an undecided parent and are evaluated for nothing.  But as many slots as it has taken so
    // far to find that many live ones: tree workloads leave most slots empty or dead, and every batch costs a
    // round trip to the work list.
    int slots_seen = 0, live_seen = 0;
    // slots of the work list that are in use, and those of the list of leaves behind them
    PlanSummary extent = {P.B * (N > 0 ? N : 1), FEW ? P.B * N : 0, 0};   // (at most, until the plan's summary has been read)
    auto batch_size = [&](int at) {
      const int share = (extent.slots + extent.leaf_slots - at) / (4 * G);
      const int live = share < 1 ? 1 : (share > 2 ? 2 : share);
      const int s = live * ((slots_seen + 1) / (live_seen + 1));
      return s < 1 ? 1 : (s > 32 ? 32 : s);
    };
    // What a lane keeps of a candidate: its slot, its context and its dead mark (the rest is read when it is taken).  Slots beyond those
    // of the contexts with children are those of the leaves.
    struct Cand {
      int slot, item, mark;
    };
    auto load_cand = [&](int start, int size) -> Cand {
      Cand c = {start + lane, -1, 0};
      const int leaf = c.slot - extent.slots;
      if (lane < size) {
        if (leaf < 0) {
          c.item = P.work[c.slot].item;
          c.mark = P.work[c.slot].mark;
        } else if (FEW && leaf < extent.leaf_slots) {
          const int w = P.leaves[leaf], b = leaf % P.B;
          if (w >= 0) c.item = b * R + (w & 0xffff), c.mark = b * R + (w >> 16);
        }
      }
      return c;
    };
    // the rest, by the candidate's lane
    auto load_item = [&](const Cand& c, int4& lo, int4& hi) {
      if (!FEW || c.slot < extent.slots) {
        lo = *reinterpret_cast<const int4*>(P.work + c.slot);
        hi = *(reinterpret_cast<const int4*>(P.work + c.slot) + 1);
      } else {                 // nothing but a draw
        lo = make_int4(c.item, 0, 0, 0), hi = make_int4(0, 0, 0, 0);
        if (P.uniforms) hi.z = __float_as_int(P.uniforms[static_cast<size_t>(c.item / R) * R + N]);
      }
    };
    auto is_dead = [&](int mark) -> bool {
      return *reinterpret_cast<const volatile unsigned char*>(P.dead + mark) != 0;
    };
    // A bonus draw ahead of time: the leaf is taken if the walk has not got there yet.
    auto claim_leaf = [&](int item) -> bool {
      return atomicCAS(&P.records[item].word, static_cast<unsigned long long>(kWalkLeaf), static_cast<unsigned long long>(kWalkPending)) ==
             static_cast<unsigned long long>(kWalkLeaf);
    };
    int n_eval = 0, n_skip = 0, n_draw = 0;
    // live candidates of a batch, as a lane mask
    auto filter = [&](const Cand& c, bool first) -> unsigned {
      const bool has = c.item >= 0;
      const bool dead = has && !first && is_dead(c.mark);
      n_skip += __popc(__ballot_sync(kFull, dead && (!FEW || c.slot < extent.slots)));
      const unsigned live = __ballot_sync(kFull, has && !dead);
      live_seen += __popc(live);
      return live;
    };
    // Tickets for the dynamic batches are asked for two batches ahead and the candidates of a batch are read one batch
    // ahead, so that a producer waits for neither.
    const int b0 = batch_size(0);
    Cand cur = {me * b0 + lane, -1, 0}, nxt;
    int4 lo = make_int4(-1, 0, 0, 0), hi = make_int4(0, 0, 0, 0);      // the description of this lane's candidate
    if (lane < b0 && cur.slot < extent.slots) load_item(cur, lo, hi);   // (the first batch at once, beside the summary)
    cur.item = lo.x, cur.mark = hi.w;
    extent = plan_extent<FEW>(P, lane);
    const int total = extent.slots + extent.leaf_slots;
    bool cur_end = me * b0 >= total, nxt_end = false, primed = false, described = true;   // (lo and hi: only of the first batch, and until used)
    if (FEW && me * b0 + b0 > extent.slots) {   // (the leaves begin earlier than was assumed)
      cur = load_cand(me * b0, b0);
      if (cur.item >= 0) load_item(cur, lo, hi);
    }
    int ticket = 0, ticket_size = 0, seen = G * b0;
    auto ask = [&]() {       // (lane 0 holds the answer)
      ticket_size = batch_size(seen < total ? seen : total);
      if (lane == 0) ticket = atomicAdd(&P.counters->work_next, ticket_size);
      slots_seen += ticket_size;
    };
    auto load_next = [&]() {
      seen = G * b0 + __shfl_sync(kFull, ticket, 0);
      nxt = load_cand(seen, ticket_size);
      nxt_end = seen >= total;
      ask();
    };
    ask();
    unsigned mask = filter(cur, true);
    auto next_batch = [&]() {   // make `mask` non-empty if any live context is left
      if (!primed) {
        primed = true;
        load_next();
      }
      while (mask == 0 && !cur_end) {
        cur = nxt;
        cur_end = nxt_end;
        described = false;
        if (!cur_end) load_next();
        mask = filter(cur, false);
      }
    };
    // A sequence's final outcome.  (Its status stood at INTERNAL until now, see the plan kernel.)
    auto finish = [&](int b, int token, int status) {
      P.out_tok[b] = token;
      if (P.out_status) P.out_status[b] = status;
      if (status) atomicOr(&P.counters->status_or, status);
    };
    // A pending draw from a context's own q, and the context handed out last (everything its result needs;
    // nc0 = nchild << 16 | node0, kDrawForWalk for a draw the walk has asked for, kDrawAhead for one made ahead of it).
    // `open`: that context's result has not been taken yet.
    constexpr int kDrawForWalk = 0, kDrawAhead = 1;
    int draw_item = -1, draw_status = 0;
    float draw_u = 0.0f;
    int p_item = 0, p_cbase = 0, p_nc0 = 0, p_span0 = 0, p_status = 0;
    float p_u = 0.0f;
    bool open = false;
    // Takes the group's result for context j, the one handed out last.  Returns false if the group never delivered.
    auto take_result = [&](int j) -> bool {
      if (!mbar_wait(&bar_done[grp][j & 1], (j >> 1) & 1, tries)) return false;
      open = false;
      const CtxResult res = S.result[j & 1];
      const int item = p_item, nc0 = p_nc0;
      const int b = item / R;
      if (nc0 == kDrawForWalk) {
        ++n_draw;
        if (lane == 0) finish(b, res.token, p_status | res.status);
        return true;
      }
      Record* recs = P.records + static_cast<size_t>(b) * R;
      // Algorithm 1 goes on from the accepted child only: every context behind another child is dead.  In
      // pre-order those are one contiguous range per child.
      const int cbase = p_cbase, span0 = p_span0, nchild = nc0 >> 16;
      unsigned char* marks = P.dead + static_cast<size_t>(b) * R;
      for (int c = 0; c < nchild; ++c) {   // (none behind a leaf)
        int node_c = nc0 & 0xffff, span_c = span0;
        if (c > 0) {
          const int4 kid = *reinterpret_cast<const int4*>(P.children + cbase + c);
          node_c = kid.x, span_c = kid.w;
        }
        if (node_c != res.accepted)
          for (int o = lane; o < (span_c & 0xffff); o += 32) marks[(span_c >> 16) + o] = 1;
      }
      // (all lanes follow the walk; lane 0 exchanges and stores)
      int at = item - b * R, accepted = res.accepted, token = res.token, status = res.status;
      auto exchange = [&](unsigned long long v) {
        unsigned long long w = 0;
        if (lane == 0) w = walk_exchange(recs + at, v);
        return __shfl_sync(kFull, w, 0);
      };
      bool drawn = nc0 == kDrawAhead;
      unsigned long long w = exchange(walk_word(kWalkDecided | (drawn ? kWalkDrawn : 0u), status, accepted + 1, token));
      if ((w & 3u) == kWalkWaiting) {   // the walk stands here already: go on with it
        int st = static_cast<int>(w >> 8) & 0xff, len = static_cast<int>(w >> 16) & 0xffff;
        const int len_before = len;
        int32_t* path = P.out_path ? P.out_path + static_cast<size_t>(b) * N : nullptr;
        unsigned long long seen0 = 0, seen1 = 0;   // (TOPK) words of contexts `lane` and `lane` + 32
        for (int steps = 0;;) {
          st |= status;
          if (status & (LANTERN_ST_NONFINITE | LANTERN_ST_INTERNAL)) {
            n_draw += drawn;                                     // (a draw from a row that is not finite is one all the same)
            if (lane == 0) finish(b, -1, st);
            break;
          }
          bool from_q = (status & LANTERN_ST_DEGENERATE) != 0;   // a residual without weight: draw from the context's own target
          if (!from_q) {
            if (accepted < 0) {
              n_draw += drawn;
              if (lane == 0) finish(b, token, st);
              break;
            }
            if (lane == 0 && path) path[len] = accepted;
            ++len;
            at = accepted + 1;
            w = 0;
            ++steps;
            if (TOPK && R <= 64) {
              if (steps > kWalkFilter) {
                if (steps == kWalkFilter + 1) {
                  if (lane < R) seen0 = walk_look(recs + lane);
                  if (lane + 32 < R) seen1 = walk_look(recs + lane + 32);
                }
                const unsigned long long w0 = __shfl_sync(kFull, seen0, at & 31), w1 = __shfl_sync(kFull, seen1, at & 31);
                w = at < 32 ? w0 : w1;
              }
            } else if (steps > kWalkAlone) {
              // the contexts that were decided in favour of the node numbered as they are, from this one on, are followed at once
              for (int run = 32; run == 32;) {
                const unsigned long long seen = at + lane < R ? walk_look(recs + at + lane) : 0;
                const bool on = (seen & 0xffffffffull) == (walk_word(kWalkDecided, 0, at + lane + 1) & 0xffffffffull);
                const unsigned off = ~__ballot_sync(kFull, on);
                run = off ? __ffs(off) - 1 : 32;
                if (lane < run && path) path[len + lane] = at + lane;
                len += run, at += run;
                if (run < 32) w = __shfl_sync(kFull, seen, run);
              }
            }
            if ((w & 3u) != kWalkDecided) w = exchange(walk_word(kWalkWaiting, st, len));   // (a decided word stays as it is)
            from_q = (w & 3u) == kWalkLeaf;                      // no drafts left on this path: bonus token from q
          }
          if (from_q) {
            draw_item = b * R + at;
            draw_status = st;
            draw_u = p_u;
            break;
          }
          if ((w & 3u) != kWalkDecided) break;                   // whoever decides that context goes on
          status = static_cast<int>(w >> 8) & 0xff;
          accepted = static_cast<int>(w >> 16 & 0xffff) - 1;
          token = static_cast<int>(w >> 32);
          drawn = (w & kWalkDrawn) != 0;
        }
        if (lane == 0 && len > len_before) atomicMax(&P.out_len[b], len);   // (pieces of the path may be stored out of order)
      }
      __syncwarp();
      return true;
    };
    int i = 0;        // contexts handed to the group so far
    int stop = 0;     // the abort flag, as it stood when the last context was handed out
    bool clean = true;
    // A context handed to a group that has siblings to try yet waits for all of them: in a small call of trees the next one is chosen
    // when the group's result is known (8 trees 38.0 -> 36.5 us per call; chains have no siblings, and lose by it).
    const bool late = FEW && P.parents;
    for (;;) {
      if (late && open && !take_result(i - 1)) {
        clean = false;
        break;
      }
      const bool drawing = __shfl_sync(kFull, draw_item, 0) >= 0;
      if (!drawing) {
        if (mask == 0) next_batch();
        if (mask == 0) {   // nothing left but what the group is working on, which may end in a draw
          if (!open) break;
          if (!take_result(i - 1)) {
            clean = false;
            break;
          }
          continue;
        }
      }
      int l = 0;               // the lane that hands it out
      bool leaf = false;
      int it_status = 0;
      if (drawing) {
        lo = make_int4(draw_item, 0, 0, 0), hi = make_int4(0, 0, __float_as_int(draw_u), 0);
        it_status = draw_status;
        draw_item = -1;
      } else {                 // (a work slot without children is a draw from the outset: a call without drafts)
        l = __ffs(mask) - 1;
        mask &= mask - 1;
        if (FEW) leaf = __shfl_sync(kFull, cur.slot, l) >= extent.slots;
        if (!described && lane == l) load_item(cur, lo, hi);   // in flight while the group is waited for
        described = false;
      }
      if (i >= 1 && !mbar_wait(&bar_next[grp], (i - 1) & 1, tries)) {
        clean = false;   // the group never came this far: it has given up, and so does its producer
        break;
      }
      if (__any_sync(kFull, stop != 0)) break;   // the call has been given up
      // as late as possible: has the context died meanwhile?  (Not the first one: nothing has been decided.)
      if (!drawing && (i > 0 || leaf)) {
        int gone = 0;
        if (lane == l) gone = (is_dead(cur.mark) ? 1 : 0) | (leaf && !claim_leaf(cur.item) ? 1 : 0);
        if (__any_sync(kFull, gone)) {
          n_skip += leaf ? 0 : 1;
          continue;
        }
      }
      if (lane == l) {
        S.work[i & 1] = {lo.x, lo.y, lo.z >> 16, lo.z & 0xffff, hi.x, lo.w, __int_as_float(hi.y), __int_as_float(hi.z)};
        mbar_arrive(&bar_item[grp]);
      }
      const int area = i % AREAS;
      auto issue = [&]() {
        if (lane == l && lo.x != P.withhold_item) {   // (self-test of the bounded waits: nothing is copied)
          fence_proxy_async();
          ctx_issue_target<UNC>(P, lo.x, smem + (grp * AREAS + area) * area_bytes, rowbytes, &bar_rows[grp][area]);
        }
      };
      bool ok = true;
      if (AREAS > 1) {
        issue();           // (the area's last context has been taken back already)
        if (open) ok = take_result(i - 1);
      } else {
        // the area is free once every warp of the group has finished the previous context
        if (i >= 1) ok = mbar_wait(&bar_done[grp][(i - 1) & 1], ((i - 1) >> 1) & 1, tries);
        if (ok) {
          issue();
          if (open) take_result(i - 1);
        }
      }
      p_item = __shfl_sync(kFull, lo.x, l), p_cbase = __shfl_sync(kFull, lo.y, l), p_span0 = __shfl_sync(kFull, lo.w, l);
      p_nc0 = __shfl_sync(kFull, lo.z, l), p_u = __int_as_float(__shfl_sync(kFull, hi.z, l));
      p_status = it_status;
      if (p_nc0 == 0) p_nc0 = leaf ? kDrawAhead : kDrawForWalk;
      else ++n_eval;
      open = true;
      ++i;
      if (!ok) {
        clean = false;
        break;
      }
      // Look ahead: the next live context (a batch swap, if the current batch is used up, happens here, where
      // nothing waits for it) and an L2 prefetch of its rows -- of a context that has passed the dead check,
      // so that hardly any prefetched row goes unused.
      stop = *reinterpret_cast<const volatile int*>(&P.counters->abort);
      next_batch();
      if (mask && __shfl_sync(kFull, draw_item, 0) < 0) {
        const int item_ahead = __shfl_sync(kFull, cur.item, __ffs(mask) - 1);
        if (lane == 0) ctx_prefetch_rows<UNC, !GREEDY, (AREAS > 1)>(P, item_ahead, rowbytes);
      }
    }
    // (a call that was given up elsewhere: the group's last context has to be finished by all its warps before the terminator is
    // published, because the first to see that overwrite what the others may still read)
    if (clean && open) clean = mbar_wait(&bar_done[grp][(i - 1) & 1], ((i - 1) >> 1) & 1, tries);
    if (lane == 0) {
      if (clean) {   // the group is waiting for its next context: hand it the terminator
        if (i == 0 || mbar_wait(&bar_next[grp], (i - 1) & 1, tries)) {
          S.work[i & 1].item = -1;
          mbar_arrive(&bar_item[grp]);
        }
      }
      if (n_eval) atomicAdd(&P.counters->n_evaluated, n_eval);
      if (n_skip) atomicAdd(&P.counters->n_skipped, n_skip);
      if (n_draw) atomicAdd(&P.counters->n_bonus, n_draw);
    }
    if (me == 0) {   // sequences that the plan found at fault
      const int faults = plan_summary<FEW>(P, lane).faults;
      if (faults && lane == 0) atomicOr(&P.counters->status_or, faults);
    }
    return;
  }

  // ======================= consumer groups =======================
  const int grp = tid >> LOG_GT;        // which group
  const int gt = tid & (GT - 1);        // thread within the group
  const int gw = gt >> 5;               // warp within the group
  GroupShared<GW, TOPK>& S = SG[grp];
  const int row_floats = rowbytes >> 2;
  auto EI = [&](int x) { return ephys<BF16>(x, row_floats); };
  // index of the slice that owns token x in the table of shifts
  auto owner_slice = [&](int x) {
    const int g = x >> 3;
    return ((g >> (LOG_GT + LOG_CP)) << LOG_GT) | (g & (GT - 1));
  };
  const bool full = V == CH * GT * 8;                 // every thread owns CH whole chunks: no bounds to check
  const bool nbr_vec = SLOTS == 4 && (k & 3) == 0 && (reinterpret_cast<uintptr_t>(P.nbr) & 15) == 0;
  const size_t branch = static_cast<size_t>(P.B) * R * V;   // elements from a conditional row to its unconditional one
  const uint32_t tries = P.wait_tries;
  auto gbar = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(GT) : "memory"); };   // the group's threads
  // this thread's slots SLOTS gt .. of a neighbour row, from slot `base` on (slot 0 is the token itself,
  // entries past the row are not looked at)
  auto load_slots = [&](int token, int base, int (&n)[SLOTS]) {
    const int32_t* row = P.nbr + static_cast<size_t>(token) * k + base + SLOTS * gt;
    if (nbr_vec) {
      int4 v = make_int4(0, 0, 0, 0);
      if (base + SLOTS * gt < k) v = ld_nc_here4(row);   // k % 4 == 0: all four slots exist
      n[0] = v.x, n[1 % SLOTS] = v.y, n[2 % SLOTS] = v.z, n[3 % SLOTS] = v.w;
    } else {
#pragma unroll
      for (int i = 0; i < SLOTS; ++i) n[i] = base + SLOTS * gt + i < k ? ld_nc_here(row + i) : 0;
    }
  };
  // Scan rounds of this group so far, mod 2 and mod 3: a round's totals are not overwritten, and its bad-slot word is
  // not cleared, before every warp has read them.
  int round2 = 0, round3 = 0;
  int search3 = 0;                      // threshold searches so far, mod 3
  for (int iter = 0;; ++iter) {
    const int area = iter % AREAS;
    // A bounded wait that runs out ends the group: the context keeps its undecided word, so the sequences that need it
    // keep INTERNAL; the call is given up (no producer hands out further work), and one thread gives
    // the copies that may still be on their way into this group's staging areas the same bounded wait before the group
    // leaves.
    auto give_up = [&]() {
      if (gt == 0) {
        *reinterpret_cast<volatile int*>(&P.counters->abort) = 1;
        atomicOr(&P.counters->status_or, LANTERN_ST_INTERNAL);
        mbar_wait(&bar_rows[grp][area], (iter / AREAS) & 1, tries);
        if (AREAS > 1) mbar_wait(&bar_rows[grp][(iter + 1) % AREAS], ((iter + 1) / AREAS) & 1, tries);
      }
    };
    // Every warp waits for the next context by itself and may run ahead of slower ones: whatever it overwrites
    // before the next group barrier they have finished with (with one staging area because the target rows land only when
    // all warps have released it; with two areas, or a threshold search, a barrier sees to it).  A wait that runs out is reported behind that
    // barrier, where every thread sees it alike.
    if (AREAS > 1 && !TOPK) gbar();
    bool there = mbar_wait(&bar_item[grp], iter & 1, tries);
    if (TOPK) {   // (every thread has to take the same path to the barriers of a threshold search)
      uint32_t all;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.u32 p, %1, 0;\n\t"
          "bar.red.and.pred q, %2, %3, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(all)
          : "r"(static_cast<uint32_t>(there)), "r"(1 + grp), "n"(GT)
          : "memory");
      there = all != 0;
    }
    if (!there) S.fail = 1;
    const GroupItem& cur = S.work[iter & 1];
    const int item = there ? cur.item : -1;
    unsigned char* stage = smem + (grp * AREAS + area) * area_bytes;   // this context's target rows, later its E
    float* E = reinterpret_cast<float*>(stage);
    const int nchild = item < 0 ? 0 : cur.nchild;                      // 0: nothing but a draw from q
    const unsigned char* drow = static_cast<const unsigned char*>(P.draft) + static_cast<size_t>(item) * rowbytes;

    // first child: its neighbour row and its raw logits (target: thread 0, drafter: thread 1); issued now, used after the
    // streaming part
    int node = cur.node0;
    int xt = cur.tok0;
    int nb[SLOTS];
    uint32_t raw_z = 0u, raw_u = 0u;
    auto fetch_single = [&]() {   // (threads 0 and 1)
      const size_t e = static_cast<size_t>(item) * V + xt;
      raw_z = ctx_raw_logit<BF16>(gt == 0 ? P.target : P.draft, e);
      if (UNC) raw_u = ctx_raw_logit<BF16>(P.target, branch + e);
    };
    float tq = ninf, tp = ninf;   // top-k thresholds of the target and the drafter row
    auto note_single = [&]() {
      float z = ctx_widen<BF16>(raw_z);
      if (UNC) {
        const float u = ctx_widen<BF16>(raw_u), l = __fmaf_rn(P.cfg_scale, __fsub_rn(z, u), u);
        z = gt == 0 ? l : z;
      }
      if (!TONE) z = __fdiv_rn(z, P.T);
      if (TOPK) z = z < (gt == 0 ? tq : tp) ? ninf : z;
      S.single[iter & 1][gt] = exp2_split(z);
    };

    // ---------------- streaming part, thread-local ----------------
    // values travel as packed pairs (tokens 2i, 2i+1 of a chunk)
    const uint64_t L2 = pack2(L2E, L2E);
    float nd = 0.0f;              // drafter: this thread's shift and its sum of numerators, in its own units
    // (sums of up to 16 numerators are formed in single precision, from there on in double: in single precision all the way a
    // normaliser of 16384 numerators was off by up to 1.9e-7 where one of a thread's 64 outweighs the others)
    double td = 1.0;
    float nq[NP <= 2 ? NP : 1] = {};  // target: the shifts of the slices, where they are few (else in S.slice)
    float tq_sum[NP <= 2 ? NP : 1] = {};   // ... and their sums, likewise
    auto shift_of = [&](int p) { return NP <= 2 ? nq[NP <= 2 ? p : 0] : S.slice[p * GT + gt]; };
    auto sum_of = [&](int p) { return NP <= 2 ? tq_sum[NP <= 2 ? p : 0] : S.slice[1024 + p * GT + gt]; };
    float z_max = ninf;               // GREEDY: this thread's largest logit
    Raw8<BF16> raw[CH];           // the drafter row
    bool fast_d = P.T_fast != 0;  // its quotients by the temperature are formed without a division
    auto load_drafter = [&](auto whole) {
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int g = c * GT + gt;
        if (decltype(whole)::value || g * 8 < V) {
          raw[c] = load_raw8<BF16>(drow, g);
        } else {
          const uint32_t w = BF16 ? 0xff80ff80u : 0xff800000u;
          raw[c].a = raw[c].b = make_uint4(w, w, w, w);
        }
      }
    };
    auto reduce_drafter = [&]() {
      uint32_t mw = BF16 ? 0xff80ff80u : 0xff800000u;
#pragma unroll
      for (int c = 0; c < CH; ++c) mw = raw8_max<BF16>(raw[c], mw);
      float m = BF16 ? fmaxf(__uint_as_float(mw << 16), __uint_as_float(mw & 0xffff0000u)) : __uint_as_float(mw);
      if (!TONE) m = __fdiv_rn(m, P.T);           // division is monotone: the maximum of the quotients
      // a slice without any finite logit (padding, masked tokens) still needs a finite shift
      nd = ceilf(fmaxf(m, -1.0e37f) * L2E);
      const uint64_t nn2 = pack2(-nd, -nd);
      uint64_t t2 = 0;
      td = 0.0;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        uint64_t z2[4];
        raw8_pairs<BF16>(raw[c], z2);
        if (!TONE) divide_by_T(P, z2, fast_d);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float lo, hi;
          if (TOPK) {
            unpack2(z2[i], lo, hi);
            z2[i] = pack2(lo < tp ? ninf : lo, hi < tp ? ninf : hi);
          }
          unpack2(fma2(z2[i], L2, nn2), lo, hi);
          z2[i] = pack2(ex2_approx(lo), ex2_approx(hi));
        }
        const uint64_t s2 = add2(add2(z2[0], z2[1]), add2(z2[2], z2[3]));
        t2 = c % CP ? add2(t2, s2) : s2;
        if (c % CP == CP - 1) {
          float lo, hi;
          unpack2(t2, lo, hi);
          td += static_cast<double>(lo + hi);
        }
      }
    };
    // target: guidance combine, slice maximum, numerators, partial sum; E replaces the raw rows
    auto stream_target = [&](auto whole) {
      const unsigned char* rc = stage;
      const unsigned char* ru = stage + rowbytes;
      const uint64_t s2 = pack2(P.cfg_scale, P.cfg_scale);
#pragma unroll (NP > 2 ? 1 : NP)
      for (int p = 0; p < NP; ++p) {   // (rolled where there are many: three groups in different phases fill the instruction cache)
        uint64_t a2[CP * 4];
        float m = ninf;
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          const int g = (p * CP + c) * GT + gt;
          if (decltype(whole)::value || g * 8 < V) {
            uint64_t c2[4], u2[4];
            if (TOPK) {   // (processed already)
              const ulonglong2 ea = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8));
              const ulonglong2 eb = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8 + 4));
              c2[0] = ea.x, c2[1] = ea.y, c2[2] = eb.x, c2[3] = eb.y;
            } else {
              staged_pairs<BF16>(rc, g, c2);
              if (UNC) staged_pairs<BF16>(ru, g, u2);
            }
            if (UNC && !TOPK) {
#pragma unroll
              for (int i = 0; i < 4; ++i) c2[i] = fma2(s2, sub2(c2[i], u2[i]), u2[i]);   // l_u + s (l_c - l_u)
            }
            if (!TONE && !TOPK) divide_by_T(P, c2, P.T_fast != 0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint64_t l2 = c2[i];
              float lo, hi;
              unpack2(l2, lo, hi);
              if (TOPK) {   // (a NaN stays, to be reported)
                lo = lo < tq ? ninf : lo, hi = hi < tq ? ninf : hi;
                l2 = pack2(lo, hi);
              }
              a2[c * 4 + i] = l2;
              m = max3(m, lo, hi);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) a2[c * 4 + i] = pack2(ninf, ninf);
          }
        }
        if (GREEDY) z_max = fmaxf(z_max, m);
        const float n_p = ceilf(fmaxf(m, -1.0e37f) * L2E);
        const uint64_t nn2 = pack2(-n_p, -n_p);
        uint64_t t2 = pack2(0.0f, 0.0f);
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          uint64_t e2[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float lo, hi;
            unpack2(fma2(a2[c * 4 + i], L2, nn2), lo, hi);
            e2[i] = pack2(ex2_approx(lo), ex2_approx(hi));
          }
          t2 = add2(t2, add2(add2(e2[0], e2[1]), add2(e2[2], e2[3])));
          const int g = (p * CP + c) * GT + gt;
          if (decltype(whole)::value || g * 8 < V) {
            *reinterpret_cast<ulonglong2*>(E + EI(g * 8)) = make_ulonglong2(e2[0], e2[1]);
            *reinterpret_cast<ulonglong2*>(E + EI(g * 8 + 4)) = make_ulonglong2(e2[2], e2[3]);
          }
        }
        float lo, hi;
        unpack2(t2, lo, hi);
        S.slice[p * GT + gt] = n_p;
        if (NP <= 2) nq[NP <= 2 ? p : 0] = n_p, tq_sum[NP <= 2 ? p : 0] = lo + hi;
        else S.slice[1024 + p * GT + gt] = lo + hi;
      }
    };
    if (nchild > 0) {
      load_slots(xt, 0, nb);
      if (!GREEDY && gt < 2) fetch_single();
      if constexpr (!GREEDY) {
        if (full) load_drafter(std::true_type{});
        else load_drafter(std::false_type{});
      }
      if constexpr (TOPK && !TONE) {
        uint32_t least = ~0u;
#pragma unroll
        for (int c = 0; c < CH; ++c) least = least_magnitude<BF16>(raw[c], least);
        fast_d = fast_d && least >= P.T_least;
      }
      if constexpr (TOPK && !GREEDY) {   // the drafter row's threshold, from the registers that hold the row
        auto own = [&](int c, float (&z)[8]) {
          uint64_t z2[4];
          raw8_pairs<BF16>(raw[c], z2);
          if (!TONE) divide_by_T(P, z2, fast_d);
#pragma unroll
          for (int i = 0; i < 4; ++i) unpack2(z2[i], z[2 * i], z[2 * i + 1]);
        };
        auto again = [&](int c, float (&z)[8]) {
          row_logits<BF16, TONE>(P, P.draft, static_cast<size_t>(item) * V, c * GT + gt, z);
        };
        auto pairs = [&](int c, uint32_t (&w)[4]) { w[0] = raw[c].a.x, w[1] = raw[c].a.y, w[2] = raw[c].a.z, w[3] = raw[c].a.w; };
        if constexpr (BF16 && TONE) tp = group_kth_largest<SHAPE, CH, CH, true>(P, own, pairs, own, again, V, S, grp, gt, search3);
        else tp = group_kth_largest<SHAPE, CH, CH, false>(P, own, own, own, again, V, S, grp, gt, search3);
      }
      if (!GREEDY) reduce_drafter();
      if (!GREEDY && !TOPK && gt < 2) note_single();
    }
    // The target rows were issued when the staging area fell free; they arrive while the drafter
    // row is streamed.  Every thread waits for itself (bounded); a wait that runs out is reported after
    // the next group barrier, where every thread sees it alike.
    if (item >= 0) {
      if (!mbar_wait(&bar_rows[grp][area], (iter / AREAS) & 1, tries)) S.fail = 1;
      if constexpr (TOPK) {   // the target row's threshold; the processed logits replace the raw ones they came from
        auto guided_value = [&](int c, float (&z)[8], auto look) {
          const int g = c * GT + gt;
          uint64_t c2[4], u2[4];
          staged_pairs<BF16>(stage, g, c2);
          if (UNC) staged_pairs<BF16>(stage + rowbytes, g, u2);
          if (UNC) {
#pragma unroll
            for (int i = 0; i < 4; ++i) c2[i] = fma2(pack2(P.cfg_scale, P.cfg_scale), sub2(c2[i], u2[i]), u2[i]);
          }
          if (!TONE) divide_by_T(P, c2, P.T_fast != 0 && (!decltype(look)::value || quotients_fast(P, c2)));
#pragma unroll
          for (int i = 0; i < 4; ++i) unpack2(c2[i], z[2 * i], z[2 * i + 1]);
        };
        auto guided = [&](int c, float (&z)[8]) { guided_value(c, z, std::false_type{}); };   // (for the sample)
        auto guided_in_place = [&](int c, float (&z)[8]) {
          const int g = c * GT + gt;
          guided_value(c, z, std::true_type{});
          *reinterpret_cast<float4*>(E + EI(g * 8)) = make_float4(z[0], z[1], z[2], z[3]);
          *reinterpret_cast<float4*>(E + EI(g * 8 + 4)) = make_float4(z[4], z[5], z[6], z[7]);
        };
        auto processed = [&](int c, float (&z)[8]) {
          const int g = c * GT + gt;
          const float4 a = *reinterpret_cast<const float4*>(E + EI(g * 8));
          const float4 b = *reinterpret_cast<const float4*>(E + EI(g * 8 + 4));
          z[0] = a.x, z[1] = a.y, z[2] = a.z, z[3] = a.w, z[4] = b.x, z[5] = b.y, z[6] = b.z, z[7] = b.w;
        };
        tq = group_kth_largest<SHAPE, CH, (NP > 2 ? 2 : CH), false>(P, guided, guided_in_place, processed, processed, V, S, grp, gt, search3);
        if (!GREEDY && gt < 2 && nchild > 0) note_single();
      }
      if (full) stream_target(std::true_type{});
      else stream_target(std::false_type{});
    }

    // ---------------- group statistics ----------------
    // per warp: the largest shift and the sum in its units, for target and drafter; then one barrier, and every
    // warp combines the partials for itself (lane l: warp l % GW)
    {
      float n = shift_of(0);      // (without a context: what the last one left; nobody looks at it)
#pragma unroll
      for (int p = 1; p < NP; ++p) n = fmaxf(n, shift_of(p));
      const float wnq = redux_max(n), wnd = redux_max(GREEDY ? z_max : nd);   // (greedy decoding: the largest logit travels instead)
      const bool up = lane & 16;
      double sq = 0.0;            // (sums of up to 16 numerators are in single precision)
#pragma unroll
      for (int p = 0; p < NP; ++p) sq += static_cast<double>(sum_of(p) * exp2_int(shift_of(p) - wnq));
      const double z = warp_pair_sum(sq, GREEDY ? 0.0 : td * pow2_double(exp2_int(nd - wnd)), lane);
      if ((lane & 15) == 0) {
        S.wz[gw][up] = z;
        S.wn[gw][up] = up ? wnd : wnq;
      }
    }
    if (GREEDY && gt == 0) S.tok = kNone;
    gbar();   // E, the slices' shifts and the per-warp partials are visible
    if (S.fail) {   // no context was published, or its target rows did not land, within the limit
      give_up();
      break;
    }
    if (item < 0) break;
    // the producer may choose (and publish) the next context
    if (lane == 0) mbar_arrive(&bar_next[grp]);
    float Nq, Np;                // common units
    double Zq, Zp;
    {
      const float2 n = *reinterpret_cast<const float2*>(S.wn[lane & (GW - 1)]);
      const double2 z = *reinterpret_cast<const double2*>(S.wz[lane & (GW - 1)]);
      Nq = redux_max(n.x);
      Np = redux_max(n.y);
      Zq = z.x * static_cast<double>(exp2_int(n.x - Nq));
      Zp = GREEDY ? 1.0 / GW : z.y * static_cast<double>(exp2_int(n.y - Np));
#pragma unroll
      for (int o = GW / 2; o > 0; o >>= 1) {
        Zq += __shfl_xor_sync(kFull, Zq, o);
        Zp += __shfl_xor_sync(kFull, Zp, o);
      }
    }

    int status = 0;              // bits every thread sets alike
    int accepted = -1;
    bool drawn = false;
    // normalisers: q'(x) = E(x) * 2^(slice shift - Nq) / Zq_c, and p' likewise
    // (Zp_c = 0 stands for a drafter distribution that has no mass left).  Comparisons are written on
    // the unnormalised sums, so that no thread divides on the way to a decision.
    double Zq_c = Zq, Zp_c = Zp;
    if (!(Zq > 0.0 && Zq < 1e300 && Zp > 0.0 && Zp < 1e300)) {
      status |= LANTERN_ST_NONFINITE;
    } else {
      const double delta = static_cast<double>(P.delta);
      const ChildInfo* kids = P.children + cur.cbase;
      float r = cur.r0;
      StruckMask<CH> struck = 0;   // this thread's tokens that were rejected in this context: bit 8 c + e for token e of chunk c
      auto mass = [&](int n) { return E[EI(n)] * exp2_int(S.slice[owner_slice(n)] - Nq); };   // common units

      for (int ci = 0; ci < nchild; ++ci) {
        // the next sibling's description, wanted only after a rejection: in flight meanwhile
        int4 sib = make_int4(0, 0, 0, 0);
        if (ci + 1 < nchild) sib = *reinterpret_cast<const int4*>(kids + ci + 1);
        if (gt == 0) atomicAdd(&P.counters->n_tested, 1);   // work accounting (a fire-and-forget reduction)
        // The tested token's two numerators in common units, in double precision from its raw logits, carried
        // through every rejection round so far (E <- max(0, E - ratio_i * ep)); the sums they are compared
        // with are sums of thousands of terms and do not suffer from cancellation.  A token that has lost its
        // mass (it lay in an earlier A, or was itself rejected before) has none.  Every thread for itself behind the scan: by one warp, which
        // the others then waited for, it took 0.5 us of a context's 5.8 (wide shape), and 0.9 for a second sibling.  With the logit filter
        // the groups are bound by what they issue, and one warp does it ahead of the scan (4976 chains of 8192 tokens 1732 -> 1707 us,
        // 1619 trees 584 -> 575; 1024 chains of 16384 tokens and small calls the same).
        double e_xt = 0.0, p_xt = 0.0;
        // What the rejections so far have left of x~.  Read here, between the barrier that publishes the residual and the scan's: behind
        // the scan a warp that is ahead may have flagged it already.
        [[maybe_unused]] float bulk = 0.0f;
        if (!GREEDY && ci > 0 && (!TOPK || gw == 0)) bulk = mass(xt);
        [[maybe_unused]] auto numerators = [&]() {   // (by whole warps)
          const Exp2Split q = S.single[iter & 1][0], p = S.single[iter & 1][1];
          e_xt = q.y * exp2_int_d(q.n - static_cast<double>(Nq));
          p_xt = p.y * exp2_int_d(p.n - static_cast<double>(Np));
          if (ci > 0) {
            if (ci <= 32) {
              for (int i = 0; i < ci; ++i) e_xt = fmax(0.0, e_xt - S.hist[i] * p_xt);
              if (bulk == 0.0f) e_xt = 0.0;
            } else {
              e_xt = static_cast<double>(bulk);
            }
            bool again = false;
            for (int j = lane; j < ci; j += 32) again |= kids[j].token == xt;
            if (__any_sync(kFull, again)) p_xt = 0.0;
          }
        };
        if constexpr (!GREEDY && TOPK) {
          if (gw == 0) {
            numerators();
            if (lane == 0) S.tested[0] = e_xt, S.tested[1] = p_xt;
          }
        }

        // ---- A_{k,delta}(x~): gather + prefix scan with the strict bound ----
        double thr = delta * Zq_c;   // the bound in the units of the unnormalised sums
        // Section 5.3.2: the mass whose JSD is delta; the group's last warp finds it together.  (Two places: greedy decoding
        // goes on to the next sibling without a barrier, while slower warps may not have read this one's yet.)
        if (JSD && gw == GW - 1) {
          const double mine = jsd_mass_bound_warp(delta, static_cast<double>(mass(xt)) / Zq_c, lane) * Zq_c;
          if (lane == 0) S.jsd_mass[round2] = mine;
        }
        double carry = 0.0, sm = 0.0;
        int m = k - 1;
        bool cut = false;
        for (int base = 0; !cut && base < k; base += SLOTS * GT) {
          if (base > 0) load_slots(xt, base, nb);
          const int j0 = base + SLOTS * gt;
          double pre[SLOTS];    // inclusive prefix over this thread's slots
          double run = 0.0;
#pragma unroll
          for (int i = 0; i < SLOTS; ++i) {
            const int j = j0 + i, n = nb[i];
            if (j >= 1 && j < k) {
              if (static_cast<unsigned>(n) < static_cast<unsigned>(V)) run += static_cast<double>(mass(n));
              else atomicMin(&S.badslot[round3], j);   // carries no mass
            }
            pre[i] = run;
          }
          const double incl = warp_incl_scan(run, lane);
          if (lane == 31) S.wt[round2 * GW + gw] = incl;
          gbar();   // [scan 1]
          if (JSD && base == 0) thr = S.jsd_mass[round2];
          // every warp: running totals of the warps (lane l: warp l % GW), the first one that reaches the bound
          double tot = S.wt[round2 * GW + (lane & (GW - 1))];
#pragma unroll
          for (int o = 1; o < GW; o <<= 1) {
            const double t = __shfl_up_sync(kFull, tot, o);
            if ((lane & (GW - 1)) >= o) tot += t;
          }
          const unsigned over = __ballot_sync(kFull, !(carry + tot < thr));
          const int bad = S.badslot[round3];
          const int after = round3 < 2 ? round3 + 1 : 0, clear = after < 2 ? after + 1 : 0;
          if (gt == 0) S.badslot[clear] = kNone;   // last read before [scan 1], next written behind the next one
          const double carry_in = carry;
          round2 ^= 1;
          round3 = after;
          if (over == 0) {
            if (bad != kNone) status |= LANTERN_ST_BAD_TABLE;
            carry += __shfl_sync(kFull, tot, GW - 1);
            sm = carry;
          } else {
            cut = true;
            const int wc = __ffs(over) - 1;   // (the first GW lanes come first)
            if (gw == wc) {
              const double below = __shfl_sync(kFull, tot, (wc + GW - 1) & (GW - 1));
              const double before = carry_in + (wc > 0 ? below : 0.0) + (incl - run);   // prefix before this thread's first slot
              int first = kNone;
              double moved = 0.0;
#pragma unroll
              for (int i = SLOTS - 1; i >= 0; --i) {
                if (j0 + i >= 1 && j0 + i < k && !(before + pre[i] < thr)) {
                  first = j0 + i;
                  moved = i > 0 ? before + pre[i > 0 ? i - 1 : 0] : before;
                }
              }
              const unsigned who = __ballot_sync(kFull, first != kNone);
              if (who ? lane == __ffs(who) - 1 : lane == 31) {
                // (no slot: the total reached the bound by rounding alone; the set ends with this warp's slots)
                S.cut_m = who ? first - 1 : min(j0 + SLOTS - 1, k - 1);
                S.cut_sum = who ? moved : before + run;
              }
            }
            gbar();   // [scan 2]
            m = S.cut_m;
            sm = S.cut_sum;
            // a bad entry is reported where Algorithm 2's loop meets it, i.e. ahead of the slot that ends the set
            if (bad <= m) status |= LANTERN_ST_BAD_TABLE;
          }
        }
        if constexpr (!GREEDY && !TOPK) numerators();
        if constexpr (!GREEDY && TOPK) e_xt = S.tested[0], p_xt = S.tested[1];
        // Section 4.3: accept iff r p(x~) < sum_A q, i.e. r p_xt / Zp_c < (e_xt + sm) / Zq_c, both sides times Zq_c Zp_c
        // (greedy decoding: x~ itself as every other numerator, so that the largest one compares equal to itself)
        const double qa_un = (GREEDY ? static_cast<double>(mass(xt)) : e_xt) + sm;
        const bool accept = GREEDY ? qa_un >= static_cast<double>(ex2_approx(__fmaf_rn(Np, L2E, -Nq)))
                            : Zp_c > 0.0 ? static_cast<double>(r) * p_xt * Zq_c < qa_un * Zp_c : 0.0 < qa_un;
        if (gt == 0 && (P.out_qa || P.out_px || P.out_m)) {
          const size_t o = static_cast<size_t>(item / R) * N + node;
          if (P.out_qa) P.out_qa[o] = static_cast<float>(qa_un / Zq_c);
          if (P.out_px) P.out_px[o] = Zp_c > 0.0 ? static_cast<float>(p_xt / Zp_c) : 0.0f;
          if (P.out_m) P.out_m[o] = m;
        }
        if (accept) {
          accepted = node;
          break;
        }
        if constexpr (GREEDY) {
          if (ci + 1 < nchild) {
            node = sib.x;
            xt = sib.y;
            load_slots(xt, 0, nb);
          }
          continue;
        } else {
        // ---- rejected: residual [q_{k,delta}(.|D = x~) - p]_+ ----
        // the first drafter logits: asked for at once, in flight while A is flagged and across the barrier
        Raw8<BF16> ahead[AHEAD];
        if (!HOLD) {
#pragma unroll
          for (int c = 0; c < AHEAD; ++c) {
            const int g = c * GT + gt;
            ahead[c] = load_raw8<BF16>(drow, g * 8 < V ? g : 0);
          }
        }
        // members of A (x~ included) leave no residual mass: flag them with a negative sign
        for (int base = 0; base <= m; base += SLOTS * GT) {
          if (base > 0 || m >= SLOTS * GT - 1) load_slots(xt, base, nb);   // (a longer scan has replaced the first slots)
#pragma unroll
          for (int i = 0; i < SLOTS; ++i) {
            const int j = base + SLOTS * gt + i;
            if (j >= 1 && j <= m && static_cast<unsigned>(nb[i]) < static_cast<unsigned>(V)) E[EI(nb[i])] = -fabsf(E[EI(nb[i])]);
          }
        }
        if (gt == 0) E[EI(xt)] = -fabsf(E[EI(xt)]);
        // x~ leaves the drafter distribution for the following siblings: the residual pass below strikes
        // every token rejected so far (children 0..ci) from the drafter logits
        if (((xt >> 3) & (GT - 1)) == gt) struck |= StruckMask<CH>(1) << ((xt >> (3 + LOG_GT)) * 8 + (xt & 7));
        const bool last = (ci + 1 == nchild);
        if (!last) {   // next sibling's neighbour row and raw logits, in flight during the residual pass
          node = sib.x;
          xt = sib.y;
          r = __int_as_float(sib.z);
          load_slots(xt, 0, nb);
          if (gt < 2) fetch_single();
        }
        gbar();   // [flags]
        // w = E - (p'/q' scale ratio) * ep in common units, i.e. E - ratio * ep in the slice's own units
        // of E; the residual replaces E (it is the next sibling's target, or what the draw reads)
        const float ratio_g = Zp_c > 0.0 ? static_cast<float>(Zq_c / Zp_c) : 0.0f;
        const float fd = exp2_int(nd - Np);   // this thread's drafter units -> common units
        double wsum = 0.0, psum = 0.0;        // common units; the thread's own units
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          // (a slice whose numerators are all negligible has factor 0; nothing of it survives anyway)
          const float fq = exp2_int(shift_of(p) - Nq);
          const float ratio = fq > 0.0f ? ratio_g * (fd / fq) : 0.0f;
          const uint64_t nr2 = pack2(-ratio, -ratio), nn2 = pack2(-nd, -nd);
          float w_p = 0.0f, p_p = 0.0f;       // the slice's part of either sum
#pragma unroll
          for (int c = p * CP; c < (p + 1) * CP; ++c) {
            const Raw8<BF16> drafted = HOLD ? raw[c] : ahead[c % AHEAD];
            if (!HOLD && c + AHEAD < CH) {   // the next groups travel during this one
              const int g = (c + AHEAD) * GT + gt;
              ahead[c % AHEAD] = load_raw8<BF16>(drow, g * 8 < V ? g : 0);
            }
            const int g = c * GT + gt;
            if (full || g * 8 < V) {
              float z[8];
              {
                uint64_t z2[4];
                raw8_pairs<BF16>(drafted, z2);
                if (!TONE) divide_by_T(P, z2, fast_d);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  unpack2(z2[i], z[2 * i], z[2 * i + 1]);
                  if (TOPK) {
                    z[2 * i] = z[2 * i] < tp ? ninf : z[2 * i];
                    z[2 * i + 1] = z[2 * i + 1] < tp ? ninf : z[2 * i + 1];
                  }
                }
              }
              if (const uint32_t gone = static_cast<uint32_t>(struck >> (8 * c)) & 0xffu) {   // tokens rejected in this context
#pragma unroll
                for (int e = 0; e < 8; ++e) z[e] = (gone >> e) & 1u ? ninf : z[e];
              }
              const ulonglong2 ea = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8));
              const ulonglong2 eb = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8 + 4));
              const uint64_t e2[4] = {ea.x, ea.y, eb.x, eb.y};
              uint64_t w2[4], ps2 = pack2(0.0f, 0.0f);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                float lo, hi;
                unpack2(fma2(pack2(z[2 * i], z[2 * i + 1]), L2, nn2), lo, hi);
                const uint64_t ep = pack2(ex2_approx(lo), ex2_approx(hi));
                ps2 = add2(ps2, ep);
                unpack2(fma2(nr2, ep, e2[i]), lo, hi);
                w2[i] = pack2(fmaxf(0.0f, lo), fmaxf(0.0f, hi));
              }
              *reinterpret_cast<ulonglong2*>(E + EI(g * 8)) = make_ulonglong2(w2[0], w2[1]);
              *reinterpret_cast<ulonglong2*>(E + EI(g * 8 + 4)) = make_ulonglong2(w2[2], w2[3]);
              float lo, hi;
              unpack2(ps2, lo, hi);
              p_p += lo + hi;
              unpack2(add2(add2(w2[0], w2[1]), add2(w2[2], w2[3])), lo, hi);
              w_p += lo + hi;
            }
          }
          if (!last) wsum += static_cast<double>(w_p * fq), psum += static_cast<double>(p_p);
        }
        if (last) break;   // the draw below takes it from here
        const double z = warp_pair_sum(wsum, psum * pow2_double(fd), lane);
        if ((lane & 15) == 0) S.wz[gw][lane >> 4] = z;
        if (gt < 2) note_single();
        if (gt == 0 && ci < 32) S.hist[ci] = static_cast<double>(ratio_g);
        gbar();   // [totals] also publishes the written-back residual
        const double2 z2 = *reinterpret_cast<const double2*>(S.wz[lane & (GW - 1)]);
        double W = z2.x, Sp = z2.y;
#pragma unroll
        for (int o = GW / 2; o > 0; o >>= 1) {
          W += __shfl_xor_sync(kFull, W, o);
          Sp += __shfl_xor_sync(kFull, Sp, o);
        }
        if (!(W > kDegenerate * Zq_c)) {
          status |= LANTERN_ST_DEGENERATE;
          break;
        }
        Zq_c = W;
        Zp_c = Sp > 0.0 ? Sp : 0.0;
        }
      }

      if constexpr (GREEDY) {   // arg max q, smallest index on ties, from the logits themselves
        if (accepted < 0) {
          if (z_max == Np) {
            int first = kNone;
#pragma unroll 1
            for (int c = CH - 1; c >= 0; --c) {
              const int g = c * GT + gt;
              if (g * 8 < V) {
                const unsigned char* row = static_cast<const unsigned char*>(P.target) + static_cast<size_t>(item) * rowbytes;
                uint64_t c2[4], u2[4];
                raw8_pairs<BF16>(load_raw8<BF16>(row, g), c2);
                if (UNC) raw8_pairs<BF16>(load_raw8<BF16>(row + static_cast<size_t>(P.B) * R * rowbytes, g), u2);
#pragma unroll
                for (int i = 3; i >= 0; --i) {
                  float lo, hi;
                  unpack2(UNC ? fma2(pack2(P.cfg_scale, P.cfg_scale), sub2(c2[i], u2[i]), u2[i]) : c2[i], lo, hi);
                  if (hi == Np) first = g * 8 + 2 * i + 1;
                  if (lo == Np) first = g * 8 + 2 * i;
                }
              }
            }
            if (first != kNone) atomicMin(&S.tok, first);
          }
          gbar();
          drawn = true;
          if (gt == 0) S.result[iter & 1] = {-1, S.tok, status};
        }
      }
      // ---- the draw, by inverse CDF over E in token order: the replacement token from the residual where the last
      // child was rejected (Algorithm 1), the bonus token from q itself where there are no children ----
      if constexpr (!GREEDY) if (accepted < 0 && !(status & LANTERN_ST_DEGENERATE)) {
        {
          float cs[CH];        // weight of each of this thread's chunks, common units
#pragma unroll
          for (int c = 0; c < CH; ++c) {
            const int g = c * GT + gt;
            cs[c] = 0.0f;
            if (full || g * 8 < V) {
              const ulonglong2 ea = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8));
              const ulonglong2 eb = *reinterpret_cast<const ulonglong2*>(E + EI(g * 8 + 4));
              float lo, hi;
              unpack2(add2(add2(ea.x, ea.y), add2(eb.x, eb.y)), lo, hi);
              cs[c] = (lo + hi) * exp2_int(shift_of(c / CP) - Nq);
            }
          }
          const double t = warp_transposed_sum<CH>(cs, lane);
          if ((lane & (32 / CH - 1)) == 0) S.wt[(lane / (32 / CH)) * GW + gw] = t;
          if (gt == 0) S.tok = -1;
        }
        gbar();   // [draw 1] totals of the (chunk, warp) blocks, in token order chunk by chunk
        double before, W;
        int blk;
        {
          // every warp: the block in which the cumulative weight first exceeds the target (two blocks per lane)
          const double t0 = 2 * lane < CH * GW ? S.wt[2 * lane] : 0.0, t1 = 2 * lane < CH * GW ? S.wt[2 * lane + 1] : 0.0;
          const double incl = warp_incl_scan(t0 + t1, lane);
          W = __shfl_sync(kFull, incl, 31);
          const double target = static_cast<double>(cur.u_final) * W;
          const unsigned over = __ballot_sync(kFull, incl > target);
          const double ex = incl - (t0 + t1);
          const bool second = !(ex + t0 > target);
          blk = over ? __shfl_sync(kFull, 2 * lane + (second ? 1 : 0), __ffs(over) - 1) : -1;
          before = __shfl_sync(kFull, second ? ex + t0 : ex, over ? __ffs(over) - 1 : 0);
        }
        const double target = static_cast<double>(cur.u_final) * W;
        if (!(W > kDegenerate * Zq_c)) {
          status |= LANTERN_ST_DEGENERATE;
        } else if (blk < 0) {
          // rounding left no block above the target: the largest token of positive weight
          int lastp = -1;
          for (int c = 0; c < CH; ++c) {
            const int g = c * GT + gt;
            if (g * 8 < V)
              for (int e = 0; e < 8; ++e)
                if (E[EI(g * 8 + e)] > 0.0f) lastp = g * 8 + e;
          }
          if (lastp >= 0) atomicMax(&S.tok, lastp);
          gbar();
          drawn = true;
          if (gt == 0) S.result[iter & 1] = {-1, S.tok, status | (S.tok < 0 ? LANTERN_ST_DEGENERATE : 0)};
        } else {
          drawn = true;
          if ((blk & (GW - 1)) == gw) {   // the block's own warp: the thread, then the token
            const int c = blk / GW, g = c * GT + gt;
            float w8[8] = {};
            float fq = 0.0f;
            if (g * 8 < V) {
              const float4 a = *reinterpret_cast<const float4*>(E + EI(g * 8));
              const float4 b = *reinterpret_cast<const float4*>(E + EI(g * 8 + 4));
              w8[0] = a.x, w8[1] = a.y, w8[2] = a.z, w8[3] = a.w, w8[4] = b.x, w8[5] = b.y, w8[6] = b.z, w8[7] = b.w;
              fq = exp2_int(S.slice[(c / CP) * GT + gt] - Nq);
            }
            const double mine = static_cast<double>(sum8(w8) * fq);
            const double incl = warp_incl_scan(mine, lane);
            const unsigned over = __ballot_sync(kFull, before + incl > target);
            const unsigned some = __ballot_sync(kFull, mine > 0.0);
            const int who = over ? __ffs(over) - 1 : 31 - __clz(some);   // (rounding: its last thread with weight)
            if (lane == who) {
              int tok = -1, lastpos = -1;
              double cum = before + (incl - mine);
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                cum += static_cast<double>(w8[e]) * static_cast<double>(fq);
                if (w8[e] > 0.0f) lastpos = e;
                if (tok < 0 && cum > target) tok = e;
              }
              if (tok < 0) tok = lastpos;
              S.result[iter & 1] = {-1, g * 8 + tok, status};
            }
          }
        }
      }
    }
    if (!drawn && gt == 0) S.result[iter & 1] = {accepted, -1, status};
    // this context's staging area (rows and E) is no longer needed by this warp, and its result is there
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar_done[grp][iter & 1]);
  }
}

}  // namespace lantern
