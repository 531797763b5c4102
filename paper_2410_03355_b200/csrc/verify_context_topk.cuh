// Top-k threshold of one row of a context (Appendix B.2: logits below the K-th largest of their row count as -inf; ties at
// that value are kept).  Included by verify_context.cuh.
//
// Found by the group that holds the row, on processed logits (guidance combine, temperature) with exactly the roundings of
// the streaming part.  Exact in the end; the sample only decides where to look:
//   1. four values per thread, spread over the row, go into a histogram of 128 bins between the smallest and
//      the largest of them; two bin edges whose sample ranks lie three standard deviations to either side of the rank
//      the K-th largest is expected to have give a bracket [lo, hi);
//   2. every thread goes over its values twice: it counts those >= hi and those inside the bracket, and, knowing its place by
//      one counter update per warp, puts the latter on a list;
//   3. if the K-th largest does lie in [lo, hi) -- count(>= hi) < K <= count(>= lo) -- the listed values go into a histogram of 256
//      bins over the bracket, every warp finds the bin that holds the wanted rank by a suffix scan of its own, and ranks
//      the handful of values of that bin; a crowded bin (ties) is left to one warp, which searches the
//      list by two pivots per pass, set where the rank should lie if the values were spread evenly;
//   4. otherwise (a sample that misleads, a list too long: ties, or a mask value that stretches the sample's range) by a radix
//      search on the order-preserving bit patterns: the patterns' range, a histogram of 256 bins over it, on with the bin that holds
//      the wanted rank.  Two passes over the row a round; a round takes eight bits off the range, which is exact after four.
//      lantern_verify_counts reports how many rows needed it.
#pragma once

#include <cuda_bf16.h>

namespace lantern {

// order-preserving bit pattern of a processed logit: NaN lowest, -0 as +0
__device__ __forceinline__ uint32_t topk_order(float z) {
  if (z != z) return 0u;
  if (z == 0.0f) z = 0.0f;
  const uint32_t u = __float_as_uint(z);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float topk_from_order(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}
constexpr uint32_t TOPK_ORDER_NINF = 0x007fffffu;
// Logits of and below this are taken for masks (-1e4, -1e9, the type's lowest value): they do not stretch the range of the sample's bins.
// (Half of the tokens masked by -1e9, 300 chains: 558 us per call with them, all rows going to step 4.)  The result does not
// depend on it.
constexpr float TOPK_MASK = -4096.0f;

// eight processed logits of 16-byte group g of a row in global memory (no guidance)
template <bool BF16, bool TONE>
__device__ __forceinline__ void row_logits(const VerifyParams& P, const void* base, size_t row, int g, float (&z)[8]) {
  const size_t elem = row + static_cast<size_t>(g) * 8;
  if (BF16) {
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(static_cast<const unsigned short*>(base) + elem));
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      z[2 * q] = __uint_as_float(w[q] << 16);
      z[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
    }
  } else {
    const float4 a = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(base) + elem));
    const float4 b = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(base) + elem) + 1);
    z[0] = a.x, z[1] = a.y, z[2] = a.z, z[3] = a.w, z[4] = b.x, z[5] = b.y, z[6] = b.z, z[7] = b.w;
  }
  if (!TONE) {
#pragma unroll
    for (int e = 0; e < 8; ++e) z[e] = __fdiv_rn(z[e], P.T);
  }
}

// The two inner steps of the sweeps, predicated: only every twentieth value ends up on the list (1024 chains, K = 1000: 523 us
// per call as C++ conditions, 506 like this).
// n += z >= t
__device__ __forceinline__ void topk_count(int& n, float z, float t) {
  asm("{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %1, %2;\n\t@p add.s32 %0, %0, 1;\n\t}" : "+r"(n) : "f"(z), "f"(t));
}
// *to++ = z if lo <= z < hi (to: an address in shared memory)
__device__ __forceinline__ void topk_append(uint32_t& to, float z, float lo, float hi) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ge.f32 p, %1, %2;\n\t"
      "setp.lt.and.f32 p, %1, %3, p;\n\t"
      "@p st.shared.f32 [%0], %1;\n\t"
      "@p add.u32 %0, %0, 4;\n\t}"
      : "+r"(to)
      : "f"(z), "f"(lo), "f"(hi)
      : "memory");
}

// the smallest bf16 value >= x
__device__ __forceinline__ float topk_bf16_up(float x) {
  const uint32_t u = __float_as_uint(x);
  return __uint_as_float((u & 0x80000000u ? u : u + 0xffffu) & 0xffff0000u);
}

// Step 3, by one warp: the rank-th largest of the n values in `list` (1 <= rank <= n, no NaN).
__device__ __forceinline__ float topk_listed(const float* list, int n, int rank, int lane) {
  const float pinf = __int_as_float(0x7f800000), ninf = __int_as_float(0xff800000);
  float vmin = pinf, vmax = ninf;
  for (int i = lane; i < n; i += 32) {
    const float v = list[i];
    vmin = fminf(vmin, v);
    vmax = fmaxf(vmax, v);
  }
  uint32_t L = __reduce_min_sync(kFull, topk_order(vmin)), H = __reduce_max_sync(kFull, topk_order(vmax)) + 1u;
  int cL = n, cH = 0;                       // count(>= L) >= rank > count(>= H), on order-preserving bit patterns
  bool even = true;                         // the last pass took enough away: go on with interpolation
  for (int pass = 0; pass < 64 && H - L > 1u && cL > rank && cH < rank - 1; ++pass) {
    uint32_t p1, p2;                        // L < p1 <= p2 < H
    p1 = p2 = L + ((H - L) >> 1);
    if (even) {
      const float a = topk_from_order(L), b = topk_from_order(H - 1u);
      const float in = static_cast<float>(cL - cH), pos = (static_cast<float>(rank - cH) - 0.5f) / in;   // from the top
      const float half = 0.8f / sqrtf(in);
      const uint32_t q1 = topk_order(b - (b - a) * fminf(pos + half, 1.0f)), q2 = topk_order(b - (b - a) * fmaxf(pos - half, 0.0f));
      if (q1 > L && q1 < H) p1 = q1;
      if (q2 > L && q2 < H) p2 = q2;
      if (p1 > p2) p1 = p2;
    }
    const float v1 = topk_from_order(p1), v2 = topk_from_order(p2);
    int c1 = 0, c2 = 0;
    for (int i = lane; i < n; i += 32) {
      const float v = list[i];
      c1 += v >= v1;
      c2 += v >= v2;
    }
    const int both = __reduce_add_sync(kFull, (c1 << 16) | c2);
    c1 = both >> 16, c2 = both & 0xffff;
    const int before = cL - cH;
    if (c2 >= rank) {
      L = p2, cL = c2;
    } else if (c1 >= rank) {
      L = p1, cL = c1, H = p2, cH = c2;
    } else {
      H = p1, cH = c1;
    }
    even = 2 * (cL - cH) <= before;
  }
  // the answer is the smallest value >= L where exactly `rank` values are, the largest below H where rank - 1 are not below
  // it, and L itself where the interval has closed
  const float vL = topk_from_order(L), vH = topk_from_order(H);
  uint32_t up = 0xffffffffu, down = 0u;
  for (int i = lane; i < n; i += 32) {
    const float v = list[i];
    const uint32_t key = topk_order(v);
    if (v >= vL) up = key < up ? key : up;
    if (H == 0xff800001u || v < vH) down = key > down ? key : down;
  }
  up = __reduce_min_sync(kFull, up);
  down = __reduce_max_sync(kFull, down);
  return topk_from_order(cL == rank ? up : (cH == rank - 1 ? down : L));
}

// The bin of a histogram of TOPK_FINE bins that holds the want-th largest value, its rank inside that bin (from the top) and the
// bin's population; every warp for itself.  False if there are fewer values.
__device__ __forceinline__ bool topk_find_bin(const int (&fine)[TOPK_FINE], int want, int lane, int& bin, int& rank, int& pop) {
  constexpr int PER = TOPK_FINE / 32;
  int h[PER];
#pragma unroll
  for (int q = 0; q < PER; q += 4) {
    const int4 v = *reinterpret_cast<const int4*>(&fine[lane * PER + q]);
    h[q] = v.x, h[q + 1] = v.y, h[q + 2] = v.z, h[q + 3] = v.w;
  }
  int mine = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) mine += h[q];
  int incl = mine;                                     // suffix sum over the lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(kFull, incl, o);
    if (lane + o < 32) incl += v;
  }
  int above = incl - mine, b = 0, r = 0, p = 0;
  const bool holds = above < want && want <= incl;     // one lane at most
#pragma unroll
  for (int q = PER - 1; q >= 0; --q) {
    if (holds && r == 0 && above + h[q] >= want) b = lane * PER + q, r = want - above, p = h[q];
    above += h[q];
  }
  const unsigned who = __ballot_sync(kFull, holds);
  const int src = who ? __ffs(who) - 1 : 0;
  bin = __shfl_sync(kFull, b, src);
  rank = __shfl_sync(kFull, r, src);
  pop = __shfl_sync(kFull, p, src);
  return who != 0;
}

// The K-th largest processed logit of a row (0 < K < V); every thread of the group calls it and gets the same value.
// The callables give the eight values of this thread's chunk c: for the sample, for the first and the second sweep (loops
// unrolled UNROLL times), and for the slow path (in a rolled loop).  PAIRS: the first sweep is given the values as pairs of
// bf16, which they are then exactly, and counts two at a time.  search3 = searches of this group so far, mod 3: its list
// counter is zero on entry, and the one after the next is cleared here.
template <class SHAPE, int CH, int UNROLL, bool PAIRS, class Z0, class Z1, class Z2, class Z3, class SH>
__device__ __forceinline__ float group_kth_largest(const VerifyParams& P, Z0& sampled, Z1& first, Z2& second, Z3& slow, int V, SH& S,
                                                   int grp, int gt, int& search3) {
  constexpr int GT = SHAPE::GT, GW = GT / 32;
  const float pinf = __int_as_float(0x7f800000), ninf = __int_as_float(0xff800000);
  auto gbar = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(GT) : "memory"); };
  auto& T = S.tk;
  float* list = S.slice;
  const int K = P.top_k, gw = gt >> 5, lane = gt & 31;
  auto here = [&](int c) { return (c * GT + gt) * 8 < V; };
  // ---- 1. ----
  float smp[4];
  constexpr int FROM = CH < 4 ? CH : 4;               // chunks the sample is taken from, 4 / FROM values of each
#pragma unroll
  for (int q = 0; q < FROM; ++q) {
    const int c = q * (CH / FROM);
    float z[8];
    const bool on = here(c);
    if (on) sampled(c, z);
#pragma unroll
    for (int e = 0; e < 4 / FROM; ++e) smp[q * (4 / FROM) + e] = on ? z[e * (2 * FROM)] : __int_as_float(0x7fc00000);
  }
  float vmin = pinf, vmax = ninf;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (smp[q] > TOPK_MASK) vmin = fminf(vmin, smp[q]);
    vmax = fmaxf(vmax, smp[q]);                        // (a NaN is passed over)
  }
  vmin = -redux_max(-vmin);
  vmax = redux_max(vmax);
  if (lane == 0) T.range[gw][0] = vmin, T.range[gw][1] = vmax;
  gbar();
  vmin = -redux_max(lane < GW ? -T.range[lane][0] : ninf);
  vmax = redux_max(lane < GW ? T.range[lane][1] : ninf);
  if (!(vmin <= vmax)) vmin = vmax;                    // (nothing but masks)
  const float width = (vmax - vmin) * (1.0f / TOPK_BINS);
  const float scale = width > 0.0f && width < pinf ? 1.0f / width : 0.0f;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (smp[q] == smp[q]) atomicAdd(&T.hist[min(static_cast<int>(fmaxf((smp[q] - vmin) * scale, 0.0f)), TOPK_BINS - 1)], 1);
  gbar();
  float lo = ninf, hi = pinf;
  {
    constexpr int PER = TOPK_BINS / 32;
    static_assert(PER == 4, "a lane reads four bins");
    const int4 h = *reinterpret_cast<const int4*>(&T.hist[lane * PER]);
    int incl = h.x + h.y + h.z + h.w;                  // suffix sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_down_sync(kFull, incl, o);
      if (lane + o < 32) incl += v;
    }
    const int s0 = incl, s1 = s0 - h.x, s2 = s1 - h.y, s3 = s2 - h.z;   // sample values in this bin and above
    const float ns = static_cast<float>(__shfl_sync(kFull, incl, 0)), share = static_cast<float>(K) / static_cast<float>(V);
    const float mean = share * ns, sd = sqrtf(mean * (1.0f - share));
    const int r_hi = static_cast<int>(floorf(mean - 3.0f * sd)) - 1, r_lo = static_cast<int>(mean + 3.0f * sd) + 2;
    const int over = (s0 > r_hi) + (s1 > r_hi) + (s2 > r_hi) + (s3 > r_hi);
    const int cover = (s0 >= r_lo) + (s1 >= r_lo) + (s2 >= r_lo) + (s3 >= r_lo);
    const int both = __reduce_add_sync(kFull, over << 16 | cover);
    const int b_hi = both >> 16, b_lo = (both & 0xffff) - 1;
    if (r_hi >= 0 && b_hi < TOPK_BINS) hi = vmin + width * static_cast<float>(b_hi);
    if (b_lo > 0) lo = vmin + width * static_cast<float>(b_lo);
  }
  // ---- 2. ----
  int c_hi = 0, n_in = 0;
  if constexpr (PAIRS) {
    // against the next bf16 value from each edge on, which leaves the same values inside; at most 32 to a half word, so the
    // counts are exact (1024 chains 506 -> 495 us per call)
    lo = topk_bf16_up(lo), hi = topk_bf16_up(hi);
    const __nv_bfloat162 lo2 = __float2bfloat162_rn(lo), hi2 = __float2bfloat162_rn(hi);
    __nv_bfloat162 n_hi = __float2bfloat162_rn(0.0f), n_lo = n_hi;
#pragma unroll UNROLL
    for (int c = 0; c < CH; ++c) {
      if (here(c)) {
        uint32_t w[4];
        first(c, w);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __nv_bfloat162 z = *reinterpret_cast<const __nv_bfloat162*>(&w[e]);
          n_hi = __hadd2(n_hi, __hge2(z, hi2));
          n_lo = __hadd2(n_lo, __hge2(z, lo2));
        }
      }
    }
    c_hi = static_cast<int>(__low2float(n_hi) + __high2float(n_hi));
    n_in = static_cast<int>(__low2float(n_lo) + __high2float(n_lo));
  } else {
#pragma unroll UNROLL
    for (int c = 0; c < CH; ++c) {
      if (here(c)) {
        float z[8];
        first(c, z);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          topk_count(c_hi, z[e], hi);
          topk_count(n_in, z[e], lo);
        }
      }
    }
  }
  n_in -= c_hi;
  {
    int incl = n_in;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    int start = 0;
    if (lane == 31) start = atomicAdd(&T.listed[search3], incl);
    int pos = __shfl_sync(kFull, start, 31) + incl - n_in;
    if (lane == 31) T.count[gw][1] = incl;
    const bool room = __all_sync(kFull, pos + n_in <= TOPK_LIST);
    if (room) {
      uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(list + pos));
#pragma unroll UNROLL
      for (int c = 0; c < CH; ++c) {
        if (here(c)) {
          float z[8];
          second(c, z);
#pragma unroll
          for (int e = 0; e < 8; ++e) topk_append(to, z[e], lo, hi);
        }
      }
    }
  }
  const int w_hi = __reduce_add_sync(kFull, c_hi);
  if (lane == 0) T.count[gw][0] = w_hi;
  gbar();
  c_hi = __reduce_add_sync(kFull, lane < GW ? T.count[lane][0] : 0);
  const int c_in = __reduce_add_sync(kFull, lane < GW ? T.count[lane][1] : 0);
  const int now = search3;
  search3 = now < 2 ? now + 1 : 0;
  if (gt == 0) T.listed[now > 0 ? now - 1 : 2] = T.picked[now > 0 ? now - 1 : 2] = 0;   // (the one before the current one comes after the next)
  if (gt < TOPK_BINS) T.hist[gt] = 0;                 // everybody has read it
  if (c_in <= TOPK_LIST && c_hi < K && K <= c_hi + c_in) {
    // ---- 3. ----
    const float f_lo = lo > ninf ? lo : vmin, f_hi = hi < pinf ? hi : vmax;
    const float f_scale = f_hi > f_lo ? static_cast<float>(TOPK_FINE) / (f_hi - f_lo) : 0.0f;
    auto bin_of = [&](float v) { return min(static_cast<int>(fmaxf((v - f_lo) * f_scale, 0.0f)), TOPK_FINE - 1); };
    for (int i = gt; i < c_in; i += GT) atomicAdd(&T.fine[bin_of(list[i])], 1);
    gbar();
    int bin, rank, pop;
    topk_find_bin(T.fine, K - c_hi, lane, bin, rank, pop);   // 1 <= K - c_hi <= c_in
    if (pop <= TOPK_TINY) {
      for (int i = gt; i < c_in; i += GT) {
        const float v = list[i];
        if (bin_of(v) == bin) T.tiny[atomicAdd(&T.picked[now], 1)] = v;
      }
    } else if (gw == 0) {
      const float t = topk_listed(list, c_in, K - c_hi, lane);
      if (lane == 0) T.threshold = t;
    }
    gbar();
    for (int q = gt; q < TOPK_FINE; q += GT) T.fine[q] = 0;
    if (pop > TOPK_TINY) return T.threshold;
    // lane l holds the bin's l-th value; the wanted one has fewer than `rank` values above it and at least `rank` not below
    // it (equal values give the same answer)
    const float v = lane < pop ? T.tiny[lane] : ninf;
    int gtr = 0, geq = 0;
    for (int j = 0; j < pop; ++j) {
      const float o = __shfl_sync(kFull, v, j);
      gtr += o > v;
      geq += o >= v;
    }
    return __shfl_sync(kFull, v, __ffs(__ballot_sync(kFull, lane < pop && gtr < rank && rank <= geq)) - 1);
  }
  // ---- 4.  (If fewer than K values lie above -inf the answer is -inf: nothing is cut.) ----
  if (gt == 0) atomicAdd(&P.counters->n_slow_topk, 1);
  uint32_t L = TOPK_ORDER_NINF + 1u, H = 0xff800000u;   // the wanted pattern lies in [L, H]: just above -inf .. +inf
  auto each_key = [&](auto take) {
#pragma unroll 1
    for (int c = 0; c < CH; ++c) {
      if (here(c)) {
        float z[8];
        slow(c, z);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t key = topk_order(z[e]);
          if (key >= L && key <= H) take(key);
        }
      }
    }
  };
  int want = K;
#pragma unroll 1
  for (int round = 0; round < 5; ++round) {
    uint32_t least = 0xffffffffu, most = 0u;
    each_key([&](uint32_t key) {
      least = key < least ? key : least;
      most = key > most ? key : most;
    });
    least = __reduce_min_sync(kFull, least);
    most = __reduce_max_sync(kFull, most);
    gbar();                                             // the previous readers of count[] and of fine[] are done
    if (lane == 0) T.count[gw][0] = static_cast<int>(least), T.count[gw][1] = static_cast<int>(most);
    if (round > 0)
      for (int q = gt; q < TOPK_FINE; q += GT) T.fine[q] = 0;
    gbar();
    L = __reduce_min_sync(kFull, lane < GW ? static_cast<uint32_t>(T.count[lane][0]) : 0xffffffffu);
    H = __reduce_max_sync(kFull, lane < GW ? static_cast<uint32_t>(T.count[lane][1]) : 0u);
    if (L > H) break;                                   // no value above -inf
    const int shift = max(0, 24 - __clz(H - L));
    each_key([&](uint32_t key) { atomicAdd(&T.fine[(key - L) >> shift], 1); });
    gbar();
    int bin, rank, pop;
    const bool found = topk_find_bin(T.fine, want, lane, bin, rank, pop);
    L = found ? L + (static_cast<uint32_t>(bin) << shift) : TOPK_ORDER_NINF;
    if (!found || shift == 0) {
      H = L;
      break;
    }
    H = min(H, L + ((1u << shift) - 1u));
    want = rank;
  }
  gbar();                                               // fine[] and count[] are free again
  for (int q = gt; q < TOPK_FINE; q += GT) T.fine[q] = 0;
  return L == H ? topk_from_order(L) : ninf;
}

}  // namespace lantern
