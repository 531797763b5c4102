// Neighbour table B_k of a VQ codebook (Algorithm 2, block "Precompute B_k for all tokens").
//
// Key of a pair (i, j): squared l2 distance accumulated in fp32 in dimension order,
// acc = fma(a_d - b_d, a_d - b_d, acc).  That exact operation sequence is kept whatever the
// tiling, so the order of neighbours does not depend on how the work is split.
//
// Small D (<= 32): a CTA takes R codes (rows of the table) at once and computes their keys against the
// whole codebook, two rows to a packed fp32 instruction.  Large D: a tiled SIMT kernel writes the keys
// of a block of rows to global scratch first (each (i, j) accumulator still runs over d in order), and the same row
// kernel reads them from there.
//
// Selection per row.  Only about k of the V keys matter, so no pass but the first looks at the others:
//   1. a sample of 1024 keys gives a bound t below which, with room to spare, the k smallest lie;
//   2. one pass over all keys keeps those <= t (composites key << 32 | index + 1; the code itself: 0);
//   3. the keep list -- some 1.5 k entries -- is counting-sorted into 2048 bins, in place through registers, every
//      entry ranked inside its bin and stored at its final position, so that ties are taken by smaller index.
// Where many keys equal the bound (codes that are the same: dead ones, say), the bound is one on (key, index): of the keys equal to t
// those of codes up to an index are kept, found in the sample like t itself, and their bins go by index.
// A row whose sample misled (fewer than k kept, or more than fit) or whose keys crowd a bin all the same
// takes the general path: radix select down to the exact threshold key over all V keys, compaction, bitonic
// sort of the composites.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <type_traits>

#include "lantern.h"
#include "lantern_device.cuh"

namespace lantern {

constexpr int SMALL_D = 32;
constexpr int TM = 128;          // distance tile edge (rows and columns of one CTA)
constexpr int DK = 16;           // dimensions staged per step
constexpr int HB = 11;           // general path: radix-select digit, 2048 bins, kept in the (still unused) list area
constexpr int HBINS = 1 << HB;
constexpr int SAMPLE = 1024;     // keys sampled per row
constexpr int NBINS = 2048;      // bins of the counting sort, 16-bit counters, two to a word
constexpr int CROWD = 1023;      // largest bin that is ranked by pairwise comparison
constexpr int KEEP = 18;         // list entries per thread of a row's team, at most
static_assert(SAMPLE <= NBINS / 2, "the sample is kept where the bins will be");

struct BuildParams {
  const float* codebook;
  const uint32_t* scratch;       // [rows, V] key bits of rows row0.. (large-D path), else null
  int32_t* idx;
  float* dist;
  int V, D, k;
  int row0, row_end;             // the rows of this launch
  const int* map;                // the rows are the codes map[row0..], *count of them at most (null: the codes themselves)
  const int* count;
  int cap;                       // entries of a row's keep list
  int want;                      // rank in the sample that bounds the k smallest keys; 0 = keep everything (cap = V)
};

// Two fp32 lanes in one 64-bit register; each lane of the packed operations rounds exactly like the
// scalar instruction, so the key sequence is unchanged.
__device__ __forceinline__ unsigned long long dup2(float a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// ---------------------------------------------------------------------------------------
// keys of a block of rows, large D: a 128 x 128 tile per CTA, 8 x 8 accumulators per thread
// (rows ty*4.. and 64+ty*4.., columns tx*4.. and 64+tx*4.., so that every shared-memory read is
// one conflict-free 16-byte load), the next 16 dimensions fetched into registers while the
// current ones are used.  Every (i, j) accumulator still runs over d in order.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float4 fetch_quad(const float* __restrict__ cb, int row, int row_end, int D, int d, bool vec) {
  float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);   // zero padding adds fma(0, 0, acc) = acc exactly
  if (row < row_end) {
    const float* p = cb + static_cast<size_t>(row) * D + d;
    if (vec && d + 3 < D) {
      v = __ldg(reinterpret_cast<const float4*>(p));
    } else {
      if (d < D) v.x = __ldg(p);
      if (d + 1 < D) v.y = __ldg(p + 1);
      if (d + 2 < D) v.z = __ldg(p + 2);
      if (d + 3 < D) v.w = __ldg(p + 3);
    }
  }
  return v;
}

// The accumulators of one tile.  `row` and `col` are the codes this thread stages (element tid & 127 of either side); a code
// of V and beyond reads as zero.
__device__ __forceinline__ void distance_tile(const float* __restrict__ cb, int V, int D, int row, int col, float (&As)[DK][TM],
                                              float (&Bs)[DK][TM], unsigned long long (&acc)[8][4]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const bool vec = (D & 3) == 0;
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
  // staging: element e = l * 256 + tid of a 128 x 16 tile is (row e & 127, dimensions 4 * (e >> 7) ..+3)
  const int srow = tid & 127, squad = tid >> 7;
  float4 ra[2], rb[2];
#pragma unroll
  for (int l = 0; l < 2; ++l) {
    ra[l] = fetch_quad(cb, row, V, D, 4 * (squad + 2 * l), vec);
    rb[l] = fetch_quad(cb, col, V, D, 4 * (squad + 2 * l), vec);
  }
  for (int d0 = 0; d0 < D; d0 += DK) {
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const int q = 4 * (squad + 2 * l);
      As[q][srow] = ra[l].x;
      As[q + 1][srow] = ra[l].y;
      As[q + 2][srow] = ra[l].z;
      As[q + 3][srow] = ra[l].w;
      Bs[q][srow] = rb[l].x;
      Bs[q + 1][srow] = rb[l].y;
      Bs[q + 2][srow] = rb[l].z;
      Bs[q + 3][srow] = rb[l].w;
    }
    __syncthreads();
    if (d0 + DK < D) {
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        ra[l] = fetch_quad(cb, row, V, D, d0 + DK + 4 * (squad + 2 * l), vec);
        rb[l] = fetch_quad(cb, col, V, D, d0 + DK + 4 * (squad + 2 * l), vec);
      }
    }
#pragma unroll
    for (int dd = 0; dd < DK; ++dd) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[dd][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[dd][64 + ty * 4]);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[dd][tx * 4]);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[dd][64 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const unsigned long long b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const unsigned long long aa = dup2(a[r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const unsigned long long t = sub2(aa, b[c]);
          acc[r][c] = fma2(t, t, acc[r][c]);
        }
      }
    }
    __syncthreads();
  }
}
__device__ __forceinline__ uint32_t low_key(unsigned long long v) { return static_cast<uint32_t>(v); }
__device__ __forceinline__ uint32_t high_key(unsigned long long v) { return static_cast<uint32_t>(v >> 32); }

// code s of the sample, spread over the codebook by the golden ratio (so that no period of the code order is sampled in step)
__device__ __forceinline__ int sampled_code(int s, int V) {
  return static_cast<int>((static_cast<unsigned long long>(static_cast<uint32_t>(s) * 2654435769u) * static_cast<unsigned>(V)) >> 32);
}

// the largest float below t >= 0 (below 0: anything negative)
__device__ __forceinline__ float key_below(float t) { return t > 0.0f ? __uint_as_float(__float_as_uint(t) - 1u) : -1.0f; }

// keys of rows x cols pairs -> out[local row, column], rows `pitch` apart
struct DistParams {
  const float* cb;
  uint32_t* out;
  int V, D;
  int row0, row_end, cols, pitch;
  const int* map;                // the rows are the codes map[row0..], *count of them at most (null: the codes themselves)
  const int* count;
  int sample;                    // the columns are the codes of the sample
};

__global__ void __launch_bounds__(256, 2) lantern_distance_tile_kernel(DistParams P) {
  __shared__ __align__(16) float As[DK][TM];
  __shared__ __align__(16) float Bs[DK][TM];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int V = P.V, cols = P.cols;
  grid_dependency_wait();
  // Not where whole tables are made block by block: CTAs put in place early take the SMs that a short grid leaves free, and
  // the grid after them is then crowded onto a few (V = 1500, D = 256: 117 -> 150 us).
  if (P.sample || P.count) grid_dependents_launch();
  const int row_end = P.count ? min(P.row_end, *P.count) : P.row_end;
  const int rbase = P.row0 + blockIdx.y * TM, cbase = blockIdx.x * TM;
  if (rbase >= row_end) return;
  const int r_mine = rbase + (tid & 127), c_mine = cbase + (tid & 127);
  const int row = r_mine < row_end ? (P.map ? P.map[r_mine] : r_mine) : V;
  const int col = c_mine < cols ? (P.sample ? sampled_code(c_mine, V) : c_mine) : V;
  unsigned long long acc[8][4];
  distance_tile(P.cb, V, P.D, row, col, As, Bs, acc);
  const bool vec_out = (P.pitch & 3) == 0;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int gr = rbase + (r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4));
    if (gr >= row_end) continue;
    uint32_t* orow = P.out + static_cast<size_t>(gr - P.row0) * P.pitch;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gc = cbase + 64 * h + tx * 4;
      const uint32_t w[4] = {low_key(acc[r][2 * h]), high_key(acc[r][2 * h]), low_key(acc[r][2 * h + 1]), high_key(acc[r][2 * h + 1])};
      if (vec_out && gc + 3 < cols) {
        *reinterpret_cast<uint4*>(orow + gc) = make_uint4(w[0], w[1], w[2], w[3]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (gc + c < cols) orow[gc + c] = w[c];
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Large D and a large codebook: every pair once.  (a - b)^2 and (b - a)^2 round alike, so key(j, i) = key(i, j) to the bit, and
// half of the distance work -- which the fp32 pipes bound -- can go; but the keys of all pairs do not fit the scratch, and a row's
// cannot be kept until the row is complete.  What fits are the rows' keep lists: with the bounds known beforehand (from 1024
// sampled keys per row: one sixteenth of the work at V = 16384), a tile on or above the diagonal appends the keys
// within the bounds to the lists of its rows and, mirrored, to those of its columns.
//
// A row's list: indices (16 bit) and as many keys as there is room for in its 1/V of the scratch, behind a counter; further keys in
// the row's own part of the outputs, idx from entry 1 on (entry 0 holds the bound until the list is read), then dist.
// ---------------------------------------------------------------------------------------
struct ListParams {
  unsigned char* scratch;
  int32_t* idx;
  float* dist;
  int V, k, cap;
  int region;                    // bytes of scratch per row
  __device__ __forceinline__ int* counter(int i) const { return reinterpret_cast<int*>(scratch + static_cast<size_t>(i) * region); }
  __device__ __forceinline__ unsigned short* index(int i) const {
    return reinterpret_cast<unsigned short*>(scratch + static_cast<size_t>(i) * region + 16);
  }
  __device__ __forceinline__ uint32_t* key(int i, int e) const {
    const int head = 16 + ((2 * cap + 3) & ~3), near = (region - head) >> 2;
    if (e < near) return reinterpret_cast<uint32_t*>(scratch + static_cast<size_t>(i) * region + head) + e;
    e -= near;
    if (e < k - 1) return reinterpret_cast<uint32_t*>(idx) + static_cast<size_t>(i) * k + 1 + e;
    return reinterpret_cast<uint32_t*>(dist) + static_cast<size_t>(i) * k + (e - (k - 1));
  }
  __device__ __forceinline__ float bound(int i) const { return __int_as_float(idx[static_cast<size_t>(i) * k]); }
  __device__ __forceinline__ int* last(int i) const { return counter(i) + 1; }   // of keys equal to the bound: codes up to this one (V: all)
};
// entries that a row's list has room for
static int list_room(int region, int k, bool dist, int cap) {
  const int head = 16 + ((2 * cap + 3) & ~3);
  return head > region ? 0 : ((region - head) >> 2) + (k - 1) + (dist ? k : 0);
}

// Bound of every row from its sampled keys (scratch[i, 0..SAMPLE)), which its list's counter replaces; one warp per row.
__global__ void __launch_bounds__(256) lantern_row_bound_kernel(ListParams L, int want) {
  grid_dependency_wait();
  grid_dependents_launch();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= L.V) return;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(L.scratch) + static_cast<size_t>(i) * SAMPLE;
  uint32_t key[SAMPLE / 32], most = 0u;
#pragma unroll
  for (int q = 0; q < SAMPLE / 32; ++q) {
    key[q] = src[q * 32 + lane];
    most = key[q] > most ? key[q] : most;
  }
  most = __reduce_max_sync(kFull, most);
  const int room = want / 16 + 2;
  uint32_t lo = 0u, hi = most;             // count(key <= hi) >= want > count(key <= lo); a few more than wanted will do
  int c_hi = SAMPLE;
  for (int pass = 0; pass < 48 && hi - lo > 1u; ++pass) {
    uint32_t m = __float_as_uint(0.5f * __uint_as_float(lo) + 0.5f * __uint_as_float(hi));
    if (!(m > lo && m < hi)) m = lo + ((hi - lo) >> 1);
    int c0 = 0, c1 = 0;
#pragma unroll
    for (int q = 0; q < SAMPLE / 32; q += 2) {
      c0 += key[q] <= m;
      c1 += key[q + 1] <= m;
    }
    const int c = __reduce_add_sync(kFull, c0 + c1);
    if (c >= want) hi = m, c_hi = c;
    else lo = m;
    if (c >= want && c <= want + room) break;
  }
  int last = L.V;
  if (c_hi > want + room) {                // ties: the same bisection on the index of the codes that lie at the bound
    int from = -1;
    last = L.V - 1;
    while (last - from > 1) {
      const int m = (from + last) >> 1;
      int c = 0;
#pragma unroll
      for (int q = 0; q < SAMPLE / 32; ++q) c += key[q] < hi || (key[q] == hi && sampled_code(q * 32 + lane, L.V) <= m);
      c = __reduce_add_sync(kFull, c);
      if (c >= want) last = m;
      else from = m;
      if (c >= want && c <= want + room) break;
    }
  }
  if (lane == 0) {
    L.idx[static_cast<size_t>(i) * L.k] = static_cast<int32_t>(hi);
    *L.counter(i) = 0;                     // (all lanes have read the row: the reduction above)
    *L.last(i) = last;
  }
}

// What a tile keeps (some 3000 entries at k = 1000) is first put in order of its lists in shared memory and then stored by
// all threads alike: the address of an entry takes thirty instructions, too many to spend on every pair.
constexpr int TILE_KEEP = 4096;
struct TileLists {
  uint32_t key[TILE_KEEP];
  unsigned short code[TILE_KEEP];
  unsigned char line[TILE_KEEP];
};

__global__ void __launch_bounds__(256, 2) lantern_distance_lists_kernel(const float* __restrict__ cb, int D, ListParams L) {
  __shared__ __align__(16) union {
    struct {
      float As[DK][TM], Bs[DK][TM];
    } in;
    TileLists out;
  } S;
  __shared__ float s_bound[2][TM];         // [0] the tile's rows, [1] its columns
  __shared__ float s_tie[2][TM];           // where only some of the other side's codes count if their keys equal the bound: the bound
  __shared__ int s_last[2][TM], s_mixed;
  __shared__ int s_n[2][TM], s_off[2][TM], s_base[2][TM], s_warp[8];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const int side = tid >> 7, line = tid & 127;
  grid_dependency_wait();
  grid_dependents_launch();
  const int V = L.V;
  // tile (tr, tc) with tr <= tc, numbered column by column: tc (tc + 1) / 2 + tr
  int tc = static_cast<int>((sqrtf(8.0f * static_cast<float>(blockIdx.x) + 1.0f) - 1.0f) * 0.5f);
  while (tc * (tc + 1) / 2 > static_cast<int>(blockIdx.x)) --tc;
  while ((tc + 1) * (tc + 2) / 2 <= static_cast<int>(blockIdx.x)) ++tc;
  const int tr = blockIdx.x - tc * (tc + 1) / 2;
  const int rbase = tr * TM, cbase = tc * TM;
  const int mine = (side ? cbase : rbase) + line;   // the code whose list this thread looks after
  s_n[side][line] = 0;
  if (tid == 0) s_mixed = 0;
  __syncthreads();
  {
    float t = __int_as_float(0xff800000), tie = __int_as_float(0x7fffffff);   // (-inf: keeps nothing; NaN: equals nothing)
    if (mine < V && (side == 0 || tr != tc)) {
      const int first = side ? rbase : cbase, last = *L.last(mine);
      t = L.bound(mine);
      if (last < min(first + TM, V) - 1) {   // keys equal to the bound count only for codes up to `last`: some here, or none
        if (last >= first) tie = t, s_last[side][line] = last, s_mixed = 1;
        t = key_below(t);
      }
    }
    s_bound[side][line] = t;
    s_tie[side][line] = tie;
  }
  unsigned long long acc[8][4];
  distance_tile(cb, V, D, rbase + line, cbase + line, S.in.As, S.in.Bs, acc);   // (its barriers publish the bounds as well)
  auto row_of = [&](int r) { return r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4); };
  auto col_of = [&](int c) { return c < 4 ? tx * 4 + c : 64 + tx * 4 + (c - 4); };
  // a pair with a code past the end is kept by nobody
  if (cbase + TM > V) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (cbase + col_of(c) >= V) {
#pragma unroll
        for (int r = 0; r < 8; ++r)
          acc[r][c >> 1] |= c & 1 ? 0x7fffffff00000000ull : 0x7fffffffull;   // NaN
      }
  }
  auto key_of = [&](int r, int c) { return c & 1 ? high_key(acc[r][c >> 1]) : low_key(acc[r][c >> 1]); };
  auto put = [&](int code, int e, int other, uint32_t key) {
    if (e < L.cap) {
      L.index(code)[e] = static_cast<unsigned short>(other);
      *L.key(code, e) = key;
    }
  };
  if (s_mixed) {                           // one tile per tied list: entry by entry
#pragma unroll
    for (int r = 0; r < 8; ++r) {
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int lr = row_of(r), lc = col_of(c);
        const uint32_t key = key_of(r, c);
        if (__uint_as_float(key) == s_tie[0][lr] && cbase + lc <= s_last[0][lr]) put(rbase + lr, atomicAdd(L.counter(rbase + lr), 1), cbase + lc, key);
        if (__uint_as_float(key) == s_tie[1][lc] && rbase + lr <= s_last[1][lc]) put(cbase + lc, atomicAdd(L.counter(cbase + lc), 1), rbase + lr, key);
      }
    }
  }
  int at_r[8], at_c[8];                    // this thread's places in the tile's part of each list
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float t = s_bound[0][row_of(r)];
    int n = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) n += __uint_as_float(key_of(r, c)) <= t;
    at_r[r] = n ? atomicAdd(&s_n[0][row_of(r)], n) : 0;
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float t = s_bound[1][col_of(c)];
    int n = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) n += __uint_as_float(key_of(r, c)) <= t;
    at_c[c] = n ? atomicAdd(&s_n[1][col_of(c)], n) : 0;
  }
  __syncthreads();
  const int n_mine = s_n[side][line];
  s_base[side][line] = n_mine ? atomicAdd(L.counter(mine), n_mine) : 0;
  int incl = n_mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_warp[tid >> 5] = incl;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w < (tid >> 5)) before += s_warp[w];
    total += s_warp[w];
  }
  s_off[side][line] = before + incl - n_mine;
  __syncthreads();
  // every kept pair: list (0 = of its row, 1 = of its column) and line, place in the tile's part, the other code, the key
  auto each = [&](auto take) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float t = s_bound[0][row_of(r)];
      int e = at_r[r];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (__uint_as_float(key_of(r, c)) <= t) take(0, row_of(r), e++, cbase + col_of(c), key_of(r, c));
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float t = s_bound[1][col_of(c)];
      int e = at_c[c];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (__uint_as_float(key_of(r, c)) <= t) take(1, col_of(c), e++, rbase + row_of(r), key_of(r, c));
    }
  };
  if (total <= TILE_KEEP) {
    each([&](int sd, int ln, int e, int other, uint32_t key) {
      const int p = s_off[sd][ln] + e;
      S.out.key[p] = key;
      S.out.code[p] = static_cast<unsigned short>(other);
      S.out.line[p] = static_cast<unsigned char>(sd << 7 | ln);
    });
    __syncthreads();
    for (int p = tid; p < total; p += 256) {
      const int sd = S.out.line[p] >> 7, ln = S.out.line[p] & 127;
      put((sd ? cbase : rbase) + ln, s_base[sd][ln] + p - s_off[sd][ln], S.out.code[p], S.out.key[p]);
    }
  } else {   // (codes of one cluster side by side)
    each([&](int sd, int ln, int e, int other, uint32_t key) { put((sd ? cbase : rbase) + ln, s_base[sd][ln] + e, other, key); });
  }
}

// the rows whose lists failed (marked by idx[i, 0] = -1), in any order; one CTA
__global__ void __launch_bounds__(1024) lantern_failed_rows_kernel(const int32_t* idx, int V, int k, int* rows, int* count) {
  __shared__ int s_n;
  grid_dependency_wait();
  grid_dependents_launch();
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
#pragma unroll 8
  for (int i = threadIdx.x; i < V; i += 1024)
    if (idx[static_cast<size_t>(i) * k] < 0) rows[atomicAdd(&s_n, 1)] = i;
  __syncthreads();
  if (threadIdx.x == 0) *count = s_n;
}

// ---------------------------------------------------------------------------------------
// one row: keys -> select -> sort -> store
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long shfl_xor_u64(unsigned long long x, int m) {
  const unsigned lo = __shfl_xor_sync(kFull, static_cast<unsigned>(x), m);
  const unsigned hi = __shfl_xor_sync(kFull, static_cast<unsigned>(x >> 32), m);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// Bitonic merge steps of strides 32..1 on one 64-element block held by a warp (elements lane and
// lane + 32), for every merge size from size_lo to size_hi whose strides all lie inside the block.
__device__ __forceinline__ void bitonic_block64(unsigned long long* list, int block, int lane, int size_lo, int size_hi) {
  const int e0 = block * 64 + lane, e1 = e0 + 32;
  unsigned long long x0 = list[e0], x1 = list[e1];
  for (int size = size_lo; size <= size_hi; size <<= 1) {
    if (size >= 64) {
      const bool up = (e0 & size) == 0;
      if ((x0 > x1) == up) {
        const unsigned long long t = x0;
        x0 = x1;
        x1 = t;
      }
    }
    for (int stride = size >= 64 ? 16 : (size >> 1); stride > 0; stride >>= 1) {
      const bool am_lo = (lane & stride) == 0;
      const unsigned long long o0 = shfl_xor_u64(x0, stride), o1 = shfl_xor_u64(x1, stride);
      const bool up0 = (e0 & size) == 0, up1 = (e1 & size) == 0;
      x0 = (am_lo == up0) ? (x0 < o0 ? x0 : o0) : (x0 > o0 ? x0 : o0);
      x1 = (am_lo == up1) ? (x1 < o1 ? x1 : o1) : (x1 > o1 ? x1 : o1);
    }
  }
  list[e0] = x0;
  list[e1] = x1;
}

// squared distance of codes i (already in `ai`) and j, in the canonical operation sequence
__device__ __forceinline__ float key_of(const float* ai, const float* __restrict__ b, int D, bool vec) {
  float acc = 0.0f;
  if (vec) {
    for (int d = 0; d < D; d += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(b + d));
      float t = __fsub_rn(ai[d], v.x);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(ai[d + 1], v.y);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(ai[d + 2], v.z);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(ai[d + 3], v.w);
      acc = __fmaf_rn(t, t, acc);
    }
  } else {
    for (int d = 0; d < D; ++d) {
      const float t = __fsub_rn(ai[d], __ldg(b + d));
      acc = __fmaf_rn(t, t, acc);
    }
  }
  return acc;
}

struct GeneralShared {
  int wcnt[32];
  uint32_t wmin[32], wmax[32];
  float ai[SMALL_D];
  int s_digit, s_below, s_ties, s_cnt;
};

// The general path for row i, by the whole CTA: dsm = V keys, then the list of P2 composites.
template <int KT>
__device__ __noinline__ void knn_row_general(const BuildParams& P, int i, int local, int P2, unsigned char* dsm, GeneralShared& S) {
  uint32_t* keys = reinterpret_cast<uint32_t*>(dsm);                                  // [V]
  unsigned long long* list =
      reinterpret_cast<unsigned long long*>(dsm + ((static_cast<size_t>(P.V) * 4 + 15) & ~size_t(15)));  // [P2]
  unsigned* hist = reinterpret_cast<unsigned*>(list);   // [HBINS] 16-bit counters, two to a word; used before the list is filled
  auto bin_count = [hist](int b) { return static_cast<int>((hist[b >> 1] >> ((b & 1) << 4)) & 0xffffu); };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int V = P.V, D = P.D, K = P.k - 1;
  constexpr int KW = KT / 32;

  // ---- keys (and their range over j != i) ----
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  if (!P.scratch && tid < D) S.ai[tid] = P.codebook[static_cast<size_t>(i) * D + tid];
  __syncthreads();
  for (int j = tid; j < V; j += KT) {
    const uint32_t key = P.scratch ? P.scratch[static_cast<size_t>(local) * V + j]
                                   : __float_as_uint(key_of(S.ai, P.codebook + static_cast<size_t>(j) * D, D, (D & 3) == 0));
    keys[j] = key;
    if (j != i) {
      kmin = key < kmin ? key : kmin;
      kmax = key > kmax ? key : kmax;
    }
  }
  kmin = __reduce_min_sync(kFull, kmin);
  kmax = __reduce_max_sync(kFull, kmax);
  if (lane == 0) {
    S.wmin[warp] = kmin;
    S.wmax[warp] = kmax;
  }
  if (tid == 0) S.s_cnt = 0;
  __syncthreads();
  const uint32_t self_key = keys[i];
  kmin = __reduce_min_sync(kFull, S.wmin[lane & (KW - 1)]);
  kmax = __reduce_max_sync(kFull, S.wmax[lane & (KW - 1)]);

  if (K > 0) {
    // ---- radix select on rel = key - kmin, 11 bits at a time from the top of the occupied range:
    //      tau = K-th smallest key over j != i; `need` ties at tau are taken, smallest index first ----
    const uint32_t range = kmax - kmin;
    int hi = range ? 32 - __clz(range) : 0;
    uint32_t prefix = 0;
    int need = K, ties_total = V - 1;
    while (hi > 0) {
      const int lo = hi > HB ? hi - HB : 0;
      const uint32_t dmask = (1u << (hi - lo)) - 1u;
      for (int t = tid; t < HBINS / 2; t += KT) hist[t] = 0u;
      __syncthreads();
      for (int j = tid; j < V; j += KT) {
        const uint32_t rel = keys[j] - kmin;
        if (j != i && (hi >= 32 || (rel >> hi) == (prefix >> hi))) {
          const uint32_t b = (rel >> lo) & dmask;
          atomicAdd(&hist[b >> 1], 1u << ((b & 1u) << 4));
        }
      }
      __syncthreads();
      int loc[HBINS / KT], s = 0;
#pragma unroll
      for (int q = 0; q < HBINS / KT; ++q) {
        loc[q] = bin_count(tid * (HBINS / KT) + q);
        s += loc[q];
      }
      int incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) S.wcnt[warp] = incl;
      __syncthreads();
      int excl = incl - s;
      for (int w = 0; w < warp; ++w) excl += S.wcnt[w];
      if (excl < need && need <= excl + s) {   // exactly one thread
        int run = excl;
#pragma unroll
        for (int q = 0; q < HBINS / KT; ++q) {
          if (run < need && need <= run + loc[q]) {
            S.s_digit = tid * (HBINS / KT) + q;
            S.s_below = run;
            S.s_ties = loc[q];
          }
          run += loc[q];
        }
      }
      __syncthreads();
      need -= S.s_below;
      ties_total = S.s_ties;
      prefix |= static_cast<uint32_t>(S.s_digit) << lo;
      hi = lo;
    }
    __syncthreads();   // the histogram's storage becomes the list
    const uint32_t tau = kmin + prefix;
    const int n_less = K - need;

    // ---- compaction (one counter update per warp) ----
    const bool all_ties = (ties_total == need);
    for (int base = 0; base < V; base += KT) {
      const int j = base + tid;
      const uint32_t key = j < V ? keys[j] : 0u;
      const bool sel = j < V && j != i && (key < tau || (all_ties && key == tau));
      const unsigned bal = __ballot_sync(kFull, sel);
      if (bal) {
        int pos = 0;
        if (lane == 0) pos = atomicAdd(&S.s_cnt, __popc(bal));
        pos = __shfl_sync(kFull, pos, 0) + __popc(bal & ((1u << lane) - 1u));
        if (sel) list[pos] = (static_cast<unsigned long long>(key) << 32) | static_cast<unsigned>(j);
      }
    }
    if (!all_ties) {   // more ties than places: take them in index order
      int run = 0;
      for (int base = 0; base < V && run < need; base += KT) {
        const int j = base + tid;
        const bool flag = j < V && j != i && keys[j] == tau;
        const unsigned bal = __ballot_sync(kFull, flag);
        if (lane == 0) S.wcnt[warp] = __popc(bal);
        __syncthreads();
        const int c = lane < KW ? S.wcnt[lane] : 0;
        const int before = __reduce_add_sync(kFull, lane < warp ? c : 0), chunk = __reduce_add_sync(kFull, c);
        const int rank = run + before + __popc(bal & ((1u << lane) - 1u));
        if (flag && rank < need)
          list[n_less + rank] = (static_cast<unsigned long long>(tau) << 32) | static_cast<unsigned>(j);
        run += chunk;
        __syncthreads();
      }
    }
    for (int t = K + tid; t < P2; t += KT) list[t] = ~0ull;
    __syncthreads();

    // ---- bitonic sort of (key, index) composites: strides below 64 in registers by shuffles ----
    const int nblk = P2 >> 6;
    for (int blk = warp; blk < nblk; blk += KW) bitonic_block64(list, blk, lane, 2, 64);
    __syncthreads();
    for (int size = 128; size <= P2; size <<= 1) {
      for (int stride = size >> 1; stride >= 64; stride >>= 1) {
        for (int t = tid; t < (P2 >> 1); t += KT) {
          const int lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1));
          const int hi2 = lo | stride;
          const bool up = (lo & size) == 0;
          const unsigned long long x = list[lo], y = list[hi2];
          if ((x > y) == up) {
            list[lo] = y;
            list[hi2] = x;
          }
        }
        __syncthreads();
      }
      for (int blk = warp; blk < nblk; blk += KW) bitonic_block64(list, blk, lane, size, size);
      __syncthreads();
    }
  }

  // ---- store ----
  int32_t* irow = P.idx + static_cast<size_t>(i) * P.k;
  float* drow = P.dist ? P.dist + static_cast<size_t>(i) * P.k : nullptr;
  if (tid == 0) {
    irow[0] = i;
    if (drow) drow[0] = __uint_as_float(self_key);
  }
  for (int t = tid; t < K; t += KT) {
    const unsigned long long c = list[t];
    irow[1 + t] = static_cast<int32_t>(c & 0xffffffffu);
    if (drow) drow[1 + t] = __uint_as_float(static_cast<uint32_t>(c >> 32));
  }
  __syncthreads();
}

// bytes of shared memory per row: keep list (and four entries that take what does not fit), bins
static __host__ __device__ constexpr size_t row_bytes(int cap) {
  return ((static_cast<size_t>(cap + 4) * 8 + 15) & ~size_t(15)) + NBINS * 2;
}

// *to++ = {who, key} if key <= t (to: an address in shared memory), predicated: one key in eleven is kept at
// V = 16384, k = 1000 (D = 8: 551 us per table as a C++ condition, 540 like this).
__device__ __forceinline__ void append_key(uint32_t& to, float key, float t, uint32_t who) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.le.f32 p, %1, %2;\n\t"
      "@p st.shared.v2.b32 [%0], {%3, %4};\n\t"
      "@p add.u32 %0, %0, 8;\n\t}"
      : "+r"(to)
      : "f"(key), "f"(t), "r"(who), "r"(__float_as_uint(key))
      : "memory");
}

// R rows per CTA of KT threads; KT / R threads rank a row; U codes per thread and step of the key pass.  FROM: where the keys come from -- computed here (small D), read
// from scratch rows, or already on lists.  ALL: every key is kept, so there is neither sample nor bound, and the
// bins cover the range that the keys turn out to have.
//
// What bounds it (V = 16384, k = 1000, cycles of a CTA of eight rows, D = 8): the key pass 40 k, of which the fp32
// pipes need 16 k and instruction issue 24 k; sample and bound 9 k; counting sort 13 k; ranking 11 k.
// 0.54 ms per table; 1.20 ms when a CTA selected from all keys of one row (73 k warp instructions per row, now 26 k).
enum { FROM_CODES = 0, FROM_SCRATCH = 1, FROM_LISTS = 2 };
template <int KT, int R, int FROM, bool ALL, int U>
__global__ void __launch_bounds__(KT, 1024 / KT) lantern_knn_rows_kernel(BuildParams P, ListParams L, int P2) {
  constexpr bool SCRATCH = FROM == FROM_SCRATCH, LISTS = FROM == FROM_LISTS;
  constexpr int RT = KT / R;         // threads of a row's team
  constexpr int RW = RT / 32;
  constexpr int OWN = NBINS / 2 / RT;   // words of bins per thread of a team
  constexpr int SMP = SAMPLE / RT;   // sampled keys per thread of a team
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ __align__(16) float As[SMALL_D][R];
  __shared__ GeneralShared S;
  __shared__ int s_cnt[R], s_wsum[R][RW], s_slow[R];
  __shared__ float s_t[R], s_lo[R], s_scale[R];
  __shared__ int s_last[R];          // of keys equal to the bound: codes up to this one (V: all)
  __shared__ int s_vote[2][R][RW];
  __shared__ uint32_t s_low[R][3 * RW], s_most[R][RW];
  const int tid = threadIdx.x, lane = tid & 31;
  const int V = P.V, D = P.D, k = P.k, cap = P.cap;
  grid_dependency_wait();
  if (LISTS || P.count) grid_dependents_launch();   // (see lantern_distance_tile_kernel)
  const int row0 = P.row0 + blockIdx.x * R, row_end = P.count ? min(P.row_end, *P.count) : P.row_end;
  if (row0 >= row_end) return;
  const bool vec = (D & 3) == 0;
  const size_t per_row = row_bytes(cap);
  auto list_of = [&](int r) { return reinterpret_cast<unsigned long long*>(dsm + r * per_row); };
  auto bins_of = [&](int r) { return reinterpret_cast<unsigned*>(dsm + (r + 1) * per_row - NBINS * 2); };

  if (FROM == FROM_CODES) {
    for (int t = tid; t < SMALL_D * R; t += KT) {
      const int d = t / R, r = t % R;
      As[d][r] = (d < D && row0 + r < row_end) ? P.codebook[static_cast<size_t>(row0 + r) * D + d] : 0.0f;
    }
  }
  if (tid < R) s_cnt[tid] = 0, s_slow[tid] = 0, s_last[tid] = V;
  __syncthreads();

  const int r = tid / RT, rt = tid % RT;   // this thread's team and its place in it
  const bool on = row0 + r < row_end;
  const int local = row0 + r - P.row0;
  const int i = on && P.map ? P.map[row0 + r] : row0 + r;
  auto team = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + r), "n"(RT) : "memory"); };
  // ---- 1. the bound, from SAMPLE keys ----
  if constexpr (!LISTS && !ALL) {
    uint32_t key[SMP];
    if constexpr (SCRATCH) {
      const uint32_t* src = P.scratch + static_cast<size_t>(on ? local : 0) * V;
#pragma unroll
      for (int q = 0; q < SMP; ++q) key[q] = src[sampled_code(q * RT + rt, V)];   // (not a read-only load: this kernel may be in place while they are written)
    } else {   // every thread takes codes of the sample against all rows of the CTA
      for (int s = tid; s < SAMPLE; s += KT) {
        const float* b = P.codebook + static_cast<size_t>(sampled_code(s, V)) * D;
        float acc[R];
#pragma unroll
        for (int q = 0; q < R; ++q) acc[q] = 0.0f;
        auto dim = [&](int d, float v) {
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const float t = __fsub_rn(As[d][q], v);
            acc[q] = __fmaf_rn(t, t, acc[q]);
          }
        };
        if (vec) {
          for (int d = 0; d < D; d += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(b + d));
            dim(d, v.x), dim(d + 1, v.y), dim(d + 2, v.z), dim(d + 3, v.w);
          }
        } else {
          for (int d = 0; d < D; ++d) dim(d, __ldg(b + d));
        }
#pragma unroll
        for (int q = 0; q < R; ++q) reinterpret_cast<uint32_t*>(bins_of(q))[s] = __float_as_uint(acc[q]);
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < SMP; ++q) key[q] = bins_of(r)[q * RT + rt];
    }
    // where the bins start: about the third smallest of the sample (of the warps' three smallest lane minima)
    const int wv = rt >> 5;
    uint32_t least = 0xffffffffu, most = 0u;
#pragma unroll
    for (int q = 0; q < SMP; ++q) {
      least = key[q] < least ? key[q] : least;
      most = key[q] > most ? key[q] : most;
    }
    most = __reduce_max_sync(kFull, most);
    if (lane == 0) s_most[r][wv] = most;
    for (int q = 0; q < 3; ++q) {
      const uint32_t low = __reduce_min_sync(kFull, least);
      if (lane == 0) s_low[r][3 * wv + q] = low;
      if (least == low) least = 0xffffffffu;
    }
    team();
    most = 0u;
#pragma unroll
    for (int w = 0; w < RW; ++w) most = s_most[r][w] > most ? s_most[r][w] : most;
    // bisection on the sampled values: count(key <= hi) >= want > count(key <= lo); a few more than wanted will do
    const int room = P.want / 16 + 2;
    uint32_t lo = 0u, hi = most;
    int pass = 0, c_hi = SAMPLE;
    auto vote = [&](int c) {                // the team's sum
      c = __reduce_add_sync(kFull, c);
      if (lane == 0) s_vote[pass & 1][r][wv] = c;
      team();
      c = 0;
#pragma unroll
      for (int w = 0; w < RW; ++w) c += s_vote[pass & 1][r][w];
      ++pass;
      return c;
    };
    while (pass < 48 && hi - lo > 1u) {
      uint32_t m = __float_as_uint(0.5f * __uint_as_float(lo) + 0.5f * __uint_as_float(hi));
      if (!(m > lo && m < hi)) m = lo + ((hi - lo) >> 1);
      int c = 0;
#pragma unroll
      for (int q = 0; q < SMP; ++q) c += key[q] <= m;
      c = vote(c);
      if (c >= P.want) hi = m, c_hi = c;
      else lo = m;
      if (c >= P.want && c <= P.want + room) break;
    }
    const uint32_t t = hi;
    if (c_hi > P.want + room) {             // ties: the same bisection on the index of the codes that lie at the bound
      int from = -1, last = V - 1;
      while (last - from > 1) {
        const int m = (from + last) >> 1;
        int c = 0;
#pragma unroll
        for (int q = 0; q < SMP; ++q) c += key[q] < t || (key[q] == t && sampled_code(q * RT + rt, V) <= m);
        c = vote(c);
        if (c >= P.want) last = m;
        else from = m;
        if (c >= P.want && c <= P.want + room) break;
      }
      if (rt == 0) s_last[r] = last;
    }
    if (rt < 32) {
      uint32_t low = 0u, mine = lane < 3 * RW ? s_low[r][lane] : 0xffffffffu;
      for (int q = 0; q < 3; ++q) {
        low = __reduce_min_sync(kFull, mine);
        if (mine == low) mine = 0xffffffffu;
      }
      if (low > most) low = most;     // (fewer than three different minima)
      if (lane == 0) {
        const float lo_f = __uint_as_float(low), hi_f = __uint_as_float(t < most ? t : most);
        s_t[r] = __uint_as_float(t);
        s_lo[r] = lo_f;
        s_scale[r] = hi_f > lo_f ? 1.0f / (hi_f - lo_f) : 0.0f;
      }
    }
    __syncthreads();
  }

  // ---- 2. all keys; those within the bound go to their row's list ----
  if constexpr (FROM == FROM_CODES) {
    float t_row[R];
#pragma unroll
    for (int q = 0; q < R; ++q) t_row[q] = ALL ? 0.0f : s_t[q];
    const uint32_t lists = static_cast<uint32_t>(__cvta_generic_to_shared(dsm));
    int tied_to = V;                         // the smallest index up to which a row takes keys equal to its bound
    if constexpr (!ALL) {
#pragma unroll
      for (int q = 0; q < R; ++q) tied_to = min(tied_to, s_last[q]);
    }
    for (int base = 0; base < V; base += U * KT) {
      unsigned long long acc[U][R / 2];
      const float* b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = base + u * KT + tid;
        b[u] = P.codebook + static_cast<size_t>(j < V ? j : 0) * D;
#pragma unroll
        for (int q = 0; q < R / 2; ++q) acc[u][q] = 0ull;
      }
      for (int d0 = 0; d0 < D; d0 += 4) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (vec) {
            v[u] = __ldg(reinterpret_cast<const float4*>(b[u] + d0));
          } else {   // zero padding (As is zero there too) adds fma(0, 0, acc) = acc exactly
            v[u].x = __ldg(b[u] + d0);
            v[u].y = d0 + 1 < D ? __ldg(b[u] + d0 + 1) : 0.0f;
            v[u].z = d0 + 2 < D ? __ldg(b[u] + d0 + 2) : 0.0f;
            v[u].w = d0 + 3 < D ? __ldg(b[u] + d0 + 3) : 0.0f;
          }
        }
#pragma unroll
        for (int dd = 0; dd < 4; ++dd) {
          unsigned long long a2[R / 2];
          if (R >= 4) {
#pragma unroll
            for (int q = 0; q < R / 2; q += 2) {
              const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&As[d0 + dd][2 * q]);
              a2[q] = a.x, a2[(q + 1) % (R / 2)] = a.y;
            }
          } else {
            a2[0] = *reinterpret_cast<const unsigned long long*>(&As[d0 + dd][0]);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const unsigned long long bb = dup2(dd == 0 ? v[u].x : (dd == 1 ? v[u].y : (dd == 2 ? v[u].z : v[u].w)));
#pragma unroll
            for (int q = 0; q < R / 2; ++q) {
              const unsigned long long t = sub2(a2[q], bb);
              acc[u][q] = fma2(t, t, acc[u][q]);
            }
          }
        }
      }
      if (base + U * KT > V) {   // codes past the end: NaN, never kept
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (base + u * KT + tid >= V) {
#pragma unroll
            for (int q = 0; q < R / 2; ++q) acc[u][q] = 0x7fffffff7fffffffull;
          }
      }
      if (!ALL && base + U * KT > tied_to) {   // (uniform, and never where no row has ties)
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int last = s_last[q];
          if (last >= base + U * KT || last >= V) continue;
          const float t = s_t[q];
          if (last < base) {
            t_row[q] = key_below(t);
          } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const float key = __uint_as_float(static_cast<uint32_t>(q & 1 ? acc[u][q / 2] >> 32 : acc[u][q / 2]));
              if (base + u * KT + tid > last && key == t) acc[u][q / 2] |= q & 1 ? 0x7fffffff00000000ull : 0x7fffffffull;   // NaN
            }
          }
        }
      }
      if constexpr (ALL) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = base + u * KT + tid;
          if (j < V) {
#pragma unroll
            for (int q = 0; q < R; ++q)
              list_of(q)[j] = (static_cast<unsigned long long>(static_cast<uint32_t>(q & 1 ? acc[u][q / 2] >> 32 : acc[u][q / 2])) << 32) |
                              static_cast<unsigned>(j + 1);
          }
        }
        continue;
      }
      // How many of this thread's keys each row keeps, four rows to a word (at most U each, 32 U per warp), and a
      // prefix over the warp; then one counter update per row and warp.  (Ballots and population counts in
      // their place kept the XU pipe busy for 24 of the pass's 51 thousand cycles.)
      constexpr int NW = (R + 3) / 4;
      auto key_of_row = [&](int u, int q) {
        return __uint_as_float(static_cast<uint32_t>(q & 1 ? acc[u][q / 2] >> 32 : acc[u][q / 2]));
      };
      uint32_t cnt[NW] = {}, incl[NW], tot[NW];
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (key_of_row(u, q) <= t_row[q]) cnt[q / 4] += 1u << (8 * (q % 4));
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        incl[w] = cnt[w];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t v = __shfl_up_sync(kFull, incl[w], o);
          if (lane >= o) incl[w] += v;
        }
        tot[w] = __shfl_sync(kFull, incl[w], 31);
        incl[w] -= cnt[w];
      }
      const int mine = ((NW > 1 && (lane & 4) ? tot[NW - 1] : tot[0]) >> (8 * (lane & 3))) & 0xffu;
      int start = 0;
      if (lane < R && mine) start = atomicAdd(&s_cnt[lane], mine);
#pragma unroll
      for (int q = 0; q < R; ++q) {
        int at = __shfl_sync(kFull, start, q) + static_cast<int>((incl[q / 4] >> (8 * (q % 4))) & 0xffu);
        at = at < cap ? at : cap;                        // (the list has room for U more)
        uint32_t to = lists + static_cast<uint32_t>(q * static_cast<int>(per_row) + at * 8);
#pragma unroll
        for (int u = 0; u < U; ++u) append_key(to, key_of_row(u, q), t_row[q], static_cast<uint32_t>(base + u * KT + tid + 1));
      }
    }
  } else if (SCRATCH && on && !ALL) {   // each team reads its own row of keys, W groups of four per thread at a time
    constexpr int W = 4;
    const uint32_t* src = P.scratch + static_cast<size_t>(local) * V;
    const float t = s_t[r];
    const int last = s_last[r];
    unsigned long long* list = list_of(r);
    const bool vec4 = (V & 3) == 0;
    for (int base = 0; base < V; base += W * 4 * RT) {
      uint4 key[W];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const int j0 = base + w * 4 * RT + 4 * rt;
        key[w] = make_uint4(0x7fffffffu, 0x7fffffffu, 0x7fffffffu, 0x7fffffffu);   // NaN: never kept
        if (vec4) {
          if (j0 < V) key[w] = __ldcs(reinterpret_cast<const uint4*>(src + j0));
        } else {
          if (j0 < V) key[w].x = __ldcs(src + j0);
          if (j0 + 1 < V) key[w].y = __ldcs(src + j0 + 1);
          if (j0 + 2 < V) key[w].z = __ldcs(src + j0 + 2);
          if (j0 + 3 < V) key[w].w = __ldcs(src + j0 + 3);
        }
      }
      if (base + W * 4 * RT > last) {   // ties beyond the last code that counts (uniform over the team)
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const int j0 = base + w * 4 * RT + 4 * rt;
          if (j0 > last && __uint_as_float(key[w].x) == t) key[w].x = 0x7fffffffu;
          if (j0 + 1 > last && __uint_as_float(key[w].y) == t) key[w].y = 0x7fffffffu;
          if (j0 + 2 > last && __uint_as_float(key[w].z) == t) key[w].z = 0x7fffffffu;
          if (j0 + 3 > last && __uint_as_float(key[w].w) == t) key[w].w = 0x7fffffffu;
        }
      }
      // thread by thread: how many of the sixteen are kept, where they go, then the entries
      int c = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t kk[4] = {key[w].x, key[w].y, key[w].z, key[w].w};
#pragma unroll
        for (int u = 0; u < 4; ++u) c += __uint_as_float(kk[u]) <= t;
      }
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&s_cnt[r], incl);
      at = __shfl_sync(kFull, at, 31) + incl - c;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t kk[4] = {key[w].x, key[w].y, key[w].z, key[w].w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (__uint_as_float(kk[u]) <= t) {
            if (at < cap) list[at] = (static_cast<unsigned long long>(kk[u]) << 32) | static_cast<unsigned>(base + w * 4 * RT + 4 * rt + u + 1);
            ++at;
          }
        }
      }
    }
  }
  if (!LISTS && !ALL && on && rt == 0 && s_last[r] < i && s_t[r] == 0.0f) {   // the code itself lies behind the last tie that counts
    const int at = atomicAdd(&s_cnt[r], 1);
    if (at < cap) list_of(r)[at] = static_cast<unsigned>(i + 1);
  }
  __syncthreads();

  // ---- 3. counting sort (in place, through registers) and ranking, a team per row ----
  if (on) {
    unsigned long long* list = list_of(r);
    unsigned* bins = bins_of(r);
    const int last = LISTS ? *L.last(i) : (ALL ? V : s_last[r]);
    const bool tied = last < V;
    const uint32_t tie = tied ? __float_as_uint(LISTS ? L.bound(i) : s_t[r]) : 0u;
    const bool self_left = LISTS && tied && tie == 0u && last < i;   // (as above)
    auto rank_row = [&](auto with_ties) {   // (rows without ties in code of their own: 542 us per table of D = 8, 570 in common code)
      constexpr bool TIED = decltype(with_ties)::value;
      const int n = LISTS ? *L.counter(i) + (TIED && self_left ? 1 : 0) : (ALL ? V : s_cnt[r]);
      const uint32_t* row = SCRATCH ? P.scratch + static_cast<size_t>(local) * V : nullptr;
      float lo = 0.0f, scale = 0.0f;
      uint32_t key[KEEP], who[KEEP];    // this thread's entries: the key; index + 1 and place of arrival in its bin
      constexpr bool ranged = LISTS || ALL;   // the range of the bins comes from the entries themselves
      if (!ranged) lo = s_lo[r], scale = s_scale[r];
      // with ties the upper half of the bins is for keys equal to the bound, by index
      constexpr int KEY_BINS = TIED ? NBINS / 2 : NBINS;
      const float per_index = TIED ? static_cast<float>(NBINS / 2) / static_cast<float>(last + 2) : 0.0f;
      auto bin_of = [&](uint32_t key, uint32_t id) {   // monotone in (key, index + 1)
        if (TIED && key == tie) return NBINS / 2 + min(static_cast<int>(static_cast<float>(id & 0xffffu) * per_index), NBINS / 2 - 1);
        // the square: near the bound the keys lie closer together (distances in D dimensions grow like the D/2-th root)
        const float x = fmaxf(__uint_as_float(key) - lo, 0.0f) * scale;
        return min(static_cast<int>(x * x * static_cast<float>(KEY_BINS)), KEY_BINS - 1);
      };
      auto bin_at = [&](int b) { return static_cast<int>((bins[b >> 1] >> ((b & 1) << 4)) & 0xffffu); };
      if (n < k || n > cap) {
        if (rt == 0) s_slow[r] = 1;
      } else {
#pragma unroll
        for (int q = 0; q < OWN; ++q) bins[q * RT + rt] = 0u;
        if (ranged) {                     // read the list; its range (without the code itself) is where the bins go
          uint32_t least = 0xffffffffu, most = 0u;
#pragma unroll
          for (int q = 0; q < KEEP; ++q) {
            const int e = q * RT + rt;
            if (e < n) {
              if (LISTS && TIED && self_left && e == n - 1) {
                key[q] = 0u, who[q] = static_cast<uint32_t>(i + 1);
              } else {
                key[q] = LISTS ? *L.key(i, e) : (SCRATCH ? __ldcs(row + e) : static_cast<uint32_t>(list[e] >> 32));
                who[q] = LISTS ? L.index(i)[e] + 1u : static_cast<uint32_t>(e + 1);
              }
              if (who[q] != static_cast<uint32_t>(i + 1)) {
                least = key[q] < least ? key[q] : least;
                most = key[q] > most ? key[q] : most;
              }
            }
          }
          least = __reduce_min_sync(kFull, least);
          most = __reduce_max_sync(kFull, most);
          if (lane == 0) s_low[r][rt >> 5] = least, s_most[r][rt >> 5] = most;
        }
        team();
        if (ranged) {
          uint32_t least = 0xffffffffu, most = 0u;
#pragma unroll
          for (int w = 0; w < RW; ++w) {
            least = s_low[r][w] < least ? s_low[r][w] : least;
            most = s_most[r][w] > most ? s_most[r][w] : most;
          }
          lo = __uint_as_float(least);
          scale = most > least ? 1.0f / (__uint_as_float(most) - lo) : 0.0f;
          if (most > 0x7f800000u) s_slow[r] = 1;   // NaN
        }
#pragma unroll
        for (int q = 0; q < KEEP; ++q) {
          const int e = q * RT + rt;
          if (e < n) {
            if (!ranged) {
              const unsigned long long c = list[e];
              key[q] = static_cast<uint32_t>(c >> 32);
              who[q] = static_cast<uint32_t>(c);
            }
            if (who[q] == static_cast<uint32_t>(i + 1)) key[q] = who[q] = 0u;   // the code itself comes first
            const int b = bin_of(key[q], who[q]), sh = (b & 1) << 4;
            who[q] |= ((atomicAdd(&bins[b >> 1], 1u << sh) >> sh) & 0xffffu) << 16;
          }
        }
        team();
        unsigned loc[OWN];
        int s = 0;
#pragma unroll
        for (int q = 0; q < OWN; ++q) {
          loc[q] = bins[rt * OWN + q];
          s += static_cast<int>((loc[q] & 0xffffu) + (loc[q] >> 16));
        }
        int incl = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += t;
        }
        if (lane == 31) s_wsum[r][rt >> 5] = incl;
        team();
        unsigned at = static_cast<unsigned>(incl - s);
#pragma unroll
        for (int w = 0; w < RW; ++w)
          if (w < (rt >> 5)) at += static_cast<unsigned>(s_wsum[r][w]);
#pragma unroll
        for (int q = 0; q < OWN; ++q) {   // every count becomes the place where its bin starts
          const unsigned c0 = loc[q] & 0xffffu, c1 = loc[q] >> 16;
          bins[rt * OWN + q] = at | ((at + c0) << 16);
          if ((c0 > CROWD && at < static_cast<unsigned>(k)) || (c1 > CROWD && at + c0 < static_cast<unsigned>(k))) s_slow[r] = 1;
          at += c0 + c1;
        }
        team();
        if (!s_slow[r]) {
#pragma unroll
          for (int q = 0; q < KEEP; ++q) {
            if (q * RT + rt < n)
              list[bin_at(bin_of(key[q], who[q])) + (who[q] >> 16)] = (static_cast<unsigned long long>(key[q]) << 32) | (who[q] & 0xffffu);
          }
          team();
          int32_t* irow = P.idx + static_cast<size_t>(i) * k;
          float* drow = P.dist ? P.dist + static_cast<size_t>(i) * k : nullptr;
          for (int p = rt; p < n; p += RT) {
            const unsigned long long c = list[p];
            const int b = bin_of(static_cast<uint32_t>(c >> 32), static_cast<uint32_t>(c));
            const int start = bin_at(b), end = b + 1 < NBINS ? bin_at(b + 1) : n;
            if (start >= k) break;
            int rank = start;
            for (int u = start; u < end; ++u) rank += list[u] < c;
            if (rank < k) {
              irow[rank] = c ? static_cast<int32_t>(static_cast<uint32_t>(c)) - 1 : i;
              if (drow) drow[rank] = __uint_as_float(static_cast<uint32_t>(c >> 32));
            }
          }
        }
      }
    };
    if (!ALL && tied) rank_row(std::true_type{});
    else rank_row(std::false_type{});
  }
  __syncthreads();
  for (int q = 0; q < R; ++q) {
    if (!s_slow[q]) continue;
    const int l = row0 + q, code = P.map ? P.map[l] : l;
    if constexpr (LISTS) {
      if (tid == 0) P.idx[static_cast<size_t>(code) * k] = -1;   // done again from all keys
    } else {
      knn_row_general<KT>(P, code, l - P.row0, P2, dsm, S);
    }
  }
}

static int next_pow2(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

constexpr size_t kRowSmem = 216 * 1024;   // dynamic shared memory of an SM that the row kernel counts on

// Rows whose keys are held in scratch at a time: 64 MB at V = 16384, which the row kernel still finds
// in L2 (1152 rows, which would fill the distance kernel's last wave of CTAs, measured slower).
static int rows_per_block(int V) {
  int r = V < 1024 ? V : 1024;
  return (r + TM - 1) / TM * TM;
}

// A launch that may be put in place while the kernel before it on the stream drains.  A build is a chain of short launches --
// two per block of rows, most of them without work where they only redo failed rows (38 at V = 16384) -- and every kernel
// waits (grid_dependency_wait) before it reads.  D = 256, k = 1000: V = 16384 3174 -> 3088 us, with k = 25 V = 4096 377 -> 348.
// First: nothing of the chain lies before it.
template <class... Arg>
static cudaError_t launch_chained(bool first, void (*kernel)(Arg...), dim3 grid, int threads, size_t smem, cudaStream_t st, Arg... arg) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &attr;
  c.numAttrs = first ? 0 : 1;
  return cudaLaunchKernelEx(&c, kernel, arg...);
}

template <int KT, int R, int FROM, bool ALL = false, int U = 2>
static cudaError_t launch_rows(const BuildParams& P, int P2, size_t smem, cudaStream_t st, const ListParams& L = {}) {
  auto kk = lantern_knn_rows_kernel<KT, R, FROM, ALL, U>;
  static DeviceFlags ready;
  const cudaError_t e = allow_shared_memory(kk, kRowSmem, ready);
  if (e != cudaSuccess) return e;
  return launch_chained(FROM == FROM_CODES, kk, dim3((P.row_end - P.row0 + R - 1) / R), KT, smem, st, P, L, P2);
}

}  // namespace lantern

using namespace lantern;

extern "C" size_t lantern_build_workspace_bytes(int V, int D, int k) {
  (void)k;
  if (V < 1 || D < 1) return 0;
  if (D <= SMALL_D) return 0;
  return static_cast<size_t>(rows_per_block(V)) * V * 4;
}

extern "C" lantern_status lantern_build_neighbors(const float* codebook, int V, int D, int k, int32_t* idx,
                                                  float* dist, void* workspace, size_t workspace_bytes,
                                                  void* cuda_stream) {
  if (V < 1 || V > 32768 || D < 1 || D > 4096 || k < 1 || k > V || k > 4097) return LANTERN_E_SHAPE;
  if (!codebook || !idx) return LANTERN_E_NULL;
  if ((reinterpret_cast<uintptr_t>(codebook) & 15)) return LANTERN_E_ALIGN;
  const size_t need_ws = lantern_build_workspace_bytes(V, D, k);
  if (need_ws && (!workspace || workspace_bytes < need_ws || (reinterpret_cast<uintptr_t>(workspace) & 15)))
    return LANTERN_E_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int P2 = next_pow2(k - 1 < 64 ? 64 : k - 1);   // the general path's sort works on whole 64-element blocks
  const size_t list_bytes = static_cast<size_t>(P2) * 8 > HBINS * 2 ? static_cast<size_t>(P2) * 8 : HBINS * 2;
  const size_t general = ((static_cast<size_t>(V) * 4 + 15) & ~size_t(15)) + list_bytes;
  BuildParams P;
  P.codebook = codebook;
  P.scratch = D > SMALL_D ? static_cast<const uint32_t*>(workspace) : nullptr;
  P.idx = idx;
  P.dist = dist;
  P.V = V;
  P.D = D;
  P.k = k;
  P.map = P.count = nullptr;
  // The k-th smallest of V keys has rank k SAMPLE / V in the sample, with a binomial spread; 3.5 standard deviations
  // above that the bound fails one row in some thousands, and the list is as long as the kept keys may be with the same
  // margin.  Few codes: every key is kept and sorted.  The line: where keys are computed here a sample costs as
  // much as the keys it stands for (V = 2048, D = 16, k = 25: 34 us per table without one, 38 with it), and a team's registers
  // hold 2304 keys; where they are read the sample is cheap and sorting all is not (V = 2048, D = 40: 50 and 48 us).
  const double f = static_cast<double>(SAMPLE) / V, mean = k * f, sd = sqrt(mean * (1.0 - static_cast<double>(k) / V));
  const int want = static_cast<int>(mean + 3.5 * sd) + 3, most = want + want / 16 + 2;
  const double kept = (most + 3.5 * sqrt(static_cast<double>(most))) / f;
  P.want = (V <= (D > SMALL_D ? SAMPLE : KEEP * 128) || kept >= V) ? 0 : want;
  P.cap = P.want ? (static_cast<int>(kept) + 7) & ~7 : V;
  // As many rows per CTA as their lists leave room for (and a team's registers hold): eight rows share every load of a
  // code.  The longest list, 7264 entries at V = 32768 and k = 4097, leaves room for two.  Rows read from
  // scratch share nothing: two CTAs of half the size then overlap one another's phases.
  const size_t per_row = row_bytes(P.cap);
  const int kt = P.scratch ? 512 : 1024;
  auto fits = [&](int R) { return R * per_row <= kRowSmem && P.cap <= KEEP * (1024 / R); };
  const int R = fits(8) ? 8 : (fits(4) ? 4 : 2);   // per 1024 threads
  // Few codes: small CTAs of two rows, four to an SM, so that the last wave is not mostly empty (V = 2400, D = 8, k = 25: 40 us
  // per table, 50 with eight rows per CTA; from scratch V = 2693, D = 40: 107 and 110).  Two rows share a code's
  // loads where eight could, which costs more the longer the codes are: D = 12 43 and 54 us, D = 16 68 and 65, D = 32 190 and 105;
  // at D = 8 the two shapes meet at V = 3600 (73 and 69).
  const bool few = (P.scratch ? V <= 4096 : D <= 12 && V <= 3072) && fits(8);
  const size_t rows_smem = few ? 2 * per_row : R * per_row * kt / 1024;
  const size_t smem = rows_smem > general ? rows_smem : general;
  if (smem > kRowSmem || P.cap > KEEP * (1024 / R)) return LANTERN_E_SHAPE;
  auto with = [&](auto all) {
    constexpr bool ALL = decltype(all)::value;
    if (few) {
      return P.scratch ? launch_rows<256, 2, FROM_SCRATCH, ALL>(P, P2, smem, st) : launch_rows<256, 2, FROM_CODES, ALL>(P, P2, smem, st);
    }
    if (P.scratch)
      return R == 8 ? launch_rows<512, 4, FROM_SCRATCH, ALL>(P, P2, smem, st)
                    : (R == 4 ? launch_rows<512, 2, FROM_SCRATCH, ALL>(P, P2, smem, st)
                              : launch_rows<512, 1, FROM_SCRATCH, ALL>(P, P2, smem, st));
    // Four codes a step instead of two halve what a step costs besides the keys (a prefix over the warp, a counter update), where the
    // codes fill such steps (V = 16384: D = 8 555 -> 544 us per table, D = 16 787 -> 763, D = 32 1580 -> 1472; V = 6000, whose second
    // step would be half empty, D = 24 215 and 261).
    if constexpr (!ALL) {
      if (R == 8 && (V + 2047) / 2048 % 2 == 0) return launch_rows<1024, 8, FROM_CODES, ALL, 4>(P, P2, smem, st);
    }
    return R == 8 ? launch_rows<1024, 8, FROM_CODES, ALL>(P, P2, smem, st)
                  : (R == 4 ? launch_rows<1024, 4, FROM_CODES, ALL>(P, P2, smem, st)
                            : launch_rows<1024, 2, FROM_CODES, ALL>(P, P2, smem, st));
  };
  auto select = [&]() { return P.want > 0 ? with(std::false_type()) : with(std::true_type()); };
  DistParams T = {};
  T.cb = codebook;
  T.out = static_cast<uint32_t*>(workspace);
  T.V = V;
  T.D = D;
  T.cols = T.pitch = V;
  auto distances = [&](int row0, int row_end) {
    T.row0 = row0;
    T.row_end = row_end;
    const dim3 grid((T.cols + TM - 1) / TM, (row_end - row0 + TM - 1) / TM);
    return launch_chained(row0 == 0 && !T.map, lantern_distance_tile_kernel, grid, 256, 0, st, T);
  };
  // all rows, or the codes of P.map, a block of rows at a time
  auto by_blocks = [&](int block) {
    for (P.row0 = 0; P.row0 < V; P.row0 += block) {
      P.row_end = V - P.row0 < block ? V : P.row0 + block;
      cudaError_t e = P.scratch ? distances(P.row0, P.row_end) : cudaSuccess;
      if (e == cudaSuccess) e = select();
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  };
  if (!P.scratch) return by_blocks(V) == cudaSuccess ? LANTERN_OK : LANTERN_E_CUDA;

  // Every pair once, through lists, where the lists fit with 2.3 to 2.7 standard deviations of room: a row in some hundreds
  // overflows its list and is done again from all its keys.  Half the distances (V^2 D) are saved, some 2 k entries per row go
  // through memory instead (V k): with k = 500, D = 40, lists / blocks of rows take 115 / 108 us at V = 2693, 165 / 145 at 4096,
  // 240 / 228 at 5000 and 253 / 279 at 6000; with D = 100, 156 / 159 at 2693 and 222 / 225 at 4096.  Below 2304 codes the
  // sample is half of them (V = 2048, D = 40, k = 25: 68 / 48).
  ListParams L;
  L.scratch = static_cast<unsigned char*>(workspace);
  L.idx = idx;
  L.dist = dist;
  L.V = V;
  L.k = k;
  L.region = rows_per_block(V) * 4;
  L.cap = static_cast<int>((most + 2.7 * sqrt(static_cast<double>(most))) / f) & ~1;
  const int least = static_cast<int>((most + 2.3 * sqrt(static_cast<double>(most))) / f);
  while (L.cap > least && list_room(L.region, k, dist != nullptr, L.cap) < L.cap) L.cap -= 2;
  const bool pays = V > 2304 && static_cast<long long>(V) * D >= 450ll * k;
  if (pays && P.want > 0 && R == 8 && L.cap > least && L.cap >= k && L.cap <= P.cap) {
    T.sample = 1;
    T.cols = T.pitch = SAMPLE;
    cudaError_t e = distances(0, V);
    if (e != cudaSuccess) return LANTERN_E_CUDA;
    e = launch_chained(false, lantern_row_bound_kernel, dim3((V + 7) / 8), 256, 0, st, L, P.want);
    if (e != cudaSuccess) return LANTERN_E_CUDA;
    const int t = (V + TM - 1) / TM;
    e = launch_chained(false, lantern_distance_lists_kernel, dim3(t * (t + 1) / 2), 256, 0, st, codebook, D, L);
    if (e != cudaSuccess) return LANTERN_E_CUDA;
    const int cap = P.cap;
    P.row0 = 0;
    P.row_end = V;
    P.cap = L.cap;
    e = launch_rows<512, 4, FROM_LISTS>(P, P2, 4 * row_bytes(P.cap), st, L);
    if (e != cudaSuccess) return LANTERN_E_CUDA;
    // the rows whose lists failed, from all their keys: the list of them takes the last rows of the scratch
    P.cap = cap;
    const int block = rows_per_block(V) - TM;
    int* rows = reinterpret_cast<int*>(static_cast<uint32_t*>(workspace) + static_cast<size_t>(block) * V);
    int* count = rows + V;
    e = launch_chained(false, lantern_failed_rows_kernel, dim3(1), 1024, 0, st, static_cast<const int32_t*>(idx), V, k, rows, count);
    if (e != cudaSuccess) return LANTERN_E_CUDA;
    P.map = T.map = rows;
    P.count = T.count = count;
    T.sample = 0;
    T.cols = T.pitch = V;
    return by_blocks(block) == cudaSuccess ? LANTERN_OK : LANTERN_E_CUDA;
  }
  if (by_blocks(rows_per_block(V)) != cudaSuccess) return LANTERN_E_CUDA;
  return LANTERN_OK;
}

// ---------------------------------------------------------------------------------------
// Cosine variant of the latent proximity (Section 5.3.1): codes scaled to unit length, then the
// same neighbour build -- on unit vectors the squared distance is 2 - 2 cos, so increasing
// distance is decreasing cosine similarity.  One thread per code runs the canonical fp32
// sequence: squared norm by one fused multiply-add per dimension in dimension order, one square
// root, one division per component; a zero code stays zero.
// ---------------------------------------------------------------------------------------
namespace lantern {
__global__ void lantern_normalize_rows_kernel(const float* __restrict__ codebook, float* __restrict__ out, int V,
                                              int D) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= V) return;
  const float* a = codebook + static_cast<size_t>(i) * D;
  float n2 = 0.0f;
  for (int d = 0; d < D; ++d) n2 = __fmaf_rn(a[d], a[d], n2);
  const float n = __fsqrt_rn(n2);
  for (int d = 0; d < D; ++d) out[static_cast<size_t>(i) * D + d] = n > 0.0f ? __fdiv_rn(a[d], n) : 0.0f;
}
}  // namespace lantern

static size_t unit_codes_bytes(int V, int D) { return (static_cast<size_t>(V) * D * 4 + 255) & ~static_cast<size_t>(255); }

extern "C" size_t lantern_build_workspace_bytes_metric(int V, int D, int k, int metric) {
  if (V < 1 || D < 1 || (metric != LANTERN_METRIC_L2 && metric != LANTERN_METRIC_COSINE)) return 0;
  const size_t base = lantern_build_workspace_bytes(V, D, k);
  return metric == LANTERN_METRIC_COSINE ? unit_codes_bytes(V, D) + base : base;
}

extern "C" lantern_status lantern_build_neighbors_metric(const float* codebook, int V, int D, int k, int metric,
                                                         int32_t* idx, float* dist, void* workspace,
                                                         size_t workspace_bytes, void* cuda_stream) {
  if (metric == LANTERN_METRIC_L2)
    return lantern_build_neighbors(codebook, V, D, k, idx, dist, workspace, workspace_bytes, cuda_stream);
  if (metric != LANTERN_METRIC_COSINE) return LANTERN_E_PARAM;
  if (V < 1 || V > 32768 || D < 1 || D > 4096 || k < 1 || k > V || k > 4097) return LANTERN_E_SHAPE;
  if (!codebook || !idx) return LANTERN_E_NULL;
  const size_t unit = unit_codes_bytes(V, D);
  if (!workspace || workspace_bytes < lantern_build_workspace_bytes_metric(V, D, k, metric) ||
      (reinterpret_cast<uintptr_t>(workspace) & 255))
    return LANTERN_E_WORKSPACE;
  float* unit_codes = static_cast<float*>(workspace);
  lantern::lantern_normalize_rows_kernel<<<(V + 127) / 128, 128, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      codebook, unit_codes, V, D);
  if (cudaGetLastError() != cudaSuccess) return LANTERN_E_CUDA;
  return lantern_build_neighbors(unit_codes, V, D, k, idx, dist, static_cast<unsigned char*>(workspace) + unit,
                                 workspace_bytes - unit, cuda_stream);
}
