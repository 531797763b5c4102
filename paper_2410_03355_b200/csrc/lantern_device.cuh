// Device-side helpers shared by the LANTERN kernels: warp reductions and scans, the JSD mass bound, mbarrier + bulk-copy (TMA) wrappers for sm_100a.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace lantern {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------------------
// warp primitives
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ double warp_incl_scan(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    double t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// ---------------------------------------------------------------------------------------
// JSD bound (Section 5.3.2).  Moving mass S onto a token of probability q0 changes the
// distribution by JSD (natural logarithm; only the collapsed tokens contribute)
//   f(S) = 1/2 [ S ln 2 + q0 ln(1 - x) + (q0 + S) ln(1 + x) ],   x = S / (2 q0 + S),
// since (q0 + S) / mid = 1 + x and q0 / mid = 1 - x for mid = q0 + S/2.  f is increasing and
// convex in S with f' = 1/2 [ln 2 + ln(1 + x)], so "f(S) < delta" is "S < S*" with f(S*) = delta,
// and the prefix test stays a comparison of a running sum with one number per draft.  It is found by a
// whole warp (all 32 lanes call it and get the same value): S ln2 / 2 <= f(S) <= S ln 2, so the root lies
// in [delta / ln 2, 2 delta / ln 2]; three rounds in which the 32 lanes evaluate f (single precision) at
// 32 points of the current interval and a ballot picks the sub-interval narrow it by 33^3, and one Newton
// step in double precision finishes (|f(S*) - delta| below 1e-8 over delta in [1e-7, 2], q0 in [0, 1] on a
// CPU replica; the decision window is 1e-6).  A third of the latency of Newton's method by one thread,
// and this sits on every context's critical path.
// ---------------------------------------------------------------------------------------
static __device__ __forceinline__ double jsd_mass_bound_warp(double delta, double q0, int lane) {
  const double LN2 = 0.69314718055994530942;
  if (!(delta > 0.0)) return 0.0;
  if (!(q0 > 0.0)) return delta / LN2;   // f(S) = S ln 2 exactly
  const float LN2F = 0.693147182464599609375f;
  const float qf = static_cast<float>(q0), df = static_cast<float>(delta);
  float lo = df / LN2F, w = lo;          // the root lies in [lo, lo + w]
#pragma unroll 1
  for (int round = 0; round < 3; ++round) {
    const float step = w * (1.0f / 33.0f);
    const float Sf = lo + step * static_cast<float>(lane + 1);
    const float x = Sf / (2.0f * qf + Sf);
    const float t = Sf * LN2F + (qf + Sf) * log1pf(x) + (x < 1.0f ? qf * log1pf(-x) : 0.0f);   // q0 ln(1 - x) -> 0 with q0
    const int below = __popc(__ballot_sync(0xffffffffu, 0.5f * t < df));   // f is increasing: a prefix of the lanes
    lo += step * static_cast<float>(below);
    w = step;
  }
  double S = static_cast<double>(lo) + 0.5 * static_cast<double>(w);
  {
    const double x = S / (2.0 * q0 + S);
    const double lp = log1p(x);
    const double t = S * LN2 + (q0 + S) * lp + q0 * log1p(-x);
    S -= (0.5 * t - delta) / (0.5 * (LN2 + lp));
  }
  return S;
}

// ---------------------------------------------------------------------------------------
// shared-memory barrier (mbarrier) and bulk asynchronous copy global -> shared
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
// One bulk copy of `bytes` (multiple of 16, both addresses 16-byte aligned) that reports its
// completion to `bar`.  No multicast: the destination is this CTA's own shared memory.
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst_smem)),
               "l"(src_gmem), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
// Bounded wait for phase `parity` of `bar`.  Returns false if the limit ran out.  Each try may suspend
// the thread in hardware for up to `suspend_ns` (it wakes when the phase completes), so a long wait costs
// few issue slots; the hint is an upper limit, the loop bound is what ends a wait that never completes.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t max_tries = (1u << 21),
                                          uint32_t suspend_ns = 4000) {
  const uint32_t a = smem_addr(bar);
  for (uint32_t i = 0; i < max_tries; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity), "r"(suspend_ns)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// ---------------------------------------------------------------------------------------
// fp32 helpers
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed pairs of fp32 values (Blackwell's two-wide fp32 instructions): each lane is rounded exactly
// like the scalar instruction, so results do not depend on the packing.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// a load that stays where it is written (issued early on purpose; the value is used much later)
__device__ __forceinline__ int ld_nc_here(const int32_t* p) {
  int v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ld_nc_here4(const int32_t* p) {
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// 16 bytes of a row that nobody reads twice from this SM
__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// maximum over the warp in one instruction (a NaN is passed over)
__device__ __forceinline__ float redux_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Programmatic dependent launch: wait for the kernels this one depends on (a no-op where it was launched normally); let
// the kernel that depends on this one be put in place.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Host side: which devices a kernel's shared-memory limit has been raised on (ordinals 0..63; beyond that it is raised every
// time).  The limit belongs to the kernel and is shared by all host threads: always the largest value that any call needs.
struct DeviceFlags {
  std::atomic<unsigned long long> bits{0};
};
template <class K>
static inline cudaError_t allow_shared_memory(K kernel, size_t bytes, DeviceFlags& ready) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (ready.bits.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  if (e == cudaSuccess) ready.bits.fetch_or(bit, std::memory_order_release);
  return e;
}

}  // namespace lantern
