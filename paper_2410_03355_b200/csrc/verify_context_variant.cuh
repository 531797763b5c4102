// One compile-time variant (TONE, JSD, TOPK, GREEDY) of the fused context kernel for every row layout:
// included by verify_context_v*.cu after defining LANTERN_VARIANT_{TONE,JSD,TOPK,GREEDY,NAME}.
#include "verify_common.cuh"
#include "verify_context.cuh"

namespace lantern {

template <class SHAPE, int CHC, bool BF16, bool UNC, bool FEW>
static cudaError_t launch_kernel(const VerifyParams& P, long long items, int sms, cudaStream_t st) {
  auto kc = lantern_context_kernel<SHAPE, CHC, BF16, UNC, LANTERN_VARIANT_TONE, LANTERN_VARIANT_JSD, LANTERN_VARIANT_TOPK,
                                   LANTERN_VARIANT_GREEDY, FEW>;
  const size_t groups = SHAPE::NGRP * SHAPE::AREAS;
  const int ctas = sms * SHAPE::CTAS;
  const int grid = static_cast<int>(items < ctas ? items : ctas);   // a few contexts get an SM each
  static DeviceFlags ready;
  const cudaError_t e = allow_shared_memory(kc, groups * ctx_area_bytes(CHC * SHAPE::GT * 8, BF16, UNC), ready);
  if (e != cudaSuccess) return e;
  return launch_dependent(kc, grid, SHAPE::THREADS, groups * ctx_area_bytes(P.V, BF16, UNC), st, P);
}
template <class SHAPE, int CHC, bool BF16, bool UNC>
static cudaError_t launch_shape(const VerifyParams& P, long long items, int sms, cudaStream_t st) {
  if (P.leaves) return launch_kernel<SHAPE, CHC, BF16, UNC, true>(P, items, sms, st);
  return launch_kernel<SHAPE, CHC, BF16, UNC, false>(P, items, sms, st);
}
template <int CHC, bool BF16, bool UNC>
static cudaError_t launch_one(const VerifyParams& P, long long items, int sms, cudaStream_t st) {
  constexpr bool LONG_F32 = CHC == 8 && !BF16;   // fp32 rows beyond 8192 tokens: greedy decoding only
  if constexpr (LONG_F32 && !LANTERN_VARIANT_GREEDY) return cudaErrorInvalidValue;
  else if constexpr (LONG_F32 && UNC) return launch_shape<CtxSingle, CHC / 2, BF16, UNC>(P, items, sms, st);
  else if constexpr (CHC == 8) {                 // rows beyond 8192 tokens whose area takes 64 KB
    const int shape = ctx_shape(P, sms);
    if (shape == 2) return launch_shape<CtxWide, CHC / 2, BF16, UNC>(P, items, sms, st);
    if (shape == 1) return launch_shape<CtxPair, CHC / 2, BF16, UNC>(P, items, sms, st);
    return launch_shape<CtxNarrow, CHC, BF16, UNC>(P, items, sms, st);
  } else {
    return launch_shape<CtxNarrow, CHC, BF16, UNC>(P, items, sms, st);
  }
}
template <int CHC>
static cudaError_t launch_layout(const VerifyParams& P, bool bf, bool un, long long items, int sms, cudaStream_t st) {
  return bf ? (un ? launch_one<CHC, true, true>(P, items, sms, st) : launch_one<CHC, true, false>(P, items, sms, st))
            : (un ? launch_one<CHC, false, true>(P, items, sms, st) : launch_one<CHC, false, false>(P, items, sms, st));
}

cudaError_t LANTERN_VARIANT_NAME(const VerifyParams& P, bool bf, bool un, long long items, int sms, cudaStream_t st) {
  // 8-token chunks per thread of a 256-thread group: the smallest power of two that covers the row
  const int chunks = (P.V + 2047) / 2048;
  return chunks > 4 ? launch_layout<8>(P, bf, un, items, sms, st)
                    : (chunks > 2 ? launch_layout<4>(P, bf, un, items, sms, st)
                                  : (chunks > 1 ? launch_layout<2>(P, bf, un, items, sms, st)
                                                : launch_layout<1>(P, bf, un, items, sms, st)));
}

}  // namespace lantern
