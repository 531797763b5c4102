// Fused context kernel, variant 9: greedy decoding, JSD bound = 1, top-k thresholds = 0.
#define LANTERN_VARIANT_TONE true
#define LANTERN_VARIANT_JSD true
#define LANTERN_VARIANT_TOPK false
#define LANTERN_VARIANT_GREEDY true
#define LANTERN_VARIANT_NAME launch_context_v9
#include "verify_context_variant.cuh"
