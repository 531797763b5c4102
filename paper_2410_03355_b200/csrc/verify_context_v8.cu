// Fused context kernel, variant 8: greedy decoding, JSD bound = 0, top-k thresholds = 0.
#define LANTERN_VARIANT_TONE true
#define LANTERN_VARIANT_JSD false
#define LANTERN_VARIANT_TOPK false
#define LANTERN_VARIANT_GREEDY true
#define LANTERN_VARIANT_NAME launch_context_v8
#include "verify_context_variant.cuh"
