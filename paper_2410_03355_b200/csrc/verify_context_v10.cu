// Fused context kernel, variant 10: greedy decoding, JSD bound = 0, top-k thresholds = 1.
#define LANTERN_VARIANT_TONE true
#define LANTERN_VARIANT_JSD false
#define LANTERN_VARIANT_TOPK true
#define LANTERN_VARIANT_GREEDY true
#define LANTERN_VARIANT_NAME launch_context_v10
#include "verify_context_variant.cuh"
