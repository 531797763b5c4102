// Fused context kernel, variant 11: greedy decoding, JSD bound = 1, top-k thresholds = 1.
#define LANTERN_VARIANT_TONE true
#define LANTERN_VARIANT_JSD true
#define LANTERN_VARIANT_TOPK true
#define LANTERN_VARIANT_GREEDY true
#define LANTERN_VARIANT_NAME launch_context_v11
#include "verify_context_variant.cuh"
