// k_vmemo_u16.cu -- memoising rollout under the variant rule semantics for boards with
// two bytes per cell (C <= 16).
#define AV_MEMO_CELL uint16_t
#define AV_MEMO_STEP VariantParams
#define AV_MEMO_VARIANT
#define AV_MEMO_CONFIGURE configure_vmemo_u16
#define AV_MEMO_LAUNCH launch_rollout_vmemo_u16
#include "k_memo_impl.cuh"
