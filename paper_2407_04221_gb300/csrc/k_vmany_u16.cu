// k_vmany_u16.cu -- memoising rollout under the variant rule semantics for rules that
// match in many places, boards with two bytes per cell (C <= 16).
#define AV_MEMO_CELL uint16_t
#define AV_MEMO_STEP VariantManyParams
#define AV_MEMO_VARIANT
#define AV_MEMO_CONFIGURE configure_vmany_u16
#define AV_MEMO_LAUNCH launch_rollout_vmany_u16
#include "k_memo_impl.cuh"
