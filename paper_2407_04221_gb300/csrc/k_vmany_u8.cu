// k_vmany_u8.cu -- memoising rollout under the variant rule semantics for rules that
// match in many places, boards with one byte per cell (C <= 8).
#define AV_MEMO_CELL uint8_t
#define AV_MEMO_STEP VariantManyParams
#define AV_MEMO_VARIANT
#define AV_MEMO_CONFIGURE configure_vmany_u8
#define AV_MEMO_LAUNCH launch_rollout_vmany_u8
#include "k_memo_impl.cuh"
