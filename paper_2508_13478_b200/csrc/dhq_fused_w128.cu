// The fused forward kernels of hidden width 128 (see dhq_fused.cuh), compiled on their own so that
// the widths build side by side.
#include "dhq_fused.cuh"

namespace dhq {

fused_fn fused_pick_128(bool per_token, bool rot, bool spread, bool ahead) { return pick_width<128, true>(per_token, rot, spread, ahead); }
fused_dump_fn fused_pick_dump_128(bool per_token, bool rot) { return pick_dump_width<128, true>(per_token, rot); }
fused_fn fused_pick_both_128(bool per_token) { return pick_both_width<128>(per_token); }
fused_dump_fn fused_pick_both_dump_128(bool per_token) { return pick_both_dump_width<128>(per_token); }
fused_fn fused_pick_narrow_128(bool per_token, bool rot, bool both, bool gabor, bool mixed) { return pick_narrow_width<128>(per_token, rot, both, gabor, mixed); }
fused_fn fused_pick_dup_128(bool per_token, bool rot, bool both, bool gabor, bool mixed) { return pick_dup_width<128>(per_token, rot, both, gabor, mixed); }
fused_calib_fn fused_pick_calib_128(bool rot, bool gabor, bool both) { return pick_calib_width<128>(rot, gabor, both); }
fused_fn fused_pick_mixed_128(bool rot, bool ahead) { return pick_mixed_width<128, true>(rot, ahead); }
fused_dump_fn fused_pick_mixed_dump_128(bool rot) { return pick_mixed_dump_width<128, true>(rot); }
fused_fn fused_pick_gabor_128(bool per_token, bool rot) { return pick_gabor_width<128>(per_token, rot); }
fused_dump_fn fused_pick_gabor_dump_128(bool per_token, bool rot) { return pick_gabor_dump_width<128>(per_token, rot); }
fused_fn fused_pick_gabor_both_128(bool per_token) { return pick_gabor_both_width<128>(per_token); }
fused_dump_fn fused_pick_gabor_both_dump_128(bool per_token) { return pick_gabor_both_dump_width<128>(per_token); }

} // namespace dhq
