// Host-side declarations of the layer's causal attention forward (k_attn_fwd.cu).
#pragma once

#include "avtp_internal.cuh"

namespace avtp {

// Workspace of avtp_attn_forward beyond the criterion-B part (which is the plan of
// plan_workspace with the forward's LSE supplied).
struct FwdWs {
  size_t qtile_cu;  // int32 [R + 1]: units of forward_unit_rows() query rows per request, prefix
  size_t total;
};
FwdWs plan_forward_workspace(const avtp_layout_t& L, const avtp_score_args_t& sa, size_t base_bytes);

// Query rows of a CTA's unit: 128 when it takes two heads of a tile, 256 when it takes two
// tiles of a head (KV groups with an odd number of heads).
int forward_unit_rows(const avtp_score_args_t& sa);

// The tcgen05 kernel that writes O and the natural-log LSE; the validation kernel has
// left the unit prefix in the workspace (PrepArgs::qtile_cu).
cudaError_t launch_attn_forward(const avtp_layout_t& L, const avtp_score_args_t& sa, const avtp_forward_args_t& fa,
                                void* ws, const WsPlan& p, const FwdWs& f, cudaStream_t s);

}  // namespace avtp
