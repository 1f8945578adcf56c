// attn_tc.cu -- the tensor-core attention path: d = 64 and the choice by shape.
#include "attn_tc.cuh"

namespace topk {

size_t attn_tc_bytes_d128(const AttnArgs& a, int num_sms);
int attn_tc_d128(const AttnArgs& a, const DevCtl& ctl, int num_sms, cudaStream_t st);

// Types, head sizes and masks served here; whether the lists of topk entries
// fit is the plan's answer (no scratch, no launch).
static bool attn_tc_supports(const AttnArgs& a) {
  if (a.dtype != 1 || a.topk > kTcMaxK || a.mask) return false;  // bit masks run on the SIMT kernel
  return a.d == 64 || a.d == 128;
}

size_t attn_tc_workspace_bytes(const AttnArgs& a, int num_sms) {
  if (!attn_tc_supports(a)) return 0;
  return a.d == 64 ? tc_bytes<64>(a, num_sms) : attn_tc_bytes_d128(a, num_sms);
}

int attn_tc(const AttnArgs& a, const DevCtl& ctl, int num_sms, cudaStream_t st) {
  if (!attn_tc_supports(a)) return 0;
  return a.d == 64 ? tc_launch<64>(a, ctl, num_sms, st) : attn_tc_d128(a, ctl, num_sms, st);
}

}  // namespace topk
