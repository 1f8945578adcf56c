// attn_tc_d128.cu -- the tensor-core attention path, d = 128 (a translation
// unit of its own, so that the two head sizes compile in parallel).
#include "attn_tc.cuh"

namespace topk {

size_t attn_tc_bytes_d128(const AttnArgs& a, int num_sms) { return tc_bytes<128>(a, num_sms); }

int attn_tc_d128(const AttnArgs& a, const DevCtl& ctl, int num_sms, cudaStream_t st) {
  return tc_launch<128>(a, ctl, num_sms, st);
}

}  // namespace topk
