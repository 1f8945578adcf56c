// attn_simt.cu -- the CUDA-core attention path: fp32 inputs and the choice by type.
#include "attn_simt.cuh"

namespace topk {

int attn_simt_bf16(const AttnArgs& a, int num_sms, cudaStream_t st);

// Returns the number of launches (>0) on success, -1 on a CUDA error, 0 if
// the shape is not served here.
int attn_simt(const AttnArgs& a, int num_sms, cudaStream_t st) {
  if (a.dtype != 0) return attn_simt_bf16(a, num_sms, st);
  switch (a.d) {
    case 16: return launch_simt<float, 16>(a, num_sms, st);
    case 32: return launch_simt<float, 32>(a, num_sms, st);
    case 64: return launch_simt<float, 64>(a, num_sms, st);
    case 128: return launch_simt<float, 128>(a, num_sms, st);
    default: return 0;
  }
}

}  // namespace topk
