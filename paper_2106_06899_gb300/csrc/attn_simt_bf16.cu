// attn_simt_bf16.cu -- the CUDA-core attention path for bf16 inputs (a
// translation unit of its own, so that it compiles in parallel).
#include "attn_simt.cuh"

namespace topk {

int attn_simt_bf16(const AttnArgs& a, int num_sms, cudaStream_t st) {
  switch (a.d) {
    case 64: return launch_simt<__nv_bfloat16, 64>(a, num_sms, st);
    case 128: return launch_simt<__nv_bfloat16, 128>(a, num_sms, st);
    default: return 0;
  }
}

}  // namespace topk
