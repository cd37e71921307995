// The streaming kernel's instantiations for rows that do not all start on a
// 16-byte boundary, in the logits or in dLogits.
#include "k_stream.cuh"

namespace milesloss {

const void* stream_kernel_unal(rl_dtype in, rl_dtype out, bool grad, bool topk, int cw, bool clu,
                               bool dec) {
  return pick_stream<true>(in, out, grad, topk, cw, clu, dec);
}

}  // namespace milesloss
