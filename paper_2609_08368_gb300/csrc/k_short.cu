// The short-row kernel's instantiations without top-K OPD; those with it are
// compiled in k_short_topk.cu (built in parallel).
#include "k_short.cuh"

namespace milesloss {

const void* short_kernel(rl_dtype in, rl_dtype out, bool grad, bool topk, int warps, int nv) {
  if (topk) return short_kernel_topk(in, out, grad, warps, nv);
  if (!grad) return in == RL_BF16 ? pick_short<InBf16, OutBf16, false, false>(warps, nv)
                                  : pick_short<InF32, OutF32, false, false>(warps, nv);
  if (in == RL_BF16) return out == RL_BF16 ? pick_short<InBf16, OutBf16, true, false>(warps, nv)
                                           : pick_short<InBf16, OutF32, true, false>(warps, nv);
  return out == RL_BF16 ? pick_short<InF32, OutBf16, true, false>(warps, nv)
                        : pick_short<InF32, OutF32, true, false>(warps, nv);
}

}  // namespace milesloss
