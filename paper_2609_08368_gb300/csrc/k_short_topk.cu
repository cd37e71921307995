// The short-row kernel's instantiations with top-K OPD (Sec. 5.2) on.
#include "k_short.cuh"

namespace milesloss {

const void* short_kernel_topk(rl_dtype in, rl_dtype out, bool grad, int warps, int nv) {
  if (!grad) return in == RL_BF16 ? pick_short<InBf16, OutBf16, false, true>(warps, nv)
                                  : pick_short<InF32, OutF32, false, true>(warps, nv);
  if (in == RL_BF16) return out == RL_BF16 ? pick_short<InBf16, OutBf16, true, true>(warps, nv)
                                           : pick_short<InBf16, OutF32, true, true>(warps, nv);
  return out == RL_BF16 ? pick_short<InF32, OutBf16, true, true>(warps, nv)
                        : pick_short<InF32, OutF32, true, true>(warps, nv);
}

}  // namespace milesloss
