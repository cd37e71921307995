// The streaming kernel's launch plan on the current device, and its
// instantiations for 16-byte aligned rows (the others are compiled in
// k_stream_unal.cu, a translation unit of their own, built in parallel).
#include "k_stream.cuh"

namespace milesloss {

bool use_stream(long long row_bytes, int es, bool in_bulk, bool unal, bool grad, bool topk,
                const rl_launch_overrides& ov) {
  if (ov.sweep_kernel == 0) return false;
  // (unaligned fp32 logits: in the cluster kernel's order, k_stream.cuh; with
  // a launch shape forced, and below kVirtRowBytes, by that kernel itself)
  if (es == 4 && !in_bulk) return !plan_forced(ov) && row_bytes >= kVirtRowBytes;
  if (ov.sweep_kernel == 1) return true;
  if (es == 2 && unal && row_bytes < unal_stream_bytes(in_bulk, grad, topk)) return false;
  return stream_ctas(row_bytes, es, grad, topk, unal && es == 2) > 0;
}

rl_status plan_stream(int dev, int extra, long long row_bytes, int es, bool grad, bool topk,
                      bool unal, bool can_cluster, const rl_launch_overrides& ov, StreamPlan* out) {
  int optin = 0, per_sm = 0, reserved = 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
          cudaSuccess)
    return RL_ERR_CUDA;
  return plan_stream_rows(row_bytes, es, grad, topk, can_cluster,
                          SmemLimits{optin, per_sm, reserved}, extra, ov, out, unal)
             ? RL_OK
             : RL_ERR_UNSUPPORTED;
}

const void* stream_kernel(rl_dtype in, rl_dtype out, bool grad, bool topk, bool unal, int cw,
                          bool clu, bool dec) {
  return unal ? stream_kernel_unal(in, out, grad, topk, cw, clu, dec)
              : pick_stream<false>(in, out, grad, topk, cw, clu, dec);
}

}  // namespace milesloss
