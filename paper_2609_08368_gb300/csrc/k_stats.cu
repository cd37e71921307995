// The masked token-mean of the loss and the reported metrics: means over
// training tokens of the PG term, k3, entropy, ratio, |r - 1|, |logp -
// rollout logp| (the train/rollout divergence of Sec. 9.2) and the
// correction ratio (Sec. 3.4), min / max ratio, and exact clip counts.
//
// Each block reduces a fixed strided set of rows into partial results
// (butterfly merges in a fixed order), which are merged in double precision in
// a fixed order: of up to kStatCluster blocks through the shared memory of a
// cluster, of more by the last block to finish (an atomic ticket, no waiting)
// through the workspace. The grid size depends only on the row
// count, so the scalar loss is bit-for-bit reproducible.
//
// Latency bounds the kernel (13 reads per row, 80 bytes, of rows the sweep has
// just written), and the double-precision merge was most of it: 14 doubles
// merged by every warp of the last block are some 1,400 warp instructions on
// a unit that takes one per 16 clocks. Here each of the 16 results has its
// own lanes, 256 threads of (result, subset of the partials), so the merge
// is one operation per 16 partials and a fixed tree.
#include <stddef.h>

#include "common.cuh"
#include "kernels.h"

namespace milesloss {

namespace {

// Per-block partial sums: fp32 within a block (a fixed-order tree over at
// most kStatThreads rows a block; its rounding is far below the statistics'
// tolerance), exact integer counts.
struct Part {
  float v[9];  // ell, pg, k3, H, r, |r-1|, |logp-rho|, rc, |rc-1|
  float rmin, rmax;
  unsigned int c[5];  // n, clip_hi, clip_lo, dual, corr_clip
};
// The 16 results of a StatPart: 0..8 the sums, 9..13 the counts, then the
// smallest and the largest ratio.
constexpr int kCount0 = 9, kMin = 14, kMax = 15;

__device__ __forceinline__ void part_zero(Part& p) {
#pragma unroll
  for (int i = 0; i < 9; ++i) p.v[i] = 0.0f;
  p.rmin = INFINITY;
  p.rmax = -INFINITY;
#pragma unroll
  for (int i = 0; i < 5; ++i) p.c[i] = 0u;
}

// The warp's results, the same in every lane.
__device__ __forceinline__ void warp_reduce(Part& p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int i = 0; i < 9; ++i) p.v[i] += __shfl_xor_sync(0xffffffffu, p.v[i], o);
    p.rmin = fminf(p.rmin, __shfl_xor_sync(0xffffffffu, p.rmin, o));
    p.rmax = fmaxf(p.rmax, __shfl_xor_sync(0xffffffffu, p.rmax, o));
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) p.c[i] = __reduce_add_sync(0xffffffffu, p.c[i]);
}

// Result `q` merged with another of the same kind.
template <class T>
__device__ __forceinline__ T merge_q(int q, T a, T b) {
  return q < kMin ? a + b : (q == kMin ? (b < a ? b : a) : (b > a ? b : a));
}
__device__ __forceinline__ double none_q(int q) {
  return q < kMin ? 0.0 : (q == kMin ? INFINITY : -INFINITY);
}

// One field of the statistics from the merged results f: means over the n
// training tokens (inv = 1 / n); zeros when there are none.
__device__ __forceinline__ void write_stat(rl_loss_stats* o, int q, double f, double n,
                                           double inv) {
  double* means = &o->loss;  // nine consecutive means, as the sums
  int64_t* counts = &o->n_tokens;
  if (q < kCount0) means[q] = n > 0.0 ? f * inv : 0.0;
  else if (q < kMin) counts[q - kCount0] = static_cast<int64_t>(f);
  else if (q == kMin) o->ratio_min = n > 0.0 ? static_cast<float>(f) : 0.0f;
  else o->ratio_max = n > 0.0 ? static_cast<float>(f) : 0.0f;
}
static_assert(offsetof(rl_loss_stats, corr_absdev_mean) == 8 * sizeof(double) &&
                  offsetof(rl_loss_stats, n_corr_clip) ==
                      offsetof(rl_loss_stats, n_tokens) + 4 * sizeof(int64_t),
              "the means and the counts are consecutive");

__global__ void __launch_bounds__(kStatThreads) k_stats(const StatArgs a) {
  constexpr int kWarps = kStatThreads / 32, kSubs = kStatThreads / kStatFields;
  static_assert(kWarps >= kStatCluster, "one row of sh_d per warp, or per block of a cluster");
  __shared__ float sh_f[kWarps][kStatFields];         // the warps' sums and extremes
  __shared__ unsigned int sh_c[kWarps][kStatFields];  // ... and counts
  __shared__ double sh_d[kWarps][kStatFields];
  __shared__ int s_last;
  WsPtrs ws = a.ws;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // one cluster of all the blocks (below): each must know that the first has
  // started before it stores into its shared memory; the wait is after the
  // rows' loads and costs nothing there
  const int NC = static_cast<int>(cluster_nctarank());
  const bool one_cluster = gridDim.x > 1 && static_cast<int>(gridDim.x) == NC;
  if (one_cluster) cluster_arrive();
  pdl_trigger();
  pdl_wait();
  // 1 / N while the rows' loads are on their way (the rows' own count is the
  // call's N; a division in double is some 0.4 us)
  const double n_call = static_cast<double>(ws.hdr->n_tokens);
  const double inv_call = warp == 0 ? 1.0 / n_call : 0.0;
  Part p;
  part_zero(p);
  const long long stride = static_cast<long long>(gridDim.x) * kStatThreads;
  for (long long t = blockIdx.x * static_cast<long long>(kStatThreads) + tid; t < a.R; t += stride) {
    // every load of a row is issued at once (a masked row's values are not used)
    const uint8_t m = a.mask[t], f = ws.flags[t];
    const float r = ws.r[t], rc = ws.rc[t], ell = ws.ell[t], pg = ws.pg[t], k3 = ws.k3[t],
                H = ws.H[t], logp = ws.logp[t], rho = a.rho[t];
    if (!m) continue;
    p.v[0] += ell;
    p.v[1] += pg;
    p.v[2] += k3;
    p.v[3] += H;
    p.v[4] += r;
    p.v[5] += fabsf(r - 1.0f);
    p.v[6] += fabsf(logp - rho);
    p.v[7] += rc;
    p.v[8] += fabsf(rc - 1.0f);
    p.rmin = fminf(p.rmin, r);
    p.rmax = fmaxf(p.rmax, r);
    p.c[0] += 1;
    p.c[1] += (f & kFlagClipHi) ? 1 : 0;
    p.c[2] += (f & kFlagClipLo) ? 1 : 0;
    p.c[3] += (f & kFlagDual) ? 1 : 0;
    p.c[4] += (f & kFlagCorrClip) ? 1 : 0;
  }
  warp_reduce(p);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 9; ++i) sh_f[warp][i] = p.v[i];
    sh_f[warp][kMin] = p.rmin;
    sh_f[warp][kMax] = p.rmax;
#pragma unroll
    for (int i = 0; i < 5; ++i) sh_c[warp][kCount0 + i] = p.c[i];
  }
  __syncthreads();
  if (one_cluster) cluster_wait();
  // the block's results: thread q < 16 merges the warps' result q, in order
  const int q = tid & (kStatFields - 1);
  const bool is_count = q >= kCount0 && q < kMin;
  double mine = 0.0;
  if (tid < kStatFields) {
    if (is_count) {
      unsigned int c = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) c += sh_c[w][q];
      mine = static_cast<double>(c);
    } else {
      float v = sh_f[0][q];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) v = merge_q(q, v, sh_f[w][q]);
      mine = static_cast<double>(v);
    }
  }
  if (one_cluster) {
    // one cluster: every block's results into the first block's shared memory
    const uint32_t rank = cluster_ctarank();
    if (tid < kStatFields)
      st_dsmem_f64(mapa_shared(smem_u32(&sh_d[rank][q]), 0), mine);
    cluster_sync_all();
    if (rank != 0) return;
    if (tid < kStatFields) {
      mine = sh_d[0][q];
      for (int b = 1; b < NC; ++b) mine = merge_q(q, mine, sh_d[b][q]);
    }
  } else if (gridDim.x > 1) {
    if (warp == 0) {
      if (lane < kStatFields) {
        ws.parts[blockIdx.x].f[lane] = mine;
        __threadfence();
      }
      __syncwarp();
      if (lane == 0) {
        const unsigned int ticket = atomicAdd(&ws.hdr->ticket, 1u);
        s_last = (ticket == gridDim.x - 1) ? 1 : 0;
      }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Last block: thread (sub, q) merges result q of the partials sub,
    // sub + 16, ... in order, then the 16 subsets in a fixed order.
    const int sub = tid / kStatFields;
    double v = none_q(q);
    for (int b = sub; b < static_cast<int>(gridDim.x); b += kSubs)
      v = merge_q(q, v, __ldcg(&ws.parts[b].f[q]));
    v = merge_q(q, v, __shfl_xor_sync(0xffffffffu, v, kStatFields));
    if (lane < kStatFields) sh_d[warp][q] = v;
    __syncthreads();
    if (tid < kStatFields) {
      mine = sh_d[0][q];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) mine = merge_q(q, mine, sh_d[w][q]);
    }
    if (tid == 0) ws.hdr->ticket = 0;
  }
  if (warp != 0) return;
  const double n = __shfl_sync(0xffffffffu, mine, kCount0);
  if (lane >= kStatFields) return;
  if (a.part_out) {
    if (q < kCount0) a.part_out->sum[q] = mine;
    else if (q < kMin) a.part_out->count[q - kCount0] = mine;
    else if (q == kMin) a.part_out->max[0] = n > 0.0 ? -mine : -INFINITY;
    else a.part_out->max[1] = n > 0.0 ? mine : -INFINITY;
  } else {
    write_stat(a.out, q, mine, n, n == n_call ? inv_call : 1.0 / n);
  }
}

// The statistics of a sharded call from its shards' combined partials, one
// result per lane.
__global__ void k_finish(const FinishArgs a) {
  const int q = threadIdx.x;
  if (q >= kStatFields || blockIdx.x != 0) return;
  const double n = a.part->count[0];
  const double f = q < kCount0 ? a.part->sum[q]
                               : (q < kMin ? a.part->count[q - kCount0]
                                           : (q == kMin ? -a.part->max[0] : a.part->max[1]));
  write_stat(a.out, q, f, n, 1.0 / n);
}

}  // namespace

const void* stats_kernel() { return reinterpret_cast<const void*>(&k_stats); }
const void* finish_kernel() { return reinterpret_cast<const void*>(&k_finish); }

}  // namespace milesloss
