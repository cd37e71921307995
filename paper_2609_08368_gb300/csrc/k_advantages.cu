// Advantages of the configured estimator (Sec. 3.4: GRPO, GSPO, REINFORCE++
// plain and baseline-relative), the per-row advantage with the one-sample
// on-policy-distillation shaping (Sec. 5.2), the masked token count N, the
// training tokens of every trajectory, and validation of group ids and row
// offsets.
//
// The inputs are a few KB of per-trajectory data plus one byte and one float
// per row, so what bounds the kernel is latency: the chain of loads, the
// double-precision group statistics (GB300 runs double precision at about two
// operations per SM and clock) and, past some ten thousand rows, one SM's
// loads and stores. One thread-block cluster of up to kAdvCluster CTAs does
// all of it: groups and trajectories are spread over its warps, counts are
// added with integer atomics, and two cluster barriers separate the group
// statistics, the row passes and (REINFORCE++) the normalisation. The sweep
// that follows is launched as a programmatic dependent (pdl_trigger below), so
// its first pass over the logits runs meanwhile.
// Every floating-point sum runs in a fixed order (lane-strided partial sums,
// xor-butterfly merges) in double precision and every count is an integer, so
// results are bit-for-bit reproducible, whatever the cluster's size.
#include "common.cuh"
#include "kernels.h"

namespace milesloss {

namespace {

constexpr int kWarps = kAdvThreads / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_maxf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Block-wide merges in a fixed order (valid in every thread): butterflies in
// the warps that hold trajectories, then one over the warps' values, by warp
// 0. A double operation holds the SM's double unit for 16 clocks a warp: when
// every thread summed the warps' values by itself, 32 x 32 of them queued, 8 us
// a merge.
constexpr int kMergeMax = 3;
template <int N>
__device__ void block_merge_d(double (&v)[N], const bool (&is_max)[N], int n_traj,
                              double (&sh)[kMergeMax][kWarps + 1]) {
  static_assert(N <= kMergeMax, "merge scratch");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (warp * 32 < n_traj) v[i] = is_max[i] ? warp_max(v[i]) : warp_sum(v[i]);
    if (lane == 0) sh[i][warp] = v[i];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      double t = lane < kWarps ? sh[i][lane] : (is_max[i] ? -INFINITY : 0.0);
      t = is_max[i] ? warp_max(t) : warp_sum(t);
      if (lane == 0) sh[i][kWarps] = t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = sh[i][kWarps];
}

// The statistics of group g, computed by one warp that scans the group ids
// for the group's members: n, mean, the standard deviation with its floor,
// and whether all rewards are equal. In double precision; a step of the scan
// that meets no member adds nothing and skips the double arithmetic.
struct Group {
  int n, flat;
  double mu, den;
};
__device__ __forceinline__ Group group_stats(const AdvArgs& a, const int* gid, const float* rew,
                                             int g, int lane) {
  Group r;
  int n = 0;
  double sum = 0.0;
  float wmax = -INFINITY, wmin = INFINITY;
#pragma unroll 4
  for (int b = 0; b < a.n_traj; b += 32) {
    const int i = b + lane;
    const bool in = i < a.n_traj && gid[i] == g;
    if (!__any_sync(0xffffffffu, in)) continue;
    if (in) {
      const float w = rew[i];
      ++n;
      sum += static_cast<double>(w);
      wmax = fmaxf(wmax, w);
      wmin = fminf(wmin, w);
    }
  }
  r.n = n = __reduce_add_sync(0xffffffffu, n);
  sum = warp_sum(sum);
  wmax = warp_maxf(wmax);
  wmin = -warp_maxf(-wmin);
  r.mu = n > 0 ? sum / n : 0.0;
  // A group whose rewards are all equal (this includes one-member groups)
  // carries no advantage signal: its GRPO advantages are exactly zero.
  r.flat = (n == 0) || (wmax == wmin);
  r.den = 1.0;
  if (a.normalize_std && !r.flat) {  // (uniform over the warp)
    double ss = 0.0;
#pragma unroll 4
    for (int b = 0; b < a.n_traj; b += 32) {
      const int i = b + lane;
      const bool in = i < a.n_traj && gid[i] == g;
      if (!__any_sync(0xffffffffu, in)) continue;
      if (in) {
        const double d = static_cast<double>(rew[i]) - r.mu;
        ss += d * d;
      }
    }
    ss = warp_sum(ss);
    const int ddof = a.unbiased_std ? 1 : 0;
    r.den = fmax(sqrt(ss / static_cast<double>(n - ddof)), static_cast<double>(a.std_floor));
  }
  return r;
}
__device__ __forceinline__ void group_store(const AdvArgs& a, const Group& r, int g) {
  a.ws.g_mu[g] = r.mu;
  a.ws.g_den[g] = r.den;
  a.ws.g_flag[g] = r.flat;
  if (a.group_sizes) a.group_sizes[g] = r.n;
}

// Group statistics for calls whose groups are too many for one cluster
// (group_kernel_pays), one 32-thread block per group over the whole GPU.
__global__ void __launch_bounds__(32) k_groups(const AdvArgs a) {
  pdl_wait();
  pdl_trigger();
  for (int g = blockIdx.x; g < a.n_groups; g += gridDim.x) {
    const Group r = group_stats(a, a.gid, a.rewards, g, threadIdx.x);
    if (threadIdx.x == 0) group_store(a, r, g);
  }
}

__global__ void __launch_bounds__(kAdvThreads, 1) k_advantages(const AdvArgs a) {
  extern __shared__ __align__(16) int dyn[];
  // whatever ran before the call has finished once this returns; only then may
  // the sweep start, which reads the call's inputs without waiting for them
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = static_cast<int>(cluster_ctarank()), NC = static_cast<int>(cluster_nctarank());
  const int gtid = rank * kAdvThreads + tid, gthreads = NC * kAdvThreads;
  const int gwarp = rank * kWarps + warp, gwarps = NC * kWarps;
  __shared__ unsigned int s_err;
  __shared__ double s_red[kMergeMax][kWarps + 1];
  __shared__ unsigned long long s_tok;
  __shared__ unsigned int s_seq;
  static_assert(sizeof(s_err) + sizeof(s_red) + sizeof(s_tok) + sizeof(s_seq) + 64 <= kAdvStaticBytes,
                "static shared memory beside the tables");
  WsPtrs ws = a.ws;
  // Shared copies, when they fit, of cu (n_traj + 1), group ids and rewards,
  // and the advantages of this CTA's trajectories.
  const bool on_chip = a.smem_traj;
  const int nt = a.n_traj;
  const int* cu = on_chip ? dyn : a.cu;
  const int* gid = on_chip ? dyn + (nt + 1) : a.gid;
  const float* rew = on_chip ? reinterpret_cast<const float*>(dyn + (2 * nt + 1)) : a.rewards;
  float* adv_s = reinterpret_cast<float*>(dyn + (3 * nt + 1));
  if (tid == 0) {
    s_err = 0;
    s_tok = 0;
    s_seq = 0;
    if (rank == 0) {
      ws.hdr->err_bits = 0;
      ws.hdr->ticket = 0;
      ws.hdr->n_tokens = 0;
      ws.hdr->n_seq = 0;
    }
  }
  if (on_chip)
    for (int i = tid; i <= nt; i += kAdvThreads) {
      dyn[i] = a.cu[i];
      if (i < nt) {
        dyn[nt + 1 + i] = a.gid[i];
        reinterpret_cast<float*>(dyn + 2 * nt + 1)[i] = a.rewards[i];
      }
    }
  for (int i = gtid; i < nt; i += gthreads) {
    ws.traj_n[i] = 0;
    if (a.counts_out) a.counts_out[i] = 0;
  }
  __syncthreads();

  // ---- validation (every CTA reads all of the row offsets)
  unsigned int err = 0;
  for (int i = tid; i < nt; i += kAdvThreads) {
    if (cu[i] > cu[i + 1]) err |= kErrSeqlens;
    const int g = gid[i];
    if (g < 0 || g >= a.n_groups) err |= kErrGroup;
  }
  if (tid == 0 && (cu[0] != 0 || static_cast<long long>(cu[nt]) != a.R_total)) err |= kErrSeqlens;
  if (err) atomicOr(&s_err, err);

  // ---- group statistics, one warp per group, the groups dealt to the CTAs in
  // turn
  if (!a.groups_done)
    for (int g = warp * NC + rank; g < a.n_groups; g += gwarps) {
      const Group r = group_stats(a, gid, rew, g, lane);
      if (lane == 0) group_store(a, r, g);
    }
  // every CTA's part of the header, the counts and the group table is written
  __syncthreads();
  cluster_sync_all();
  const bool cu_ok = (s_err & kErrSeqlens) == 0;
  const bool rpp = a.estimator == RL_EST_REINFORCEPP || a.estimator == RL_EST_REINFORCEPP_BASELINE;

  // ---- a trajectory's base value, in double from the group table
  auto base_value = [&](int i) -> double {
    const int g = gid[i];
    const bool gok = g >= 0 && g < a.n_groups;
    const double w = rew[i];
    if (a.estimator == RL_EST_REINFORCEPP) return w;
    if (a.estimator == RL_EST_REINFORCEPP_BASELINE) return gok ? w - ws.g_mu[g] : 0.0;
    if (!gok || ws.g_flag[g]) return 0.0;  // GRPO, GSPO
    return (w - ws.g_mu[g]) / ws.g_den[g];
  };
  auto publish = [&](int i, float A) {
    ws.a_traj[i] = A;
    if (a.advantages) a.advantages[i] = A;
  };

  // ---- passes over the rows, one warp per trajectory (its rows are the
  // contiguous range [cu[i], cu[i+1]); several warps per trajectory when
  // there are fewer trajectories than warps): the lanes count the trajectory's
  // training tokens from 16-byte blocks of the mask and fill its row
  // advantages with 16-byte stores, with the one-sample OPD shaping. GRPO and
  // GSPO know the advantage here and make both in one pass. With invalid row
  // offsets every row gets advantage 0 (plus the shaping) and only N is
  // counted, row by row. A shard sees the part of each trajectory that falls
  // in its rows [row0, row0 + R) (local indices from 0); given the counts of
  // every shard (counts_in), it takes N and the trajectories' counts from
  // them instead of counting.
  const bool lookup = cu_ok && nt > 0;
  const bool mask_vec = (reinterpret_cast<uintptr_t>(a.mask) & 15u) == 0;
  const bool row_vec = (reinterpret_cast<uintptr_t>(ws.a_row) & 15u) == 0;
  const bool opd_vec = a.teacher && ((reinterpret_cast<uintptr_t>(a.rho) |
                                      reinterpret_cast<uintptr_t>(a.teacher)) & 15u) == 0;
  auto opd = [&](long long t) { return a.teacher ? a.opd_coef * (a.rho[t] - a.teacher[t]) : 0.0f; };
  // trajectory i's rows in this call, as local indices [lo, hi)
  auto local_lo = [&](int i) { return max(static_cast<long long>(cu[i]), a.row0) - a.row0; };
  auto local_hi = [&](int i) {
    return max(min(static_cast<long long>(cu[i + 1]), a.row0 + a.R) - a.row0, local_lo(i));
  };
  // With fewer trajectories than warps, wpt warps share each trajectory
  // (warp `sub` of them takes every wpt-th 512-row or 128-row piece).
  const int wpt = nt > 0 ? max(1, gwarps / nt) : 1;
  const int traj_groups = gwarps / wpt;
  const int group = gwarp / wpt, sub = gwarp % wpt;
  auto count_rows = [&](long long lo, long long hi) {  // training tokens in [lo, hi), warp-wide
    int c = 0;
#pragma unroll 2
    for (long long b = (lo & ~15LL) + 16LL * (lane + 32 * sub); b < hi; b += 16LL * 32 * wpt) {
      if (mask_vec && b >= lo && b + 16 <= hi) {
        const uint4 v = *reinterpret_cast<const uint4*>(a.mask + b);
        c += (__popc(__vcmpne4(v.x, 0u)) + __popc(__vcmpne4(v.y, 0u)) +
              __popc(__vcmpne4(v.z, 0u)) + __popc(__vcmpne4(v.w, 0u))) >> 3;
      } else {
        for (long long t = max(b, lo); t < min(b + 16, hi); ++t) c += a.mask[t] != 0;
      }
    }
    return static_cast<int>(__reduce_add_sync(0xffffffffu, c));
  };
  auto write_rows = [&](long long lo, long long hi, float A) {  // row advantages of [lo, hi)
#pragma unroll 2
    for (long long b = (lo & ~3LL) + 4LL * (lane + 32 * sub); b < hi; b += 4LL * 32 * wpt) {
      if (row_vec && b >= lo && b + 4 <= hi && (!a.teacher || opd_vec)) {
        float4 v = make_float4(A, A, A, A);
        if (a.teacher) {
          const float4 r = *reinterpret_cast<const float4*>(a.rho + b);
          const float4 q = *reinterpret_cast<const float4*>(a.teacher + b);
          v.x -= a.opd_coef * (r.x - q.x);
          v.y -= a.opd_coef * (r.y - q.y);
          v.z -= a.opd_coef * (r.z - q.z);
          v.w -= a.opd_coef * (r.w - q.w);
        }
        *reinterpret_cast<float4*>(ws.a_row + b) = v;
      } else {
        for (long long t = max(b, lo); t < min(b + 4, hi); ++t) ws.a_row[t] = A - opd(t);
      }
    }
  };
  // The advantages of the trajectories whose rows this CTA writes, one thread
  // each (a warp's lanes share each double operation), before the row pass.
  // A trajectory shared by several CTAs is published by its first.
  auto own_adv = [&](auto value_of) {
    if (on_chip) {
      const int g0 = rank * kWarps / wpt, g1 = (rank * kWarps + kWarps - 1) / wpt;
      for (int i = tid; i < nt; i += kAdvThreads) {
        const int g = i % traj_groups;
        if (g < g0 || g > g1) continue;
        const float A = value_of(i);
        adv_s[i] = A;
        if (g * wpt >= rank * kWarps) publish(i, A);
      }
      __syncthreads();
    }
  };
  auto adv_of = [&](int i, auto value_of) {
    if (on_chip) return adv_s[i];
    const float A = value_of(i);
    if (sub == 0 && lane == 0) publish(i, A);
    return A;
  };
  auto direct = [&](int i) { return static_cast<float>(base_value(i)); };
  unsigned long long n_tok = 0;  // (lane 0 of each warp, or every thread's own)
  unsigned int n_seq = 0;
  if (lookup) {
    if (a.counts_in)
      for (int i = gtid; i < nt; i += gthreads) {
        const int c = a.counts_in[i];
        ws.traj_n[i] = c;
        n_tok += static_cast<unsigned long long>(c);
        n_seq += c > 0;
      }
    if (!rpp) own_adv(direct);
    if (group < traj_groups)
      for (int i = group; i < nt; i += traj_groups) {
        const long long lo = local_lo(i), hi = local_hi(i);
        if (!a.counts_in) {
          const int c = count_rows(lo, hi);
          if (lane == 0 && c) {  // integers: exact in any order
            n_seq += atomicAdd(&ws.traj_n[i], c) == 0;
            if (a.counts_out) atomicAdd(&a.counts_out[i], c);
            n_tok += static_cast<unsigned long long>(c);
          }
        }
        if (!rpp) write_rows(lo, hi, adv_of(i, direct));
      }
  } else {
    for (long long t = gtid; t < a.R; t += gthreads) {
      n_tok += a.mask[t] != 0;
      if (!rpp) ws.a_row[t] = -opd(t);
    }
    for (int i = gtid; i < nt; i += gthreads)
      if (!rpp) publish(i, static_cast<float>(base_value(i)));
  }
  if (n_tok) atomicAdd(&s_tok, n_tok);
  if (n_seq) atomicAdd(&s_seq, n_seq);
  __syncthreads();
  if (tid == 0) {
    if (s_tok) atomicAdd(reinterpret_cast<unsigned long long*>(&ws.hdr->n_tokens), s_tok);
    if (s_seq)
      atomicAdd(reinterpret_cast<unsigned long long*>(&ws.hdr->n_seq),
                static_cast<unsigned long long>(s_seq));
    if (s_err) atomicOr(&ws.hdr->err_bits, s_err);
  }
  if (!rpp) return;

  // ---- REINFORCE++: normalise the returns over the training tokens, then a
  // second pass writes the row advantages. Every CTA forms the moments, over
  // all trajectories in the same order.
  __syncthreads();
  cluster_sync_all();  // every CTA's counts are in
  const double N = static_cast<double>(__ldcg(&ws.hdr->n_tokens));
  double sb = 0.0, bmax = -INFINITY, bmin = INFINITY;
  for (int i = tid; i < nt; i += kAdvThreads) {
    const int n_i = __ldcg(&ws.traj_n[i]);
    if (n_i == 0) continue;
    const double b = base_value(i);
    sb += b * n_i;
    bmax = fmax(bmax, b);
    bmin = fmin(bmin, b);
  }
  {
    double v[3] = {sb, bmax, -bmin};
    block_merge_d<3>(v, {false, true, true}, nt, s_red);
    sb = v[0];
    bmax = v[1];
    bmin = -v[2];
  }
  const bool zero_all = !(N > 0.0) || !(bmax != bmin);
  const double mu = N > 0.0 ? sb / N : 0.0;
  double ss = 0.0;
  for (int i = tid; i < nt; i += kAdvThreads) {
    const int n_i = __ldcg(&ws.traj_n[i]);
    if (n_i == 0) continue;
    const double d = base_value(i) - mu;
    ss += d * d * n_i;
  }
  {
    double v[1] = {ss};
    block_merge_d<1>(v, {false}, nt, s_red);
    ss = v[0];
  }
  double den = 1.0;
  if (a.normalize_std) {
    const double ddof = a.unbiased_std ? 1.0 : 0.0;
    const double var = N > ddof ? ss / (N - ddof) : 0.0;
    den = fmax(sqrt(var), static_cast<double>(a.std_floor));
  }
  auto final_value = [&](int i) {
    return static_cast<float>(zero_all ? 0.0 : (base_value(i) - mu) / den);
  };
  if (lookup) {
    own_adv(final_value);
    if (group < traj_groups)
      for (int i = group; i < nt; i += traj_groups)
        write_rows(local_lo(i), local_hi(i), adv_of(i, final_value));
  } else {
    for (int i = gtid; i < nt; i += gthreads) publish(i, final_value(i));
    for (long long t = gtid; t < a.R; t += gthreads) ws.a_row[t] = -opd(t);
  }
}

// The usual call: GRPO, with the trajectory tables on chip and no counts asked
// for (k_advantages does the rest). No CTA waits for another: the last counts
// N, checks the inputs and writes the header and the group sizes; every other
// one has a run of trajectories (or, with few trajectories, a piece of one),
// forms the statistics of the groups they belong to (each by one warp, in
// k_advantages' order: the same bits), and writes their advantages and rows.
// What bounds it is one chain: tables, a group's double arithmetic, the rows;
// it ends before the sweep's first row needs it. k_advantages, with two
// barriers of the cluster and the group table's way through L2 in the chain,
// took 7.3-8.3 us from its start on 2,048 rows: with this kernel an eager call of
// 2,048 x 4,096 went from 19.1 to 16.6 us, 3,136 x 15,616 (224 trajectories) 56.2 ->
// 49.8, 27,456 x 33,247 710 -> 682, 32,768 x 32,768 fp32 1,307 -> 1,290.
__global__ void __launch_bounds__(kAdvThreads, 1) k_adv_grpo(const AdvArgs a) {
  extern __shared__ __align__(16) int dyn[];
  pdl_wait();  // as in k_advantages
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = a.n_traj;
  __shared__ unsigned int s_err;
  __shared__ unsigned int s_cnt[kWarps];
  static_assert(sizeof(s_err) + sizeof(s_cnt) + 64 <= kAdvStaticBytes,
                "static shared memory beside the tables");
  int* cu = dyn;
  int* gid = dyn + (nt + 1);
  float* rew = reinterpret_cast<float*>(dyn + (2 * nt + 1));
  float* adv_s = reinterpret_cast<float*>(dyn + (3 * nt + 1));
  WsPtrs ws = a.ws;
  if (tid == 0) s_err = 0;
  for (int i = tid; i <= nt; i += kAdvThreads) {
    cu[i] = a.cu[i];
    if (i < nt) {
      gid[i] = a.gid[i];
      rew[i] = a.rewards[i];
    }
  }
  const int n_row_ctas = static_cast<int>(gridDim.x) - 1;
  const bool counts = static_cast<int>(blockIdx.x) == n_row_ctas;
  unsigned int n_tok = 0;
  if (counts && !a.counts_in) {
    const long long whole = (reinterpret_cast<uintptr_t>(a.mask) & 15u) == 0 ? a.R / 16 : 0;
#pragma unroll 4
    for (long long b = tid; b < whole; b += kAdvThreads) {
      const uint4 v = reinterpret_cast<const uint4*>(a.mask)[b];
      n_tok += (__popc(__vcmpne4(v.x, 0u)) + __popc(__vcmpne4(v.y, 0u)) +
                __popc(__vcmpne4(v.z, 0u)) + __popc(__vcmpne4(v.w, 0u))) >> 3;
    }
    for (long long t = whole * 16 + tid; t < a.R; t += kAdvThreads) n_tok += a.mask[t] != 0;
  }
  __syncthreads();
  unsigned int err = 0;
  for (int i = tid; i < nt; i += kAdvThreads) {
    if (cu[i] > cu[i + 1]) err |= kErrSeqlens;
    const int g = gid[i];
    if (g < 0 || g >= a.n_groups) err |= kErrGroup;
    if (counts && a.counts_in) n_tok += static_cast<unsigned int>(a.counts_in[i]);
  }
  if (tid == 0 && (cu[0] != 0 || static_cast<long long>(cu[nt]) != a.R_total)) err |= kErrSeqlens;
  if (err) atomicOr(&s_err, err);
  n_tok = __reduce_add_sync(0xffffffffu, n_tok);
  if (lane == 0) s_cnt[warp] = n_tok;

  if (counts) {
    __syncthreads();
    if (tid == 0) {
      long long N = 0;
      for (int w = 0; w < kWarps; ++w) N += s_cnt[w];
      ws.hdr->err_bits = s_err;
      ws.hdr->ticket = 0;
      ws.hdr->n_tokens = N;
      ws.hdr->n_seq = 0;  // (GSPO's)
    }
    if (a.group_sizes)
      for (int g = warp; g < a.n_groups; g += kWarps) {
        int n = 0;
        for (int i = lane; i < nt; i += 32) n += gid[i] == g;
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) a.group_sizes[g] = n;
      }
    return;
  }

  // This CTA's trajectories [i0, i1) and, with more CTAs than trajectories,
  // which of `pieces` pieces of its one trajectory's rows.
  const int pieces = max(1, n_row_ctas / nt);
  const int b = static_cast<int>(blockIdx.x);
  const int per = (nt + n_row_ctas - 1) / n_row_ctas;
  const int i0 = min(nt, pieces > 1 ? b / pieces : b * per);
  const int i1 = min(nt, pieces > 1 ? i0 + 1 : i0 + per);
  const int piece = pieces > 1 ? b % pieces : 0;
  for (int i = i0 + warp; i < i1; i += kWarps) {
    // the first of the run's members of a group does the group
    const int g = gid[i];
    bool later = false;
    for (int m = i0 + lane; m < i; m += 32) later |= gid[m] == g;
    if (__any_sync(0xffffffffu, later)) continue;
    Group r{0, 1, 0.0, 1.0};
    if (g >= 0 && g < a.n_groups) r = group_stats(a, gid, rew, g, lane);
    for (int m = i0 + lane; m < i1; m += 32) {
      if (gid[m] != g) continue;
      const float A =
          r.flat ? 0.0f : static_cast<float>((static_cast<double>(rew[m]) - r.mu) / r.den);
      adv_s[m] = A;
      if (piece == 0) {
        ws.a_traj[m] = A;
        if (a.advantages) a.advantages[m] = A;
      }
    }
  }
  __syncthreads();
  const bool cu_ok = (s_err & kErrSeqlens) == 0;
  auto opd = [&](long long t) { return a.teacher ? a.opd_coef * (a.rho[t] - a.teacher[t]) : 0.0f; };
  if (!cu_ok) {  // rows cannot be attributed: advantage 0 (plus the shaping)
    for (long long t = static_cast<long long>(b) * kAdvThreads + tid; t < a.R;
         t += static_cast<long long>(n_row_ctas) * kAdvThreads)
      ws.a_row[t] = -opd(t);
    return;
  }
  // the rows of the run, four to a thread, a warp (or a piece's warps) per trajectory
  const int wpt = max(1, kWarps / max(1, i1 - i0));
  const int n_par = max(1, kWarps / wpt);
  const bool vec = ((reinterpret_cast<uintptr_t>(ws.a_row) |
                     (a.teacher ? reinterpret_cast<uintptr_t>(a.rho) |
                                      reinterpret_cast<uintptr_t>(a.teacher)
                                : 0u)) & 15u) == 0;
  if (warp / wpt >= n_par) return;
  for (int i = i0 + warp / wpt; i < i1; i += n_par) {
    const long long lo = max(static_cast<long long>(cu[i]), a.row0) - a.row0;
    const long long hi = max(min(static_cast<long long>(cu[i + 1]), a.row0 + a.R) - a.row0, lo);
    const float A = adv_s[i];
    const long long step = 4LL * 32 * wpt * pieces;
    for (long long t0 = (lo & ~3LL) + 4LL * (lane + 32 * (warp % wpt + wpt * piece)); t0 < hi;
         t0 += step) {
      if (vec && t0 >= lo && t0 + 4 <= hi) {
        float4 v = make_float4(A, A, A, A);
        if (a.teacher) {
          const float4 p = *reinterpret_cast<const float4*>(a.rho + t0);
          const float4 q = *reinterpret_cast<const float4*>(a.teacher + t0);
          v.x -= a.opd_coef * (p.x - q.x);
          v.y -= a.opd_coef * (p.y - q.y);
          v.z -= a.opd_coef * (p.z - q.z);
          v.w -= a.opd_coef * (p.w - q.w);
        }
        *reinterpret_cast<float4*>(ws.a_row + t0) = v;
      } else {
        for (long long t = max(t0, lo); t < min(t0 + 4, hi); ++t) ws.a_row[t] = A - opd(t);
      }
    }
  }
}

}  // namespace

const void* adv_grpo_kernel() { return reinterpret_cast<const void*>(&k_adv_grpo); }
const void* adv_kernel() { return reinterpret_cast<const void*>(&k_advantages); }
const void* groups_kernel() { return reinterpret_cast<const void*>(&k_groups); }

}  // namespace milesloss
