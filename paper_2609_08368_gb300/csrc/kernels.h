// Internal interface between the C-ABI layer (abi.cu) and the kernels.
#pragma once

#include <cstdlib>

#include "common.cuh"
#include "stream_plan.h"

namespace milesloss {

constexpr int kMaxStages = 4;
constexpr int kMaxCluster = 8;
constexpr uint32_t kBulkChunk = 16384;    // bytes per cp.async.bulk
// Calls of up to this many rows start while what ran before them ends (their
// first kernel waits there for it). That gives about a launch, 1 to 3 us, at any
// size, so the line is where it is some per cent of a call. Late / early, us,
// calls back to back: 1,024 x 8,192 bf16 16.4 / 15.0, 2,048 x 4,096 16.7 / 15.4,
// 4,096 x 4,096 26.1 / 26.6, 8,192 x 4,096 38.1 / 38.4; streamed, 2,048 x 32,768 56.3 /
// 54.7, 8,192 x 32,768 182.7 / 180.8, 4,096 x 151,936 408.5 / 407.7. The cluster
// kernel loses by it back to back and gains behind another kernel (a matrix
// product of 14 us included): 2,048 x 45,056 75.5 / 78.2 and 90.8 / 86.3, 8,192 x
// 45,056 247.8 / 255.2 and 265.7 / 260.9, with top-K 2,048 x 43,648 81.0 / 84.2 and
// 95.3 / 92.6.
constexpr int kEarlyStartRows = 2048;
constexpr int kAdvThreads = 512;
// CTAs of k_advantages (one cluster). With 1 / 4 / 8, us a call: REINFORCE++, 128
// trajectories of 4 rows x 2,048 39.4 / 26.1 / 24.2, 512 of 4 141 / 54 / 40, 4,096 of 4
// 804 / 274 / 186, 128 of 64 rows x 20,480 154 / 140 / 138; GSPO, 2,048 of 4 306 / 141 /
// 117; 16 trajectories 22.9 / 22.2 / 21.9.
constexpr int kAdvCluster = 8;
constexpr int kBwdThreads = 256;
// k_stream's block: cw consumer warps (16 with one CTA per SM, 8 with two, 4
// with four),
// the producer warp and, with top-K OPD, the top-K warp
// and, where it is decoupled, the epilogue warp: forward-only calls on aligned
// rows, with four CTAs per SM up to 64 KB (calls without / with it: 64 KB rows
// 91.7 / 90.7 us, 80 KB 107.8 / 109.8, 112 KB 143.6 / 148.6, unaligned 56 KB rows
// 113 / 123: the fourth part of an SM's registers is tight for a sixth warp), and
// with fewer where top-K OPD makes the epilogue longer (without top-K equal:
// 8,192 x 65,536 167 / 163, but in a split call of 6,144 rows 343 / 351).
inline bool stream_decoupled(long long row_bytes, bool grad, bool topk, bool unal, int cw) {
  if (grad || unal) return false;
  return cw == 4 ? row_bytes <= 64 * 1024 : topk;
}
__host__ __device__ constexpr int stream_threads(bool topk, int cw, bool dec) {
  return cw * 32 + (topk ? 64 : 32) + (dec ? 32 : 0);
}
constexpr int kShortThreads = 128;
constexpr int kSeqThreads = 256;
constexpr int kAdvSmemBytes = 48 * 1024;  // on-chip trajectory tables when they fit
// The advantage kernels' own (static) shared memory, at most (asserted there).
// It counts towards the 48 KB that a launch gets unasked.
constexpr int kAdvStaticBytes = 1024;
constexpr int kVirtSmem = kMaxCluster * 8 * 16;     // the warps' sums of a row's virtual slices
constexpr int kTopKSmem = 2 * (2 * kMaxTopK * 4);  // two rows of top-K ids + teacher values

struct SweepArgs {
  const void* logits;
  long long ld, R;
  int V;
  int slice;        // columns per CTA (multiple of 16 bytes of input)
  int stages;       // ring depth S
  int stage_bytes;  // bytes per stage (multiple of 128)
  int in_bulk;      // rows are 16-byte aligned: bulk-copy path
  int out_vec;      // dLogits rows are 16-byte aligned: vector stores
  const int* targets;
  const float* rho;
  const float* q;
  const float* old;
  const uint8_t* mask;
  float* out_logp;
  float* out_H;
  void* dlogits;
  long long ld_out;
  float grad_loss;
  const float* grad_loss_dev;
  LossScalars s;
  WsPtrs ws;
  // Test hook (0 = off): the first wait of every CTA waits instead on a
  // barrier nothing completes, bounded by this many nanoseconds, so that the
  // timeout path runs (see rl_launch_overrides).
  unsigned long long stall_ns;
  // A vocabulary-sharded call (forward only): the logits are columns
  // [col0, col0 + V) of a vocabulary of vocab_total ids, a target or top-K
  // candidate outside them is another shard's, and each row's partial sums
  // go to part_rows (two float4 per row, see k_vshard.cu) in place of the
  // epilogue. Unsharded calls: col0 0, vocab_total V, part_rows null.
  long long col0;
  int vocab_total;
  float4* part_rows;
};

struct StreamArgs {
  const void* logits;
  long long ld, R;
  int V;
  int chunk_bytes;  // bytes per ring slot (multiple of 128)
  int n_slots;      // ring depth
  int n_hold;       // last chunks of a row that pass B reads from shared memory (<= n_slots)
  int split_first;  // 1: the first chunk takes the ragged remainder (rounded up to 128 bytes)
  int prefetch;     // bytes of the next row to ask L2 for once a row's first pass is issued
  int first;        // the call's first kernel, launched as a dependent all the same: it waits
                    // for what ran before the call, before anything else
  int virt_slice;   // > 0: unaligned fp32 rows, summed as virt_c slices of this many
  int virt_c;       // elements are by the cluster kernel (k_stream.cuh)
  int slice_vec;    // launched in clusters (one per row): whole vectors of a row per CTA, a
                    // multiple of 8 (the cluster's last CTA may take fewer, or none)
  const int* targets;
  const float* rho;
  const float* q;
  const float* old;
  const uint8_t* mask;
  float* out_logp;
  float* out_H;
  void* dlogits;
  long long ld_out;
  float grad_loss;
  const float* grad_loss_dev;
  LossScalars s;
  WsPtrs ws;
  unsigned long long stall_ns;  // test hook, as in SweepArgs (the consumers' first wait)
  long long col0;               // vocabulary-sharded calls, as in SweepArgs
  int vocab_total;
  float4* part_rows;
};

struct ShortArgs {  // k_short; the fields of SweepArgs that it needs
  const void* logits;
  long long ld, R;
  int V;
  int first_wave;   // CTAs that may start before the advantage kernel has finished
  const int* targets;
  const float* rho;
  const float* q;
  const float* old;
  const uint8_t* mask;
  float* out_logp;
  float* out_H;
  void* dlogits;
  long long ld_out;
  float grad_loss;
  const float* grad_loss_dev;
  LossScalars s;
  WsPtrs ws;
  long long col0;
  int vocab_total;
  float4* part_rows;
};

struct AdvArgs {
  long long R;          // rows of this call (the local rows of a shard)
  long long row0;       // global index of local row 0 (0 unless sharded)
  long long R_total;    // rows of the whole call: cu_seqlens ends here (R unless sharded)
  const int* counts_in; // sharded calls: every trajectory's training tokens over all
                        // shards (then N and the per-trajectory counts come from these)
  int* counts_out;      // sharded calls: this shard's training tokens per trajectory
  int n_traj, n_groups;
  const float* rewards;
  const int* gid;
  const int* cu;
  const uint8_t* mask;
  const float* rho;
  const float* teacher;
  float opd_coef;
  int normalize_std, unbiased_std;
  float std_floor;
  int estimator;   // rl_estimator
  int smem_traj;   // trajectory tables (cu_seqlens, group ids, rewards, advantages)
                   // staged in shared memory
  int groups_done; // k_groups has computed the group statistics
  float* advantages;   // may be null
  int* group_sizes;    // may be null
  WsPtrs ws;
};

struct SeqArgs {
  const int* cu;        // row offsets of the whole call
  const float* rho;     // per-row arrays: this call's rows (local indices)
  const float* old;
  const float* q;
  const uint8_t* mask;
  long long row0, R;    // the call's rows are [row0, row0 + R) of the whole call
  // Sharded calls: sums_out receives, per trajectory, the sums over this
  // call's rows (sum of logp - base, sum of correction weights; [n_traj][2])
  // and nothing else is written; sums_in gives those sums added over every
  // shard, in place of the kernel's own.
  double* sums_out;
  const double* sums_in;
  LossScalars s;
  WsPtrs ws;
};

struct StatArgs {
  long long R;
  const uint8_t* mask;
  const float* rho;
  rl_loss_stats* out;
  rl_loss_partials* part_out;  // a shard: its partial sums instead of the statistics
  WsPtrs ws;
};

struct FinishArgs {
  const rl_loss_partials* part;
  rl_loss_stats* out;
};

struct BwdArgs {
  const void* logits;
  long long ld, R;
  int V;
  int tiles_per_row;
  long long n_tiles;
  const int* targets;
  const uint8_t* mask;
  void* dlogits;
  long long ld_out;
  float grad_loss;
  const float* grad_loss_dev;
  float invT, k, gamma;
  int col0;  // the logits are columns [col0, col0 + V) of the vocabulary
  WsPtrs ws;
};

// The merge of a vocabulary-sharded call: each row's record from every
// column shard (two float4, shard-major: all[2 (k R + row)] and the one after
// it) in shard order, then the row's statistics and per-token objective, as
// the fused sweep's epilogue writes them.
constexpr int kMaxColShards = 64;
constexpr int kMergeThreads = 256;
struct MergeArgs {
  long long R;
  int n_shards;
  long long col_starts[kMaxColShards + 1];
  const float4* all;
  const int* targets;  // vocabulary ids
  const float* rho;
  const float* q;
  const float* old;
  const uint8_t* mask;
  float* out_logp;
  float* out_H;
  LossScalars s;
  WsPtrs ws;
};

constexpr int kBwdTile = kBwdThreads * 8 * 4;  // elements of one row per backward tile

// Kernel entry points (device function pointers usable with cudaLaunchKernelEx).
// topk: top-K OPD on (a separate instantiation, so that calls without it
// carry none of its code)
const void* sweep_kernel(rl_dtype in, rl_dtype out, bool grad, int threads, bool topk);
const void* sweep_kernel_topk(rl_dtype in, rl_dtype out, bool grad, int threads);
// k_short: warps per row and vectors per lane as short_shape gives them
const void* short_kernel(rl_dtype in, rl_dtype out, bool grad, bool topk, int warps, int nv);
const void* short_kernel_topk(rl_dtype in, rl_dtype out, bool grad, int warps, int nv);
// clu: the instantiation that runs in clusters of CTAs per row (fused
// calls without top-K only; nullptr otherwise)
// unal: the instantiations for rows that do not all start on a 16-byte boundary
const void* stream_kernel(rl_dtype in, rl_dtype out, bool grad, bool topk, bool unal, int cw,
                          bool clu, bool dec);
const void* stream_kernel_unal(rl_dtype in, rl_dtype out, bool grad, bool topk, int cw, bool clu,
                               bool dec);

// The process-wide launch-plan overrides set by rl_set_launch_overrides (a
// copy; every field -1 when none are set).
rl_launch_overrides current_overrides();
// The status a workspace's error bits report: the lowest recorded code.
rl_status status_of_bits(uint32_t bits);

// The streaming kernel's launch plan (k_stream.cu, from the pure plan in
// stream_plan.h): whether rows of row_bytes go to it, and its ring of
// shared-memory slots.
// (in_bulk: every row of the logits starts on a 16-byte boundary; unal: not
// every row of the logits and of dLogits does)
bool use_stream(long long row_bytes, int es, bool in_bulk, bool unal, bool grad, bool topk,
                const rl_launch_overrides& ov);
// extra: shared memory beyond the ring and the fixed scratch (kTopKSmem with
// top-K OPD on, else 0); the ring's shape depends on the row length and on
// whether the call writes dLogits
// (can_cluster: the call may run a row over a cluster of CTAs)
rl_status plan_stream(int dev, int extra, long long row_bytes, int es, bool grad, bool topk,
                      bool unal, bool can_cluster, const rl_launch_overrides& ov, StreamPlan* out);
const void* bwd_kernel(rl_dtype in, rl_dtype out, bool unal);
const void* adv_kernel();
const void* adv_grpo_kernel();  // GRPO without counts: a grid of adv_grpo_ctas
// CTAs of k_adv_grpo: one that counts, and one per four groups' worth of
// trajectories (a group's double arithmetic is some 0.3 us of its SM) or per
// 2,048 rows.
inline int adv_grpo_ctas(long long rows, int n_traj) {
  const long long by_rows = (rows + 2047) / 2048, by_traj = (n_traj + 15) / 16;
  const long long n = by_rows > by_traj ? by_rows : by_traj;
  return static_cast<int>(n < 1 ? 1 : (n > 32 ? 32 : n)) + 1;
}
const void* groups_kernel();  // one 32-thread block per group (grid-stride)
constexpr int kMaxGroupBlocks = 65535;
// Whether k_groups spreads the group statistics over the whole GPU before the
// advantage kernel, which else forms them itself. k_advantages' 128 warps deal
// the groups among them and queue for the SMs' double units: from some 64
// groups on that is longer than another launch (REINFORCE++, 3,072 rows x 2,048,
// inside / in k_groups, us: 64 groups of 16 62 / 64, 128 of 4 56 / 50, 128 of 8
// 76 / 64, 256 of 4 105 / 64; 4,096 rows, 512 of 4 268 / 94; GRPO of 4,096
// trajectories, 16 / 64 / 256 groups 157 / 179 / 326 against 168 / 172 / 179).
// k_adv_grpo spreads the trajectories over up to 33 CTAs and forms a group in
// every CTA that meets it, so groups times trajectories count: 128 x 1,024
// 35 / 47, 256 x 1,024 37 / 47, 128 x 2,048 80 / 74, 512 x 2,048 86 / 77,
// 1,024 x 2,048 125 / 81.
inline bool group_kernel_pays(bool grpo_kernel, long long n_groups, long long n_traj) {
  return grpo_kernel ? n_groups * n_traj > (1LL << 20) : n_groups > 64;
}
const void* seq_kernel();
const void* merge_kernel();   // vocabulary-sharded calls: k_vmerge
const void* stats_kernel();
const void* finish_kernel();  // rl_loss_stats from combined partials (one thread)

}  // namespace milesloss
