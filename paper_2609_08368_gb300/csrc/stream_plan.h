// The streaming kernel's launch plan, in host-only C++ (no CUDA headers), so
// that the plan can be built and checked without a GPU: which rows k_stream
// takes, with how many CTAs per SM, and the shape of each CTA's ring of
// shared-memory slots. k_stream.cu reads the device's shared-memory limits
// and calls plan_ring; the host tests compile this header on its own.
#pragma once

#include <algorithm>

#include "milesloss.h"

namespace milesloss {

constexpr int kSweepSmemExtra = 1024;  // mbarriers + exchange + reduction scratch
constexpr int kMaxSlots = 16;          // ring slots of k_stream
constexpr int kUnalPad = 16;           // a slot's bytes past its chunk when rows are unaligned

// Which kernel sweeps rows of row_bytes, and with how many streaming CTAs per
// SM: 0 = the cluster kernel, 1 = one streaming CTA per SM (sixteen consumer
// warps, the whole shared memory for its ring), 2 or 4 = that many CTAs per SM
// (eight or four consumer warps, a half or a quarter of the shared memory),
// so that one CTA's per-row merge and epilogue overlap the other CTAs'
// passes. The table is for rows that start 16-byte aligned (others: below). Measured on GB300 (fractions of the copy peak, A/B on one box,
// bf16 and fp32 rows):
//   fused: rows of 192-310 KB one CTA 0.966-0.984 against 0.939-0.959 in
//   clusters; 56-80 KB rows two CTAs 0.956-1.00 against 0.91-0.94; 20-56 KB
//   rows four CTAs 0.93-1.00 against 0.90-0.94 (48 KB fp32 rows: equal);
//   80-192 KB rows in clusters (0.93-0.99 by box; two CTAs ran from 2 % ahead
//   to 1 % behind on 96 KB rows, and one CTA with equal chunks from 3 % ahead
//   to 2 % behind on 136-184 KB bf16 rows, depending on the box), except fp32
//   rows of 120-136 KB (fp32_mid_row) and 136-192 KB (halves_row); 16 KB rows
//   in clusters (fp32 0.91 against 0.79 with four CTAs). With top-K OPD, four
//   CTAs per SM ran 6 % behind the clusters on 32 KB rows; two ran 3-4 %
//   ahead on 64 KB rows.
//   forward only: 200-310 KB rows one CTA (224 / 288 / 302 KB: 1.13 / 1.10
//   / 1.10 against 1.10 / 1.07 / 1.06 with two); 112-200 KB rows two CTAs
//   (151 KB: 1.05 against 0.94 with one, 192 KB: 1.08 against 1.06; a
//   read-only stream can pass the copy peak); 20-112 KB rows four CTAs
//   0.84-1.06 against 0.71-0.96 in clusters (64 KB fp32 rows: 1.07 against
//   1.08).
// The sweep_kernel override forces either kernel, stream_ctas_per_sm the
// CTAs per SM.

// fp32 rows of 120-136 KB (the fp32 workload's 32,768 columns), fused: two
// CTAs per SM with 18 KB chunks, 0.976 / 0.979 / 0.983 / 0.976 / 0.976
// against 0.970 / 0.960 / 0.969 / 0.968 / 0.962 in clusters on five boxes
// (bf16 rows of that length with those chunks: 0.87; with 24-36 KB chunks
// equal to the clusters).
inline bool fp32_mid_row(long long row_bytes, int es, bool grad, bool topk) {
  return grad && !topk && es == 4 && row_bytes > 120 * 1024 && row_bytes <= 136 * 1024;
}

// Fused fp32 rows of 136-192 KB: one CTA per SM with the row in two equal
// chunks (three ring slots up to 150 KB rows, two above), neither kept:
// against the clusters, rows of 136 / 144 / 152 / 160 / 176 KB ran +0.3 /
// +2.9 / +1.8 / +1.7 / +1.3 % on one box, 144 / 160 KB +4.1 / +3.5 % on
// another. (bf16 rows of that length: from 3 % ahead on one box to 2 % behind
// on another, where the clusters ran 0.96-0.99; they stay in clusters.)
inline bool halves_row(long long row_bytes, int es, bool grad, bool unal) {
  constexpr long long KB = 1024;
  return grad && (es == 4 || unal) && row_bytes >= 136 * KB && row_bytes < 192 * KB;
}

// unal: bf16 rows that do not all start on a 16-byte boundary. The cluster
// kernel reads and writes those element by element (4,096 x 45,003: 937 us
// against 135), so all but the shortest (unal_stream_bytes) stream: those the
// table above gives to the cluster kernel with the CTAs per SM that came
// closest to it there.
inline int stream_ctas(long long row_bytes, int es, bool grad, bool topk, bool unal = false) {
  constexpr long long KB = 1024;
  if (unal) {
    const int n = stream_ctas(row_bytes, es, grad, topk);
    if (n > 0) return n;
    if (grad && row_bytes >= 136 * KB) return 1;
    return (topk || row_bytes > 56 * KB) ? 2 : 4;
  }
  if (grad) {
    if (row_bytes >= 192 * KB || halves_row(row_bytes, es, grad, false)) return 1;
    if (fp32_mid_row(row_bytes, es, grad, topk)) return 2;
    if (row_bytes > 56 * KB && row_bytes <= 80 * KB) return 2;
    if (!topk && row_bytes >= 20 * KB && row_bytes <= 56 * KB) return 4;
    return 0;
  }
  if (row_bytes >= 200 * KB) return 1;
  if (row_bytes > 112 * KB) return 2;
  if (row_bytes > 56 * KB) return topk ? 2 : 4;
  if (!topk && row_bytes >= 20 * KB) return 4;
  return 0;
}

// Rows of up to kShortRowBytes that start 16-byte aligned (logits and
// dLogits): k_short, with the row in registers, unless an override asks for a
// launch shape of the other kernels. With top-K OPD (topk = K) one of a row's
// four warps has the candidates while the others wait: past 16 KB and K = 32
// the cluster kernel is faster (k_short / k_sweep, us, 18 KB rows, K = 64: bf16
// fused 16,384 rows 153 / 142, 65,536 577 / 530, forward only 65,536 395 / 380, fp32
// fused 65,536 512 / 476; but 1,024 rows 18.4 / 19.8. K = 32: bf16 fused 4,096 44 /
// 46, 16,384 146 / 140, 65,536 552 / 519, forward only 325 / 372, fp32 fused 435 / 461).
constexpr long long kShortRowBytes = 20 * 1024;
constexpr long long kShortTopKBytes = 16 * 1024;
inline bool plan_forced(const rl_launch_overrides& ov) {
  return ov.sweep_kernel >= 0 || ov.cluster_size > 0 || ov.cluster_stages > 0 ||
         ov.cluster_threads > 0 || ov.cluster_ctas_per_sm > 0 ||
         ov.stream_chunk_bytes > 0 || ov.stream_slots > 0 || ov.stream_hold >= 0 ||
         ov.stream_split_first >= 0 || ov.stream_prefetch_bytes >= 0 ||
         ov.stream_ctas_per_sm > 0 || ov.stream_cluster > 0 ||
         ov.stall_first_wait_ns > 0;
}
inline bool use_short(long long row_bytes, bool unal, int topk, const rl_launch_overrides& ov) {
  if (topk > 32 && row_bytes > kShortTopKBytes) return false;
  return !plan_forced(ov) && !unal && row_bytes < kShortRowBytes;
}
// Unaligned rows stream from these lengths on; shorter ones take the cluster
// kernel, element by element (streamed / that kernel, us a call; 16,384 rows,
// or 1,024 where said). fp32, in the cluster kernel's order: 4 KB 178 / 128, 6
// KB 184 / 163, 8 KB 186 / 198 (1,024: 22.3 / 21.8), 12 KB 189 / 272.
constexpr long long kVirtRowBytes = 8 * 1024;
// bf16: fused 0.4 KB 105 / 81, 1.5 KB 112 / 107 (1,024: 17.7 / 18.8), 3 KB 115 /
// 127; forward only 0.6 KB 71 / 68, 1 KB 73 / 69, 1.5 KB 73 / 83; with top-K, whose
// warp waits for every row's copy, 1 KB 202 / 107, 4 KB 212 / 191, 6 KB 220 / 259
// (1,024: 4 KB 24.3 / 22.9, 6 KB 24.7 / 24.8). Where only dLogits are unaligned the
// cluster kernel still copies its rows whole: 2 KB 102 / 94, 3 KB 106 / 101 (1,024:
// 17.1 / 18.4), 4 KB 108 / 109; with top-K 12 KB 227 / 190, 16 KB 235 / 222 (6,144
// rows: 97 / 103).
inline long long unal_stream_bytes(bool in_bulk, bool grad, bool topk) {
  if (in_bulk) return topk ? 16 * 1024 : 3 * 1024;
  if (topk) return 5 * 1024;
  return grad ? 1536 : 1280;
}
// Warps per row and vectors per lane that hold a row of n_vec vectors.
inline void short_shape(long long n_vec, int* warps, int* nv) {
  *warps = n_vec <= 512 ? 1 : (n_vec <= 1024 ? 2 : 4);
  *nv = n_vec <= 256 ? 8 : (n_vec <= 1024 ? 16 : 10);
}

// The ring. One CTA per SM, measured on GB300 among 44-112 KB chunks and 0-3
// kept chunks (bf16, fused): rows of 240 KB and more run best with three 74
// KB slots, the ragged remainder as the first chunk and the last two chunks
// kept for pass B (0.966-0.984 of the copy peak, against 0.959-0.973 with two
// 112 KB slots); shorter rows with two 112 KB slots and the last chunk kept
// (200 KB rows: 0.972-0.979, against 0.944 with 74 KB slots); a forward-only
// call has no pass B: two 112 KB slots. Several CTAs per SM, measured among
// 8-36 KB chunks and 1-3 kept chunks: two CTAs with three 36 KB slots (every
// chunk kept, up to three; six 18 KB slots for fp32_mid_row rows, three
// kept); four CTAs with the whole row in one slot up to 24 KB rows, else 16
// KB slots up to 44 KB rows, 12 KB slots up to 56 KB rows and 18 KB slots
// past that (forward only), the last chunk kept; chunks of 12 KB or less with
// two CTAs, or 8 KB with four, ran 10-45 % slower. The stream_* overrides
// force a chunk size, slot count, kept chunks, split and CTAs per SM.
constexpr long long kLongRowBytes = 240 * 1024;

struct SmemLimits {
  int optin;     // largest dynamic shared memory one CTA may opt in to
  int per_sm;    // shared memory of one SM
  int reserved;  // shared memory the system reserves per CTA
};

// The streaming kernel's launch plan (ring slots, kept chunks, split, shared
// memory per CTA, consumer warps, CTAs per row).
struct StreamPlan {
  int chunk, slots, hold, split_first, prefetch, smem;
  int cw;         // consumer warps per CTA: 16, 8 or 4 (one, two or four CTAs per SM)
  int cluster;    // CTAs per row: 1, or a cluster of 2, 4 or 8 (one CTA per SM)
  int slice_vec;  // with a cluster: whole 16-byte vectors of a row per CTA
};

// Fused calls without top-K: how many CTAs share a row (a thread-block
// cluster, each CTA streaming one slice of the row through its own ring, one
// CTA per SM). With one CTA per row and per SM, 152 rows are live at once and
// the second read of each row comes from L2 only while they fit in it; each
// row of a cluster costs one exchange between its CTAs, which short slices
// do not repay. Measured on
// GB300 (fractions of the copy peak, the glm recipe's rows with the
// vocabulary shown; one CTA / two / four per row):
//   bf16 400 KB 0.972 / 0.903, 448 KB 0.965 / 0.946, 512 KB 0.916 / 0.934 /
//   0.740, 1 MB - / 0.939 / 0.861, 1.5 MB - / 0.850 / 0.933, 2 MB 0.751 /
//   0.815 / 0.943 (eight: 0.724); fp32 400 KB 0.957 / 0.964, 620 KB 0.899 /
//   0.935 / 0.836; 310 KB (the glm rows) 0.978 / 0.831.
inline int stream_cluster(long long row_bytes, int es, bool grad, bool topk) {
  (void)es;
  constexpr long long KB = 1024;
  if (!grad || topk) return 1;
  if (row_bytes >= 1280 * KB) return 4;
  if (row_bytes >= 480 * KB) return 2;
  return 1;
}

// The whole 16-byte vectors of a row each CTA of a cluster of C takes: an
// even split rounded up to a multiple of 8 (every slice starts 128-byte
// aligned; the last CTA takes the rest, possibly nothing).
inline int slice_vectors(long long row_vec, int C) {
  return static_cast<int>(std::max(8LL, ((row_vec + C - 1) / C + 7) / 8 * 8));
}

// The plan for rows of row_bytes (elements of es bytes), given the SM's
// shared-memory limits, the extra shared memory beyond the ring and the
// fixed scratch (with top-K OPD on, its candidate buffers) and the
// overrides; false when a forced value does not fit.
inline bool plan_ring(long long row_bytes, int es, bool grad, bool topk, const SmemLimits& lim,
                      int extra, const rl_launch_overrides& ov, StreamPlan* out,
                      bool unal = false) {
  const int per = ov.stream_ctas_per_sm > 0 ? ov.stream_ctas_per_sm
                                            : std::max(1, stream_ctas(row_bytes, es, grad, topk, unal));
  if (per != 1 && per != 2 && per != 4) return false;
  const bool lng = grad && row_bytes >= kLongRowBytes;
  const int budget = per > 1 ? std::min(lim.optin, lim.per_sm / per - lim.reserved) : lim.optin;
  int chunk_d = lng ? 75776 : 114688, hold_d = lng ? 2 : 1, split_d = lng ? 1 : 0;
  if (per == 1 && halves_row(row_bytes, es, grad, unal)) {
    chunk_d = static_cast<int>(((row_bytes + 1) / 2 + 127) / 128 * 128);
    hold_d = 0;
    split_d = 1;
  } else if (per == 2) {
    chunk_d = fp32_mid_row(row_bytes, es, grad, topk) ? 18432 : 36864;
    hold_d = 3;
    split_d = 1;
  } else if (per == 4) {
    // (rows up to 56 KB take the same chunks in fused and forward-only
    // calls, so that both sum a row in the same order: the same bits)
    const long long whole = (row_bytes + 127) / 128 * 128;
    chunk_d = whole <= 24576 ? static_cast<int>(std::max(1024LL, whole))
                             : (row_bytes <= 44 * 1024 ? 16384
                                                       : (row_bytes <= 56 * 1024 ? 12288 : 18432));
    hold_d = 1;
    split_d = 1;
  }
  const int chunk = ov.stream_chunk_bytes > 0 ? ov.stream_chunk_bytes : chunk_d;
  if (chunk < 1024 || chunk > 131072 || chunk % 128) return false;
  const int slot = chunk + (unal ? kUnalPad : 0);
  int slots = (budget - kSweepSmemExtra - extra) / slot;
  if (slots > kMaxSlots) slots = kMaxSlots;
  if (ov.stream_slots > 0) {
    if (ov.stream_slots > slots) return false;
    slots = ov.stream_slots;
  }
  if (slots < 1) return false;
  const int hold = ov.stream_hold >= 0 ? ov.stream_hold : std::min(hold_d, slots);
  if (hold > slots) return false;
  out->chunk = chunk;
  out->slots = slots;
  out->hold = hold;
  out->split_first = ov.stream_split_first >= 0 ? ov.stream_split_first : split_d;
  out->prefetch = ov.stream_prefetch_bytes >= 0 ? ov.stream_prefetch_bytes : 0;
  out->smem = slots * slot + kSweepSmemExtra + extra;
  out->cw = 16 / per;
  out->cluster = 1;
  out->slice_vec = 0;
  return true;
}

// The plan with the row's CTAs: one (plan_ring over the whole row), or a
// cluster of C, whose CTAs each run plan_ring's one-CTA ring over their
// slice. Only fused calls without top-K run in clusters, and only when
// can_cluster (a call that writes the row's own results, not a vocabulary
// shard's records); other calls take one CTA per row whatever the
// stream_cluster override says, and so does a row whose CTAs per SM are
// forced above one (unless stream_cluster is forced too: no plan). False
// when a forced value does not fit.
inline bool plan_stream_rows(long long row_bytes, int es, bool grad, bool topk, bool can_cluster,
                             const SmemLimits& lim, int extra, const rl_launch_overrides& ov,
                             StreamPlan* out, bool unal = false) {
  const bool can = can_cluster && grad && !topk;
  int C = 1;
  if (can && ov.stream_cluster > 0) C = ov.stream_cluster;
  else if (can && ov.stream_ctas_per_sm <= 1) C = stream_cluster(row_bytes, es, grad, topk);
  if (C == 1) return plan_ring(row_bytes, es, grad, topk, lim, extra, ov, out, unal);
  if (C != 2 && C != 4 && C != 8) return false;
  if (ov.stream_ctas_per_sm > 1) return false;
  const int sv = slice_vectors(row_bytes / 16, C);
  rl_launch_overrides one = ov;
  one.stream_ctas_per_sm = 1;
  if (!plan_ring(static_cast<long long>(sv) * 16, es, grad, topk, lim, extra, one, out, unal))
    return false;
  out->cluster = C;
  out->slice_vec = sv;
  return true;
}

}  // namespace milesloss
