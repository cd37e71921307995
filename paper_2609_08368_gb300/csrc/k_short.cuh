// The vocabulary sweep for short rows (up to kShortRowBytes): the same per-row
// results as k_sweep and k_stream, with the whole row in the registers of one
// to four warps.
//
// A row of a few KB is over before a ring of shared-memory slots pays: per row
// the other sweeps spend a copy's latency, two block barriers and one thread's
// epilogue, in a chain that too few CTAs per SM hide (2,048 rows x 4,096 bf16,
// k_sweep: 16.3 us against 5 of traffic). Here kW warps own a row: every lane
// loads its kNV vectors at once (16-byte streaming loads, 8 KB in flight per
// warp), sums them from registers, the warps merge their sums by shuffles and
// one exchange in shared memory, every lane evaluates the per-token objective
// (nothing to broadcast), and dLogits are formed from the same registers: each
// logit is read once. With 128 threads a CTA and up to 128 registers, 16 or
// more warps an SM keep 64-128 KB of loads in flight; CTAs hold no state
// between rows, so the grid is the rows and the hardware balances them.
//
// The sums are k_sweep's, to the bit: its block has 256 threads, of which
// thread v sums the vectors v, v + 256, ... against the maximum of the first;
// the warps here stand in for its eight (kJ of them each, their lanes the
// same), with its fixed orders of merging. The eight warps' butterfly sums
// share their shuffles (at each step a lane keeps half of the values and sends
// the other half, which adds the same pairs).
// Instruction issue bounds it (19 warp instructions per 32 logits and some 950 a
// row, 62 % of the issue slots, before the usual sums skipped the floor, a
// row's mode was chosen outside pass B and the rescale had one test: 32,768
// rows x 2,048 / 4,096 / 9,600 73.1 / 120 / 231 -> 68.3 / 110 / 222 us).
// Measured against k_sweep, whole calls: 32,768 rows x 2,048 / 4,096 / 9,600 bf16
// 179 / 198 / 248 -> 68 / 110 / 222 us; 65,536 x 8,192 435 -> 366; 32,768 x 4,096
// fp32 230 -> 176; forward only, 32,768 x 4,096 / 8,192 bf16 156 / 174 -> 71 / 116.
// Definitions: Sec. 3.4 (ratio), Sec. 2 / 9.1 (advantage), Sec. 2.4 (mask).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace milesloss {

namespace {

constexpr float kLn2s = 0.69314718055994531f;

// The warp's maximum (fp32 order by an order-preserving map to integers).
__device__ __forceinline__ float warp_max_redux(float v) {
  const int i = __float_as_int(v);
  const int r = __reduce_max_sync(0xffffffffu, i ^ ((i >> 31) & 0x7fffffff));
  return __int_as_float(r ^ ((r >> 31) & 0x7fffffff));
}

// The sums over the warp's lanes of N values per lane (N = 4, 8 or 16), as N
// xor butterflies (16, 8, 4, 2, 1) would give them: lane l returns value
// l / (32 / N).
template <int N>
__device__ __forceinline__ float warp_sum_scatter(float* v, int lane) {
  int o = 16;
#pragma unroll
  for (int n = N; n > 1; n /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float send = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// kW warps per row, kNV vectors per lane: rows of up to kW kNV 512 bytes.
template <class In, class Out, bool kGrad, bool kTopK, int kW, int kNV>
__global__ void __launch_bounds__(kShortThreads, kNV > 10 ? 4 : 5) k_short(const ShortArgs a) {
  using St = typename In::storage;
  constexpr int V8 = In::kVec, P = V8 / 2;
  constexpr int kT = kW * 32;                       // threads per row
  constexpr int kRows = kShortThreads / kT;         // rows per CTA
  constexpr int kJ = 8 / kW;                        // warps of k_sweep's block per warp
  constexpr int kI = (kNV + kJ - 1) / kJ;           // vectors per thread of that block
  // m, s, u of that block's eight warps
  __shared__ __align__(16) float red_m[kRows][8], red_su[kRows][2][8];
  __shared__ TopKPart tkp[kRows];
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31;
  const int grp = tid / kT, t = tid % kT, w = t >> 5;
  const long long row = static_cast<long long>(blockIdx.x) * kRows + grp;
  if (row >= a.R) return;  // (whole groups of warps)
  const char* grow = static_cast<const char*>(a.logits) + row * a.ld * static_cast<long long>(sizeof(St));
  const int n_vec = a.V / V8, tail0 = n_vec * V8;

  // ---------------- loads: the row, its scalars
  // top-K OPD: the row's candidates in these columns (the group's first
  // warp): the ids and the teacher's values first, their logits once the row is
  // on its way, the part after pass A. (The values behind pass A, where they
  // are used, cost a load's latency a row: 65,536 rows x 2,048 / 4,096 fp32, K =
  // 32, 216 / 397 -> 198 / 363 us. With sixteen vectors of bf16 a lane there are no
  // registers for them: x 4,096 261 us early, 252 late.)
  constexpr bool kTeachEarly = !(kW == 1 && kNV > 8 && V8 == 8);
  TopKLane tk{-1, -1, 0.0f, 0.0f, false};
  float teach0 = 0.0f, teach1 = 0.0f;
  const float* teacher = a.s.topk_teacher + (kTopK ? row * a.s.topk : 0);
  if (kTopK && w == 0) {
    if (kTeachEarly && lane < a.s.topk) teach0 = teacher[lane];
    if (kTeachEarly && lane + 32 < a.s.topk) teach1 = teacher[lane + 32];
    tk = topk_ids(a.s.topk_ids + row * a.s.topk, static_cast<int>(a.col0), a.V, a.vocab_total,
                  a.s.topk, lane);
  }
  uint4 raw[kNV];
#pragma unroll
  for (int i = 0; i < kNV; ++i)
    if (i * kT + t < n_vec) raw[i] = ld_stream_u4(grow + static_cast<size_t>(i * kT + t) * 16);
  const bool has_tail = tail0 + t < a.V;            // an element past the last whole vector
  float z_tail = -INFINITY;
  if (has_tail) z_tail = In::load1(grow, tail0 + t);
  const long long yl = a.targets[row] - a.col0;
  const int y = (yl >= 0 && yl < a.V) ? static_cast<int>(yl) : -1;
  const bool yok = y >= 0;
  const float rho = a.rho[row];
  const float q = a.q ? a.q[row] : 0.0f;
  const float old = a.old ? a.old[row] : 0.0f;
  const bool trains = a.mask[row] != 0;
  const float zy = yok ? In::load1(grow, y) : 0.0f;
  // The advantage kernel may still run while the first CTAs load and sum
  // their rows; for later ones it is over, and its results are loaded early.
  const bool early = blockIdx.x >= static_cast<unsigned>(a.first_wave);
  float A = 0.0f, cscale = 0.0f;
  auto dependent = [&]() {
    pdl_wait();
    A = a.ws.a_row[row];
    const long long N = a.ws.hdr->n_tokens;
    float g = a.grad_loss;
    if (a.grad_loss_dev) g *= *a.grad_loss_dev;
    cscale = (N > 0) ? g / static_cast<float>(N) * a.s.invT : 0.0f;
  };
  if (early) dependent();
  if (kTopK && w == 0) topk_gather<In>(tk, grow, 0, a.V);
  // ---------------- pass A: raw[j + kJ ii] is vector ii of the thread that
  // has this lane in warp kW j + w of k_sweep's block
  const float k = a.s.k;
  const float2 k2 = make_float2(k, k);
  float vm[kJ], vs[kJ], vu[kJ];
  // against the reference r; safe: with floor_t (the usual sums skip that)
  auto sums = [&](auto safe, int j, float r, float& s, float& u) {
    const float2 nr2 = make_float2(-r, -r);
    float2 s0 = make_float2(0.0f, 0.0f), s1 = s0, u0 = s0, u1 = s0;
#pragma unroll
    for (int ii = 0; ii < kI; ++ii) {
      const int i = j + kJ * ii;
      if (i < kNV && i * kT + t < n_vec) {
        float2 f[P];
        In::unpack2(raw[i], f);
#pragma unroll
        for (int e = 0; e < P; ++e) {
          float2 x2 = ffma2(f[e], k2, nr2);
          if (decltype(safe)::value) x2 = floor_t2(x2);
          const float2 x = ex2x2(x2);
          if (ii & 1) {
            s1 = fadd2(s1, x);
            u1 = ffma2(x, x2, u1);
          } else {
            s0 = fadd2(s0, x);
            u0 = ffma2(x, x2, u0);
          }
        }
      }
    }
    const float2 s2 = fadd2(s0, s1), u2 = fadd2(u0, u1);
    s = s2.x + s2.y;
    u = u2.x + u2.y;
  };
  uint32_t redo = 0;  // threads whose sums are not finite
#pragma unroll
  for (int j = 0; j < kJ; ++j) {
    vm[j] = -INFINITY;
    vs[j] = vu[j] = 0.0f;
    if (j * kT + t < n_vec) {
      const float r = In::vmax(raw[j]) * k;
      sums(std::false_type{}, j, r, vs[j], vu[j]);
      vm[j] = r;
      if (!(fabsf(vs[j]) < INFINITY) || !(fabsf(vu[j]) < INFINITY) || r < kNoLogit) redo |= 1u << j;
    }
  }
  if (redo) {  // (rare: an overflow, or a masked logit) the thread's own maximum
#pragma unroll
    for (int j = 0; j < kJ; ++j) {
      if (!(redo >> j & 1u)) continue;
      typename In::MaxAcc macc = In::kMaxInit;
#pragma unroll
      for (int ii = 0; ii < kI; ++ii) {
        const int i = j + kJ * ii;
        if (i < kNV && i * kT + t < n_vec) macc = In::max_acc(macc, raw[i]);
      }
      vm[j] = In::max_val(macc) * k;
      vs[j] = vu[j] = 0.0f;
      if (vm[j] < kNoLogit) vm[j] = -INFINITY;
      else sums(std::true_type{}, j, vm[j], vs[j], vu[j]);
    }
  }
  float most = vs[0];
#pragma unroll
  for (int j = 1; j < kJ; ++j) most = fmaxf(most, vs[j]);
  if (most >= 131072.0f) {  // sums past 2^16 move the reference up by their binary exponent
#pragma unroll
    for (int j = 0; j < kJ; ++j) {
      const int e = ((__float_as_int(vs[j]) >> 23) & 0xff) - 127;
      if (e > 16) {
        const float f = __int_as_float((127 - e) << 23), d = static_cast<float>(e);
        vu[j] = f * fmaf(-d, vs[j], vu[j]);
        vs[j] *= f;
        vm[j] += d;
      }
    }
  }
  const float zk = z_tail * k;
  if (has_tail && !(zk < kNoLogit)) {  // (the block's first threads: j = 0 of warp 0)
    if (zk > vm[0]) {
      if (vs[0] > 0.0f) {
        const float d = vm[0] - zk, f = ex2(d);
        vu[0] = f * fmaf(d, vs[0], vu[0]);
        vs[0] *= f;
      }
      vm[0] = zk;
    }
    const float tt = fmaf(z_tail, k, -vm[0]), x = ex2(tt);
    vs[0] += x;
    vu[0] = fmaf(x, tt, vu[0]);
  }
  // ---------------- merge: each warp of the block, then the eight in order
  float sum[2 * kJ];
#pragma unroll
  for (int j = 0; j < kJ; ++j) {
    const float M = warp_max_redux(vm[j]);
    sum[j] = sum[kJ + j] = 0.0f;
    if (vs[j] > 0.0f) {
      const float d = vm[j] - M, f = ex2(d);
      sum[j] = f * vs[j];
      sum[kJ + j] = f * fmaf(d, vs[j], vu[j]);
    }
    if (lane == 0) red_m[grp][kW * j + w] = M;
  }
  const float mine = warp_sum_scatter<2 * kJ>(sum, lane);
  {
    constexpr int kL = 32 / (2 * kJ);  // lanes that hold one value
    const int idx = lane / kL;
    if (lane % kL == 0) red_su[grp][idx / kJ][kW * (idx % kJ) + w] = mine;
  }
  TopKPart part{-INFINITY, 0.0f, 0.0f, 0};
  if (kTopK && w == 0) {
    auto value = [=](int i) { return kTeachEarly ? (i < 32 ? teach0 : teach1) : teacher[i]; };
    part = topk_part(tk, value, lane, a.s.invT, k, [](int) { return true; });
    if (lane == 0) tkp[grp] = part;
  }
  if (kW > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(kT) : "memory");
  else __syncwarp();
  if (kTopK && kW > 1) part = tkp[grp];
  float M = -INFINITY, s = 0.0f, u = 0.0f;
  {
    float ms[8], ss[8], us[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      ms[r] = red_m[grp][r];
      ss[r] = red_su[grp][0][r];
      us[r] = red_su[grp][1][r];
      M = fmaxf(M, ms[r]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float d = ms[r] - M, f = ex2(d);
      us[r] = ss[r] > 0.0f ? f * fmaf(d, ss[r], us[r]) : 0.0f;
      ss[r] = ss[r] > 0.0f ? f * ss[r] : 0.0f;
    }
    s = ((ss[0] + ss[4]) + (ss[2] + ss[6])) + ((ss[1] + ss[5]) + (ss[3] + ss[7]));
    u = ((us[0] + us[4]) + (us[2] + us[6])) + ((us[1] + us[5]) + (us[3] + us[7]));
  }
  const bool first = t == 0;
  if (!kGrad && a.part_rows) {
    // vocabulary-sharded forward: the row's partial sums over these columns
    if (!early) pdl_wait();
    if (first) {
      a.part_rows[2 * row] = make_float4(M, s, u, yok ? zy : 0.0f);
      a.part_rows[2 * row + 1] = make_float4(part.m, part.sw, part.acc, part.bad ? 1.0f : 0.0f);
    }
    return;
  }
  if (!early) dependent();

  // ---------------- epilogue (every lane)
  const bool bad = !yok || (kTopK && part.bad);
  const float lnS = logf(s);
  const float lse = fmaf(M, kLn2s, lnS);  // the reference is in log2 units
  float H = lnS - u * kLn2s / s;
  float logp = zy * a.s.invT - lse;
  if (bad) { logp = 0.0f; H = 0.0f; }
  if (kTopK && !bad) A -= a.s.opd_coef * topk_value(part, lse);
  TokenTerms tt = token_terms(logp, H, rho, q, a.q != nullptr, old, a.old != nullptr, A, a.s);
  if (bad) tt = TokenTerms{0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, kFlagBad};
  const WsPtrs& ws = a.ws;
  if (first) {
    if (!yok) atomicOr(&ws.hdr->err_bits, kErrTarget);
    if (kTopK && part.bad) atomicOr(&ws.hdr->err_bits, kErrTopK);
    if (a.out_logp) a.out_logp[row] = logp;
    if (a.out_H) a.out_H[row] = H;
    ws.logp[row] = logp;
    ws.H[row] = H;
    ws.lse[row] = lse;
    ws.G[row] = tt.G;
    ws.ell[row] = tt.ell;
    ws.pg[row] = tt.pg;
    ws.k3[row] = tt.k3;
    ws.r[row] = tt.r;
    ws.rc[row] = tt.rc;
    ws.flags[row] = tt.flags;
  }
  if constexpr (kGrad) {
    // ---------------- pass B: dZ_j = p_j (ca + cb z_j) + cc G 1[j = y]
    char* drow = static_cast<char*>(a.dlogits) + row * a.ld_out * static_cast<long long>(Out::kSize);
    const float cc = (trains && !bad) ? cscale : 0.0f;
    const float ca = cc * (-tt.G + a.s.gamma * (H - lse));
    const float cb = cc * a.s.gamma * a.s.invT;
    const float L2 = M + __log2f(s);
    const bool zero = (cc == 0.0f) || (ca == 0.0f && cb == 0.0f);
    const bool fold = !zero && cb == 0.0f;  // |ca| goes into the exponent
    const float off = fold ? (__log2f(fabsf(ca)) - L2) : -L2;
    // cc [G (1 - p_y) + gamma p_y (log p_y + H)], 1 - p_y = -expm1(logp)
    const float dzy = zero ? 0.0f
                           : cc * (tt.G * -expm1f(logp) + a.s.gamma * expf(logp) * (logp + H));
    const float2 off2 = make_float2(off, off), ca2 = make_float2(ca, ca), cb2 = make_float2(cb, cb);
    const float sgn = (fold && ca < 0.0f) ? -1.0f : 1.0f;
    const int yv = yok ? y / V8 : -1;
    // mode 0: p |ca| with ca's sign, 1: p (ca + cb z), 2: zeros. (The two signs
    // share their code: a small call fetches each form's instructions once per
    // SM, and rows of both signs meet there; a third form cost 2,048 x 4,096
    // in a graph 18.5 -> 20.8 us.)
    const float2 sgn2 = make_float2(sgn, sgn);
    auto pass_b = [&](auto mode) {
      constexpr int kMode = decltype(mode)::value;
#pragma unroll
      for (int i = 0; i < kNV; ++i) {
        const int v = i * kT + t;
        if (v < n_vec) {
          float2 f[P];
          if (kMode == 2) {
#pragma unroll
            for (int e = 0; e < P; ++e) f[e] = make_float2(0.0f, 0.0f);
          } else {
            In::unpack2(raw[i], f);
#pragma unroll
            for (int e = 0; e < P; ++e) {
              const float2 p = ex2x2(ffma2(f[e], k2, off2));
              f[e] = fmul2(p, kMode == 1 ? ent_factor2(f[e], ca2, cb2) : sgn2);
            }
            if (v == yv) {
              float* fv = reinterpret_cast<float*>(f);
#pragma unroll
              for (int e = 0; e < V8; ++e)
                if (v * V8 + e == y) fv[e] = dzy;
            }
          }
          Out::template storev<V8>(drow + static_cast<size_t>(v) * V8 * Out::kSize,
                                   reinterpret_cast<const float*>(f), 0u);
        }
      }
    };
    if (zero) pass_b(std::integral_constant<int, 2>{});
    else if (fold) pass_b(std::integral_constant<int, 0>{});
    else pass_b(std::integral_constant<int, 1>{});
    if (has_tail) {
      float x = 0.0f;
      if (!zero) x = ex2(fmaf(z_tail, k, off)) * (fold ? sgn : ent_factor(z_tail, ca, cb));
      Out::store1(drow, tail0 + t, tail0 + t == y ? dzy : x);
    }
  }
}

template <class In, class Out, bool kGrad, bool kTopK>
const void* pick_short(int warps, int nv) {
  if (warps == 1)
    return nv <= 8 ? reinterpret_cast<const void*>(&k_short<In, Out, kGrad, kTopK, 1, 8>)
                   : reinterpret_cast<const void*>(&k_short<In, Out, kGrad, kTopK, 1, 16>);
  if (warps == 2) return reinterpret_cast<const void*>(&k_short<In, Out, kGrad, kTopK, 2, 16>);
  return reinterpret_cast<const void*>(&k_short<In, Out, kGrad, kTopK, 4, 10>);
}

}  // namespace

}  // namespace milesloss
