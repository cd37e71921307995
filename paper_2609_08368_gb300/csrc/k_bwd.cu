// dLogits from the per-row state a forward call saved (split forward /
// backward path): the logits are read once more, row statistics come from
// the workspace.
//   dZ_tj = g (m_t / N) (1/T) [G_t (1[j = y_t] - p_j) + gamma p_j (log p_j + H_t)]
// A tile is a contiguous run of kTile columns of one row; blocks stride
// over tiles. Each thread issues all of its 16-byte streaming loads of a tile
// (L1 skipped) before using any, then writes 16-byte streaming stores. Rows
// that do not all start on a 16-byte boundary take an instantiation of their
// own (kUnal): a row's vectors start at its first boundary, and the elements
// before it and after the last whole vector go one by one (1,456 x 130,894
// fp32: 1,034 -> 201 us). Where dLogits are misaligned against the logits
// the whole row goes element by element.
#include "common.cuh"
#include "kernels.h"

namespace milesloss {

namespace {

template <class In, class Out, bool kUnal>
__global__ void __launch_bounds__(kBwdThreads) k_bwd(const BwdArgs a) {
  constexpr int V8 = In::kVec;
  using St = typename In::storage;
  pdl_trigger();
  WsPtrs ws = a.ws;

  constexpr int kTile = kBwdTile;
  constexpr int kPer = kTile / V8 / kBwdThreads;  // vectors per thread per tile
  // Tile (row, t) of this block, advanced by gridDim.x tiles per step
  // without a division in the loop.
  const int tpr = a.tiles_per_row;
  const long long dq = gridDim.x / tpr;
  const int dr = static_cast<int>(gridDim.x % tpr);
  auto advance = [&](long long& row, int& t) {
    row += dq;
    t += dr;
    if (t >= tpr) { t -= tpr; ++row; }
  };
  // the elements before a row's first vector (-1: no vectors)
  auto head_of = [&](const char* zrow, const char* drow) {
    if (!kUnal) return 0;
    constexpr uintptr_t kAlignOut = V8 * Out::kSize < 16 ? V8 * Out::kSize : 16;
    const int h = static_cast<int>((-reinterpret_cast<uintptr_t>(zrow) & 15u) / sizeof(St));
    const uintptr_t d0 = reinterpret_cast<uintptr_t>(drow) + h * Out::kSize;
    return d0 % kAlignOut == 0 ? h : -1;
  };
  auto row_ptrs = [&](long long row, const char*& zrow, char*& drow) {
    zrow = static_cast<const char*>(a.logits) + row * a.ld * static_cast<long long>(sizeof(St));
    drow = static_cast<char*>(a.dlogits) + row * a.ld_out * static_cast<long long>(Out::kSize);
  };
  // vectors of tile t, which starts at element t * kTile + head (the last
  // tile of a row may be partial)
  auto tile_nv = [&](int t, int head) {
    if (kUnal && head < 0) return 0;
    const int jv = t * kTile + head;
    return max(0, min(a.V - jv, kTile)) / V8;
  };
  // All of a thread's 16-byte streaming loads of a tile are issued before
  // any is used, and the next tile's loads are issued before this tile's
  // arithmetic, so each thread keeps up to 2 kPer loads in flight.
  // rows that do not train (or have a bad target) get zeros: no read
  auto reads = [&](long long row) { return a.mask[row] != 0 && !(ws.flags[row] & kFlagBad); };
  // (rd: whether the row is read; the block's first tile is loaded before the
  // kernel in front has finished, so by the mask alone. bf16 asks for the next
  // tile once and carries the answer over, fp32 asks in here and again: us, bf16
  // 131,072 x 151,936 (T = 0.7) carried 8,560, asked twice 8,760, in here 8,670,
  // 65,536 x 154,880 5,365 / 5,415 / 5,490; fp32 32,768 x 32,768 1,143 / 1,158 /
  // 1,115. Known two tiles ahead it is 7,190 on the first and 1-4 % slower on
  // other calls.)
  constexpr bool kAskInside = V8 == 4;
  auto load_tile = [&](long long row, int t, uint4* raw, bool rd, bool first) {
    const char* zrow;
    char* drow;
    row_ptrs(row, zrow, drow);
    const int head = head_of(zrow, drow);
    const int nv = ((kAskInside && !first) ? reads(row) : rd) ? tile_nv(t, head) : 0;
    zrow += (static_cast<long long>(t) * kTile + head) * static_cast<long long>(sizeof(St));
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int v = threadIdx.x + i * kBwdThreads;
      if (v < nv) raw[i] = ld_stream_u4(zrow + static_cast<size_t>(v) * 16);
    }
  };
  long long row = blockIdx.x / tpr;
  int t = static_cast<int>(blockIdx.x % tpr);
  uint4 raw[kPer], nxt[kPer];
  // (the first tile's loads need nothing of the kernel before this one)
  if (row < a.R) load_tile(row, t, raw, a.mask[row] != 0, true);
  pdl_wait();
  const long long N = ws.hdr->n_tokens;
  float g = a.grad_loss;
  if (a.grad_loss_dev) g *= *a.grad_loss_dev;
  const float cscale = (N > 0) ? g / static_cast<float>(N) * a.invT : 0.0f;
  bool rd = !kAskInside && row < a.R && reads(row);
  while (row < a.R) {
    long long nrow = row;
    int nt = t;
    advance(nrow, nt);
    const bool rd_next = !kAskInside && nrow < a.R && reads(nrow);
    if (nrow < a.R) load_tile(nrow, nt, nxt, rd_next, false);
    const char* zrow;
    char* drow;
    row_ptrs(row, zrow, drow);
    const int head = head_of(zrow, drow);
    const int nv = tile_nv(t, head);
    // the tile's elements [j0, j1), its vectors from jv on
    const int jv = t * kTile + (kUnal ? max(head, 0) : 0);
    const int j0 = (kUnal && t == 0) ? 0 : min(a.V, jv);
    const int j1 = (kUnal && t == tpr - 1) ? a.V : min(a.V, jv + kTile);
    if (kAskInside) rd = reads(row);
    const float cc = rd ? cscale : 0.0f;
    const float G = ws.G[row], H = ws.H[row], lse = ws.lse[row];
    const float ca = cc * (-G + a.gamma * (H - lse));
    const float cb = cc * a.gamma * a.invT;
    const float L2 = lse * 1.4426950408889634f;
    // the target's column in this call's logits (outside [0, V): another
    // shard's, which no tile of this row holds)
    const int y = a.targets[row] - a.col0;
    const bool has_y = y >= j0 && y < j1;
    // The sampled token's entry (only in the tile that holds it):
    // cc [G (1 - p_y) + gamma p_y (log p_y + H)] with 1 - p_y = -expm1(logp),
    // accurate when p_y is close to 1.
    float dzy = 0.0f;
    if (has_y) {
      const float logp = ws.logp[row];
      dzy = cc * (G * -expm1f(logp) + a.gamma * expf(logp) * (logp + H));
    }
    auto value = [&](float z, int j) {
      if (j == y) return dzy;
      return (cc == 0.0f) ? 0.0f : ex2(fmaf(z, a.k, -L2)) * ent_factor(z, ca, cb);
    };
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int v = threadIdx.x + i * kBwdThreads;
      if (v >= nv) continue;
      const int jb = jv + v * V8;
      float f[V8];
      if (cc == 0.0f) {  // (a row that does not train was not read)
#pragma unroll
        for (int e = 0; e < V8; ++e) f[e] = 0.0f;
      } else {
        In::unpack(raw[i], f);
#pragma unroll
        for (int e = 0; e < V8; ++e) f[e] = ex2(fmaf(f[e], a.k, -L2)) * ent_factor(f[e], ca, cb);
        if (has_y && static_cast<unsigned>(y - jb) < static_cast<unsigned>(V8)) {
#pragma unroll
          for (int e = 0; e < V8; ++e)
            if (jb + e == y) f[e] = dzy;
        }
      }
      Out::template storev<V8>(drow + static_cast<size_t>(jb) * Out::kSize, f, 0u);
    }
    // the elements that no vector holds
    const int skip = nv * V8;
    auto element = [&](int j) {
      Out::store1(drow, j, cc == 0.0f ? 0.0f : value(In::load1(zrow, j), j));
    };
    if constexpr (kUnal) {
      if (head < 0) {
        // (a loop of its own, which the compiler can unroll: 4,096 rows x 16,632
        // bf16 376 -> 209 us, x 45,003 727 -> 560)
        for (int j = j0 + skip + threadIdx.x; j < j1; j += kBwdThreads) element(j);
      } else {
        const int before = min(jv, j1) - j0;
        for (int e = threadIdx.x; e < j1 - j0 - skip; e += kBwdThreads)
          element(j0 + e + (e >= before ? skip : 0));
      }
    } else {
      for (int e = threadIdx.x; e < j1 - j0 - skip; e += kBwdThreads) element(j0 + e + skip);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) raw[i] = nxt[i];
    row = nrow;
    t = nt;
    rd = rd_next;
  }
}

}  // namespace

template <bool kUnal>
static const void* pick_bwd(rl_dtype in, rl_dtype out) {
  if (in == RL_BF16)
    return out == RL_BF16 ? reinterpret_cast<const void*>(&k_bwd<InBf16, OutBf16, kUnal>)
                          : reinterpret_cast<const void*>(&k_bwd<InBf16, OutF32, kUnal>);
  return out == RL_BF16 ? reinterpret_cast<const void*>(&k_bwd<InF32, OutBf16, kUnal>)
                        : reinterpret_cast<const void*>(&k_bwd<InF32, OutF32, kUnal>);
}

const void* bwd_kernel(rl_dtype in, rl_dtype out, bool unal) {
  return unal ? pick_bwd<true>(in, out) : pick_bwd<false>(in, out);
}

}  // namespace milesloss
