// Attention over 128 query rows and 128-key tiles on tcgen05, shared by the
// training attention and the prefill: the pipeline is here, a policy says
// which rows and keys an item has, how its operands are loaded and where its
// output goes.
//
// A CTA of six warps takes items of 128 query rows of one (sequence, head):
//   warp 0   copies Q, K and V tiles (128-byte swizzled) into shared memory;
//   warp 1   issues S = Q K^T (M = N = 128, K = 64) into TMEM columns 0..127
//            and O += P V (N = 64, K = 128) into columns 192..255, P read from
//            TMEM columns 128..191 (bf16 pairs);
//   warps 2..5  the softmax, one thread per query row (its TMEM lane), so the
//            maximum and the sum need no exchange between threads; P goes back to
//            TMEM, not through shared memory.
// Two CTAs share an SM (113 KB of shared memory, 256 TMEM columns and 150 of at most
// 168 registers a thread each): while one's chain of MMA, TMEM loads and exponentials waits, the
// other's runs.  The scores are taken against a reference per row that is fixed by
// the first tile the row sees keys in and stays while no later score exceeds it by
// 2^8, so a tile is one pass over its scores, and S is released before the last
// exponentials: the next S product runs under them.  A tile with a score past the
// bound is started again.  With the bound P stays below 2^8, l and |O| below 2^8
// times the keys and the largest |V|; a bound of 2^64 restarts fewer tiles (4 x 12
// heads, N = 1024, k = 4, scores of standard deviation 1, 2 and 4: 93, 93 and 93 us
// against 93, 95 and 125) but lets O overflow from |V| near 2^63 / keys.  32-key chunks that no row of a warp sees (a window tile's
// other windows, a prefix tile past the diagonal) are zeros in P and nothing else.
// Measured (training attention, 4 x 12 heads, N = 1024, k = 4, SingleForward; and 3 x
// 7 heads, N = 301, k = 3, DoubleForward): 131 -> 94 us (343 TFLOP/s over the mask's
// pairs) and 45 -> 22.8 us, against one CTA per SM with two threads per row, P through
// shared memory and a maximum exchanged per tile.  A tile takes an SM about 2,700
// clocks: 512 of exponentials, 700 of MMA, about 950 issue slots per scheduler; the
// rest is latency (TMEM loads, barriers, instruction fetch) that two chains do not
// cover.  Measured and not kept: all 128 scores in registers at once (spills, 168 us),
// two threads per row in this layout (118 us: the per-tile overhead of twice the
// warps), packed scale-and-shift of the scores (moves into register pairs, 104 against
// 94 us).
#pragma once

#include "kf_mma.cuh"
#include "kf_tc.cuh"

namespace kf {
namespace fa {

constexpr int kRows = 128;                            // query rows of an item
constexpr int kKeys = 128;                            // keys of a tile
constexpr int kHD = 64;
constexpr float kRaise = 8.f;                          // a row's reference follows scores past 2^kRaise of it
constexpr int kKSt = 3, kVSt = 3;                     // K and V ring stages
constexpr uint32_t kTileBytes = kRows * kHD * 2;      // 16 KB: Q, a K tile, a V tile
constexpr int kSoftWarps = 4;
constexpr int kThreads = 64 + 32 * kSoftWarps;
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kColP = 128, kColO = 192;
// [Q][K stages][V stages][barriers]; the base must be 1024-byte aligned (it is: no static shared memory lies before it), so two CTAs
// fit an SM's 228 KB
constexpr size_t kSmemBytes = (1 + kKSt + kVSt) * (size_t)kTileBytes + 256;

// the keys a query row sees: keys <= ctx, and [w1lo, w1hi), [w2lo, w2hi)
struct RowVis {
  int ctx, w1lo, w1hi, w2lo, w2hi;
};
// An item's key ranges (an empty one has lo == hi), the smallest ctx of its
// valid rows, and the key tiles of the first, the first two and all ranges
struct Ranges {
  int lo[3], hi[3], cmin, n0, n01, n;
};
__device__ __forceinline__ void count_tiles(Ranges& r) {
  r.n0 = ceil_div(r.hi[0] - r.lo[0], kKeys);
  r.n01 = r.n0 + ceil_div(r.hi[1] - r.lo[1], kKeys);
  r.n = r.n01 + ceil_div(r.hi[2] - r.lo[2], kKeys);
}
// first key and range end of tile j
__device__ __forceinline__ void tile_at(const Ranges& r, int j, int* lo, int* hi) {
  const bool a = j < r.n0, b = j < r.n01;
  *lo = (a ? r.lo[0] : b ? r.lo[1] : r.lo[2]) + (j - (a ? 0 : b ? r.n0 : r.n01)) * kKeys;
  *hi = a ? r.hi[0] : b ? r.hi[1] : r.hi[2];
}
// bits [lo, hi) of the 32-bit word of keys 32 w .. 32 w + 31 of a tile
__device__ __forceinline__ uint32_t word_bits(int w, int lo, int hi) {
  lo = max(lo - 32 * w, 0);
  const int n = max(hi - 32 * w - lo, 0);
  uint32_t r;
  asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(r) : "r"(lo), "r"(n));   // n bits from bit lo, none past bit 31
  return r;
}

// D += A . B with A (M = 128 rows, bf16 pairs) in TMEM
__device__ __forceinline__ void mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 16 columns of this thread's TMEM lane, without the wait
__device__ __forceinline__ void tmem_st16_async(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Policy P:
//   Args, Maps           kernel arguments
//   Item                 one item; item(a, w, lane, Item&, Ranges&) is warp-collective
//   n_items(a)
//   kQByRows             false: load_q(maps, it, sQ, bar) by lane 0 of warp 0 (kTileBytes);
//                        true: q_rows(a, it, sm, first, lane): 32 rows by each softmax warp
//   tile(a, it, kt, kend, lane, d_err)   what a key tile copies: TileRef, by warp 0's lanes
//   tile_bytes / load_k / load_v   the bytes of a K (or V) tile and its copies
//   clear_v(ref, lane, dst)   the V rows that no copy of this tile writes become zeros
//   has_row(a, it, row)  whether the item has this row
//   vis(a, it, row)      the row's visible keys; a row that the item does not have is
//                        given those of a row that it has (its result is not stored):
//                        a row without keys would cost its warp the separate maximum
//                        and the masks in every tile
//   store(a, it, row, o, inv)   the finished row
template <class P>
__global__ void __launch_bounds__(kThreads, 2)
k_attn_tc(const __grid_constant__ typename P::Maps maps, const typename P::Args a, int* d_err, int clear_err) {
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t sQ = smem_u32(sm);
  const uint32_t sK = sQ + kTileBytes;
  const uint32_t sV = sK + kKSt * kTileBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + (1 + kKSt + kVSt) * kTileBytes);
  uint64_t* q_full = bars;
  uint64_t* q_empty = bars + 1;                 // the item's last S product is done
  uint64_t* k_full = bars + 2;                  // [kKSt]
  uint64_t* k_empty = k_full + kKSt;
  uint64_t* v_full = k_empty + kKSt;            // [kVSt]
  uint64_t* v_empty = v_full + kVSt;
  uint64_t* s_full = v_empty + kVSt;            // S_g is complete
  uint64_t* s_free = s_full + 1;                // ... and in registers
  uint64_t* p_full = s_full + 2;                // P_g is in TMEM (and O scaled)
  uint64_t* o_full = s_full + 3;                // P_g V_g is complete
  uint64_t* o_free = s_full + 4;                // the item's O is in registers
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_full + 5);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // (the word is set below, or after a wait of about 2 s)
  if (clear_err && t == 0 && blockIdx.x == 0) atomicExch(d_err, 0);
  if (sQ & 1023) {                              // (uniform) swizzle atoms need the alignment
    if (t == 0) atomicOr(d_err, kErrInternal);
    return;
  }
  const int n_items = P::n_items(a);
  // the CTA's i-th item: rounds of gridDim.x items, walked forwards in even
  // rounds and backwards in odd ones, so that each CTA's items (most keys
  // first) add up to about the same number of tiles; -1 past the last
  auto item_at = [&](int i) -> int {
    const int G = gridDim.x, c = blockIdx.x;
    const long long w = (long long)i * G + ((i & 1) ? G - 1 - c : c);
    return w < n_items ? (int)w : -1;
  };
  if (t == 0) {
    mbar_init(smem_u32(q_full), P::kQByRows ? kSoftWarps : 1);
    mbar_init(smem_u32(q_empty), 1);
    for (int i = 0; i < kKSt; ++i) {
      mbar_init(smem_u32(&k_full[i]), 1);
      mbar_init(smem_u32(&k_empty[i]), 1);
    }
    for (int i = 0; i < kVSt; ++i) {
      mbar_init(smem_u32(&v_full[i]), 1);
      mbar_init(smem_u32(&v_empty[i]), 1);
    }
    mbar_init(smem_u32(s_full), 1);
    mbar_init(smem_u32(s_free), kSoftWarps);
    mbar_init(smem_u32(p_full), kSoftWarps);
    mbar_init(smem_u32(o_full), 1);
    mbar_init(smem_u32(o_free), kSoftWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    bool ok = true;
    int g = 0, it = 0, q_issued = 0, k_issued = 0, v_issued = 0;
    for (int w = item_at(0); ok && w >= 0; w = item_at(++it)) {
      typename P::Item im;
      Ranges r;
      P::item(a, w, lane, im, r);
      if (!P::kQByRows) {
        // the Q buffer is free once the previous item's last S product is done
        if (it > 0) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(q_empty), (it - 1) & 1, d_err));
        if (ok && lane == 0) {
          mbar_expect_tx(smem_u32(q_full), kTileBytes);
          P::load_q(maps, im, sQ, smem_u32(q_full));
        }
        if (ok) q_issued = it + 1;
      }
      for (int j = 0; ok && j < r.n; ++j, ++g) {
        const int ks = g % kKSt, vs = g % kVSt;
        int kt, kend;
        tile_at(r, j, &kt, &kend);
        typename P::TileRef ref = P::tile(a, im, kt, kend, lane, d_err);
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&k_empty[ks]), ((g / kKSt) & 1) ^ 1, d_err));
        if (!ok) break;
        if (lane == 0) mbar_expect_tx(smem_u32(&k_full[ks]), P::tile_bytes(ref));
        __syncwarp();
        P::load_k(maps, a, im, ref, lane, sK + ks * kTileBytes, smem_u32(&k_full[ks]));
        k_issued = g + 1;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&v_empty[vs]), ((g / kVSt) & 1) ^ 1, d_err));
        if (!ok) break;
        P::clear_v(ref, lane, sm + (1 + kKSt + vs) * kTileBytes);
        if (lane == 0) mbar_expect_tx(smem_u32(&v_full[vs]), P::tile_bytes(ref));
        __syncwarp();
        P::load_v(maps, a, im, ref, lane, sV + vs * kTileBytes, smem_u32(&v_full[vs]));
        v_issued = g + 1;
      }
    }
    if (!ok && lane == 0) {
      // let the copies still in flight land before the CTA ends (bounded)
      if (q_issued) mbar_wait(smem_u32(q_full), (q_issued - 1) & 1, d_err);
      for (int n = max(0, k_issued - kKSt); n < k_issued; ++n)
        mbar_wait(smem_u32(&k_full[n % kKSt]), (n / kKSt) & 1, d_err);
      for (int n = max(0, v_issued - kVSt); n < v_issued; ++n)
        mbar_wait(smem_u32(&v_full[n % kVSt]), (n / kVSt) & 1, d_err);
    }
    __syncwarp();
  } else if (warp == 1) {
    constexpr uint32_t idesc_s = idesc_bf16(kRows, kKeys);
    constexpr uint32_t idesc_o = idesc_bf16(kRows, kHD) | (1u << 16);   // B (V) MN-major
    bool ok = true;
    int g = 0, it = 0, o_items = 0;
    // O (+)= P_i V_i once P_i is in TMEM; an item's first tile overwrites O
    // once the softmax has read the previous item's
    auto issue_pv = [&](int i, bool first) -> bool {
      if (first) {
        if (o_items > 0 && !mbar_wait(smem_u32(o_free), (o_items - 1) & 1, d_err)) return false;
        ++o_items;
      }
      const int st = i % kVSt;
      if (!mbar_wait(smem_u32(&v_full[st]), (i / kVSt) & 1, d_err)) return false;
      if (!mbar_wait(smem_u32(p_full), i & 1, d_err)) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t vb = sV + st * kTileBytes;
#pragma unroll
      for (int kk = 0; kk < kKeys / 16; ++kk)
        mma_bf16_ts(tmem + kColO, tmem + kColP + 8 * kk, sdesc_mn(vb + kk * 16 * 128), idesc_o,
                    (!first || kk > 0) ? 1u : 0u);
      mma_commit(smem_u32(o_full));
      mma_commit(smem_u32(&v_empty[st]));
      return true;
    };
    for (int w = item_at(0); ok && w >= 0; w = item_at(++it)) {
      typename P::Item im;
      Ranges r;
      P::item(a, w, lane, im, r);
      if (lane == 0) {
        ok = mbar_wait(smem_u32(q_full), it & 1, d_err);
        for (int j = 0; ok && j < r.n; ++j, ++g) {
          const int st = g % kKSt;
          if (!mbar_wait(smem_u32(&k_full[st]), (g / kKSt) & 1, d_err)) { ok = false; break; }
          if (g >= 1 && !mbar_wait(smem_u32(s_free), (g - 1) & 1, d_err)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t kb = sK + st * kTileBytes;
#pragma unroll
          for (int kk = 0; kk < kHD / 16; ++kk)
            mma_bf16(tmem, sdesc(sQ + kk * 32), sdesc(kb + kk * 32), idesc_s, kk > 0 ? 1u : 0u);
          mma_commit(smem_u32(s_full));
          mma_commit(smem_u32(&k_empty[st]));
          if (j == r.n - 1) mma_commit(smem_u32(q_empty));
          if (j > 0 && !issue_pv(g - 1, j == 1)) { ok = false; break; }
        }
        // the item's last P V follows at once: the softmax's read of O does
        // not wait for the next item's copies
        if (ok && r.n > 0) ok = issue_pv(g - 1, r.n == 1);
        if (ok && r.n == 0) mma_commit(smem_u32(q_empty));
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      g = __shfl_sync(0xffffffffu, g, 0);
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3;                 // TMEM lanes 32 quarter ..
    const int row = 32 * quarter + lane;          // this thread's query row
    const float sc = 1.4426950408889634f * rsqrtf((float)kHD);
    const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16);
    constexpr int NC = kKeys / 32;                // 32-key chunks of a tile
    // A bounded wait that runs out ends this warp's loops; the other warps'
    // waits then run out in turn.
    auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity, d_err));
    };
    auto arrive = [&](uint64_t* bar) {
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(bar));
    };
    auto put_q = [&](int w) {
      typename P::Item im;
      Ranges r;
      P::item(a, w, lane, im, r);
      P::q_rows(a, im, sm, 32 * quarter, lane);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      arrive(q_full);
    };
    bool ok = true;
    int g = 0, it = 0;
    if (P::kQByRows && item_at(0) >= 0) put_q(item_at(0));
    for (int w = item_at(0); ok && w >= 0; w = item_at(++it)) {
      typename P::Item im;
      Ranges r;
      P::item(a, w, lane, im, r);
      const RowVis v = P::vis(a, im, row);
      // m: the reference (in base-2 units) the probabilities so far are taken
      // against; l: their sum
      float m = -INFINITY, l = 0.f;
      for (int j = 0; j < r.n; ++j, ++g) {
        int kt, kend;
        tile_at(r, j, &kt, &kend);
        const bool open = P::all_open(a) && kt + kKeys <= kend && kt + kKeys - 1 <= r.cmin;
        const bool masked = __any_sync(0xffffffffu, !open);
        // the keys of chunk c that this row sees (each key belongs to one
        // range's tiles)
        auto vis_word = [&](int c) -> uint32_t {
          uint32_t vis = word_bits(c, 0, v.ctx - kt + 1);
          if (P::kWindows) vis |= word_bits(c, v.w1lo - kt, v.w1hi - kt) | word_bits(c, v.w2lo - kt, v.w2hi - kt);
          return vis & word_bits(c, 0, kend - kt);
        };
        auto mask_chunk = [&](uint32_t vis, uint32_t* su) {
#pragma unroll
          for (int e = 0; e < 32; ++e) su[e] = (vis >> e) & 1u ? su[e] : 0xff800000u;   // -inf
        };
        float mq[4];
        auto max_chunk = [&](const uint32_t* su) {
#pragma unroll
          for (int e = 0; e < 32; e += 8)
#pragma unroll
            for (int c = 0; c < 4; ++c)
              mq[c] = max3f(mq[c], __uint_as_float(su[e + 2 * c]), __uint_as_float(su[e + 2 * c + 1]));
        };
        // raw scores: sc > 0, so the maximum commutes with the scaling
        auto tile_max = [&] { return fmaxf(fmaxf(mq[0], mq[1]), fmaxf(mq[2], mq[3])) * sc; };
        // a new reference where the row's maximum exceeds it by more than
        // 2^kRaise; O (once P_{g-1} V_{g-1} has been added) and l follow it
        auto raise_to = [&](float mx) -> bool {
          const bool raise = mx > m + kRaise;
          const float f = (raise && m != -INFINITY) ? mma::ex2(m - mx) : 1.f;
          if (__any_sync(0xffffffffu, f != 1.f)) {
            if (!wait(o_full, (g - 1) & 1)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int c = 0; c < kHD / 32; ++c) {
              float rr[32];
              tmem_ld32(lane_base + kColO + 32 * c, rr);
#pragma unroll
              for (int d = 0; d < 32; ++d) rr[d] *= f;
              tmem_st32(lane_base + kColO + 32 * c, rr);
            }
          }
          if (raise) {
            l *= f;
            m = mx;
          }
          return true;
        };
        if (!wait(s_full, g & 1)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // the first tile that a row of this warp sees keys in: the reference
        // is its maximum, a pass of its own
        bool known = __any_sync(0xffffffffu, m == -INFINITY);
        if (known) {
#pragma unroll
          for (int c = 0; c < 4; ++c) mq[c] = -INFINITY;
#pragma unroll 1
          for (int c = 0; c < NC; ++c) {
            const uint32_t vis = masked ? vis_word(c) : ~0u;
            if (masked && !__any_sync(0xffffffffu, vis != 0u)) continue;
            uint32_t su[32];
            tmem_ld32_async(lane_base + 32 * c, su);
            tmem_wait32(su);
            if (masked && !__all_sync(0xffffffffu, vis == ~0u)) mask_chunk(vis, su);
            max_chunk(su);
          }
          if (!raise_to(tile_max())) { ok = false; break; }
        }
        // P = 2^(S sc - m) rounded to bf16 (2^-inf = 0 for masked keys) and the
        // sum of the rounded values, in one pass against the reference so
        // far; only a maximum past 2^kRaise of it (seen before S is released)
        // raises the reference and starts the tile again
        uint64_t ps[4];
        bool again;
        do {
          again = false;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            ps[c] = 0ull;
            mq[c] = -INFINITY;
          }
          const float nm = m == -INFINITY ? 0.f : -m;
          uint32_t su[2][32];
          tmem_ld32_async(lane_base, su[0]);
#pragma unroll 1
          for (int c2 = 0; c2 < NC && !again; c2 += 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int c = c2 + h;
              tmem_wait32(su[h]);
              if (c + 1 < NC) tmem_ld32_async(lane_base + 32 * (c + 1), su[h ^ 1]);
              const uint32_t vis = masked ? vis_word(c) : ~0u;
              const bool some = !masked || __any_sync(0xffffffffu, vis != 0u);
              if (some) {
                if (masked && !__all_sync(0xffffffffu, vis == ~0u)) mask_chunk(vis, su[h]);
                if (!known) max_chunk(su[h]);
              }
              if (h == 1 && c2 == NC - 2) {
                if (!known && __any_sync(0xffffffffu, tile_max() > m + kRaise)) {
                  again = known = true;
                  ok = raise_to(tile_max());
                  break;
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                arrive(s_free);
              }
              uint32_t pk[16];
              if (some) {
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                  pk[u] = mma::pack_bf16(mma::ex2(fmaf(__uint_as_float(su[h][2 * u]), sc, nm)),
                                         mma::ex2(fmaf(__uint_as_float(su[h][2 * u + 1]), sc, nm)));
                  // (the pair's rounded values: shifts, not conversions)
                  ps[u & 3] = add_f2(ps[u & 3], f2(__uint_as_float(pk[u] << 16), __uint_as_float(pk[u] & 0xffff0000u)));
                }
              } else {
#pragma unroll
                for (int u = 0; u < 16; ++u) pk[u] = 0u;
              }
              if (h == 0 && c2 == 0 && g > 0) {      // P_{g-1} V_{g-1} has read P
                if (!wait(o_full, (g - 1) & 1)) ok = false;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              }
              tmem_st16_async(lane_base + kColP + 16 * c, pk);
            }
          }
        } while (again && ok);
        if (!ok) break;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        arrive(p_full);
        const float2 s2 = f2_split(add_f2(add_f2(ps[0], ps[1]), add_f2(ps[2], ps[3])));
        l += s2.x + s2.y;
      }
      if (!ok) break;
      // the next item's rows while the last P V runs (its last S product is
      // done: Q is free)
      if (P::kQByRows && item_at(it + 1) >= 0) put_q(item_at(it + 1));
      if (r.n > 0) {
        if (!wait(o_full, (g - 1) & 1)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float o[kHD];
        tmem_ld32(lane_base + kColO, o);
        tmem_ld32(lane_base + kColO + 32, o + 32);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        arrive(o_free);
        // every row of the item is written: one whose scores are NaN as NaN, not left
        // as the buffer was (a row with finite scores has l > 0)
        if (P::has_row(a, im, row)) P::store(a, im, row, o, 1.f / l);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

}  // namespace fa
}  // namespace kf
