// Prefill attention on tcgen05 (bf16 cache, head_dim 64): items of up to 128
// consecutive query rows of one (sequence, head) against the paged cache, on the
// pipeline of kf_attn_tc.cuh.  The warp-level MMA kernel takes 16 rows per CTA, so
// a prompt of n rows reads its keys n / 16 times from L2 and multiplies 16-row
// tiles; here a key tile serves 128 rows.  What bounds it: the chain of the
// longest items (a 900-row prompt's last 128 rows walk eight tiles).  Measured,
// 16-row -> 128-row groups: 16 prompts of 128 to 896 tokens, 12 layers, and an AR
// step 3.25 -> 2.76 ms; where
// few or short rows leave the items idle the 16-row kernel stays (the rule and
// its figures are at the caller).
#include <algorithm>

#include "kf_attn_tc.cuh"

namespace kf {
namespace {
constexpr uint32_t kPageBytes = kPage * fa::kHD * 2;   // one (page, K or V, head) block

struct PrefillPolicy {
  struct Args {
    const float* q;               // [R][H][64]
    const int32_t* page_table;    // [slots][max_pages]
    const int4* groups;           // {slot, first row, rows <= 128, first position}, most keys first
    __nv_bfloat16* out;           // [R][H * 64]
    int n_groups, H, max_pages, n_pages;
  };
  struct Maps { CUtensorMap kv; };     // this layer's pages as rows of 64 bf16
  struct Item { int slot, row0, rows, pos0, h; };
  struct TileRef { int page; uint32_t mask; };   // this lane's page, the lanes that copy one
  static constexpr bool kQByRows = true, kWindows = false;

  static __device__ __forceinline__ int n_items(const Args& a) { return a.n_groups * a.H; }
  static __device__ __forceinline__ bool all_open(const Args&) { return true; }
  static __device__ __forceinline__ void item(const Args& a, int w, int, Item& im, fa::Ranges& r) {
    const int gi = w / a.H;
    const int4 gg = a.groups[gi];
    im.slot = gg.x; im.row0 = gg.y; im.rows = gg.z; im.pos0 = gg.w;
    im.h = w - gi * a.H;
#pragma unroll
    for (int i = 0; i < 3; ++i) r.lo[i] = r.hi[i] = 0;
    r.hi[0] = im.pos0 + im.rows;
    r.cmin = im.pos0;
    fa::count_tiles(r);
  }
  static __device__ __forceinline__ bool has_row(const Args&, const Item& im, int row) { return row < im.rows; }
  static __device__ __forceinline__ fa::RowVis vis(const Args&, const Item& im, int row) {
    return {im.pos0 + min(row, im.rows - 1), 0, 0, 0, 0};
  }
  static __device__ __forceinline__ void load_q(const Maps&, const Item&, uint32_t, uint32_t) {}
  // 32 rows of Q to bf16, swizzled as the MMA reads them (rows past the item: zeros)
  static __device__ __forceinline__ void q_rows(const Args& a, const Item& im, uint8_t* sQ, int first, int lane) {
    const int c4 = lane & 15;          // 4 columns
#pragma unroll 8
    for (int i = 0; i < 16; ++i) {
      const int r = first + 2 * i + (lane >> 4);
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < im.rows) x = *reinterpret_cast<const float4*>(a.q + ((size_t)(im.row0 + r) * a.H + im.h) * fa::kHD + 4 * c4);
      *reinterpret_cast<uint2*>(sQ + r * 128 + (((c4 >> 1) ^ (r & 7)) << 4) + (c4 & 1) * 8) =
          make_uint2(mma::pack_bf16(x.x, x.y), mma::pack_bf16(x.z, x.w));
    }
  }
  // a tile is 8 pages, one per lane; pages past the last key are not copied
  static __device__ __forceinline__ TileRef tile(const Args& a, const Item& im, int kt, int kend, int lane, int* d_err) {
    const int key = kt + lane * kPage, pi = key / kPage;
    int page = -1;
    bool go = lane < fa::kKeys / kPage && key < kend;
    if (go) {
      page = pi < a.max_pages ? __ldg(a.page_table + (size_t)im.slot * a.max_pages + pi) : -1;
      if (page < 0 || page >= a.n_pages) {
        atomicOr(d_err, kErrBadPage);
        go = false;
      }
    }
    return {go ? page : -1, __ballot_sync(0xffffffffu, go)};
  }
  static __device__ __forceinline__ uint32_t tile_bytes(const TileRef& r) { return __popc(r.mask) * kPageBytes; }
  static __device__ __forceinline__ void load_k(const Maps& m, const Args& a, const Item& im, const TileRef& r, int lane,
                                                uint32_t dst, uint32_t bar) {
    if (r.page >= 0) tma_load_2d(dst + lane * kPageBytes, &m.kv, bar, 0, (r.page * 2 * a.H + im.h) * kPage);
  }
  static __device__ __forceinline__ void load_v(const Maps& m, const Args& a, const Item& im, const TileRef& r, int lane,
                                                uint32_t dst, uint32_t bar) {
    if (r.page >= 0) tma_load_2d(dst + lane * kPageBytes, &m.kv, bar, 0, ((r.page * 2 + 1) * a.H + im.h) * kPage);
  }
  // The pages that are not copied (past the last key) are cleared for each tile:
  // their probabilities are 0 and 0 * V must be 0, and the stage may hold another
  // sequence's values, which need not be finite
  static __device__ __forceinline__ void clear_v(const TileRef& r, int lane, uint8_t* dst) {
    if (r.mask == (1u << (fa::kKeys / kPage)) - 1) return;
    for (int p = 0; p < fa::kKeys / kPage; ++p)
      if (!((r.mask >> p) & 1u))
#pragma unroll
        for (int i = 0; i < (int)kPageBytes; i += 32 * 16)
          *reinterpret_cast<uint4*>(dst + p * kPageBytes + i + 16 * lane) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
  }
  static __device__ __forceinline__ void store(const Args& a, const Item& im, int row, const float* o, float inv) {
    uint4* dst = reinterpret_cast<uint4*>(a.out + ((size_t)(im.row0 + row) * a.H + im.h) * fa::kHD);
#pragma unroll
    for (int d = 0; d < fa::kHD; d += 8)
      dst[d / 8] = make_uint4(mma::pack_bf16(o[d] * inv, o[d + 1] * inv), mma::pack_bf16(o[d + 2] * inv, o[d + 3] * inv),
                              mma::pack_bf16(o[d + 4] * inv, o[d + 5] * inv), mma::pack_bf16(o[d + 6] * inv, o[d + 7] * inv));
  }
};
}  // namespace

int launch_attention_prefill(const AttnArgs& a, int n_groups, cudaStream_t s) {
  if (n_groups == 0) return 0;
  PrefillPolicy::Args p{a.q, a.page_table, a.groups, static_cast<__nv_bfloat16*>(a.out), n_groups, a.H, a.max_pages,
                        a.n_pages};
  const size_t layer_elems = (size_t)a.n_pages * 2 * a.H * kPage * fa::kHD;
  PrefillPolicy::Maps maps;
  if (!encode_rows_map_bf16(&maps.kv, static_cast<const __nv_bfloat16*>(a.kv) + (size_t)a.layer * layer_elems,
                            (uint64_t)a.n_pages * 2 * a.H * kPage, fa::kHD, kPage))
    return -1;
  static PerDevice attr;
  set_smem_attr(attr, fa::k_attn_tc<PrefillPolicy>, fa::kSmemBytes);
  const long long items = (long long)n_groups * a.H;
  if (items > (1ll << 30)) return -1;
  const dim3 grid((unsigned)std::min<long long>(items, 2ll * device_sms()));
  kf_launch(fa::k_attn_tc<PrefillPolicy>, grid, dim3(fa::kThreads), fa::kSmemBytes, s, maps, p, a.d_err, 0);
  return 0;
}

}  // namespace kf
