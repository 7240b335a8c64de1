// render.cu -- front-to-back compositing (gs_render_fwd) and the batched
// information-gain pass (gs_info_gain_batch).
//
// Sec. III of RT-GuIDE: C(p) = sum_i c_i f_i(p) prod_{j<i} (1 - f_j(p)), depth with
// d_i in place of c_i; Sec. IV-A: the per-Gaussian uncertainty u_i composited the
// same way gives the rendered information channel, whose per-view mean scores a
// candidate view (Eq. (nbv) with the Jacobian replaced by the blend weights).
//
// One warp per 8x4-pixel block of a screen tile, one pixel per lane.  The tile's depth-sorted
// list is walked in groups of 32 entries; those that reach a live pixel of the block are staged
// in a shared-memory ring and composited in whole chunks, so no warp waits for another and each
// leaves its list as soon as all of its pixels are saturated.
#include "gs_common.cuh"
#include "gs_internal.h"
#include "render_common.cuh"

namespace gs {
namespace {

constexpr int kFwdWarps = 2;   // warps (work items) per CTA: small CTAs free their slot as soon as both finish
constexpr int kIgWarps = 4;    // the same for the persistent information-gain kernel (which shares out long lists)
constexpr int kRing = 64;      // staged entries per warp (a ring): a group of 32 and a partial chunk
constexpr uint32_t kLongList = 1024;   // entries that a list has at least to be shared by a block's warps
// Chunk depth: staged entries whose alphas are computed together, a template argument of both
// compositing kernels chosen per launch by gs_params (forward 1, 2 or 4, default 4; 1 runs as 2,
// the pair of one packed evaluation; information gain 4, 8 or 16, default 8)
constexpr int kFwdBatchDefault = 4;
constexpr int kIgBatchDefault = 8;

// The list walk of all compositing kernels is a four-stage software pipeline
// over groups of 32 entries (one per lane).  While group g is composited, the
// alpha/colour data of group g+32 is fetched -- only for entries whose support
// box touches the live pixels of the warp's block, decided from their means fetched one
// iteration earlier -- the means of group g+64 are fetched, and the list
// indices of group g+96.  Every fetch is issued one iteration before it is
// used and none depends on a value loaded in the same iteration.
//
// Both kernels are bound by instruction issue where a batch fills the chip (about 0.75 of the
// cycles issue one) and by the chain of transmittance updates of one long list where it does
// not, so both are short per entry:
//  - the exponents of two entries are evaluated by one packed fused multiply-add each
//    (alpha_raw2), from a layout staged for it;
//  - whole chunks leave the ring and a partial one waits for the next group, so only a list's
//    last chunk is padded;
//  - T runs through a chunk as if nothing stopped in it (one multiply and one subtraction per
//    entry); the stop rule is a predicate beside that chain, and the sums follow it;
//  - entries are culled against the bounding box of the pixels still live.
// Measured against one entry per evaluation, a stop test inside the chain and (forward) a chunk
// of 2 without the ring: forward 354 -> 307 us (500k Gaussians, four 640x480 views), 1551 ->
// 1338 us (3M, eight 1280x720), 45 -> 28 us (20k, two 321x243: bound by its longest list);
// information gain 3.07 -> 2.63 ms (1M, 256 views), 517 -> 428 us (200k, 27 views), 6.83 -> 6.22
// ms (3M, 384 views).  Registers are held to 24 warps per SM in both: without the bound the
// information gain takes 105 registers, 16 warps, and 3.10 ms.

// Narrows the block's cull box to the bounding box of its live pixels (lane l holds pixel
// (l mod 8, l div 8); lm = ballot of the live lanes, not zero; (x0, y0) = the centre of the
// block's first pixel): an entry that reaches only saturated pixels adds nothing.
__device__ __forceinline__ void live_box(uint32_t lm, float x0, float y0, WarpBlock& wb) {
  const uint32_t cols = (lm | (lm >> 8) | (lm >> 16) | (lm >> 24)) & 0xFFu;
  const uint32_t rows = ((lm & 0xFFu) ? 1u : 0u) | ((lm & 0xFF00u) ? 2u : 0u) | ((lm & 0xFF0000u) ? 4u : 0u) |
                        ((lm & 0xFF000000u) ? 8u : 0u);
  wb.bx0 = x0 + (float)(__ffs(cols) - 1);
  wb.bx1 = x0 + (float)(31 - __clz(cols));
  wb.by0 = y0 + (float)(__ffs(rows) - 1);
  wb.by1 = y0 + (float)(31 - __clz(rows));
}

// kPairs: packed pairs per chunk.  kCount: the per-pixel counts are asked for (n_contrib).
// kRest = false: block b takes the items 2 b and 2 b + 1.  kRest = true: the blocks share the items
// from block first_rest on, usually none (launch_items).  One kernel that loops over its items
// keeps more registers across them: 1,365 instead of 1,324 us for eight 1280x720 views.
template <int kPairs, bool kCount, bool kRest>
__global__ void __launch_bounds__(kFwdWarps * 32, 12) k_render_fwd(gs_map map, gs_proj proj, gs_bins bins,
                                                                const gs_camera* __restrict__ cams, int n_views,
                                                                gs_params p, gs_image img, uint32_t n_items,
                                                                uint32_t first_rest) {
  pdl_begin();
  constexpr int kChunk = 2 * kPairs;
  __shared__ __align__(16) float s_exp[kFwdWarps][kRing / 2 * kPairFloats];   // staged exponents (stage_pair)
  __shared__ float4 s_col[kFwdWarps][kRing];                                  // (r, g, b, depth)
  __shared__ float2 s_up[kFwdWarps][kRing];                                   // (u, position in the list + 1)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t b = blockIdx.x + (kRest ? first_rest : 0u);
  if (kRest && !more_items(proj, n_views, n_items, b, kFwdWarps)) return;
  do {
    const uint32_t item = ordered_item(bins, proj.view_info, n_views, b * kFwdWarps + warp);
    TileInfo ti;
    if (!warp_item_setup(proj, bins, cams, n_views, item, ti)) continue;
    WarpBlock wb;
    warp_block(ti, wb);
    float* sx = s_exp[warp];
    float4* sk = s_col[warp];
    float2* su = s_up[warp];
    const float ln_amin = __logf(p.alpha_min);
    const LaneOffsets2 lo = lane_offsets2(lane);
    const float ccx = wb.bx0 + 3.5f, ccy = wb.by0 + 1.5f;   // centre of the 8x4 block
    const bool inside = wb.px < ti.W && wb.py < ti.H;
    bool alive = inside;
    float T = 1.f, cu = 0.f;
    f32x2 rg = 0ull, bd = 0ull;
    int32_t last = 0, n_contrib = 0;
    const uint32_t n = ti.end - ti.beg;
    const uint32_t* rl = bins.rec + ti.beg;
    const float4* SP = reinterpret_cast<const float4*>(proj.splat);
    const float4* CD = reinterpret_cast<const float4*>(proj.color_d);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t rA = 0, rB = 0, rC = 0;
    if ((uint32_t)lane < n) rA = __ldg(rl + lane);
    if (32u + lane < n) rB = __ldg(rl + 32 + lane);
    if (64u + lane < n) rC = __ldg(rl + 64 + lane);
    float4 mA = z4, mB = z4;
    if ((uint32_t)lane < n) mA = __ldg(SP + 2 * (size_t)rA);
    if (32u + lane < n) mB = __ldg(SP + 2 * (size_t)rB);
    bool ovA = (uint32_t)lane < n && box_overlaps(mA, wb);
    float4 cA = z4, kA = z4;
    if (ovA) {
      cA = __ldg(SP + 2 * (size_t)rA + 1);
      kA = __ldg(CD + rA);
    }
    // Composites the chunk at ring position i0, of which the first `valid` entries exist: the alphas
    // are independent and computed together, the transmittance updates run in list order.
    auto chunk = [&](int i0, int valid) {
      float al[kChunk];
#pragma unroll
      for (int k = 0; k < kPairs; ++k) {
        const float2 a = alpha_raw2(sx, (i0 >> 1) + k, lo);
        al[2 * k] = fminf(p.alpha_max, a.x);
        al[2 * k + 1] = fminf(p.alpha_max, a.y);
      }
      float w[kChunk];
      bool add[kChunk];
      float Tc = T;   // transmittance as if no entry of the chunk stopped the pixel
#pragma unroll
      for (int k = 0; k < kChunk; ++k) {
        const bool hit = !(al[k] < p.alpha_min);
        w[k] = (hit ? al[k] : 0.f) * Tc;
        Tc = Tc - w[k];              // T (1 - alpha)
        alive = alive && !(Tc < p.T_min);
        add[k] = hit && alive && k < valid;
        if (alive) T = Tc;
      }
#pragma unroll
      for (int k = 0; k < kChunk; ++k) {
        const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(sk + i0 + k);
        const float2 e = su[i0 + k];
        if (add[k]) {
          const f32x2 w2 = pack2(w[k], w[k]);
          rg = fma2(w2, c.x, rg);
          bd = fma2(w2, c.y, bd);
          cu += w[k] * e.x;
          last = __float_as_int(e.y);
          if (kCount) ++n_contrib;
        }
      }
    };
    uint32_t head = 0, tail = 0;   // ring entries [head, tail) are staged and not yet composited
    uint32_t lm_prev = 0;
    for (uint32_t g = 0; g < n; g += 32) {
      const uint32_t lm = __ballot_sync(0xffffffffu, alive);
      if (!lm) break;
      if (lm != lm_prev) live_box(lm, ccx - 3.5f, ccy - 1.5f, wb);
      lm_prev = lm;
      const bool ovB = g + 32 + lane < n && box_overlaps(mB, wb);
      float4 cB = z4, kB = z4;
      if (ovB) {
        cB = __ldg(SP + 2 * (size_t)rB + 1);
        kB = __ldg(CD + rB);
      }
      float4 mC = z4;
      if (g + 64 + lane < n) mC = __ldg(SP + 2 * (size_t)rC);
      uint32_t rD = 0;
      if (g + 96 + lane < n) rD = __ldg(rl + g + 96 + lane);
      ovA = ovA && ellipse_reaches(mA, cA, wb, ln_amin);
      const uint32_t m = __ballot_sync(0xffffffffu, ovA);
      if (m) {
        // the overlapping entries join the ring in list order; whole chunks are composited at once
        // and a partial chunk waits for the next group's entries
        if (ovA) {
          const uint32_t s = (tail + __popc(m & lt)) & (kRing - 1);
          stage_pair(sx, s, stage_exponent(mA.x, mA.y, cA, ccx, ccy));
          sk[s] = kA;
          su[s] = make_float2(mA.w, __int_as_float((int)(g + lane + 1)));
        }
        tail += __popc(m);
        __syncwarp();
        const uint32_t end = head + (tail - head) / kChunk * kChunk;
        for (uint32_t h = head; h != end && alive; h += kChunk) {
          chunk((int)(h & (kRing - 1)), kChunk);
        }
        head = end;
        __syncwarp();
      }
      mA = mB; ovA = ovB; cA = cB; kA = kB;
      rB = rC; mB = mC;
      rC = rD;
    }
    // the last partial chunk, padded with entries of c0 = -inf (alpha = 0)
    if (tail != head && __any_sync(0xffffffffu, alive)) {
      const int i0 = (int)(head & (kRing - 1));
      if ((uint32_t)lane >= tail - head && lane < kChunk)
        stage_pair(sx, i0 + lane, Exponent{-INFINITY, 0.f, 0.f, 0.f, 0.f, 0.f});
      __syncwarp();
      if (alive) chunk(i0, (int)(tail - head));
    }
    __syncwarp();   // (the next round stages over this one's entries)
    if (!inside) continue;
    const float2 vrg = unpack2(rg), vbd = unpack2(bd);
    const size_t P = (size_t)ti.W * ti.H;
    const size_t pix = (size_t)wb.py * ti.W + wb.px;
    const size_t o = (size_t)ti.pix_base + pix;
    if (img.rgb) {
      float* base = img.rgb + 3 * (size_t)ti.pix_base;
      base[pix] = vrg.x;
      base[P + pix] = vrg.y;
      base[2 * P + pix] = vbd.x;
    }
    if (img.depth) img.depth[o] = vbd.y;
    if (img.unc) img.unc[o] = cu;
    if (img.T) img.T[o] = T;
    if (img.last) img.last[o] = last;
    if (kCount) img.n_contrib[o] = n_contrib;
  } while (kRest && more_items(proj, n_views, n_items, b += gridDim.x, kFwdWarps));
}

// Composites `chunks` whole chunks of kIgBatch entries staged in a ring of kSlots, starting at position
// `head` (a multiple of kIgBatch, so no chunk wraps): the alphas of a chunk are independent
// and computed together, two to an instruction; the transmittance updates then run in list
// order.  A lane leaves as soon as its pixel is saturated.
template <int kIgBatch, int kSlots>
__device__ __forceinline__ void composite_chunks(const float* sx, const float* su, uint32_t head, uint32_t chunks,
                                                 const LaneOffsets2& lo, const gs_params& p, float& T, float& cu) {
  for (uint32_t c = 0; c < chunks && T != 0.f; ++c) {
    const uint32_t b0 = (head + c * kIgBatch) & (kSlots - 1);
    float al[kIgBatch], uu[kIgBatch];
#pragma unroll
    for (int k = 0; k < kIgBatch; k += 2) {
      const float2 a = alpha_raw2(sx, (b0 + k) >> 1, lo);
      al[k] = fminf(p.alpha_max, a.x);
      al[k + 1] = fminf(p.alpha_max, a.y);
    }
#pragma unroll
    for (int k = 0; k < kIgBatch; k += 4) {
      const float4 u = *reinterpret_cast<const float4*>(su + b0 + k);
      uu[k] = u.x;
      uu[k + 1] = u.y;
      uu[k + 2] = u.z;
      uu[k + 3] = u.w;
    }
    bool alive = true;
    float Tc = T;   // transmittance as if no entry of the chunk stopped the pixel
#pragma unroll
    for (int k = 0; k < kIgBatch; ++k) {
      const bool hit = !(al[k] < p.alpha_min);
      const float w = Tc * (hit ? al[k] : 0.f);
      Tc = Tc - w;   // T (1 - alpha) taken as T - w: one instruction less
      alive = alive && !(Tc < p.T_min);
      if (hit && alive) cu += w * uu[k];
    }
    T = alive ? Tc : 0.f;
  }
}

// One item by a whole block: warp 0 composites, the others look for the entries that reach the item's
// live pixels, 32 of the list each and round, and stage them in list order in one ring of the block,
// while warp 0 composites what earlier rounds staged.  The entries and their order are those of a
// warp on its own (the live pixels that the others know are a round old, which only keeps entries
// that add nothing), so the sum is the same bit for bit.  sx, su: the block's rings as one.
template <int kIgBatch>
__device__ __forceinline__ void composite_long(const TileInfo& ti, WarpBlock wb, const float4* SP, const gs_bins& bins,
                                               const gs_params& p, float* sx, float* su, uint32_t (*s_cnt)[kIgWarps],
                                               uint32_t* s_live, float* out) {
  constexpr int kSlots = kRing * kIgWarps;
  constexpr uint32_t kStep = 32u * (kIgWarps - 1);
  static_assert(kSlots >= 2 * (int)kStep + kIgBatch, "a round's entries beside the round before it");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const float x0 = wb.bx0, y0 = wb.by0;
  const float ccx = x0 + 3.5f, ccy = y0 + 1.5f;   // centre of the 8x4 block
  const uint32_t n = ti.end - ti.beg;
  const uint32_t* rl = bins.rec + ti.beg;
  uint32_t tail = 0;   // entries staged by the rounds before this one
  if (warp == 0) {
    const LaneOffsets2 lo = lane_offsets2(lane);
    float T = (wb.px < ti.W && wb.py < ti.H) ? 1.f : 0.f, cu = 0.f;
    uint32_t head = 0, r = 0;
    for (uint32_t g = 0; g < n; g += kStep, r ^= 1u) {
      const uint32_t chunks = (tail - head) / kIgBatch;
      composite_chunks<kIgBatch, kSlots>(sx, su, head, chunks, lo, p, T, cu);
      head += chunks * kIgBatch;
      const uint32_t lm = __ballot_sync(0xffffffffu, T != 0.f);
      if (lane == 0) s_live[r] = lm;
      __syncthreads();
      for (int w = 1; w < kIgWarps; ++w) tail += s_cnt[r][w];
      if (!lm) break;
    }
    const uint32_t rest = (tail - head) % kIgBatch;
    if (rest && (uint32_t)lane >= rest && (uint32_t)lane < kIgBatch) {   // pad the last chunk (alpha = 0)
      const uint32_t s = (tail - rest + lane) & (kSlots - 1);
      stage_pair(sx, s, Exponent{-INFINITY, 0.f, 0.f, 0.f, 0.f, 0.f});
      su[s] = 0.f;
    }
    __syncwarp();
    composite_chunks<kIgBatch, kSlots>(sx, su, head, (tail - head + kIgBatch - 1) / kIgBatch, lo, p, T, cu);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) cu += __shfl_down_sync(0xffffffffu, cu, d);
    if (lane == 0) *out = cu;
  } else {
    const float ln_amin = __logf(p.alpha_min);
    const uint32_t i0 = 32u * (warp - 1) + lane;
    uint32_t rB = 0, rC = 0, r = 0, lm_prev = 0;
    float4 mA = z4, mB = z4;
    if (i0 < n) mA = __ldg(SP + 2 * (size_t)__ldg(rl + i0));
    float4 cA = z4;
    bool ovA = i0 < n && box_overlaps(mA, wb);
    if (ovA) cA = __ldg(SP + 2 * (size_t)__ldg(rl + i0) + 1);
    if (i0 + kStep < n) rB = __ldg(rl + i0 + kStep);
    if (i0 + 2 * kStep < n) rC = __ldg(rl + i0 + 2 * kStep);
    if (i0 + kStep < n) mB = __ldg(SP + 2 * (size_t)rB);
    for (uint32_t g = 0; g < n; g += kStep, r ^= 1u) {
      const uint32_t i = g + i0;   // (below 2^32: list positions of one batch)
      const bool ovB = i + kStep < n && box_overlaps(mB, wb);
      float4 cB = z4;
      if (ovB) cB = __ldg(SP + 2 * (size_t)rB + 1);
      float4 mC = z4;
      if (i + 2 * kStep < n) mC = __ldg(SP + 2 * (size_t)rC);
      uint32_t rD = 0;
      if (i + 3 * kStep < n) rD = __ldg(rl + i + 3 * kStep);
      ovA = ovA && ellipse_reaches(mA, cA, wb, ln_amin);
      const uint32_t m = __ballot_sync(0xffffffffu, ovA);
      if (lane == 0) s_cnt[r][warp] = __popc(m);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * (kIgWarps - 1)) : "memory");   // the staging warps' counts
      uint32_t s = tail, all = 0;
      for (int w = 1; w < kIgWarps; ++w) {
        const uint32_t c = s_cnt[r][w];
        if (w < warp) s += c;
        all += c;
      }
      if (ovA) {
        s = (s + __popc(m & lt)) & (kSlots - 1);
        stage_pair(sx, s, stage_exponent(mA.x, mA.y, cA, ccx, ccy));
        su[s] = mA.w;
      }
      tail += all;
      __syncthreads();   // the round's entries are staged, the live pixels are known
      const uint32_t lm = s_live[r];
      if (!lm) break;
      if (lm != lm_prev) live_box(lm, x0, y0, wb);
      lm_prev = lm;
      mA = mB; ovA = ovB; cA = cB;
      rB = rC; mB = mC;
      rC = rD;
    }
  }
  __syncthreads();   // the rings and counts are free again
}

// Persistent U-only compositing: every warp takes (tile, pixel block) work items
// from a device counter, longest tile list first, until the batch is exhausted,
// and writes the sum of U over its pixels to the item's own slot (fixed shuffle
// tree), never accumulating, so the result does not depend on scheduling.
// A list that is long against a warp's share of all the lists is still being walked when the others
// are done (200k Gaussians, 27 views: multiprocessors busy 42% of the time); such lists, which come
// first, are composited by the whole block (composite_long).  That kernel 435 -> 172 us, the pass
// over 1M Gaussians and 6 views 2,395 -> 962 us, 400k and 12 views 1,087 -> 529 us; batches whose
// share is larger than their lists (256 views) have none and are unchanged.  From a quarter of the
// share and 1,024 entries on: 64 views of 800k Gaussians 1.70 ms, from the whole share 1.91 ms.
template <int kIgBatch>
__global__ void __launch_bounds__(kIgWarps * 32, 24 / kIgWarps) k_ig_items(gs_proj proj, gs_bins bins,
                                                             const gs_camera* __restrict__ cams, int n_views,
                                                             gs_params p, const uint32_t* __restrict__ order,
                                                             float* __restrict__ item_sum, int64_t item_cap,
                                                             uint32_t* __restrict__ work) {
  pdl_begin();
  // staged entries of each warp, a ring of kRing: exponents (stage_pair) and u
  __shared__ __align__(16) float s_exp[kIgWarps][kRing / 2 * kPairFloats];
  __shared__ __align__(16) float s_u[kIgWarps][kRing];
  static_assert(kRing % kIgBatch == 0 && kRing >= 32 + kIgBatch, "ring holds a group plus a partial chunk");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  float* sx = s_exp[warp];
  float* su = s_u[warp];
  uint32_t n_items = proj.view_info[kVI * n_views + 2];
  if ((int64_t)n_items > item_cap) n_items = (uint32_t)item_cap;
  const float4* SP = reinterpret_cast<const float4*>(proj.splat);
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  // a warp's share of the entries of all items' lists: pairs x items per tile / warps
  const uint64_t tiles = proj.view_info[kVI * n_views];
  const uint64_t share = tiles ? (uint64_t)*bins.count * n_items / (tiles * gridDim.x * kIgWarps) : 0ull;
  const uint32_t long_list = (uint32_t)max((uint64_t)kLongList, min(share / 4, (uint64_t)0xFFFFFFFFu));
  __shared__ uint32_t s_item, s_cnt[2][kIgWarps], s_live[2];
  uint32_t next = 0xFFFFFFFFu;   // warp 0: an item taken and not yet done
  for (;;) {   // long lists, by the block
    if (threadIdx.x == 0) s_item = atomicAdd(work, 1u);
    __syncthreads();
    const uint32_t item = s_item;
    __syncthreads();
    if (item >= n_items) return;
    const uint32_t slot = __ldg(order + item);
    TileInfo ti;
    if (!warp_item_setup(proj, bins, cams, n_views, slot, ti) || ti.end - ti.beg <= long_list) {
      if (warp == 0) next = item;
      break;
    }
    WarpBlock wb;
    warp_block(ti, wb);
    composite_long<kIgBatch>(ti, wb, SP, bins, p, s_exp[0], s_u[0], s_cnt, s_live, item_sum + slot);
  }
  for (;;) {
    uint32_t item = next;
    next = 0xFFFFFFFFu;
    if (item == 0xFFFFFFFFu) {
      if (lane == 0) item = atomicAdd(work, 1u);
      item = __shfl_sync(0xffffffffu, item, 0);
    }
    if (item >= n_items) break;
    // items are handed out longest tile list first; each writes its own slot
    const uint32_t slot = __ldg(order + item);
    TileInfo ti;
    if (!warp_item_setup(proj, bins, cams, n_views, slot, ti)) {
      if (lane == 0) item_sum[slot] = 0.f;
      continue;
    }
    WarpBlock wb;
    warp_block(ti, wb);
    const float ln_amin = __logf(p.alpha_min);
    const float bx_full = wb.bx0, by_full = wb.by0;   // centre of the block's first pixel
    const float ccx = bx_full + 3.5f, ccy = by_full + 1.5f;   // centre of the 8x4 block
    const LaneOffsets2 lo = lane_offsets2(lane);
    // T = 0 marks a saturated pixel (and one outside the image): the stop rule sets it,
    // and a zero T adds nothing and stays zero, so no separate flag is kept
    float T = (wb.px < ti.W && wb.py < ti.H) ? 1.f : 0.f, cu = 0.f;
    const uint32_t n = ti.end - ti.beg;
    const uint32_t* rl = bins.rec + ti.beg;
    uint32_t rA = 0, rB = 0, rC = 0;
    if ((uint32_t)lane < n) rA = __ldg(rl + lane);
    if (32u + lane < n) rB = __ldg(rl + 32 + lane);
    if (64u + lane < n) rC = __ldg(rl + 64 + lane);
    float4 mA = z4, mB = z4;
    if ((uint32_t)lane < n) mA = __ldg(SP + 2 * (size_t)rA);
    if (32u + lane < n) mB = __ldg(SP + 2 * (size_t)rB);
    bool ovA = (uint32_t)lane < n && box_overlaps(mA, wb);
    float4 cA = z4;
    if (ovA) cA = __ldg(SP + 2 * (size_t)rA + 1);
    uint32_t lm_prev = 0;
    uint32_t head = 0, tail = 0;   // ring entries [head, tail) are staged and not yet composited
    for (uint32_t g = 0; g < n; g += 32) {
      const uint32_t lm = __ballot_sync(0xffffffffu, T != 0.f);
      if (!lm) break;
      if (lm != lm_prev) live_box(lm, bx_full, by_full, wb);
      lm_prev = lm;
      const bool ovB = g + 32 + lane < n && box_overlaps(mB, wb);
      float4 cB = z4;
      if (ovB) cB = __ldg(SP + 2 * (size_t)rB + 1);
      float4 mC = z4;
      if (g + 64 + lane < n) mC = __ldg(SP + 2 * (size_t)rC);
      uint32_t rD = 0;
      if (g + 96 + lane < n) rD = __ldg(rl + g + 96 + lane);
      ovA = ovA && ellipse_reaches(mA, cA, wb, ln_amin);
      const uint32_t m = __ballot_sync(0xffffffffu, ovA);
      if (m) {
        // the overlapping entries join the ring in list order; whole chunks of kIgBatch
        // are composited at once and a partial chunk waits for the next group's entries
        if (ovA) {
          const uint32_t s = (tail + __popc(m & lt)) & (kRing - 1);
          stage_pair(sx, s, stage_exponent(mA.x, mA.y, cA, ccx, ccy));
          su[s] = mA.w;
        }
        tail += __popc(m);
        __syncwarp();
        const uint32_t chunks = (tail - head) / kIgBatch;
        composite_chunks<kIgBatch, kRing>(sx, su, head, chunks, lo, p, T, cu);
        head += chunks * kIgBatch;
        __syncwarp();
      }
      mA = mB; ovA = ovB; cA = cB;
      rB = rC; mB = mC;
      rC = rD;
    }
    // the last partial chunk, padded with entries of C0 = -inf (alpha = 0: adds nothing)
    if (tail != head && __any_sync(0xffffffffu, T != 0.f)) {
      const uint32_t b0 = head & (kRing - 1);
      if ((uint32_t)lane >= tail - head && (uint32_t)lane < kIgBatch) {
        stage_pair(sx, b0 + lane, Exponent{-INFINITY, 0.f, 0.f, 0.f, 0.f, 0.f});
        su[b0 + lane] = 0.f;
      }
      __syncwarp();
      composite_chunks<kIgBatch, kRing>(sx, su, head, 1u, lo, p, T, cu);
      __syncwarp();
    }
    float sum = cu;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, d);
    if (lane == 0) item_sum[slot] = sum;
  }
}

// IG_v = (1 / P_v) * sum over the view's warp items, in a fixed order.
__global__ void __launch_bounds__(256) k_ig_views(const uint32_t* view_info,
                                                   const gs_camera* cams, int n_views,
                                                   const float* item_sum, int64_t item_cap,
                                                   float* __restrict__ ig) {
  pdl_begin();
  __shared__ float s_red[32];
  const int v = blockIdx.x;
  const uint32_t i0 = view_info[kVI * v + 2];
  uint32_t i1 = view_info[kVI * (v + 1) + 2];
  if ((int64_t)i1 > item_cap) i1 = (uint32_t)item_cap;
  const int W = cams[v].width, H = cams[v].height;
  float s = 0.f;
  // fixed assignment of items to threads and a fixed reduction tree: deterministic
  for (int64_t i = (int64_t)i0 + threadIdx.x; i < (int64_t)i1; i += blockDim.x) s += item_sum[i];
  s = block_sum_fixed(s, s_red);
  if (threadIdx.x == 0) ig[v] = (W > 0 && H > 0) ? s / ((float)W * (float)H) : 0.f;
}

__global__ void k_zero_words(uint32_t* p, int n) {
  pdl_begin();
  for (int i = threadIdx.x; i < n; i += blockDim.x) p[i] = 0u;
}

// The persistent compositing kernel at one chunk depth: one CTA per resident slot.
template <int kB>
cudaError_t launch_ig_items(const gs_proj& proj, const gs_bins& bins, const gs_camera* cams, int n_views,
                            const gs_params& p, const uint32_t* order, float* item_sum, int64_t item_cap,
                            uint32_t* work, cudaStream_t st) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_ig_items<kB>, kIgWarps * 32, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)device_sm_count() * per_sm;
  if (grid * kIgWarps > item_cap) grid = (item_cap + kIgWarps - 1) / kIgWarps;
  if (grid < 1) grid = 1;
  launch_spread(k_ig_items<kB>, (unsigned)grid, kIgWarps * 32, 0, st, proj, bins, cams, n_views, p, order, item_sum,
                item_cap, work);
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_render_fwd(const gs_map& map, const gs_proj& proj, const gs_bins& bins, const gs_camera* cams,
                              int n_views, const gs_params& p, const gs_image& img, cudaStream_t st) {
  const int64_t items = bins.tile_capacity * 32;   // upper bound: at most 32 items per tile
  if (items > 0) {
    const int b = p.fwd_batch ? p.fwd_batch : kFwdBatchDefault;
    auto run = [&](auto kern, auto rest) {
      launch_items(bins, items, kFwdWarps, 12, st, kern, rest, map, proj, bins, cams, n_views, p, img);
    };
    if (img.n_contrib && b == 4) run(k_render_fwd<2, true, false>, k_render_fwd<2, true, true>);
    else if (img.n_contrib) run(k_render_fwd<1, true, false>, k_render_fwd<1, true, true>);
    else if (b == 4) run(k_render_fwd<2, false, false>, k_render_fwd<2, false, true>);
    else run(k_render_fwd<1, false, false>, k_render_fwd<1, false, true>);
  }
  return cudaGetLastError();
}

size_t ig_ws_bytes(int64_t n, int n_views, int64_t rec_cap, int64_t pair_cap, int64_t tile_cap) {
  if (rec_cap <= 0) rec_cap = n * (int64_t)n_views;
  Carver c(nullptr);
  c.take<uint32_t>(1);                                   // record count
  c.take<uint32_t>(kVI * (size_t)(n_views + 1));         // view info
  c.take<float4>(2 * (size_t)rec_cap);                   // splat (no view ids: segments from grp_base)
  c.take<ushort4>(rec_cap);                              // rect
  c.take<uint32_t>(rec_cap);                             // depth key
  const int64_t slots = ((n + 31) / 32) * (int64_t)n_views;
  c.take<uint32_t>(slots);                               // grp_mask
  c.take<uint32_t>(slots + 1);                           // grp_base
  c.take<uint32_t>(1);                                   // pair count
  c.take<uint32_t>(pair_cap);                            // rec
  c.take<uint32_t>(2 * tile_cap);                        // ranges
  size_t a = project_ws_bytes(n, n_views), b = bin_ws_bytes(rec_cap, pair_cap, tile_cap, n_views);
  const size_t o = ig_composite_ws_bytes(tile_cap);
  c.take<char>(a > b ? (a > o ? a : o) : (b > o ? b : o));
  return align_up(c.off, 256);
}

size_t ig_composite_ws_bytes(int64_t tile_cap) {
  const int64_t item_cap = 32 * tile_cap;
  Carver c(nullptr);
  c.take<float>(item_cap);                   // per-item sums
  c.take<uint32_t>(4 + 2 * kOrderBuckets);   // work counter; item order: bucket counts and cursors
  c.take<uint32_t>(item_cap);                // item order
  return align_up(c.off, 256);
}

cudaError_t launch_ig_composite(const gs_proj& proj, const gs_bins& bins, const gs_camera* cams, int n_views,
                                const gs_params& p, float* ig_out, void* ws, cudaStream_t st) {
  const int64_t item_cap = 32 * bins.tile_capacity;
  Carver c(ws);
  float* item_sum = c.take<float>(item_cap);
  uint32_t* work = c.take<uint32_t>(4 + 2 * kOrderBuckets);
  uint32_t* order = c.take<uint32_t>(item_cap);
  launch(k_zero_words, 1, 160, 0, st, work, 4 + 2 * kOrderBuckets);
  // longest tile lists first: a counting sort over buckets of list length (an exact radix sort of
  // the lengths took 6 launches and 75 us of the 1M-Gaussian, 256-view pass instead of 2 and 19 us,
  // for the same compositing time)
  launch_item_order(proj.view_info, n_views, bins.ranges, bins.tile_capacity, item_cap, true, work + 4, order, st);
  const int b = p.ig_batch ? p.ig_batch : kIgBatchDefault;
  cudaError_t e = b == 4 ? launch_ig_items<4>(proj, bins, cams, n_views, p, order, item_sum, item_cap, work, st)
                : b == 16 ? launch_ig_items<16>(proj, bins, cams, n_views, p, order, item_sum, item_cap, work, st)
                          : launch_ig_items<8>(proj, bins, cams, n_views, p, order, item_sum, item_cap, work, st);
  if (e != cudaSuccess) return e;
  launch(k_ig_views, n_views, 256, 0, st, proj.view_info, cams, n_views, item_sum, item_cap, ig_out);
  return cudaGetLastError();
}

cudaError_t launch_info_gain(const gs_map& map, const gs_camera* cams, int n_views, const gs_params& p,
                             float* ig_out, uint32_t* status, int64_t rec_cap, int64_t pair_cap, int64_t tile_cap,
                             void* ws, cudaStream_t st) {
  if (rec_cap <= 0) rec_cap = map.n * (int64_t)n_views;
  Carver c(ws);
  gs_proj proj;
  proj.capacity = rec_cap;
  proj.count = c.take<uint32_t>(1);
  proj.status = status;
  proj.view_info = c.take<uint32_t>(kVI * (size_t)(n_views + 1));
  proj.gid = nullptr;    // Gaussian ids are not needed to score views
  proj.view = nullptr;   // nor view ids: binning finds each view's records through grp_base
  proj.splat = (float*)c.take<float4>(2 * (size_t)rec_cap);
  proj.color_d = nullptr;   // not needed to score views: the projection skips the colours
  proj.rect = (uint16_t*)c.take<ushort4>(rec_cap);
  proj.depth_key = c.take<uint32_t>(rec_cap);
  const int64_t slots = ((map.n + 31) / 32) * (int64_t)n_views;
  proj.grp_mask = c.take<uint32_t>(slots);
  proj.grp_base = c.take<uint32_t>(slots + 1);
  gs_bins bins;
  bins.pair_capacity = pair_cap;
  bins.tile_capacity = tile_cap;
  bins.count = c.take<uint32_t>(1);
  bins.tile = nullptr;   // compositing needs only the record of each pair and the ranges
  bins.rec = c.take<uint32_t>(pair_cap);
  bins.ranges = c.take<uint32_t>(2 * tile_cap);
  bins.item_order = nullptr;   // the compositing orders its items itself
  bins.item_capacity = 0;
  size_t a = project_ws_bytes(map.n, n_views), b = bin_ws_bytes(rec_cap, pair_cap, tile_cap, n_views);
  const size_t o = ig_composite_ws_bytes(tile_cap);
  void* inner = c.take<char>(a > b ? (a > o ? a : o) : (b > o ? b : o));

  cudaError_t e = launch_project(map, cams, n_views, p, proj, inner, st);
  if (e != cudaSuccess) return e;
  e = launch_bin_sort(proj, cams, n_views, p, bins, inner, st);
  if (e != cudaSuccess) return e;
  // the inner workspace is free again once binning is done
  return launch_ig_composite(proj, bins, cams, n_views, p, ig_out, inner, st);
}

}  // namespace gs
