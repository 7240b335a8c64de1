// render_bwd.cu -- gs_render_bwd: adjoint of the compositing and the projection.
//
// Eq. (2) of RT-GuIDE refines the map by back-propagating the rendering loss.
// For a pixel with contributors i = 1..n (front to back), w_i = alpha_i T_i and
// out_ch = sum_i w_i x_i,ch, the derivative with respect to alpha_i is
//   dL/dalpha_i = sum_ch g_ch (x_i,ch T_i - S_i,ch / (1 - alpha_i)),
//   S_i,ch = sum_{j>i} w_j x_j,ch.
// The kernel replays each tile back to front starting from the saved final
// transmittance and last index, recovering T_i = T_{i+1} / (1 - alpha_i), so no
// per-pixel contributor list is stored.  (The four S_i enter only through sum_ch g_ch S_i,ch:
// one suffix sum is kept.)  Per-Gaussian screen-space gradients are summed over the 32 pixels
// of a warp through shared memory, sixteen entries at a time, and added with three vector
// atomics per (warp, entry); a second kernel maps them through the projection per Gaussian
// (records of one Gaussian are contiguous), without atomics.
#include "gs_common.cuh"
#include "gs_internal.h"
#include "render_common.cuh"

namespace gs {
namespace {

constexpr int kBwdWarps = 2;   // warps (work items) per CTA
// The gradient terms of an entry are sums over the warp's 32 pixels of two per-pixel values
// times factors that do not depend on the entry or not on the pixel's history: dL/dq times
// 1, dx, dy, dx^2, dx dy, dy^2 and the blend weight w times the pixel's image gradient.  So a
// lane stores only dL/dq and w, as two rows of 32 lane values per entry, and when kRedBatch
// entries are waiting, lanes e and e + 16 form entry e's ten sums, each over 16 pixels (two
// image rows), add their halves and add them to the record's gradient slots with 16-byte
// vector reductions.  Per entry and lane that is two shared-memory stores and about nine
// instructions of the batch's sums (packed two to an FFMA2), where ten stored terms summed
// row by row took ten stores and about thirty.  Batches of 32 (a lane per entry) would need
// twice the shared memory.  Four 640x480 keyframes of a 500k-Gaussian map: 836 -> 577 us of this
// kernel (507 M warp instructions, 71% of cycles issue one); 80 registers (12 CTAs per SM)
// against 72 with a few spills (14 CTAs): 577 / 601 us; the whole mapping iteration of the 3M
// map 8.00 -> 6.96 ms.
constexpr int kRedBatch = 16;
constexpr int kRedPitch = 36;   // floats per row: 16-byte aligned, conflict-free vector reads

// kRest = false: block b takes the items 2 b and 2 b + 1.  kRest = true: the blocks share the items
// from block first_rest on, usually none (launch_items).  One kernel that loops over its items
// spills 28 bytes: 2,797 instead of 2,592 us for eight 1280x720 views.
template <bool kRest>
__global__ void __launch_bounds__(kBwdWarps * 32, 12) k_render_bwd(gs_map map, gs_proj proj, gs_bins bins,
                                                                const gs_camera* __restrict__ cams, int n_views,
                                                                gs_params p, gs_image fwd, gs_image_grad grad,
                                                                float4* __restrict__ g2d, uint32_t n_items,
                                                                uint32_t first_rest) {
  pdl_begin();
  // staged entries: (c0, cu, cv, k.x), (k.y, k.z, position in the list, record), (colour, depth)
  __shared__ float4 s_stage[kBwdWarps][3][32];
  __shared__ __align__(16) float s_red[kBwdWarps][2][kRedBatch * kRedPitch];   // dL/dq and w rows
  __shared__ __align__(16) float s_gpix[kBwdWarps][4][32];                     // image gradient (d, r, g, b) per pixel
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t b = blockIdx.x + (kRest ? first_rest : 0u);
  if (kRest && !more_items(proj, n_views, n_items, b, kBwdWarps)) return;
  do {   // longest tile lists first
    const uint32_t item = ordered_item(bins, proj.view_info, n_views, b * kBwdWarps + warp);
    TileInfo ti;
    if (!warp_item_setup(proj, bins, cams, n_views, item, ti)) continue;
    WarpBlock wb;
    warp_block(ti, wb);
    float4* sa = s_stage[warp][0];
    float4* sb = s_stage[warp][1];
    float4* sk = s_stage[warp][2];
    float* rq = s_red[warp][0];
    float* rw = s_red[warp][1];
    const float4* SP = reinterpret_cast<const float4*>(proj.splat);
    const float4* CD = reinterpret_cast<const float4*>(proj.color_d);
    uint32_t my_rec = 0;   // record of batched entry `lane & 15`
    int nb = 0;            // entries waiting in the batch (warp-uniform)
    // Sums the batched entries' terms and adds them to their records' gradient slots:
    // (P, Q, dL/da, dL/db), (dL/dc, o dL/do, dL/dt_z, -), (dL/dr, dL/dg, dL/db, -).
    auto flush = [&](int count) {
      __syncwarp();
      const int e = lane & (kRedBatch - 1), h = lane >> 4;
      const float2 mu = __ldg(reinterpret_cast<const float2*>(SP + 2 * (size_t)my_rec));   // (a record read before)
      // w times the image gradient, two pixels at a time
      const ulonglong2* W = reinterpret_cast<const ulonglong2*>(rw + e * kRedPitch + 16 * h);
      const ulonglong2* G = reinterpret_cast<const ulonglong2*>(&s_gpix[warp][0][16 * h]);
      f32x2 gs[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const ulonglong2 w = W[k];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const ulonglong2 g = G[8 * c + k];
          gs[c] = fma2(w.y, g.y, fma2(w.x, g.x, gs[c]));
        }
      }
      // dL/dq times (1, dx, dy, dx^2, dx dy, dy^2), dx = mu_x - pixel centre
      const ulonglong2* D = reinterpret_cast<const ulonglong2*>(rq + e * kRedPitch + 16 * h);
      const f32x2 mx = pack2(mu.x, mu.x);
      f32x2 dx[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) dx[j] = add2(mx, pack2(-(wb.bx0 + (float)(2 * j)), -(wb.bx0 + (float)(2 * j + 1))));
      f32x2 a2 = 0ull;
      float sP = 0.f, sQ = 0.f, sB = 0.f, sC = 0.f, s0 = 0.f;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const ulonglong2 x0 = D[2 * r], x1 = D[2 * r + 1];
        const f32x2 x[4] = {x0.x, x0.y, x1.x, x1.y};
        f32x2 o2 = 0ull, p2 = 0ull;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const f32x2 t = mul2(x[j], dx[j]);
          o2 = add2(o2, x[j]);
          p2 = add2(p2, t);
          a2 = fma2(t, dx[j], a2);
        }
        const float dy = __fsub_rn(mu.y, wb.by0 + (float)(2 * h + r));
        const float o = sum2(o2), pr = sum2(p2), q = o * dy;
        s0 += o;
        sP += pr;
        sQ += q;
        sB = fmaf(pr, dy, sB);
        sC = fmaf(q, dy, sC);
      }
      float v[10] = {sP, sQ, sum2(a2), 2.f * sB, sC, -2.f * s0, sum2(gs[0]), sum2(gs[1]), sum2(gs[2]), sum2(gs[3])};
#pragma unroll
      for (int j = 0; j < 10; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], 16);
      if (e < count) {
        // the two vectors that share a 32-byte sector go in one instruction, so a record's 48 bytes
        // are two sectors for the L2 and not three (200k Gaussians, one 640x480 view 128 -> 120 us;
        // large near Gaussians, on whose few records all warps meet, 122 -> 88 us; leaving out
        // vectors of zeros costs more than it saves)
        const uint32_t odd = my_rec & 1u, k = odd + h;
        const float4 v0 = make_float4(v[0], v[1], v[2], v[3]), v1 = make_float4(v[4], v[5], v[6], 0.f),
                     v2 = make_float4(v[7], v[8], v[9], 0.f);
        float4* dst = g2d + 3 * (size_t)my_rec;
        atomicAdd(dst + k, k == 0u ? v0 : k == 1u ? v1 : v2);
        if (h) atomicAdd(odd ? dst : dst + 2, odd ? v0 : v2);
      }
      __syncwarp();
    };
    const float ln_amin = __logf(p.alpha_min);
    const LaneOffsets lo = lane_offsets(lane);
    const float ccx = wb.bx0 + 3.5f, ccy = wb.by0 + 1.5f;   // centre of the 8x4 block
    const size_t P = (size_t)ti.W * ti.H;
    float T = 1.f, gr = 0.f, gg = 0.f, gb = 0.f, gd = 0.f;
    float S = 0.f;   // sum over the entries behind of w_j (image gradient . x_j)
    int last = 0;    // 0 outside the image
    if (wb.px < ti.W && wb.py < ti.H) {
      const size_t pix = (size_t)wb.py * ti.W + wb.px;
      const size_t o = (size_t)ti.pix_base + pix;
      T = fwd.T[o];
      last = fwd.last[o];
      if (grad.rgb) {
        const float* base = grad.rgb + 3 * (size_t)ti.pix_base;
        gr = base[pix];
        gg = base[P + pix];
        gb = base[2 * P + pix];
      }
      if (grad.depth) gd = grad.depth[o];
    }
    const int wlast = (int)__reduce_max_sync(0xffffffffu, (unsigned)(last > 0 ? last : 0));
    if (wlast == 0) continue;
    s_gpix[warp][0][lane] = gd;
    s_gpix[warp][1][lane] = gr;
    s_gpix[warp][2][lane] = gg;
    s_gpix[warp][3][lane] = gb;
    // groups of 32 entries are walked from the last one any lane used back to the
    // first, with the same four-stage pipeline as the forward kernel (alpha and
    // colour data of the next group, means of the one after, list indices of the
    // one after that)
    const uint32_t* rl = bins.rec + ti.beg;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int g = ((wlast - 1) >> 5) << 5;
    uint32_t rA = 0, rB = 0, rC = 0;
    if (g + lane < wlast) rA = __ldg(rl + g + lane);
    if (g >= 32) rB = __ldg(rl + g - 32 + lane);
    if (g >= 64) rC = __ldg(rl + g - 64 + lane);
    float4 mA = z4, mB = z4;
    if (g + lane < wlast) mA = __ldg(SP + 2 * (size_t)rA);
    if (g >= 32) mB = __ldg(SP + 2 * (size_t)rB);
    bool ovA = g + lane < wlast && box_overlaps(mA, wb);
    float4 cA = z4, kA = z4;
    if (ovA) {
      cA = __ldg(SP + 2 * (size_t)rA + 1);
      kA = __ldg(CD + rA);
    }
    for (; g >= 0; g -= 32) {
      const bool ovB = g >= 32 && box_overlaps(mB, wb);
      float4 cB = z4, kB = z4;
      if (ovB) {
        cB = __ldg(SP + 2 * (size_t)rB + 1);
        kB = __ldg(CD + rB);
      }
      float4 mC = z4;
      if (g >= 64) mC = __ldg(SP + 2 * (size_t)rC);
      uint32_t rD = 0;
      if (g >= 96) rD = __ldg(rl + g - 96 + lane);
      ovA = ovA && ellipse_reaches(mA, cA, wb, ln_amin);
      const uint32_t m = __ballot_sync(0xffffffffu, ovA);
      if (m) {
        // the overlapping entries, compacted in list order
        if (ovA) {
          const int s = __popc(m & lt);
          const Exponent e = stage_exponent(mA.x, mA.y, cA, ccx, ccy);
          sa[s] = make_float4(e.c0, e.cu, e.cv, e.kx);
          sb[s] = make_float4(e.ky, e.kz, __int_as_float(g + lane), __uint_as_float(rA));
          sk[s] = kA;
        }
        __syncwarp();
        for (int k = __popc(m) - 1; k >= 0; --k) {
          const float4 ea = sa[k], eb = sb[k];
          // the alpha of the forward pass (same staged coefficients, same operations); ar = o G.
          // A lane that does not contribute runs the same arithmetic with alpha = 0: its T and
          // suffix sum stay exactly unchanged (T * 1, S + 0) and its terms are zero.
          const float ar = alpha_raw(ea.x, ea.y, ea.z, ea.w, eb.x, eb.y, lo);
          float al = fminf(p.alpha_max, ar);
          const bool contrib = __float_as_int(eb.z) < last && !(al < p.alpha_min);
          if (!__any_sync(0xffffffffu, contrib)) continue;
          if (!contrib) al = 0.f;
          const float4 c = sk[k];
          const float inv = __fdividef(1.f, 1.f - al);   // 1 - alpha in [1 - alpha_max, 1]: approximate reciprocal
          T *= inv;
          const float w = al * T;
          const float gc = gr * c.x + gg * c.y + gb * c.z + gd * c.w;   // image gradient . x_i
          const float dalpha = gc * T - S * inv;
          S += w * gc;
          // dL/dq = -alpha/2 dL/dalpha where alpha is not clamped (there o dL/do = -2 dL/dq)
          rq[nb * kRedPitch + lane] = ar < p.alpha_max ? -0.5f * al * dalpha : 0.f;
          rw[nb * kRedPitch + lane] = w;
          if ((lane & (kRedBatch - 1)) == nb) my_rec = __float_as_uint(eb.w);
          if (++nb == kRedBatch) {
            flush(kRedBatch);
            nb = 0;
          }
        }
        __syncwarp();
      }
      mA = mB; ovA = ovB; cA = cB; kA = kB; rA = rB;
      rB = rC; mB = mC;
      rC = rD;
    }
    if (nb) flush(nb);   // (synchronises the warp: the next round stages over this one's entries)
    else __syncwarp();
  } while (kRest && more_items(proj, n_views, n_items, b += gridDim.x, kBwdWarps));
}

__global__ void k_zero_g2d(float4* __restrict__ g2d, const uint32_t* count, int64_t cap) {
  pdl_begin();
  int64_t n = (int64_t)*count;
  if (n > cap) n = cap;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 3 * n; i += (int64_t)gridDim.x * blockDim.x)
    g2d[i] = z;
}

// Projection adjoint: one thread per Gaussian, gathering its records (one per
// view it is visible in, found through the group masks) without atomics.
__global__ void __launch_bounds__(256) k_proj_adjoint(gs_map map, gs_proj proj, const gs_camera* __restrict__ cams,
                                                      int n_views, const float4* __restrict__ g2d, gs_map_grad out) {
  pdl_begin();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= map.n) return;
  const int64_t nrec = (int64_t)*proj.count;
  const int64_t grp = g >> 5, n_grp = (map.n + 31) >> 5;   // mask entry of (view v, group) at v * n_grp + group
  const uint32_t bit = 1u << (g & 31), lt = bit - 1u;
  bool any = false;
  for (int v = 0; v < n_views; ++v) any |= (proj.grp_mask[v * n_grp + grp] & bit) != 0;
  float gmu[3] = {0.f, 0.f, 0.f}, go = 0.f, grgb[3] = {0.f, 0.f, 0.f};
  float M3[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  const float4 mo = reinterpret_cast<const float4*>(map.mo)[g];
  const float4 su = reinterpret_cast<const float4*>(map.su)[g];
  const float4 qv = reinterpret_cast<const float4*>(map.q)[g];
  float Rq[9], s2[3], S3[3][3], qn[4], qnorm = 1.f;
  if (any) {
    qnorm = sqrtf(qv.x * qv.x + qv.y * qv.y + qv.z * qv.z + qv.w * qv.w);
    const float w = qv.x / qnorm, x = qv.y / qnorm, y = qv.z / qnorm, z = qv.w / qnorm;
    qn[0] = w; qn[1] = x; qn[2] = y; qn[3] = z;
    Rq[0] = 1.f - 2.f * (y * y + z * z); Rq[1] = 2.f * (x * y - w * z);       Rq[2] = 2.f * (x * z + w * y);
    Rq[3] = 2.f * (x * y + w * z);       Rq[4] = 1.f - 2.f * (x * x + z * z); Rq[5] = 2.f * (y * z - w * x);
    Rq[6] = 2.f * (x * z - w * y);       Rq[7] = 2.f * (y * z + w * x);       Rq[8] = 1.f - 2.f * (x * x + y * y);
    s2[0] = expf(2.f * su.x); s2[1] = expf(2.f * su.y); s2[2] = expf(2.f * su.z);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        S3[i][j] = Rq[3 * i] * s2[0] * Rq[3 * j] + Rq[3 * i + 1] * s2[1] * Rq[3 * j + 1] + Rq[3 * i + 2] * s2[2] * Rq[3 * j + 2];
  }
  for (int v = 0; v < n_views && any; ++v) {
    const uint32_t m = proj.grp_mask[v * n_grp + grp];
    if (!(m & bit)) continue;
    const uint32_t r = proj.grp_base[v * n_grp + grp] + __popc(m & lt);
    if ((int64_t)r >= nrec) continue;
    const float4 A = g2d[3 * (size_t)r], Bv = g2d[3 * (size_t)r + 1], Cv = g2d[3 * (size_t)r + 2];
    const float4 con = reinterpret_cast<const float4*>(proj.splat)[2 * (size_t)r + 1];
    grgb[0] += Cv.x; grgb[1] += Cv.y; grgb[2] += Cv.z;
    go += Bv.y / con.w;   // the compositing summed o dL/do (o = con.w >= alpha_min > 0)
    // slots A.x, A.y hold P = sum dq dx, Q = sum dq dy: dL/dmu_2D = 2 (a P + b Q, b P + c Q)
    const float gmx = 2.f * (con.x * A.x + con.y * A.y), gmy = 2.f * (con.y * A.x + con.z * A.y);
    const float ga = A.z, gb = A.w, gc = Bv.x, gdep = Bv.z;
    const gs_camera& cam = cams[v];
    const float* R = cam.R;
    const float dx = mo.x - cam.T[0], dy = mo.y - cam.T[1], dz = mo.z - cam.T[2];
    const float tx = R[0] * dx + R[3] * dy + R[6] * dz;
    const float ty = R[1] * dx + R[4] * dy + R[7] * dz;
    const float tz = R[2] * dx + R[5] * dy + R[8] * dz;
    // dL/dSigma2D = -C G_C C (symmetric-matrix gradients)
    const float C00 = con.x, C01 = con.y, C11 = con.z;
    const float G00 = ga, G01 = 0.5f * gb, G11 = gc;
    const float t00 = G00 * C00 + G01 * C01, t01 = G00 * C01 + G01 * C11;
    const float t10 = G01 * C00 + G11 * C01, t11 = G01 * C01 + G11 * C11;
    const float S00 = -(C00 * t00 + C01 * t10), S01 = -(C00 * t01 + C01 * t11);
    const float S11 = -(C01 * t01 + C11 * t11);
    const float iz = 1.f / tz, iz2 = iz * iz;
    const float J00 = cam.fx * iz, J02 = -cam.fx * tx * iz2, J11 = cam.fy * iz, J12 = -cam.fy * ty * iz2;
    float T3[2][3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      T3[0][m] = J00 * R[3 * m + 0] + J02 * R[3 * m + 2];
      T3[1][m] = J11 * R[3 * m + 1] + J12 * R[3 * m + 2];
    }
    const float GS[2][2] = {{S00, S01}, {S01, S11}};
    // M3 += T3^T GS T3
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float u0 = GS[0][0] * T3[0][i] + GS[1][0] * T3[1][i];
      const float u1 = GS[0][1] * T3[0][i] + GS[1][1] * T3[1][i];
#pragma unroll
      for (int j = 0; j < 3; ++j) M3[i][j] += u0 * T3[0][j] + u1 * T3[1][j];
    }
    // GT3 = 2 GS T3 S3; GJ = GT3 R (GJ[r][k] = sum_m GT3[r][m] R[m][k])
    float GT3[2][3];
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const float h0 = GS[rr][0] * T3[0][0] + GS[rr][1] * T3[1][0];
      const float h1 = GS[rr][0] * T3[0][1] + GS[rr][1] * T3[1][1];
      const float h2 = GS[rr][0] * T3[0][2] + GS[rr][1] * T3[1][2];
#pragma unroll
      for (int m = 0; m < 3; ++m) GT3[rr][m] = 2.f * (h0 * S3[0][m] + h1 * S3[1][m] + h2 * S3[2][m]);
    }
    float GJ[2][3];
#pragma unroll
    for (int rr = 0; rr < 2; ++rr)
#pragma unroll
      for (int kk = 0; kk < 3; ++kk) GJ[rr][kk] = GT3[rr][0] * R[kk] + GT3[rr][1] * R[3 + kk] + GT3[rr][2] * R[6 + kk];
    const float iz3 = iz2 * iz;
    const float gtx = GJ[0][2] * (-cam.fx * iz2) + gmx * cam.fx * iz;
    const float gty = GJ[1][2] * (-cam.fy * iz2) + gmy * cam.fy * iz;
    const float gtz = GJ[0][0] * (-cam.fx * iz2) + GJ[0][2] * (2.f * cam.fx * tx * iz3) + GJ[1][1] * (-cam.fy * iz2) +
                      GJ[1][2] * (2.f * cam.fy * ty * iz3) - gmx * cam.fx * tx * iz2 - gmy * cam.fy * ty * iz2 + gdep;
#pragma unroll
    for (int m = 0; m < 3; ++m) gmu[m] += R[3 * m + 0] * gtx + R[3 * m + 1] * gty + R[3 * m + 2] * gtz;
  }
  float4 dmo = make_float4(0.f, 0.f, 0.f, 0.f), dsu = dmo, dq = dmo, drgb = dmo;
  if (any) {
    // dL/dRq = 2 M3 Rq diag(s2); dL/ds2_k = (Rq^T M3 Rq)_kk
    float GR[9], gs2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int kk = 0; kk < 3; ++kk)
        GR[3 * i + kk] = 2.f * (M3[i][0] * Rq[kk] + M3[i][1] * Rq[3 + kk] + M3[i][2] * Rq[6 + kk]) * s2[kk];
#pragma unroll
    for (int kk = 0; kk < 3; ++kk) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) s += Rq[3 * i + kk] * M3[i][j] * Rq[3 * j + kk];
      gs2[kk] = s;
    }
    const float w = qn[0], x = qn[1], y = qn[2], z = qn[3];
    const float gw = 2.f * (-z * GR[1] + y * GR[2] + z * GR[3] - x * GR[5] - y * GR[6] + x * GR[7]);
    const float gx = 2.f * (y * GR[1] + z * GR[2] + y * GR[3] - 2.f * x * GR[4] - w * GR[5] + z * GR[6] + w * GR[7] -
                            2.f * x * GR[8]);
    const float gy = 2.f * (-2.f * y * GR[0] + x * GR[1] + w * GR[2] + x * GR[3] + z * GR[5] - w * GR[6] + z * GR[7] -
                            2.f * y * GR[8]);
    const float gz = 2.f * (-2.f * z * GR[0] - w * GR[1] + x * GR[2] + w * GR[3] - 2.f * z * GR[4] + y * GR[5] + x * GR[6] +
                            y * GR[7]);
    const float dot = w * gw + x * gx + y * gy + z * gz;
    const float inv = 1.f / qnorm;
    dq = make_float4((gw - w * dot) * inv, (gx - x * dot) * inv, (gy - y * dot) * inv, (gz - z * dot) * inv);
    const float o = 1.f / (1.f + expf(-mo.w));
    dmo = make_float4(gmu[0], gmu[1], gmu[2], go * o * (1.f - o));
    dsu = make_float4(2.f * s2[0] * gs2[0], 2.f * s2[1] * gs2[1], 2.f * s2[2] * gs2[2], 0.f);
    drgb = make_float4(grgb[0], grgb[1], grgb[2], 0.f);
  }
  reinterpret_cast<float4*>(out.dmo)[g] = dmo;
  reinterpret_cast<float4*>(out.dsu)[g] = dsu;
  reinterpret_cast<float4*>(out.dq)[g] = dq;
  reinterpret_cast<float4*>(out.drgb)[g] = drgb;
}

}  // namespace

size_t bwd_ws_bytes(int64_t rec_cap) { return align_up(sizeof(float4) * 3 * (size_t)rec_cap, 256); }

cudaError_t launch_render_bwd(const gs_map& map, const gs_proj& proj, const gs_bins& bins, const gs_image& fwd,
                              const gs_image_grad& g, const gs_camera* cams, int n_views, const gs_params& p,
                              const gs_map_grad& out, void* ws, cudaStream_t st) {
  float4* g2d = (float4*)ws;
  int64_t zb = (3 * proj.capacity + 255) / 256;
  if (zb > 4096) zb = 4096;
  if (zb < 1) zb = 1;
  launch(k_zero_g2d, (unsigned)zb, 256, 0, st, g2d, proj.count, proj.capacity);
  const int64_t items = bins.tile_capacity * 32;   // upper bound: at most 32 items per tile
  if (items > 0) {
    launch_items(bins, items, kBwdWarps, 12, st, k_render_bwd<false>, k_render_bwd<true>, map, proj, bins, cams,
                 n_views, p, fwd, g, g2d);
  }
  if (map.n > 0) {
    launch_spread(k_proj_adjoint, (unsigned)((map.n + 255) / 256), 256, 0, st, map, proj, cams, n_views, g2d, out);
  }
  return cudaGetLastError();
}

}  // namespace gs
