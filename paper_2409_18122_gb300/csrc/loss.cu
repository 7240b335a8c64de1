// loss.cu -- the mapping loss of Eq. 3 (L1 depth + L1 colour + SSIM) and its gradient
// with respect to the rendered images.
//
// Two tiled passes over 32x54-pixel output tiles of each (view, channel), one CTA each:
//   pass 1  loads the tile of x (render) and y (reference) with a 5-pixel halo into shared
//           memory, blurs the four moments x, y, (x - y)^2, xy with the separable 11-tap window
//           (rows, then columns; S needs the two variances only as their sum, which is
//           var(x - y) + 2 cov(x, y)), evaluates S(p)
//           and the partial derivatives of S with respect to the three moments that depend on x
//           (m1 = G*x, m2 = G*x^2, m12 = G*xy), stores those as three planes and reduces S and
//           the L1 terms of the tile into one FP64 partial per CTA;
//   pass 2  blurs the three derivative planes with the same window (the adjoint of the
//           zero-padded correlation with a symmetric window is itself) and forms
//           dS/dx = G*dm1 + 2 x G*dm2 + y G*dm12, then dL/dx with the L1 sign term.
// Both are bound by the multiply-adds and shared-memory traffic of the blur (pass 1: about 100
// fused multiply-adds and 30 shared wavefronts per 32 pixels), so the window slides in registers:
// a thread blurs four neighbouring pixels of a row from five 16-byte loads per plane, then seven
// pixels of a column from seventeen loads; the moments' products are formed on the way.  54 rows
// and the halo are 64, two row quads per thread, 1.19 row blurs per output row; a tile that the view
// ends in blurs only the rows it needs (one 4000x11 view 27 -> 23 us, eight 1280x720 views 484 -> 464).  Eight 1280x720
// views: pass 1 478 -> 283 us, pass 2 276 -> 184 us, the sum of the partials 57 -> 17 us.
// A one-CTA kernel sums the partials in FP64 in a fixed order.  Without the SSIM term
// (w_ssim = 0) the loss is elementwise: one flat kernel over the colour and the depth array
// (contiguous chunks per block, fixed partial slots) replaces both passes.
#include <math.h>

#include "gs_internal.h"

namespace gs {
namespace {

constexpr int kR = 5, kWin = 2 * kR + 1;      // 11-tap window
constexpr int kLTW = 32, kLTH = 54;           // output tile
constexpr int kInH = kLTH + 2 * kR;           // 64 rows of input
constexpr int kPitch = 48;                    // input columns x0 - 8 .. x0 + 39: quads of columns are 16-byte aligned
constexpr int kPad = 8;                       // columns before the output tile in a row of shared memory
constexpr int kLossThreads = 256;             // 8 warps
constexpr int kColRows = 7;                   // output rows of a thread in the column pass: warp w owns 7w .. 7w + 6
constexpr int kRowsH = kColRows * kLossThreads / 32 + kWin - 1;   // ... whose inputs reach past the 64 rows (not used)
constexpr int kLossViewsPerLaunch = 64;
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;
static_assert(kLTW == 32 && kInH * kLTW / 4 == 2 * kLossThreads, "two row quads per thread");
static_assert(kColRows * (kLossThreads / 32) >= kLTH, "the warps cover the output rows");

struct LossView {
  int64_t pix_base;  // first pixel of the view in the concatenated images
  int32_t W, H, tile_base, pad;
};

struct LossArgs {
  const float* rgb;
  const float* depth;
  const float* rgb_ref;
  const float* depth_ref;
  float* d_rgb;
  float* d_depth;
  float* dm;        // [3][3P] derivative planes (dS/dm1, dS/dm2, dS/dm12), rgb layout
  double* part;     // [slots][3] per-CTA (sum S, sum |dc|, sum |dd|)
  int64_t P;        // total pixels of all views
  float w_d, w_c, w_s, inv_n, inv_3n;
  float g[kWin];
  int32_t n_views;  // views in this launch
  int32_t part_base;
  LossView v[kLossViewsPerLaunch];
};

__device__ __forceinline__ int loss_view_of(const LossArgs& a, int t) {
  int v = 0;
  for (int i = 1; i < a.n_views; ++i) v = (a.v[i].tile_base <= t) ? i : v;
  return v;
}

__device__ __forceinline__ float sgnf(float d) { return (float)(d > 0.f) - (float)(d < 0.f); }

struct TileGeo {
  int W, H, x0, y0;
  int rows;           // input rows that an output row of the view takes: the rest of a ragged tile is left out
  int64_t pix, base;  // first pixel of the view; first element of this (view, channel) plane
};

__device__ __forceinline__ TileGeo tile_geo(const LossArgs& a, int t, int ch) {
  const int vi = loss_view_of(a, t);
  TileGeo g;
  g.W = a.v[vi].W;
  g.H = a.v[vi].H;
  const int tiles_x = (g.W + kLTW - 1) / kLTW;
  const int lt = t - a.v[vi].tile_base;
  g.x0 = (lt % tiles_x) * kLTW;
  g.y0 = (lt / tiles_x) * kLTH;
  g.rows = min(kInH, g.H - g.y0 + 2 * kR);
  g.pix = a.v[vi].pix_base;
  g.base = 3 * g.pix + (int64_t)ch * g.W * g.H;
  return g;
}

// Copies NP planes (src[k] + base) of a halo tile into s[k], zero outside the image: a warp per row,
// columns x0 - 5 .. x0 + 36.  The copies are asynchronous, so that all of a thread's are in flight
// together (through registers, the few loads that are in flight at a time made the
// tiles wait for memory: 421 and 386 us).
template <int NP>
__device__ __forceinline__ void load_halo(const float* const* src, const TileGeo& g, float (*s)[kInH][kPitch]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < kInH / (kLossThreads / 32); ++i) {
    const int r = (threadIdx.x >> 5) + i * (kLossThreads / 32);
    const int gy = g.y0 - kR + r;
    const bool row = gy >= 0 && gy < g.H;
    const int64_t o = g.base + (int64_t)gy * g.W;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h * 32 + lane, gx = g.x0 - kR + c;
      const bool in = row && gx >= 0 && gx < g.W;
      if (c < kLTW + 2 * kR && r < g.rows) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s[k][r][kPad - kR + c]);
          const float* from = src[k] + (in ? o + gx : g.base);   // (nothing is read outside the image)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(from), "r"(in ? 4 : 0) : "memory");
        }
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Row pass: plane k of the NP blurred ones at input column t is val(k, v) of the NI loaded values v
// of that column; each thread blurs two quads of four columns.
template <int NI, int NP, class F>
__device__ __forceinline__ void blur_rows(const LossArgs& a, int rows, const float (*s_in)[kInH][kPitch],
                                          float (*s_h)[kRowsH][kLTW], F val) {
#pragma unroll 1
  for (int i = threadIdx.x; i < kInH * kLTW / 4; i += kLossThreads) {
    const int r = i >> 3, c = 4 * (i & 7);
    if (r >= rows) break;
    float acc[NP][4];
#pragma unroll
    for (int k = 0; k < NP; ++k)
#pragma unroll
      for (int o = 0; o < 4; ++o) acc[k][o] = 0.f;
    // output column c + o takes input columns c + o - 5 .. c + o + 5, which are at kPad further on
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      float v[NI][4];
#pragma unroll
      for (int n = 0; n < NI; ++n) {
        const float4 w = *reinterpret_cast<const float4*>(&s_in[n][r][c + 4 * q]);
        v[n][0] = w.x; v[n][1] = w.y; v[n][2] = w.z; v[n][3] = w.w;
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = 4 * q + t - (kPad - kR);   // tap of output column c
        if (j < 0 || j > kWin + 2) continue;
        float in[NI], m[NP];
#pragma unroll
        for (int n = 0; n < NI; ++n) in[n] = v[n][t];
        val(in, m);
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          if (j - o < 0 || j - o >= kWin) continue;
#pragma unroll
          for (int k = 0; k < NP; ++k) acc[k][o] = fmaf(a.g[j - o], m[k], acc[k][o]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k)
      *reinterpret_cast<float4*>(&s_h[k][r][c]) = make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
  }
}

// Column pass of one plane: out[q] = blurred value at output row r0 + q, column c.
__device__ __forceinline__ void blur_column(const LossArgs& a, const float (*s_h)[kLTW], int r0, int c,
                                            float (&out)[kColRows]) {
#pragma unroll
  for (int q = 0; q < kColRows; ++q) out[q] = 0.f;
#pragma unroll
  for (int j = 0; j < kColRows + kWin - 1; ++j) {
    const float h = s_h[r0 + j][c];
#pragma unroll
    for (int q = 0; q < kColRows; ++q)
      if (j - q >= 0 && j - q < kWin) out[q] = fmaf(a.g[j - q], h, out[q]);
  }
}

// Block sum of three per-thread values into one FP64 partial (fixed order).
__device__ __forceinline__ void block_partial(float v0, float v1, float v2, double* dst) {
  __shared__ float s_red[3][kLossThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v0 += __shfl_xor_sync(0xffffffffu, v0, o);
    v1 += __shfl_xor_sync(0xffffffffu, v1, o);
    v2 += __shfl_xor_sync(0xffffffffu, v2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    s_red[0][threadIdx.x >> 5] = v0;
    s_red[1][threadIdx.x >> 5] = v1;
    s_red[2][threadIdx.x >> 5] = v2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t0 = 0.0, t1 = 0.0, t2 = 0.0;
    for (int w = 0; w < kLossThreads / 32; ++w) {
      t0 += (double)s_red[0][w];
      t1 += (double)s_red[1][w];
      t2 += (double)s_red[2][w];
    }
    dst[0] = t0;
    dst[1] = t1;
    dst[2] = t2;
  }
}

constexpr size_t kFwdSmem = sizeof(float) * (2 * kInH * kPitch + 4 * kRowsH * kLTW);
constexpr size_t kBwdSmem = sizeof(float) * (3 * kInH * kPitch + 3 * kRowsH * kLTW);

__global__ void __launch_bounds__(kLossThreads) k_loss_fwd(const __grid_constant__ LossArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float s_mem[];
  float (*s_in)[kInH][kPitch] = reinterpret_cast<float (*)[kInH][kPitch]>(s_mem);   // x, y
  float (*s_h)[kRowsH][kLTW] = reinterpret_cast<float (*)[kRowsH][kLTW]>(s_mem + 2 * kInH * kPitch);
  const int t = blockIdx.x, ch = blockIdx.y;
  const TileGeo g = tile_geo(a, t, ch);
  const int c = threadIdx.x & 31, r0 = kColRows * (threadIdx.x >> 5);
  const int px = g.x0 + c;
  float s_sum = 0.f, l1c = 0.f, l1d = 0.f;

  const float* src[2] = {a.rgb, a.rgb_ref};
  load_halo<2>(src, g, s_in);
  __syncthreads();
  blur_rows<2, 4>(a, g.rows, s_in, s_h, [](const float* v, float* m) {
    m[0] = v[0];
    m[1] = v[1];
    const float d = v[0] - v[1];
    m[2] = d * d;
    m[3] = v[0] * v[1];
  });
  __syncthreads();
  float m1[kColRows] = {}, m2[kColRows] = {}, m3[kColRows] = {}, m4[kColRows] = {};
  if (g.y0 + r0 < g.H) {
    blur_column(a, s_h[0], r0, c, m1);
    blur_column(a, s_h[1], r0, c, m2);
    blur_column(a, s_h[2], r0, c, m3);
    blur_column(a, s_h[3], r0, c, m4);
  }
#pragma unroll
  for (int q = 0; q < kColRows; ++q) {
    const int py = g.y0 + r0 + q;
    if (px >= g.W || py >= g.H || r0 + q >= kLTH) continue;
    const int64_t o = g.base + (int64_t)py * g.W + px;
    const float mx = m1[q], my = m2[q];
    // the variances' sum is 2 cov(x, y) + var(x - y): less cancellation than two variances
    const float dm = mx - my, sxy = m4[q] - mx * my;
    const float A1 = 2.f * mx * my + kC1, A2 = 2.f * sxy + kC2;
    const float B1 = A1 + dm * dm, B2 = A2 + (m3[q] - dm * dm);
    const float iD = __frcp_rn(B1 * B2);
    const float S = A1 * A2 * iD;
    s_sum += S;
    if (a.d_rgb) {
      // dS/dm1 = 2 my (A2 - A1) / D - 2 mx S (1/B1 - 1/B2);  dS/dm2 = -S / B2;  dS/dm12 = 2 A1 / D
      a.dm[o] = 2.f * iD * (my * (A2 - A1) - mx * S * (B2 - B1));
      a.dm[3 * a.P + o] = -S * B1 * iD;
      a.dm[6 * a.P + o] = 2.f * A1 * iD;
    }
    l1c += fabsf(s_in[0][r0 + q + kR][c + kPad] - s_in[1][r0 + q + kR][c + kPad]);
  }

  if (ch == 0 && (a.depth || a.d_depth)) {
#pragma unroll
    for (int q = 0; q < kColRows; ++q) {
      const int py = g.y0 + r0 + q;
      if (px >= g.W || py >= g.H || r0 + q >= kLTH) continue;
      const int64_t o = g.pix + (int64_t)py * g.W + px;
      const float dd = a.depth ? a.depth[o] - a.depth_ref[o] : 0.f;
      l1d += fabsf(dd);
      if (a.d_depth) a.d_depth[o] = a.w_d * sgnf(dd) * a.inv_n;
    }
  }
  block_partial(s_sum, l1c, l1d, a.part + 3 * ((int64_t)a.part_base + 3 * t + ch));
}

__global__ void __launch_bounds__(kLossThreads) k_loss_ssim_bwd(const __grid_constant__ LossArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float s_mem[];
  float (*s_in)[kInH][kPitch] = reinterpret_cast<float (*)[kInH][kPitch]>(s_mem);   // dS/dm1, dS/dm2, dS/dm12
  float (*s_h)[kRowsH][kLTW] = reinterpret_cast<float (*)[kRowsH][kLTW]>(s_mem + 3 * kInH * kPitch);
  const int t = blockIdx.x, ch = blockIdx.y;
  const TileGeo g = tile_geo(a, t, ch);
  const float* src[3] = {a.dm, a.dm + 3 * a.P, a.dm + 6 * a.P};
  const int c = threadIdx.x & 31, r0 = kColRows * (threadIdx.x >> 5);
  const int px = g.x0 + c;
  float x[kColRows], y[kColRows];
#pragma unroll
  for (int q = 0; q < kColRows; ++q) {
    const int py = g.y0 + r0 + q;
    const bool in = px < g.W && py < g.H && r0 + q < kLTH;
    const int64_t o = g.base + (int64_t)py * g.W + px;
    x[q] = in ? a.rgb[o] : 0.f;
    y[q] = in ? a.rgb_ref[o] : 0.f;
  }
  load_halo<3>(src, g, s_in);
  __syncthreads();
  blur_rows<3, 3>(a, g.rows, s_in, s_h, [](const float* v, float* m) {
    m[0] = v[0];
    m[1] = v[1];
    m[2] = v[2];
  });
  __syncthreads();
  float b0[kColRows], b1[kColRows], b2[kColRows];
  if (g.y0 + r0 >= g.H) return;
  blur_column(a, s_h[0], r0, c, b0);
  blur_column(a, s_h[1], r0, c, b1);
  blur_column(a, s_h[2], r0, c, b2);
#pragma unroll
  for (int q = 0; q < kColRows; ++q) {
    const int py = g.y0 + r0 + q;
    if (px >= g.W || py >= g.H || r0 + q >= kLTH) continue;
    const int64_t o = g.base + (int64_t)py * g.W + px;
    const float dS = fmaf(y[q], b2[q], fmaf(2.f * x[q], b1[q], b0[q]));
    a.d_rgb[o] = a.w_c * sgnf(x[q] - y[q]) * a.inv_n - a.w_s * a.inv_3n * dS;
  }
}

// Loss without the SSIM term: elementwise over the flat arrays.  The first nb_c blocks take the
// colour, the others the depth: block b of an array the contiguous elements [b chunk, (b + 1) chunk),
// storing its sum of |x - y| in its own partial slot (other fields zero) and g = w sign(x - y) / N_p
// if g.  x == NULL (no depth): differences are zero.
struct L1Array {
  const float* x;
  const float* y;
  float* g;
  int64_t n;
  float w;
};

__global__ void __launch_bounds__(kLossThreads) k_loss_l1(const L1Array colour, const L1Array depth, int64_t chunk,
                                                          int nb_c, float inv_n, double* __restrict__ part) {
  pdl_begin();
  const bool is_c = (int)blockIdx.x < nb_c;
  const L1Array a = is_c ? colour : depth;
  const int64_t b0 = (int64_t)(is_c ? blockIdx.x : blockIdx.x - nb_c) * chunk;
  const int64_t b1 = b0 + chunk < a.n ? b0 + chunk : a.n;
  float acc = 0.f;
  // four elements' loads in flight at a time (the compiler cannot know that the stores leave x and y alone)
  for (int64_t i0 = b0 + threadIdx.x; i0 < b1; i0 += 4 * kLossThreads) {
    float d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = i0 + k * kLossThreads;
      d[k] = a.x && i < b1 ? a.x[i] - a.y[i] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = i0 + k * kLossThreads;
      acc += fabsf(d[k]);
      if (a.g && i < b1) a.g[i] = a.w * sgnf(d[k]) * inv_n;
    }
  }
  block_partial(0.f, is_c ? acc : 0.f, is_c ? 0.f : acc, part + 3 * (int64_t)blockIdx.x);
}

// Sums the partials in a fixed order: thread t takes slots t, t + 1024, ..., then a fixed tree.
constexpr int kFinishThreads = 1024;
__global__ void __launch_bounds__(kFinishThreads)
    k_loss_finish(const double* part, int64_t n_slots, float w_d, float w_c, float w_s, bool ssim, double n_pix,
                  float* out) {
  pdl_begin();
  __shared__ double s[3][kFinishThreads];
  double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
  for (int64_t i = threadIdx.x; i < n_slots; i += kFinishThreads)
    for (int k = 0; k < 3; ++k) acc[k] += part[3 * i + k];
  for (int k = 0; k < 3; ++k) s[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int h = kFinishThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h)
      for (int k = 0; k < 3; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double l1d = s[2][0] / n_pix, l1c = s[1][0] / n_pix;
    const double ss = ssim ? s[0][0] / (3.0 * n_pix) : (double)NAN;
    double L = (double)w_d * l1d + (double)w_c * l1c;
    if (ssim) L += (double)w_s * (1.0 - ss);
    out[0] = (float)L;
    out[1] = (float)l1d;
    out[2] = (float)l1c;
    out[3] = (float)ss;
  }
}

struct LossLayout {
  int64_t P = 0, tiles = 0;
};

bool loss_layout(const int32_t* sizes, int n_views, LossLayout& lay) {
  if (!sizes || n_views < 1) return false;
  for (int v = 0; v < n_views; ++v) {
    const int64_t W = sizes[2 * v], H = sizes[2 * v + 1];
    if (W < 1 || H < 1 || W > 65536 || H > 65536) return false;
    lay.P += W * H;
    lay.tiles += ((W + kLTW - 1) / kLTW) * ((H + kLTH - 1) / kLTH);
  }
  return lay.P <= ((int64_t)1 << 36) && lay.tiles <= ((int64_t)1 << 30);
}

}  // namespace

size_t image_loss_ws_bytes(const int32_t* sizes, int n_views) {
  LossLayout lay;
  if (!loss_layout(sizes, n_views, lay)) return 0;
  Carver cv(nullptr);
  cv.take<float>(9 * lay.P);
  cv.take<double>(9 * lay.tiles);
  return align_up(cv.off, 256);
}

cudaError_t launch_image_loss(const int32_t* sizes, int n_views, const float* rgb, const float* depth,
                              const float* rgb_ref, const float* depth_ref, const gs_loss_weights& w,
                              float* loss_out, float* d_rgb, float* d_depth, void* ws, cudaStream_t st) {
  LossLayout lay;
  if (!loss_layout(sizes, n_views, lay)) return cudaErrorInvalidValue;
  Carver cv(ws);
  float* dm = cv.take<float>(9 * lay.P);
  double* part = cv.take<double>(9 * lay.tiles);
  const bool ssim = w.w_ssim != 0.f;

  LossArgs a{};
  a.rgb = rgb;
  a.depth = depth;
  a.rgb_ref = rgb_ref;
  a.depth_ref = depth_ref;
  a.d_rgb = d_rgb;
  a.d_depth = d_depth;
  a.dm = dm;
  a.part = part;
  a.P = lay.P;
  a.w_d = w.w_depth;
  a.w_c = w.w_rgb;
  a.w_s = w.w_ssim;
  a.inv_n = (float)(1.0 / (double)lay.P);
  a.inv_3n = (float)(1.0 / (3.0 * (double)lay.P));
  {  // normalised Gaussian window, sigma 1.5
    double gw[kWin], sum = 0.0;
    for (int j = 0; j < kWin; ++j) {
      const double k = j - kR;
      gw[j] = exp(-k * k / (2.0 * 1.5 * 1.5));
      sum += gw[j];
    }
    for (int j = 0; j < kWin; ++j) a.g[j] = (float)(gw[j] / sum);
  }

  if (ssim) {
    cudaError_t e = allow_smem<k_loss_fwd>(kFwdSmem);
    if (e == cudaSuccess) e = allow_smem<k_loss_ssim_bwd>(kBwdSmem);
    if (e != cudaSuccess) return e;
  }
  int64_t pix = 0, slot = 0;
  if (!ssim) {
    // elementwise: contiguous chunks of at least 4096 elements (at most P / 1024 + 2 partial
    // slots, within the 3 x tiles the workspace holds), about 8 blocks per SM of 152
    int64_t chunk = (3 * lay.P + 152 * 8 - 1) / (152 * 8);
    chunk = (chunk + 4 * kLossThreads - 1) / (4 * kLossThreads) * (4 * kLossThreads);
    if (chunk < 4096) chunk = 4096;
    const int64_t nb_c = (3 * lay.P + chunk - 1) / chunk, nb_d = (lay.P + chunk - 1) / chunk;
    const L1Array colour{rgb, rgb_ref, d_rgb, 3 * lay.P, w.w_rgb}, dep{depth, depth_ref, d_depth, lay.P, w.w_depth};
    launch(k_loss_l1, (unsigned)(nb_c + nb_d), kLossThreads, 0, st, colour, dep, chunk, (int)nb_c, a.inv_n, part);
    slot = nb_c + nb_d;
  }
  for (int v0 = 0; v0 < n_views && ssim; v0 += kLossViewsPerLaunch) {
    const int nv = n_views - v0 < kLossViewsPerLaunch ? n_views - v0 : kLossViewsPerLaunch;
    a.n_views = nv;
    a.part_base = (int32_t)slot;
    int32_t tb = 0;
    for (int i = 0; i < nv; ++i) {
      const int W = sizes[2 * (v0 + i)], H = sizes[2 * (v0 + i) + 1];
      a.v[i].pix_base = pix;
      a.v[i].W = W;
      a.v[i].H = H;
      a.v[i].tile_base = tb;
      a.v[i].pad = 0;
      pix += (int64_t)W * H;
      tb += ((W + kLTW - 1) / kLTW) * ((H + kLTH - 1) / kLTH);
    }
    const dim3 grid((unsigned)tb, 3);
    launch_spread(k_loss_fwd, grid, kLossThreads, kFwdSmem, st, a);
    if (d_rgb) {
      launch_spread(k_loss_ssim_bwd, grid, kLossThreads, kBwdSmem, st, a);
    }
    slot += 3 * (int64_t)tb;
  }
  launch(k_loss_finish, 1, kFinishThreads, 0, st, part, slot, w.w_depth, w.w_rgb, w.w_ssim, ssim, (double)lay.P,
         loss_out);
  return cudaGetLastError();
}

}  // namespace gs
