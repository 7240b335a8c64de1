// utility.cu -- the render-free view utility of RT-GuIDE (Sec. IV-A / IV-B):
// per-Gaussian uncertainty from mean displacements, the high / low uncertainty
// classes, the batched view utility xi (Eq. view_util) and the mean uncertainty
// of cuboid regions.
//
// Visibility v(x, g) of a Gaussian's mean in a view is decided in FP32 with a
// fixed sequence of separately rounded IEEE operations (no fused multiply-add),
// so a plain float32 program can take the same decisions.  Per-view results are
// reduced per block into fixed slots and then in a fixed order: deterministic.
#include "gs_common.cuh"
#include "gs_internal.h"

namespace gs {
namespace {

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;
constexpr int kViewChunk = 256;   // views whose partial results a block keeps in shared memory at once

// Camera constants of the visibility test, as seven 16-byte vectors (a stride of 28 words:
// lanes reading different cameras with 16-byte loads meet no bank conflict).
struct __align__(16) VisCam {
  float4 a;   // T, R2
  float4 b;   // R5, R8, R0, R3
  float4 c;   // R6, R1, R4, R7
  float4 k;   // fx, fy, cx, cy
  float4 w;   // W, H, |dt_z/dmu|, scale of the rounding margin
  float4 g;   // |d(fx t_x + cx t_z)/dmu|, the same with cx - W, and both for y
  float4 e;   // 1e-6 (|cx| + |W|), 1e-6 (|cy| + |H|), cx - W, cy - H
};

__device__ inline void load_vis_cam(const gs_camera& g, VisCam& c) {
  const float* R = g.R;
  const float W = (float)g.width, H = (float)g.height;
  c.a = make_float4(g.T[0], g.T[1], g.T[2], R[2]);
  c.b = make_float4(R[5], R[8], R[0], R[3]);
  c.c = make_float4(R[6], R[1], R[4], R[7]);
  c.k = make_float4(g.fx, g.fy, g.cx, g.cy);
  const float n0 = norm3df(R[0], R[3], R[6]), n1 = norm3df(R[1], R[4], R[7]), n2 = norm3df(R[2], R[5], R[8]);
  auto plane = [&](int j, float f, float k) {   // norm of the gradient of f t_j + k t_z
    return norm3df(f * R[j] + k * R[2], f * R[3 + j] + k * R[5], f * R[6 + j] + k * R[8]);
  };
  c.g = make_float4(plane(0, g.fx, g.cx), plane(0, g.fx, g.cx - W), plane(1, g.fy, g.cy), plane(1, g.fy, g.cy - H));
  const float mx = fabsf(g.fx) * n0 + (fabsf(g.cx) + fabsf(W)) * n2;
  const float my = fabsf(g.fy) * n1 + (fabsf(g.cy) + fabsf(H)) * n2;
  c.w = make_float4(W, H, n2, 1e-4f * fmaxf(mx, my));
  c.e = make_float4(1e-6f * (fabsf(g.cx) + fabsf(W)), 1e-6f * (fabsf(g.cy) + fabsf(H)), g.cx - W, g.cy - H);
}

// v(x, g): t = R^T (mu - T) with each product and sum rounded separately, in the
// order ((R0 dx + R3 dy) + R6 dz); visible iff near < t_z <= range and the
// projection (fx t_x / t_z + cx, fy t_y / t_z + cy) lies in [0, W) x [0, H).
// The two correctly rounded divisions (most of the test's instructions) are only made when
// fx t_x + cx t_z is within 1e-6 of its terms from 0 or from W t_z: further away, the few
// units of 2^-24 by which the separately rounded quotient and sum can be off do not matter.
__device__ __forceinline__ bool visible(float mx, float my, float mz, const VisCam& c, float near_plane,
                                        float range) {
  const float4 ca = c.a, cb = c.b;
  const float dx = __fsub_rn(mx, ca.x), dy = __fsub_rn(my, ca.y), dz = __fsub_rn(mz, ca.z);
  const float tz = __fadd_rn(__fadd_rn(__fmul_rn(ca.w, dx), __fmul_rn(cb.x, dy)), __fmul_rn(cb.y, dz));
  if (!(tz > near_plane) || !(tz <= range)) return false;
  const float4 cc = c.c, k = c.k, e = c.e;
  const float tx = __fadd_rn(__fadd_rn(__fmul_rn(cb.z, dx), __fmul_rn(cb.w, dy)), __fmul_rn(cc.x, dz));
  const float ty = __fadd_rn(__fadd_rn(__fmul_rn(cc.y, dx), __fmul_rn(cc.z, dy)), __fmul_rn(cc.w, dz));
  const float ax = __fmul_rn(k.x, tx), ay = __fmul_rn(k.y, ty);
  const float ex = fmaf(e.x, tz, 1e-6f * fabsf(ax)), ey = fmaf(e.y, tz, 1e-6f * fabsf(ay));
  const float x0 = fmaf(k.z, tz, ax), x1 = fmaf(e.z, tz, ax);   // t_z u, t_z (u - W)
  const float y0 = fmaf(k.w, tz, ay), y1 = fmaf(e.w, tz, ay);
  if (tz > 1e-20f) {   // (the relative bound holds while nothing is subnormal)
    if (x0 < -ex || x1 > ex || y0 < -ey || y1 > ey) return false;
    if (x0 > ex && x1 < -ex && y0 > ey && y1 < -ey) return true;
  }
  const float u = __fadd_rn(__fdiv_rn(ax, tz), k.z);
  const float v = __fadd_rn(__fdiv_rn(ay, tz), k.w);
  return u >= 0.f && u < c.w.x && v >= 0.f && v < c.w.y;
}

// Group cull: false only if no mean within `rad` of (gx, gy, gz) can be visible.  t_z and the
// four functions fx t_x + cx t_z >= 0, fx t_x + (cx - W) t_z < 0 (and the same in y) are
// linear in the mean, so over the sphere each differs from its value at the centre by at most
// rad times the norm of its gradient; the margin (1e-4 of the terms' magnitudes, against a few
// units of 2^-24 that the separately rounded test can be off) covers both evaluations.
// Comparisons with a NaN keep the view.
__device__ __forceinline__ bool group_may_see(float gx, float gy, float gz, float rad, const VisCam& c,
                                              float near_plane, float range) {
  const float4 ca = c.a, cb = c.b, cc = c.c, k = c.k, w = c.w, g = c.g;
  const float dx = gx - ca.x, dy = gy - ca.y, dz = gz - ca.z;
  const float tx = cb.z * dx + cb.w * dy + cc.x * dz;
  const float ty = cc.y * dx + cc.z * dy + cc.w * dz;
  const float tz = ca.w * dx + cb.x * dy + cb.y * dz;
  const float ext = fabsf(dx) + fabsf(dy) + fabsf(dz) + rad;
  const float mz = w.z * (rad * 1.0001f + 1e-4f * ext) + 1e-6f;
  if (tz + mz <= near_plane || tz - mz > range * 1.0001f) return false;
  const float m = w.w * ext + 1e-6f, r = rad * 1.0001f;
  if (k.x * tx + k.z * tz < -(g.x * r + m)) return false;
  if (k.x * tx + (k.z - w.x) * tz > g.y * r + m) return false;
  if (k.y * ty + k.w * tz < -(g.z * r + m)) return false;
  if (k.y * ty + (k.w - w.y) * tz > g.w * r + m) return false;
  return true;
}

// u_i = |mu_cur - mu_prev| (or its square); unchanged means keep their u.
__global__ void k_uncertainty_update(const float4* mo_prev, const float4* mo_cur,
                                     float4* __restrict__ su, int64_t n, int squared) {
  pdl_begin();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = mo_prev[i], b = mo_cur[i];
    const float dx = __fsub_rn(b.x, a.x), dy = __fsub_rn(b.y, a.y), dz = __fsub_rn(b.z, a.z);
    if (dx == 0.f && dy == 0.f && dz == 0.f) continue;
    const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    su[i].w = squared ? d2 : __fsqrt_rn(d2);
  }
}

constexpr int kMomThreads = 512;   // threads of the threshold kernels
constexpr int kMomBlocks = 340;    // at most: sums, counts and squares of every block fill 1,020 of 1,024 slots

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
  return v;   // valid in lane 0
}

// Fixed-order block sum of doubles; valid in thread 0.  (A warp's FP64 addition holds the
// SM's FP64 unit for many cycles whatever the number of active lanes: only one warp adds the
// warps' sums.)
__device__ double block_sum_d(double v, double* s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_sum_d(v);
  __syncthreads();
  if (lane == 0) s[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (warp == 0) t = warp_sum_d(lane < (int)(blockDim.x >> 5) ? s[lane] : 0.0);
  return t;
}

// Sum of g per-block partials in a fixed order by one warp; valid in lane 0.
__device__ double sum_partials(const double* __restrict__ part, int g) {
  double v = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x & 31; b < g; b += 32) v += part[b];
  return warp_sum_d(v);
}

// Mean and spread of u over the Gaussians with mu_z >= ground_z, two passes over contiguous
// block ranges.  Pass 0: part[b] = sum of u, part[g + b] = number of Gaussians (exact in FP64).
// Pass 1: every block first forms the mean from pass 0's partials (a few hundred values from
// L2, in the same order everywhere) and stores its sum of squared deviations in
// part[2 g + b].  The last kernel forms the statistics.  Three launches; at first the count
// and the two sums were finished in kernels of their own, by a single thread adding 304 values
// one after the other (1M Gaussians: 80 us in six launches, now 34 us).
template <int kPass>
__global__ void __launch_bounds__(kMomThreads) k_u_moments(const float4* __restrict__ mo,
                                                           const float4* __restrict__ su, int64_t n, float ground_z,
                                                           double* __restrict__ part) {
  pdl_begin();
  __shared__ double s[kMomThreads / 32];
  const int g = gridDim.x, warp = threadIdx.x >> 5;
  double mean = 0.0;
  if (kPass) {
    if (warp < 2) {   // warp 0 the sum, warp 1 the count
      const double t = sum_partials(part + warp * g, g);
      if ((threadIdx.x & 31) == 0) s[warp] = t;
    }
    __syncthreads();
    mean = s[1] > 0.0 ? s[0] / s[1] : 0.0;
  }
  double acc = 0.0;
  uint32_t cnt = 0;
  const int64_t per = (n + g - 1) / g;
  const int64_t i0 = (int64_t)blockIdx.x * per;
  int64_t i1 = i0 + per;
  if (i1 > n) i1 = n;
#pragma unroll 4
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kMomThreads) {
    const float z = mo[i].z, uf = su[i].w;
    if (!(z >= ground_z)) continue;
    const double u = (double)uf;
    acc += kPass ? (u - mean) * (u - mean) : u;
    ++cnt;
  }
  const double t = block_sum_d(acc, s);
  if (kPass == 0) {
    const uint32_t w = __reduce_add_sync(0xffffffffu, cnt);
    __shared__ unsigned long long s_cnt;
    if (threadIdx.x == 0) s_cnt = 0ull;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_cnt, (unsigned long long)w);
    __syncthreads();
    if (threadIdx.x == 0) {
      part[blockIdx.x] = t;
      part[g + blockIdx.x] = (double)s_cnt;
    }
  } else if (threadIdx.x == 0) {
    part[2 * g + blockIdx.x] = t;
  }
}

// stats = (mean, sigma, t_high = mean + sigma/2, t_low = mean - sigma/2, count); 96 threads
__global__ void __launch_bounds__(96) k_u_finish(const double* part, int g, double* __restrict__ stats) {
  pdl_begin();
  __shared__ double s[3];
  const int warp = threadIdx.x >> 5;
  const double t = sum_partials(part + warp * g, g);
  if ((threadIdx.x & 31) == 0) s[warp] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    const double m = s[1], mean = m > 0.0 ? s[0] / m : 0.0, sigma = m > 0.0 ? sqrt(s[2] / m) : 0.0;
    stats[0] = mean;
    stats[1] = sigma;
    stats[2] = mean + 0.5 * sigma;
    stats[3] = mean - 0.5 * sigma;
    stats[4] = m;
  }
}

// Per block and view: xi mode: count of visible high-uncertainty Gaussians minus
// lambda * count of visible low ones (both counted exactly as integers, combined in
// the final pass); sum mode: sum of u over the visible Gaussians.
//
// Bound: FP32 issue on the visibility tests.  A warp holds 32 consecutive Gaussians, which a
// map built keyframe by keyframe has close together: 32 views at a time, one per lane, are
// first tested against a sphere around the warp's Gaussians that count (group_may_see), and
// only the views that pass are tested lane by lane.  A map in random order pays one group
// test per 32 lane tests.  1M room Gaussians, 256 views: 672 us with every pair tested, 206 us
// with the group cull, 146 us with the test's divisions left out where they cannot matter and
// the warps' groups strided over the map.  20k Gaussians occupied a block in two with eight warps,
// each a chain of 256 views; spread over blocks and views 62 -> 27 us in patches, 86 -> 33 us in
// random order (with every pair tested 84 and 83 us).
template <bool kSum>
__global__ void __launch_bounds__(kBlock) k_view_utility(const float4* __restrict__ mo, const float4* __restrict__ su,
                                                         int64_t n, const gs_camera* __restrict__ cams, int v0, int nv,
                                                         gs_utility_params prm, const double* __restrict__ stats,
                                                         uint32_t* __restrict__ cnt_part, float* __restrict__ sum_part,
                                                         int n_views) {
  pdl_begin();
  __shared__ VisCam s_cam[kViewChunk];
  __shared__ uint32_t s_acc[kSum ? 1 : 2][kWarps][kViewChunk];   // visible high, low; or the sum of u (float)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < nv; i += blockDim.x) load_vis_cam(cams[v0 + i], s_cam[i]);
  for (int i = threadIdx.x; i < (kSum ? 1 : 2) * kWarps * kViewChunk; i += blockDim.x) (&s_acc[0][0][0])[i] = 0u;
  __syncthreads();
  uint32_t* a_hi = s_acc[0][warp];
  uint32_t* a_lo = s_acc[kSum ? 0 : 1][warp];
  float* a_sum = reinterpret_cast<float*>(a_hi);
  const double t_hi = kSum ? 0.0 : stats[2], t_lo = kSum ? 0.0 : stats[3];
  // 32 Gaussians per warp at a time, strided over the map: what a stretch of it costs depends
  // on how many views see that part of the room.  The groups of a map with fewer of them than warps
  // are spread over the blocks, and each is shared by up to eight warps with a part of the views each
  const int64_t groups = (n + 31) >> 5, warps = (int64_t)gridDim.x * kWarps;
  int lp = 0;   // log2 of the warps per group
  while (lp < 3 && (groups << (lp + 1)) <= warps) ++lp;
  const int part = (((nv + 31) >> 5) + (1 << lp) - 1) >> lp << 5;   // views of one warp
  const bool few = (groups << lp) <= warps;
  for (int64_t unit = few ? (int64_t)warp * gridDim.x + blockIdx.x : (int64_t)blockIdx.x * kWarps + warp;
       unit < groups << lp; unit += warps) {
    const int64_t i = ((unit >> lp) << 5) + lane;
    const int v_lo = (int)(unit & ((1 << lp) - 1)) * part, v_hi = v_lo + part < nv ? v_lo + part : nv;
    float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
    float u = 0.f;
    bool use = false;
    if (i < n) {
      m = mo[i];
      u = su[i].w;
      use = m.z >= prm.ground_z;
    }
    const bool hi = use && !kSum && (double)u > t_hi;
    const bool lo = use && !kSum && (double)u < t_lo;
    const bool in = kSum ? use : (hi || lo);
    const uint32_t mask = __ballot_sync(0xffffffffu, in);
    if (!mask) continue;
    // sphere around the group's counted means
    float gx = in ? m.x : 0.f, gy = in ? m.y : 0.f, gz = in ? m.z : 0.f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      gx += __shfl_xor_sync(0xffffffffu, gx, d);
      gy += __shfl_xor_sync(0xffffffffu, gy, d);
      gz += __shfl_xor_sync(0xffffffffu, gz, d);
    }
    const float inv = 1.f / (float)__popc(mask);
    gx *= inv;
    gy *= inv;
    gz *= inv;
    const float ex = m.x - gx, ey = m.y - gy, ez = m.z - gz;
    // (a NaN or infinite mean makes the radius infinite: nothing is culled)
    const float r2 = in ? ex * ex + ey * ey + ez * ez : 0.f;
    const bool odd = __any_sync(0xffffffffu, !(r2 < INFINITY));
    const float rad = odd ? INFINITY : sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(r2)))) * 1.0001f;
    for (int vb = v_lo; vb < v_hi; vb += 32) {
      const int iv = vb + lane;
      const bool may = iv < v_hi && (odd || group_may_see(gx, gy, gz, rad, s_cam[iv], prm.near_plane, prm.range));
      uint32_t cand = __ballot_sync(0xffffffffu, may);
      while (cand) {
        const int v = vb + __ffs(cand) - 1;
        cand &= cand - 1u;
        const bool vis = in && visible(m.x, m.y, m.z, s_cam[v], prm.near_plane, prm.range);
        if (kSum) {
          float s = vis ? u : 0.f;
          if (!__any_sync(0xffffffffu, vis)) continue;
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
          if (lane == 0) a_sum[v] += s;
        } else {
          const uint32_t bh = __ballot_sync(0xffffffffu, vis && hi), bl = __ballot_sync(0xffffffffu, vis && lo);
          if (lane == 0 && (bh | bl)) {
            a_hi[v] += __popc(bh);
            a_lo[v] += __popc(bl);
          }
        }
      }
    }
  }
  __syncthreads();
  for (int v = threadIdx.x; v < nv; v += blockDim.x) {
    const size_t o = (size_t)blockIdx.x * n_views + v0 + v;
    if (kSum) {
      float s = 0.f;
      for (int w = 0; w < kWarps; ++w) s += __uint_as_float(s_acc[0][w][v]);
      sum_part[o] = s;
    } else {
      uint32_t h = 0, l = 0;
      for (int w = 0; w < kWarps; ++w) {
        h += s_acc[0][w][v];
        l += s_acc[kSum ? 0 : 1][w][v];
      }
      *reinterpret_cast<uint2*>(cnt_part + 2 * o) = make_uint2(h, l);
    }
  }
}

// One warp per view adds the g blocks' partials (lanes take every 32nd, then a fixed tree).
// One thread per view, walking all partials by itself, took 41 us for 256 views.
template <bool kSum>
__global__ void __launch_bounds__(kBlock) k_view_utility_finish(const uint32_t* cnt_part,
                                                                const float* sum_part, int g,
                                                                int n_views, float lambda, float* __restrict__ xi,
                                                                uint32_t* __restrict__ counts) {
  pdl_begin();
  const int v = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (v >= n_views) return;
  if (kSum) {
    float s = 0.f;
    for (int b = lane; b < g; b += 32) s += sum_part[(size_t)b * n_views + v];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if (lane == 0) xi[v] = s;
  } else {
    unsigned long long h = 0, l = 0;
    for (int b = lane; b < g; b += 32) {
      const uint2 c = *reinterpret_cast<const uint2*>(cnt_part + 2 * ((size_t)b * n_views + v));
      h += c.x;
      l += c.y;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      h += __shfl_down_sync(0xffffffffu, h, d);
      l += __shfl_down_sync(0xffffffffu, l, d);
    }
    if (lane == 0) {
      xi[v] = (float)((double)h - (double)lambda * (double)l);
      if (counts) {
        counts[2 * v] = (uint32_t)h;
        counts[2 * v + 1] = (uint32_t)l;
      }
    }
  }
}

// Mean uncertainty of cuboid regions: region (ix, iy, iz) with i = floor((mu - origin) / size)
// holds the Gaussians inside the grid; sums in FP64, counts exact.
//
// Bound at first: FP64 atomics on few addresses (regions are metres wide, so neighbouring
// Gaussians share one), then FP64 additions themselves (a warp's addition holds the SM's FP64
// unit for 16 cycles: a shuffle reduction per region and warp step took 42 us).  So every
// warp keeps a table of the first kRegSlots regions it meets in its stretch of the map, with
// one FP64 sum per slot and lane in shared memory: one addition per 32 Gaussians, and one
// reduction and one global atomic per slot at the end.  Lanes whose region finds no slot (a
// map in random order) add for themselves, and then meet few others on an address; a full table is
// looked through slot by slot (region by region, 81,920 regions took 64 us instead of 60).
// 1M Gaussians, 32 regions: 702 us with one atomic per Gaussian, now 25 us.
constexpr int kRegSlots = 8;

__global__ void __launch_bounds__(kBlock) k_regions(const float4* __restrict__ mo, const float4* __restrict__ su,
                                                    int64_t n, gs_region_grid grid, double* __restrict__ sum,
                                                    uint32_t* __restrict__ count) {
  pdl_begin();
  __shared__ double s_acc[kWarps][kRegSlots][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < kRegSlots; ++k) s_acc[warp][k][lane] = 0.0;
  __syncwarp();
  int tab = -1;        // lane k < n_tab: region of slot k
  uint32_t cnt = 0;    // ... and its number of Gaussians
  int n_tab = 0;       // slots in use (warp-uniform)
  const int64_t n_warps = (int64_t)gridDim.x * kWarps;
  const int64_t per = ((n + n_warps - 1) / n_warps + 31) / 32 * 32;
  const int64_t i0 = ((int64_t)blockIdx.x * kWarps + warp) * per;
  const int64_t i1 = i0 + per < n ? i0 + per : n;
  float4 m_next = make_float4(0.f, 0.f, 0.f, 0.f);
  float u_next = 0.f;
  if (i0 + lane < i1) {
    m_next = mo[i0 + lane];
    u_next = su[i0 + lane].w;
  }
  for (int64_t b = i0; b < i1; b += 32) {
    const float4 m = m_next;
    const float uf = u_next;
    const bool have = b + lane < i1;
    if (b + 32 + lane < i1) {
      m_next = mo[b + 32 + lane];
      u_next = su[b + 32 + lane].w;
    }
    int r = -1;
    if (have) {
      const float fx = floorf(__fdiv_rn(__fsub_rn(m.x, grid.origin[0]), grid.size));
      const float fy = floorf(__fdiv_rn(__fsub_rn(m.y, grid.origin[1]), grid.size));
      const float fz = floorf(__fdiv_rn(__fsub_rn(m.z, grid.origin[2]), grid.size));
      if (fx >= 0.f && fy >= 0.f && fz >= 0.f && fx < (float)grid.dims[0] && fy < (float)grid.dims[1] &&
          fz < (float)grid.dims[2])
        r = (int)(((int64_t)fz * grid.dims[1] + (int64_t)fy) * grid.dims[0] + (int64_t)fx);   // at most 2^30 regions
    }
    uint32_t left = __ballot_sync(0xffffffffu, r >= 0);
    int slot = -1;
    if (n_tab == kRegSlots) {   // a full table is looked through once, whatever the number of regions here
#pragma unroll
      for (int k = 0; k < kRegSlots; ++k) {
        const uint32_t same = __ballot_sync(0xffffffffu, r == __shfl_sync(0xffffffffu, tab, k));
        if (lane == k) cnt += __popc(same);
        if ((same >> lane) & 1u) slot = k;
      }
      left = 0u;
    }
    while (left) {
      const int rr = __shfl_sync(0xffffffffu, r, __ffs(left) - 1);
      const uint32_t same = __ballot_sync(0xffffffffu, r == rr);
      int k = __ffs(__ballot_sync(0xffffffffu, tab == rr)) - 1;
      if (k < 0) {
        if (n_tab == kRegSlots) {   // the table is full: its lanes add for themselves
          left &= ~same;
          continue;
        }
        k = n_tab++;
        if (lane == k) tab = rr;
      }
      if (lane == k) cnt += __popc(same);
      if (r == rr) slot = k;
      left &= ~same;
    }
    if (slot >= 0) {
      s_acc[warp][slot][lane] += (double)uf;
    } else if (r >= 0) {
      atomicAdd(&sum[r], (double)uf);
      atomicAdd(&count[r], 1u);
    }
  }
  __syncwarp();
  for (int k = 0; k < n_tab; ++k) {
    const int rr = __shfl_sync(0xffffffffu, tab, k);
    double v = s_acc[warp][k][lane];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    if (lane == 0) atomicAdd(&sum[rr], v);
  }
  if (lane < n_tab) atomicAdd(&count[tab], cnt);
}

__global__ void k_region_mean(const double* sum, const uint32_t* count, int64_t n_reg,
                              float* __restrict__ omega) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_reg; r += (int64_t)gridDim.x * blockDim.x)
    omega[r] = count[r] ? (float)(sum[r] / (double)count[r]) : 0.f;
}

// Trajectory information (Eq. traj_utility): per trajectory the sum over its states
// of xi (states l = 0..L in order, FP64), and the first trajectory with the largest sum.
__global__ void k_traj_sum(const float* xi, int n_traj, int n_states, float* __restrict__ out,
                           int32_t* __restrict__ best) {
  pdl_begin();
  __shared__ double s_best[256];
  __shared__ int s_idx[256];
  double bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int t = threadIdx.x; t < n_traj; t += blockDim.x) {
    double acc = 0.0;
    for (int l = 0; l < n_states; ++l) acc += (double)xi[(size_t)t * n_states + l];
    out[t] = (float)acc;
    if (acc > bv) { bv = acc; bi = t; }
  }
  s_best[threadIdx.x] = bv;
  s_idx[threadIdx.x] = bi;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = -INFINITY;
    int i = 0x7fffffff;
    for (int k = 0; k < (int)blockDim.x; ++k)
      if (s_best[k] > v || (s_best[k] == v && s_idx[k] < i)) { v = s_best[k]; i = s_idx[k]; }
    *best = n_traj > 0 ? i : -1;
  }
}

// Collision check (Sec. IV-B).  Minimum of floats by integer atomics on their bits: among
// non-negative floats the signed order, among negative ones the reversed unsigned order, and
// any negative float is below any non-negative one in the signed order.  (Never -0 or NaN.)
__device__ __forceinline__ void atomic_min_float(float* p, float v) {
  if (v >= 0.f) atomicMin(reinterpret_cast<int*>(p), __float_as_int(v));
  else atomicMax(reinterpret_cast<unsigned*>(p), __float_as_uint(v));
}

// gamma of a Gaussian (negative or NaN: takes part in nothing)
__device__ __forceinline__ float col_gamma(const float4& s, float r_robot, float lambda_g) {
  return __fadd_rn(r_robot, __fmul_rn(lambda_g, ex32(fmaxf(fmaxf(s.x, s.y), s.z))));   // principal axis
}

// |p - mu|^2 < gamma^2, and the pair's margin (infinite when it changes nothing)
__device__ __forceinline__ bool pair_collides(const float4& p, const float4& mu, float gamma, float& margin) {
  const float dx = __fsub_rn(p.x, mu.x), dy = __fsub_rn(p.y, mu.y), dz = __fsub_rn(p.z, mu.z);
  const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
  const bool use = gamma >= 0.f;
  margin = use && d2 < INFINITY ? sqrtf(d2) - gamma : INFINITY;
  return use && d2 < __fmul_rn(gamma, gamma);
}

constexpr int kColChunk = 2048;               // Gaussians per block of the collision kernel
constexpr int kColGroups = kColChunk / 32;    // groups of 32, each with a bounding sphere
static_assert(kColGroups == 64, "two groups per lane below");
// A point to which more groups than this still matter after its nearest one takes the whole chunk
// instead.  Whole, a group of 32 costs about 17 instructions (the pair test; every lane keeps its own
// minimum), chosen group by group about 50 (the test, a vote, five exchanges with minima, the bounds
// again), so the line lies near 64 x 17 / 50 = 22; 12 and 20 measure alike, 32 is slower by up to a
// quarter.
constexpr int kColAll = 12;

// Each block stages a chunk of Gaussians (mu, gamma) with a sphere (centre, radius + largest
// gamma) around every 32 of them and one around the chunk.  |p - c| - radius - gamma bounds
// the margins inside a sphere from below, so Gaussians whose bound is not below the smallest
// margin known so far (k_collision_seed's, other blocks', this warp's) and that cannot
// collide are skipped: first the chunk, 256 points at a time, one per thread; then, for the
// points that are left, one per warp, the 64 groups, two per lane, the nearest evaluated
// first, one Gaussian per lane.  The results are the minimum margin over all Gaussians and
// whether some Gaussian has |p - mu|^2 < gamma^2 (separately rounded FP32), whatever the
// order, because what is skipped can change neither.
// A map in random order has wide spheres, so most groups matter to most points, which then take whole
// chunks (kColAll): 3M shuffled Gaussians and 129 points 1,200 -> 316 us, 1,000 points 9,050 -> 2,260
// us (every pair with one point per thread: 466 and 2,640 us); in patches 60 -> 45 us and 183 -> 134.
// Bound: the staging (32 B and an exponential per Gaussian) and the latency of the chain of
// evaluations near the points.  3M Gaussians, 129 points: 453 us with every pair evaluated (one point per thread),
// 153 us with groups of 32 only, 96 us with first bounds, 64 us with the chunk test (and 7 us for the
// first bounds).
__global__ void __launch_bounds__(kBlock) k_collision(const float4* __restrict__ mo, const float4* __restrict__ su,
                                                      int64_t n, const float4* __restrict__ pts, int n_pts,
                                                      float r_robot, float lambda_g, float ground_z, float* margin,
                                                      uint32_t* hit) {
  pdl_begin();
  __shared__ float4 s_g[kColChunk];        // (mu, gamma); gamma < 0: no Gaussian
  __shared__ float4 s_c[kColGroups];       // (centre, radius + largest gamma); -inf: empty group
  __shared__ float4 s_all;                 // the same for the whole chunk
  __shared__ uint16_t s_pt[kBlock];        // points of the current 256 that the chunk may matter to
  __shared__ uint32_t s_n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t g0 = (int64_t)blockIdx.x * kColChunk;
#pragma unroll 2
  for (int q = warp; q < kColGroups; q += kWarps) {   // warp-uniform
    const int64_t gi = g0 + q * 32 + lane;
    float4 e = make_float4(INFINITY, 0.f, 0.f, -1.f);   // (infinitely far: no pair with it counts)
    if (gi < n) {
      const float4 m = mo[gi];
      const float4 s = su[gi];
      const float gamma = col_gamma(s, r_robot, lambda_g);
      if (m.z >= ground_z && gamma >= 0.f) e = make_float4(m.x, m.y, m.z, gamma);
    }
    s_g[q * 32 + lane] = e;
    const bool use = e.w >= 0.f;
    const uint32_t mask = __ballot_sync(0xffffffffu, use);
    float cx = use ? e.x : 0.f, cy = use ? e.y : 0.f, cz = use ? e.z : 0.f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      cx += __shfl_xor_sync(0xffffffffu, cx, d);
      cy += __shfl_xor_sync(0xffffffffu, cy, d);
      cz += __shfl_xor_sync(0xffffffffu, cz, d);
    }
    const float inv = 1.f / (float)__popc(mask);
    cx *= inv;
    cy *= inv;
    cz *= inv;
    const float ex = e.x - cx, ey = e.y - cy, ez = e.z - cz;
    const float reach = use ? (sqrtf(ex * ex + ey * ey + ez * ez) + e.w) * 1.0001f : 0.f;
    // a NaN or infinite reach (a non-finite mean) makes the bound -inf: the group is evaluated
    const bool odd = __any_sync(0xffffffffu, !(reach < INFINITY));
    const float rg = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(reach)));
    if (lane == 0)
      s_c[q] = !mask ? make_float4(0.f, 0.f, 0.f, -INFINITY)
               : odd ? make_float4(0.f, 0.f, 0.f, INFINITY) : make_float4(cx, cy, cz, rg);
  }
  __syncthreads();
  // one sphere around the chunk, from the groups' spheres
  if (warp == 0) {
    const float4 a = s_c[lane], b = s_c[lane + 32];
    const bool ua = a.w != -INFINITY, ub = b.w != -INFINITY;
    float cx = (ua ? a.x : 0.f) + (ub ? b.x : 0.f), cy = (ua ? a.y : 0.f) + (ub ? b.y : 0.f);
    float cz = (ua ? a.z : 0.f) + (ub ? b.z : 0.f);
    const uint32_t k = __popc(__ballot_sync(0xffffffffu, ua)) + __popc(__ballot_sync(0xffffffffu, ub));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      cx += __shfl_xor_sync(0xffffffffu, cx, d);
      cy += __shfl_xor_sync(0xffffffffu, cy, d);
      cz += __shfl_xor_sync(0xffffffffu, cz, d);
    }
    const float inv = 1.f / (float)k;
    cx *= inv;
    cy *= inv;
    cz *= inv;
    auto far = [&](const float4& c) {
      const float dx = c.x - cx, dy = c.y - cy, dz = c.z - cz;
      return (sqrtf(dx * dx + dy * dy + dz * dz) + c.w) * 1.0001f;
    };
    const float ra = ua ? far(a) : 0.f, rb = ub ? far(b) : 0.f;
    const bool odd = __any_sync(0xffffffffu, !(ra < INFINITY) || !(rb < INFINITY));
    const float rg = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(ra, rb))));
    if (lane == 0)
      s_all = !k ? make_float4(0.f, 0.f, 0.f, -INFINITY)
              : odd ? make_float4(0.f, 0.f, 0.f, INFINITY) : make_float4(cx, cy, cz, rg);
  }
  __syncthreads();
  const float4 call = s_all, ca = s_c[lane], cb = s_c[lane + 32];
  if (call.w == -INFINITY) return;   // no Gaussian takes part
  for (int p0 = blockIdx.y * kBlock; p0 < n_pts; p0 += gridDim.y * kBlock) {
    // 256 points at a time, one per thread, against the chunk's sphere
    __syncthreads();
    if (threadIdx.x == 0) s_n = 0u;
    __syncthreads();
    const int pt = p0 + threadIdx.x;
    if (pt < n_pts) {
      const float4 p = pts[pt];
      const float best = *(volatile float*)(margin + pt);
      const bool col = *(volatile uint32_t*)(hit + pt) != 0u;
      const float dx = p.x - call.x, dy = p.y - call.y, dz = p.z - call.z;
      const float l = sqrtf(dx * dx + dy * dy + dz * dz) * 0.9999f - call.w - 1e-6f;
      if (!(l >= best) || (!col && !(l > 0.f))) s_pt[atomicAdd(&s_n, 1u)] = (uint16_t)threadIdx.x;
    }
    __syncthreads();
    const int todo = (int)s_n;
    for (int t = warp; t < todo; t += kWarps) {
      const int pi = p0 + s_pt[t];
      const float4 p = pts[pi];
      const float seed = *(volatile float*)(margin + pi);
      float best = seed;                                   // warp-uniform
      bool col = *(volatile uint32_t*)(hit + pi) != 0u;    // warp-uniform
      const bool seen = col;
      // lower bound of a group's margins; rounding (a few 2^-24 of the distances) is covered by 1e-4
      auto bound = [&](const float4& c) {
        const float dx = p.x - c.x, dy = p.y - c.y, dz = p.z - c.z;
        return sqrtf(dx * dx + dy * dy + dz * dz) * 0.9999f - c.w - 1e-6f;
      };
      float la = bound(ca), lb = bound(cb);
      bool wa = ca.w != -INFINITY, wb = cb.w != -INFINITY;   // still to be looked at
      auto evaluate = [&](int q) {
        const float4 g = s_g[q * 32 + lane];
        float m;
        col |= __any_sync(0xffffffffu, pair_collides(p, g, g.w, m)) != 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, d));
        best = fminf(best, m);
      };
      // a group matters unless its margins cannot be below `best` nor any of it collide anew
      auto matters = [&](float l) { return !(l >= best) || (!col && !(l > 0.f)); };
      uint32_t na = __ballot_sync(0xffffffffu, wa && matters(la));
      uint32_t nb = __ballot_sync(0xffffffffu, wb && matters(lb));
      if (na | nb) {   // the nearest group first
        const float l = fminf(wa ? la : INFINITY, wb ? lb : INFINITY);
        const uint32_t key = __float_as_uint(l) ^ (__float_as_uint(l) >> 31 ? 0xFFFFFFFFu : 0x80000000u);
        const int who = __ffs(__ballot_sync(0xffffffffu, key == __reduce_min_sync(0xffffffffu, key))) - 1;
        const int q = __shfl_sync(0xffffffffu, wa && !(la > l) ? lane : lane + 32, who);
        evaluate(q);
        if (lane == (q & 31)) (q < 32 ? wa : wb) = false;
        na = __ballot_sync(0xffffffffu, wa && matters(la));
        nb = __ballot_sync(0xffffffffu, wb && matters(lb));
      }
      if (__popc(na) + __popc(nb) > kColAll) {
        na = nb = 0u;
        float low = best;    // of this lane's Gaussians
        bool in = false;
#pragma unroll 4
        for (int q = 0; q < kColGroups; ++q) {
          const float4 g = s_g[q * 32 + lane];
          const float dx = __fsub_rn(p.x, g.x), dy = __fsub_rn(p.y, g.y), dz = __fsub_rn(p.z, g.z);
          const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
          in |= d2 < __fmul_rn(g.w, g.w);
          const float lim = fmaxf(__fadd_ru(g.w, low), 0.f);   // a smaller margin needs |p - mu| < gamma + low
          if (d2 < lim * lim * 1.0001f) low = fminf(low, sqrtf(d2) - g.w);
        }
        col |= __any_sync(0xffffffffu, in) != 0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) low = fminf(low, __shfl_xor_sync(0xffffffffu, low, d));
        best = low;
      }
      while (na | nb) {
        const int q = na ? __ffs(na) - 1 : 31 + __ffs(nb);
        evaluate(q);
        if (lane == (q & 31)) (q < 32 ? wa : wb) = false;
        na = __ballot_sync(0xffffffffu, wa && matters(la));
        nb = __ballot_sync(0xffffffffu, wb && matters(lb));
      }
      if (lane == 0) {
        if (best < seed) atomic_min_float(margin + pi, best);
        if (col && !seen) atomicOr(hit + pi, 1u);
      }
    }
  }
}

// First bounds: one block per point over at most kColSamples Gaussians spread over the map
// (every one of them a true pair, so margin and hit are bounds of the results).  Without
// them the blocks of the first wave know no margin and evaluate all their groups.
constexpr int kColSamples = 2048;
constexpr int kSeedThreads = 512;

__global__ void __launch_bounds__(kSeedThreads) k_collision_seed(const float4* mo,
                                                                 const float4* su, int64_t n,
                                                                 const float4* pts, float r_robot,
                                                                 float lambda_g, float ground_z,
                                                                 float* __restrict__ margin,
                                                                 uint32_t* __restrict__ hit) {
  pdl_begin();
  constexpr int kPer = kColSamples / kSeedThreads;
  __shared__ float s_m[kSeedThreads / 32];
  __shared__ uint32_t s_h[kSeedThreads / 32];
  const float4 p = pts[blockIdx.x];
  const int64_t step = (n + kColSamples - 1) / kColSamples;
  float best = INFINITY;
  bool col = false;
  float4 m[kPer], s[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {   // all loads in flight together
    const int64_t i = (int64_t)(threadIdx.x + k * kSeedThreads) * step;
    m[k] = i < n ? mo[i] : make_float4(0.f, 0.f, NAN, 0.f);
    s[k] = i < n ? su[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    float margin_i;
    const bool c = pair_collides(p, m[k], col_gamma(s[k], r_robot, lambda_g), margin_i);
    if (m[k].z >= ground_z) {   // (false for the NaN of no Gaussian)
      col |= c;
      best = fminf(best, margin_i);
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, d));
  const uint32_t any = __any_sync(0xffffffffu, col);
  if ((threadIdx.x & 31) == 0) {
    s_m[threadIdx.x >> 5] = best;
    s_h[threadIdx.x >> 5] = any;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t h = 0;
    for (int w = 0; w < kSeedThreads / 32; ++w) {
      best = fminf(best, s_m[w]);
      h |= s_h[w];
    }
    margin[blockIdx.x] = best;
    hit[blockIdx.x] = h ? 1u : 0u;
  }
}

__global__ void k_zero_bytes(uint8_t* p, size_t n) {
  pdl_begin();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) p[i] = 0;
}

// Blocks of the view-utility kernel: four of 256 threads fit an SM (45 KB of shared memory
// each), within the 1,024 partial slots of the workspace.
int utility_grid() {
  const int g = 4 * device_sm_count();
  return g > 1024 ? 1024 : g;
}

}  // namespace

cudaError_t launch_uncertainty_update(const float* mo_prev, const float* mo_cur, float* su, int64_t n, int squared,
                                      cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t g = (n + kBlock - 1) / kBlock;
  if (g > 4096) g = 4096;
  launch(k_uncertainty_update, (unsigned)g, kBlock, 0, st, reinterpret_cast<const float4*>(mo_prev),
         reinterpret_cast<const float4*>(mo_cur), reinterpret_cast<float4*>(su), n, squared);
  return cudaGetLastError();
}

size_t thresholds_ws_bytes() {
  return align_up(sizeof(double) * 1024, 256);
}

cudaError_t launch_uncertainty_thresholds(const float* mo, const float* su, int64_t n, float ground_z, double* stats,
                                          void* ws, cudaStream_t st) {
  Carver c(ws);
  double* part = c.take<double>(1024);
  int g = 2 * device_sm_count();
  if (g > kMomBlocks) g = kMomBlocks;
  const float4* m = reinterpret_cast<const float4*>(mo);
  const float4* s = reinterpret_cast<const float4*>(su);
  launch_spread(k_u_moments<0>, g, kMomThreads, 0, st, m, s, n, ground_z, part);
  launch_spread(k_u_moments<1>, g, kMomThreads, 0, st, m, s, n, ground_z, part);
  launch(k_u_finish, 1, 96, 0, st, part, g, stats);
  return cudaGetLastError();
}

size_t utility_ws_bytes(int n_views) {
  const int g = 1024;
  return align_up(sizeof(uint32_t) * 2 * (size_t)g * n_views, 256) + align_up(sizeof(float) * (size_t)g * n_views, 256);
}

cudaError_t launch_view_utility(const float* mo, const float* su, int64_t n, const gs_camera* cams, int n_views,
                                const gs_utility_params& prm, int mode, const double* stats, float* xi,
                                uint32_t* counts, void* ws, cudaStream_t st) {
  Carver c(ws);
  uint32_t* cnt_part = c.take<uint32_t>(2 * (size_t)1024 * n_views);
  float* sum_part = c.take<float>((size_t)1024 * n_views);
  const int g = utility_grid();
  const bool sum = mode == GS_XI_SUM;
  for (int v0 = 0; v0 < n_views; v0 += kViewChunk) {
    const int nv = n_views - v0 < kViewChunk ? n_views - v0 : kViewChunk;
    if (sum)
      launch_spread(k_view_utility<true>, g, kBlock, 0, st, reinterpret_cast<const float4*>(mo),
                    reinterpret_cast<const float4*>(su), n, cams, v0, nv, prm, stats, cnt_part, sum_part, n_views);
    else
      launch_spread(k_view_utility<false>, g, kBlock, 0, st, reinterpret_cast<const float4*>(mo),
                    reinterpret_cast<const float4*>(su), n, cams, v0, nv, prm, stats, cnt_part, sum_part, n_views);
  }
  const int fb = (n_views + kWarps - 1) / kWarps;
  if (sum) launch(k_view_utility_finish<true>, fb, kBlock, 0, st, cnt_part, sum_part, g, n_views, prm.lambda, xi,
                  counts);
  else launch(k_view_utility_finish<false>, fb, kBlock, 0, st, cnt_part, sum_part, g, n_views, prm.lambda, xi,
              counts);
  return cudaGetLastError();
}

size_t regions_ws_bytes(int64_t n_regions) {
  return align_up(sizeof(double) * (size_t)n_regions, 256) + align_up(sizeof(uint32_t) * (size_t)n_regions, 256);
}

cudaError_t launch_regions(const float* mo, const float* su, int64_t n, const gs_region_grid& grid, float* omega,
                           uint32_t* count_out, void* ws, cudaStream_t st) {
  const int64_t nr = (int64_t)grid.dims[0] * grid.dims[1] * grid.dims[2];
  Carver c(ws);
  double* sum = c.take<double>((size_t)nr);
  uint32_t* cnt = c.take<uint32_t>((size_t)nr);
  if (count_out) cnt = count_out;
  int64_t zb = ((int64_t)sizeof(double) * nr + 255) / 256;
  if (zb > 4096) zb = 4096;
  launch(k_zero_bytes, (unsigned)(zb < 1 ? 1 : zb), 256, 0, st, reinterpret_cast<uint8_t*>(sum), sizeof(double) * nr);
  launch(k_zero_bytes, (unsigned)(zb < 1 ? 1 : zb), 256, 0, st, reinterpret_cast<uint8_t*>(cnt),
         sizeof(uint32_t) * nr);
  if (n > 0) {
    int64_t g = (n + kBlock - 1) / kBlock;
    const int64_t most = 8 * (int64_t)device_sm_count();
    if (g > most) g = most;
    launch_spread(k_regions, (unsigned)g, kBlock, 0, st, reinterpret_cast<const float4*>(mo),
                  reinterpret_cast<const float4*>(su), n, grid, sum, cnt);
  }
  int64_t g2 = (nr + 255) / 256;
  if (g2 > 4096) g2 = 4096;
  launch(k_region_mean, (unsigned)(g2 < 1 ? 1 : g2), 256, 0, st, sum, cnt, nr, omega);
  return cudaGetLastError();
}

size_t trajectory_ws_bytes(int n_states_total) {
  return utility_ws_bytes(n_states_total) + align_up(sizeof(float) * (size_t)n_states_total, 256);
}

cudaError_t launch_trajectory_utility(const float* mo, const float* su, int64_t n, const gs_camera* cams, int n_traj,
                                      int n_states, const gs_utility_params& prm, int mode, const double* stats,
                                      float* traj_out, int32_t* best_out, void* ws, cudaStream_t st) {
  const int total = n_traj * n_states;
  Carver c(ws);
  void* uws = c.take<char>(utility_ws_bytes(total));
  float* xi = c.take<float>((size_t)total);
  cudaError_t e = launch_view_utility(mo, su, n, cams, total, prm, mode, stats, xi, nullptr, uws, st);
  if (e != cudaSuccess) return e;
  launch(k_traj_sum, 1, 256, 0, st, xi, n_traj, n_states, traj_out, best_out);
  return cudaGetLastError();
}

cudaError_t launch_collision_check(const float* mo, const float* su, int64_t n, const float* pts, int n_pts,
                                   float r_robot, float lambda_g, float ground_z, float* margin_out,
                                   uint32_t* collides_out, cudaStream_t st) {
  if (n_pts <= 0) return cudaSuccess;
  launch(k_collision_seed, (unsigned)n_pts, kSeedThreads, 0, st, reinterpret_cast<const float4*>(mo),
         reinterpret_cast<const float4*>(su), n, reinterpret_cast<const float4*>(pts), r_robot, lambda_g, ground_z,
         margin_out, collides_out);
  if (n > kColSamples) {   // (a smaller map has been seen whole)
    // small maps: the points are shared out over several blocks per chunk, so that about three
    // blocks per SM run (each block stages its chunk again)
    const int64_t chunks = (n + kColChunk - 1) / kColChunk;
    const int64_t want = 3 * (int64_t)device_sm_count();
    int64_t split = (want + chunks - 1) / chunks;
    const int64_t most = (n_pts + kBlock - 1) / kBlock;
    if (split > most) split = most;
    if (split > 65535) split = 65535;
    launch_spread(k_collision, dim3((unsigned)chunks, (unsigned)split), kBlock, 0, st,
                  reinterpret_cast<const float4*>(mo), reinterpret_cast<const float4*>(su), n,
                  reinterpret_cast<const float4*>(pts), n_pts, r_robot, lambda_g, ground_z, margin_out, collides_out);
  }
  return cudaGetLastError();
}

}  // namespace gs
