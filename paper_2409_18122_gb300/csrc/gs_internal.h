// gs_internal.h -- host-side launchers shared between the translation units of
// libgs103.so.  Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <nvtx3/nvToolsExt.h>

#include "../../include/gs.h"
#include "smem_limit.h"

namespace gs {

// NVTX range over one C-ABI call (host side: argument checks and the enqueue of its
// kernels), named after the entry point, so that a profiler's timeline shows which call
// launched which kernels.  With no tool attached a push or pop is one indirect call.
struct TraceRange {
  explicit TraceRange(const char* name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange&) = delete;
  TraceRange& operator=(const TraceRange&) = delete;
};
#define GS_TRACE(name) ::gs::TraceRange gs_trace_range_(name)

// ------------------------------------------------------------------ helpers
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Carves consecutive 256-byte aligned sub-buffers out of a workspace.
struct Carver {
  char* base;
  size_t off = 0;
  explicit Carver(void* b) : base((char*)b) {}
  template <class T>
  T* take(size_t count) {
    off = align_up(off, 256);
    T* p = base ? (T*)(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

int device_sm_count();

// Host-side count of kernel launches enqueued by this library (work accounting).
void note_launch();
uint64_t launch_count();

// Launches a kernel behind the work already in the stream, with its start overlapped: the launch
// may place the kernel's blocks while the kernel before it still runs, and every kernel of the
// library begins with pdl_begin, which lets the next one be placed in turn (once all blocks of this
// one have started) and then waits until everything before it in the stream has finished and its
// writes are visible.  So the order of the work is that of plain launches; what is saved is the gap
// between kernels, which small calls are made of (some 32 launches for one view): one 640x480 view of 200k
// Gaussians 288 -> 232 us, 27 scored candidates 750 -> 685 us, 3M Gaussians and eight 1280x720 views
// 5.91 -> 5.85 ms.
// Its lifetime begins before the wait, while kernels before it still write, so nothing that they may
// write is read-only "for the lifetime of the kernel": a kernel launched this way takes no input
// through the non-coherent path (no __ldg, no `const ... __restrict__` parameter, which the compiler
// reads the same way and may read early).  A kernel launched plainly may.
template <class... P, class... A>
inline void launch_as(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                      A&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);   // (an error stays for cudaGetLastError)
  note_launch();
}

template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  launch_as(true, kernel, grid, block, smem, st, static_cast<A&&>(args)...);
}

// The same without the overlapped start, for the kernels that do most of a call's work: blocks placed
// early crowd onto the multiprocessors that are free first, and stay there (pair placement of four
// keyframes, 417 blocks: 106 us after a plain launch, 162 us after an overlapped one).
template <class... P, class... A>
inline void launch_spread(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  launch_as(false, kernel, grid, block, smem, st, static_cast<A&&>(args)...);
}

__device__ __forceinline__ void pdl_begin() {
#if defined(__CUDA_ARCH__)
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
#endif
}

// ------------------------------------------------------------------ scan
// Exclusive prefix sum of n uint32 values into out[0..n]; out[n] = total.
// n = min(*n_dev, n_cap) when n_dev != NULL, else n_cap.  Prefixes saturate at
// 0xFFFFFFFF.  If total_out != NULL, the (saturated) total is also stored there.
size_t scan_temp_bytes(int64_t n_cap);
cudaError_t scan_exclusive(const uint32_t* in, uint32_t* out, const uint32_t* n_dev, int64_t n_cap,
                           uint32_t* total_out, void* temp, cudaStream_t st);

// ------------------------------------------------------------------ record sort
// Stable sort of record indices by their keys within each segment (view): the elements
// [seg[s], seg[s+1]) of every segment s < n_seg (seg non-decreasing, seg[n_seg] = n =
// min(*n_dev, n_cap)) are sorted among themselves and stay in place.  Buffers a/b are ping-pong
// storage of n_cap entries each; ctl: two words that stay valid as long as the result is used.
struct SortBufs {
  uint32_t* keys_a;
  uint32_t* vals_a;
  uint32_t* keys_b;
  uint32_t* vals_b;
};
// Work of the last pass: for the record r written to position i, out_rect[i] = rect[r] and
// out_cnt[i] = its number of tiles (0, with an empty out_rect[i], for an empty rectangle or one
// outside its view's tile grid -- the latter also sets GS_FLAG_BAD_RECORDS).
struct SortRectEpilogue {
  const ushort4* rect;
  const uint32_t* view_info;
  ushort4* out_rect;
  uint32_t* out_cnt;
  uint32_t* status;
};
// Whether three 9-bit passes sort the keys (ctl = smallest and largest key): their top 14 bits
// differ by less than 512.
__host__ __device__ inline bool sorted_in_three(const uint32_t* ctl) { return (ctl[1] >> 18) - (ctl[0] >> 18) < 512u; }
// The sorted record indices: which buffer holds them is known on the device.
struct SortedRecords {
  const uint32_t* three;   // after three passes
  const uint32_t* four;    // after four
  const uint32_t* ctl;
  __device__ const uint32_t* get() const { return sorted_in_three(ctl) ? three : four; }
};
size_t record_sort_temp_bytes(int64_t n_cap, int n_seg);
cudaError_t record_sort(const uint32_t* keys, SortBufs bufs, const uint32_t* n_dev, int64_t n_cap, const uint32_t* seg,
                        int n_seg, const SortRectEpilogue& epi, uint32_t* ctl, void* temp, cudaStream_t st,
                        SortedRecords* out);

// ------------------------------------------------------------------ pipeline stages
size_t project_ws_bytes(int64_t n, int n_views);
cudaError_t launch_project(const gs_map& map, const gs_camera* cams, int n_views, const gs_params& p,
                           const gs_proj& out, void* ws, cudaStream_t st);

size_t bin_ws_bytes(int64_t rec_cap, int64_t pair_cap, int64_t tile_cap, int n_views);
// proj.view == NULL: records written by launch_project without view ids; the view segments
// come from proj.grp_base and the group count in view_info[V][3].
cudaError_t launch_bin_sort(const gs_proj& proj, const gs_camera* cams, int n_views, const gs_params& p,
                            const gs_bins& out, void* ws, cudaStream_t st);

// The warp items of the batch (n of them, view_info[V][2]) ordered longest tile list first.
// cnt: 2 * kOrderBuckets words, zero.  n > item_cap: the first item_cap items if `clamp`, else
// nothing is written.
constexpr int kOrderBuckets = 64;
void launch_item_order(const uint32_t* view_info, int n_views, const uint32_t* ranges, int64_t tile_cap,
                       int64_t item_cap, bool clamp, uint32_t* cnt, uint32_t* order, cudaStream_t st);

cudaError_t launch_render_fwd(const gs_map& map, const gs_proj& proj, const gs_bins& bins, const gs_camera* cams,
                              int n_views, const gs_params& p, const gs_image& img, cudaStream_t st);

// the one-launch forward render of a small map (small.cu)
cudaError_t launch_render_small(const gs_map& map, const gs_camera* cams, int n_views, const gs_params& p,
                                const gs_image& img, uint32_t* status, cudaStream_t st);

size_t bwd_ws_bytes(int64_t rec_cap);
// Every argument check of gs_render_bwd except the workspace's (api.cu); GS_OK if the
// arguments are valid.  Shared by the workspace and the allocation-free entry points.
gs_status validate_render_bwd(const gs_map* map, const gs_proj* proj, const gs_bins* bins, const gs_image* fwd,
                              const gs_image_grad* grad, const gs_camera* cams, int32_t n_views, const gs_params* prm,
                              const gs_map_grad* out);
cudaError_t launch_render_bwd(const gs_map& map, const gs_proj& proj, const gs_bins& bins, const gs_image& fwd,
                              const gs_image_grad& g, const gs_camera* cams, int n_views, const gs_params& p,
                              const gs_map_grad& out, void* ws, cudaStream_t st);

size_t ig_composite_ws_bytes(int64_t tile_cap);
cudaError_t launch_ig_composite(const gs_proj& proj, const gs_bins& bins, const gs_camera* cams, int n_views,
                                const gs_params& p, float* ig_out, void* ws, cudaStream_t st);

// rec_cap: record capacity of the batch (n * n_views when 0).
size_t ig_ws_bytes(int64_t n, int n_views, int64_t rec_cap, int64_t pair_cap, int64_t tile_cap);
cudaError_t launch_info_gain(const gs_map& map, const gs_camera* cams, int n_views, const gs_params& p,
                             float* ig_out, uint32_t* status, int64_t rec_cap, int64_t pair_cap, int64_t tile_cap,
                             void* ws, cudaStream_t st);

// render-free view utility (utility.cu)
cudaError_t launch_uncertainty_update(const float* mo_prev, const float* mo_cur, float* su, int64_t n, int squared,
                                      cudaStream_t st);
size_t thresholds_ws_bytes();
cudaError_t launch_uncertainty_thresholds(const float* mo, const float* su, int64_t n, float ground_z, double* stats,
                                          void* ws, cudaStream_t st);
size_t utility_ws_bytes(int n_views);
cudaError_t launch_view_utility(const float* mo, const float* su, int64_t n, const gs_camera* cams, int n_views,
                                const gs_utility_params& prm, int mode, const double* stats, float* xi,
                                uint32_t* counts, void* ws, cudaStream_t st);
size_t trajectory_ws_bytes(int n_states_total);
cudaError_t launch_trajectory_utility(const float* mo, const float* su, int64_t n, const gs_camera* cams, int n_traj,
                                      int n_states, const gs_utility_params& prm, int mode, const double* stats,
                                      float* traj_out, int32_t* best_out, void* ws, cudaStream_t st);
cudaError_t launch_collision_check(const float* mo, const float* su, int64_t n, const float* pts, int n_pts,
                                   float r_robot, float lambda_g, float ground_z, float* margin_out,
                                   uint32_t* collides_out, cudaStream_t st);
size_t regions_ws_bytes(int64_t n_regions);

// ------------------------------------------------------------------ Adam step
cudaError_t launch_adam(float* const* params, const float* const* grads, float* const* m, float* const* v,
                        const int64_t* sizes, int n_tensors, const gs_adam_params& prm, uint32_t* step,
                        cudaStream_t st);

// ------------------------------------------------------------------ mapping loss (Eq. 3)
// 0 if the sizes are invalid.
size_t image_loss_ws_bytes(const int32_t* sizes, int n_views);
cudaError_t launch_image_loss(const int32_t* sizes, int n_views, const float* rgb, const float* depth,
                              const float* rgb_ref, const float* depth_ref, const gs_loss_weights& w,
                              float* loss_out, float* d_rgb, float* d_depth, void* ws, cudaStream_t st);
cudaError_t launch_regions(const float* mo, const float* su, int64_t n, const gs_region_grid& grid, float* omega,
                           uint32_t* count_out, void* ws, cudaStream_t st);

}  // namespace gs
