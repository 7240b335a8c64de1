// sort.cu -- stable LSD radix sort of the records of each view by their 32-bit depth keys.
//
// The records of a view are a contiguous segment; partitions never cross a segment and digit
// offsets are scanned per segment, so every pass keeps each segment in place and the result is
// sorted within each segment.  Each pass is reduce-then-scan: (1) every partition block counts
// its digits, (2) the counts of each (segment, digit) are scanned over the segment's partitions,
// (3) every partition block walks its tiles in order, ranks each key stably inside the tile with
// warp ballots, stages the tile in shared memory in digit order and writes it out at the running
// digit offsets.  No block ever waits on another, the result is deterministic, and the launch
// shape depends only on the host-side capacity.
//
// Digits have 9 bits, so three passes cover 27.  Depth keys are the bits of positive floats, and
// a batch whose depths lie within a factor of about 2^16 (0.2 m to 13 km: 2^27 keys apart) differs
// in no more: the low two digits are taken as they are, the third is the rest of the key minus the
// rest of the smallest key, which fits in 9 bits when the rests differ by less than 512.  The device
// finds the smallest and largest key during the first counts; only a batch with a wider span runs
// a fourth pass over the top 5 bits (its blocks leave at once otherwise).  Against four 8-bit
// passes with tiles of 2,048 keys: 8.3 -> 6.0 ms for the 209M records of a 384-view batch, 0.50 ->
// 0.29 ms for the 8.4M of eight keyframes; 1.29 and 1.30 ms for the 40.6M of a 256-view batch.
// Bound: per tile, the ranking's instructions (135 per 32 keys and pass, 62% of cycles issue one)
// and, for large batches, output lines that leave L2 half written.  Warp matches instead of ballots
// are slower for digits that are nearly random (950 against 740 us), 512 or 1,024 threads per block
// wait at their barriers (890 / 1,150 us), and a persistent grid loses the overlap of blocks (890 us).
#include "gs_internal.h"

namespace gs {
namespace {

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;
// Keys per thread of a scatter block, so the tile is 256 times as many.  Large batches: 16 (4,096
// keys, 8 keys or 32 bytes per digit and store on average, and few open output lines; 128
// registers, two blocks per SM): with 8 the sort of 209M records takes 10.6 instead of 6.5 ms.
// Small ones (up to kSmallSort records): 4, more blocks on a chip they leave idle anyway (one
// 640x480 view of 200k Gaussians: 286 instead of 306 us); equal at 2M records.  Segments of at most
// kSmallSegs records, a tile and a half, also 4, however many they are: they fill no larger tile (512
// rendered views of a 5,000-Gaussian map 2,949 -> 2,851 us, 16,384 views of 1,000 9,013 -> 8,281; at
// 8,000 Gaussians the larger tile is 1% faster).
constexpr int kItemsLarge = 16, kItemsSmall = 4;
constexpr int64_t kSmallSort = 1 << 20;
constexpr int64_t kSmallSegs = 6144;
constexpr int kBits = 9;
constexpr int kRadix = 1 << kBits;
constexpr int kLastShift = 2 * kBits;    // the third digit's first bit
constexpr int kPitch = kRadix + 2;       // a warp's counts and one slot for absent keys
// Partitions of a large sort: kFewParts of at most kPartKeys records each, more of them up to
// kMaxParts for more records.  Small partitions keep the blocks that run at the same time on few
// segments, so the last pass, which gathers each record's rectangle by record index within its
// view, finds them in L2, and neighbouring blocks fill the same output lines; the histograms and
// their scans grow with the count.  209M records (25,600 per partition at 8,192): 20.5 -> 19.9 ms
// for the whole 384-view pass with 16,384; 40M records are faster with 8,192.
constexpr int kFewParts = 8192, kMaxParts = 16384;
constexpr int64_t kPartKeys = 16384;


inline bool small_sort(int64_t n_cap, int n_seg) { return n_cap <= kSmallSort || n_cap / n_seg <= kSmallSegs; }
inline int tile_keys(int64_t n_cap, int n_seg) {
  return kBlock * (small_sort(n_cap, n_seg) ? kItemsSmall : kItemsLarge);
}

inline int64_t parts_for(int64_t n_cap, int n_seg) {
  const int64_t t = tile_keys(n_cap, n_seg);
  int64_t g = (n_cap + t - 1) / t;
  if (g < 1) g = 1;
  if (g > kFewParts) g = n_cap <= kFewParts * kPartKeys ? kFewParts : kMaxParts;
  return g;
}

__device__ inline int64_t count_of(const uint32_t* n_dev, int64_t n_cap) {
  int64_t n = (int64_t)*n_dev;
  return n < n_cap ? n : n_cap;
}

// Partition map: pmap[0] = partition size, pmap[1 + s] = first
// partition of segment s (s = 0 .. n_seg).  Segment s of n_s elements gets
// ceil(n_s / size) partitions; size is chosen so that all fit in the grid.
__global__ void __launch_bounds__(1024) k_part_map(const uint32_t* seg, int n_seg, const uint32_t* n_dev,
                                                   int64_t n_cap, int grid, int tile, uint32_t* __restrict__ pmap,
                                                   uint32_t* __restrict__ ctl) {
  pdl_begin();
  __shared__ unsigned long long s_sum[32];
  const int64_t n = count_of(n_dev, n_cap);
  const int64_t avail = grid - n_seg > 1 ? grid - n_seg : 1;
  const int64_t few = avail < kFewParts ? avail : kFewParts;
  int64_t size = (n + few - 1) / few;
  if (size > kPartKeys) size = (n + avail - 1) / avail;
  size = (size + tile - 1) / tile * tile;
  if (size < tile) size = tile;
  const int per = (n_seg + blockDim.x - 1) / blockDim.x;
  const int s0 = threadIdx.x * per;
  int s1 = s0 + per;
  if (s1 > n_seg) s1 = n_seg;
  unsigned long long acc = 0;
  for (int t = s0; t < s1; ++t) {
    const int64_t a = seg[t], b = seg[t + 1];
    if (b > a) acc += (unsigned long long)((b - a + size - 1) / size);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long x = acc;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s_sum[warp] = x;
  __syncthreads();
  unsigned long long e = x - acc;
  for (int w = 0; w < warp; ++w) e += s_sum[w];
  for (int t = s0; t < s1; ++t) {
    pmap[1 + t] = (uint32_t)e;
    const int64_t a = seg[t], b = seg[t + 1];
    if (b > a) e += (unsigned long long)((b - a + size - 1) / size);
  }
  if (threadIdx.x == blockDim.x - 1) pmap[1 + n_seg] = (uint32_t)e;
  if (threadIdx.x == 0) {
    pmap[0] = (uint32_t)size;
    ctl[0] = 0xFFFFFFFFu;   // smallest and largest key: found by the first pass's counts
    ctl[1] = 0u;
  }
}

// Element range of this block's partition: empty past the last.
// Returns the partition's segment.
__device__ inline int seg_part_range(const uint32_t* __restrict__ seg, int n_seg, const uint32_t* __restrict__ pmap,
                                     int64_t& beg, int64_t& end) {
  const int64_t p = blockIdx.x;
  beg = end = 0;
  if (p >= (int64_t)pmap[1 + n_seg]) return 0;
  int lo = 0, hi = n_seg - 1;   // segment: the largest s with first partition <= p
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((int64_t)pmap[1 + mid] <= p) lo = mid;
    else hi = mid - 1;
  }
  const int64_t size = pmap[0];
  const int64_t a = seg[lo], b = seg[lo + 1];
  beg = a + (p - (int64_t)pmap[1 + lo]) * size;
  end = beg + size;
  if (end > b) end = b;
  if (beg > end) beg = end;
  return lo;
}

// The digit of a key in pass kPass (third pass: `base` = the smallest key's rest if the sort ends
// there, else 0).
template <int kPass>
__device__ __forceinline__ uint32_t digit_of(uint32_t key, uint32_t base) {
  if (kPass < 2) return (key >> (kPass * kBits)) & (kRadix - 1);
  if (kPass == 2) return ((key >> kLastShift) - base) & (kRadix - 1);
  return key >> (3 * kBits);
}

// (1) digit counts of each partition: hist[part][digit]; the first pass also finds the smallest
// and largest key.
template <int kPass>
__global__ void __launch_bounds__(kBlock) k_upsweep(const uint32_t* keys,
                                                    const uint32_t* seg, int n_seg,
                                                    const uint32_t* pmap, uint32_t* __restrict__ ctl,
                                                    uint32_t* __restrict__ hist) {
  pdl_begin();
  constexpr int kCopies = kWarps / 2;   // two warps share a copy of the counts
  __shared__ uint32_t cnt[kCopies][kRadix];
  const bool three = kPass >= 2 && sorted_in_three(ctl);
  if (kPass == 3 && three) return;
  if (blockIdx.x >= pmap[1 + n_seg]) return;
  const uint32_t base = three ? ctl[0] >> kLastShift : 0u;
  const int copy = threadIdx.x >> 6;
  for (int i = threadIdx.x; i < kCopies * kRadix; i += kBlock) (&cnt[0][0])[i] = 0;
  __syncthreads();
  int64_t beg, end;
  seg_part_range(seg, n_seg, pmap, beg, end);
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll 4
  for (int64_t i = beg + threadIdx.x; i < end; i += kBlock) {
    const uint32_t k = keys[i];
    atomicAdd(&cnt[copy][digit_of<kPass>(k, base)], 1u);
    if (kPass == 0) {
      lo = min(lo, k);
      hi = max(hi, k);
    }
  }
  if (kPass == 0) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0 && lo <= hi) {   // (most warps find both bounds wide enough already)
      const volatile uint32_t* now = ctl;
      if (lo < now[0]) atomicMin(&ctl[0], lo);
      if (hi > now[1]) atomicMax(&ctl[1], hi);
    }
  }
  __syncthreads();
#pragma unroll
  for (int d = threadIdx.x; d < kRadix; d += kBlock) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < kCopies; ++w) s += cnt[w][d];
    hist[(size_t)blockIdx.x * kRadix + d] = s;
  }
}

// (2) per segment and digit: hist[part][digit] -> exclusive prefix over the segment's
// partitions (in place) and the digit's total in the segment.  Block (s, y) takes 32 digits of
// segment s: lane = digit, warp w a contiguous range of the partitions, eight loads in flight;
// the warps' sums are scanned in shared memory.  (The scatter adds the digits' bases itself.)
// One block per segment with a thread per digit took 194 us of the 3M-Gaussian mapping
// iteration's four passes (eight segments: eight blocks); this
// takes 14 us.  At least kEachSegs segments with at most kEachParts partitions each on average are
// blocks enough with one each (k_scan_hist_each), and sixteen of 1,024 threads for a handful of
// partitions are a waste: 4,096 views of a 20k map 5,743 -> 4,904 us, 128 of a 100k map 609 -> 585.
constexpr int kEachSegs = 32, kEachParts = 64;
template <int kPass>
__global__ void __launch_bounds__(1024) k_scan_hist(uint32_t* __restrict__ hist, int g,
                                                    const uint32_t* pmap,
                                                    const uint32_t* ctl, uint32_t* __restrict__ tot) {
  pdl_begin();
  __shared__ uint32_t s_sum[32][33];
  if (kPass == 3 && sorted_in_three(ctl)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, s = blockIdx.x;
  const int d = blockIdx.y * 32 + lane;
  // (malformed segments can ask for more partitions than the grid has: those are never run)
  const int64_t p0 = pmap[1 + s] < (uint32_t)g ? pmap[1 + s] : g;
  const int64_t p1 = pmap[2 + s] < (uint32_t)g ? pmap[2 + s] : g;
  const int64_t per = (p1 - p0 + 31) / 32;
  const int64_t a = p0 + warp * per;
  const int64_t b = a + per < p1 ? a + per : p1;
  uint32_t sum = 0;
  for (int64_t p = a; p < b; p += 8) {
    uint32_t c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = p + k < b ? hist[(size_t)(p + k) * kRadix + d] : 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) sum += c[k];
  }
  s_sum[warp][lane] = sum;
  __syncthreads();
  uint32_t x = s_sum[lane][warp];   // warp = digit, lane = partition range
  const uint32_t own = x;
#pragma unroll
  for (int k = 1; k < 32; k <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, k);
    if (lane >= k) x += y;
  }
  if (lane == 31) tot[(size_t)s * kRadix + blockIdx.y * 32 + warp] = x;
  s_sum[lane][warp] = x - own;      // (read and written by this warp alone)
  __syncthreads();
  uint32_t run = s_sum[warp][lane];
  for (int64_t p = a; p < b; p += 8) {
    uint32_t c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = p + k < b ? hist[(size_t)(p + k) * kRadix + d] : 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (p + k < b) hist[(size_t)(p + k) * kRadix + d] = run;
      run += c[k];
    }
  }
}

// The same with one block per segment and a thread per digit, for many segments of few partitions.
template <int kPass>
__global__ void __launch_bounds__(kRadix) k_scan_hist_each(uint32_t* __restrict__ hist, int g, const uint32_t* pmap,
                                                           const uint32_t* ctl, uint32_t* __restrict__ tot) {
  pdl_begin();
  if (kPass == 3 && sorted_in_three(ctl)) return;
  const int s = blockIdx.x, d = threadIdx.x;
  const int64_t p0 = pmap[1 + s] < (uint32_t)g ? pmap[1 + s] : g;
  const int64_t p1 = pmap[2 + s] < (uint32_t)g ? pmap[2 + s] : g;
  uint32_t run = 0;
  for (int64_t p = p0; p < p1; p += 8) {
    uint32_t c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = p + k < p1 ? hist[(size_t)(p + k) * kRadix + d] : 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (p + k < p1) hist[(size_t)(p + k) * kRadix + d] = run;
      run += c[k];
    }
  }
  tot[(size_t)s * kRadix + d] = run;
}

// Exclusive prefix over the block of one value per thread (wsum: kWarps words; ends unsynchronised).
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int k = 1; k < 32; k <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, k);
    if (lane >= k) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  uint32_t e = x - v;
  for (int w = 0; w < warp; ++w) e += wsum[w];
  return e;
}

// (3) stable scatter of each partition's tiles.  The last pass writes the record indices, their
// rectangles and pair counts (SortRectEpilogue) instead of keys and values.
template <int kPass, int kItems>
__global__ void __launch_bounds__(kBlock, kItems > 8 ? 2 : 4) k_downsweep(const uint32_t* keys_in,
                                                          const uint32_t* vals_in,
                                                          const uint32_t* seg, int n_seg,
                                                          const uint32_t* pmap,
                                                          const uint32_t* ctl,
                                                          uint32_t* __restrict__ keys_out,
                                                          uint32_t* __restrict__ vals_out,
                                                          const uint32_t* hist,
                                                          const uint32_t* tot,
                                                          const SortRectEpilogue epi) {
  pdl_begin();
  constexpr int kTile = kBlock * kItems;
  constexpr int kG = kItems < 8 ? kItems : 8;   // rectangle gathers of a thread in flight
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* s_keys = smem;                    // kTile
  uint32_t* s_vals = s_keys + kTile;          // kTile
  uint32_t* whist = s_vals + kTile;           // kWarps * kPitch
  uint32_t* start = whist + kWarps * kPitch;  // kRadix: first position of each digit in the tile
  uint32_t* base = start + kRadix;            // kRadix: global slot minus position in the tile
  uint32_t* wsum = base + kRadix;             // kWarps

  const bool three = kPass >= 2 && sorted_in_three(ctl);
  if (kPass == 3 && three) return;
  const bool last = kPass == 3 || three;
  const uint32_t kbase = three ? ctl[0] >> kLastShift : 0u;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  int64_t beg, end;
  const int segment = seg_part_range(seg, n_seg, pmap, beg, end);
  if (beg >= end) return;
  // thread t owns digits 2t and 2t + 1: next free slot of each in this partition = segment start +
  // smaller digits + earlier partitions
  uint2 first;
  {
    const uint2 c = reinterpret_cast<const uint2*>(tot + (size_t)segment * kRadix)[tid];
    const uint2 h = reinterpret_cast<const uint2*>(hist + (size_t)blockIdx.x * kRadix)[tid];
    const uint32_t e = seg[segment] + block_exclusive(c.x + c.y, wsum);
    first.x = e + h.x;
    first.y = e + c.x + h.y;
    __syncthreads();
  }

  uint32_t tiles_x = 0, tiles_y = 0;   // epilogue: the tile grid of this partition's view
  if (kPass >= 2) {
    tiles_x = epi.view_info[4 * segment + 3] >> 16;
    const uint32_t nt = epi.view_info[4 * (segment + 1)] - epi.view_info[4 * segment];
    tiles_y = tiles_x ? nt / tiles_x : 0u;
  }
  uint32_t* wh = whist + warp * kPitch;   // this warp's counts, zeroed and filled by it alone
  uint32_t nkey[kItems], nval[kItems];
  auto load_tile = [&](int64_t t0) {
    const int tn = (int)((end - t0) < kTile ? (end - t0) : kTile);
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int li = warp * (kItems * 32) + i * 32 + lane;
      const bool ok = li < tn;
      nkey[i] = ok ? keys_in[t0 + li] : 0u;
      nval[i] = ok ? (kPass ? vals_in[t0 + li] : (uint32_t)(t0 + li)) : 0u;
    }
  };
  load_tile(beg);
  for (int64_t t0 = beg; t0 < end; t0 += kTile) {
    const int tile_n = (int)((end - t0) < kTile ? (end - t0) : kTile);
    uint32_t key[kItems], val[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      key[i] = nkey[i];
      val[i] = nval[i];
    }
    if (t0 + kTile < end) load_tile(t0 + kTile);   // in flight while this tile is ranked and scattered
    for (int i = lane; i < kPitch; i += 32) wh[i] = 0;
    __syncwarp();
    uint16_t rank[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int li = warp * (kItems * 32) + i * 32 + lane;
      const bool ok = li < tile_n;
      const uint32_t d = ok ? digit_of<kPass>(key[i], kbase) : (uint32_t)kRadix;
      // lanes holding the same digit: intersect the digit's bit ballots (and validity)
      uint32_t peers = __ballot_sync(0xffffffffu, ok);
      if (!ok) peers = ~peers;
#pragma unroll
      for (int b = 0; b < (kPass == 3 ? 32 - 3 * kBits : kBits); ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t bb = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? bb : ~bb;
      }
      const uint32_t before = wh[d];
      rank[i] = (uint16_t)(before + __popc(peers & lt_mask));
      __syncwarp();
      if ((peers & lt_mask) == 0 && ok) wh[d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // the warps' exclusive offsets per digit in place, first positions of the digits
    {
      uint2 run = make_uint2(0u, 0u);
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        uint2* q = reinterpret_cast<uint2*>(whist + w * kPitch) + tid;
        const uint2 c = *q;
        *q = run;
        run.x += c.x;
        run.y += c.y;
      }
      const uint32_t e = block_exclusive(run.x + run.y, wsum);
      reinterpret_cast<uint2*>(start)[tid] = make_uint2(e, e + run.x);
      reinterpret_cast<uint2*>(base)[tid] = make_uint2(first.x - e, first.y - e - run.x);
      first.x += run.x;
      first.y += run.y;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int li = warp * (kItems * 32) + i * 32 + lane;
      if (li < tile_n) {
        const uint32_t d = digit_of<kPass>(key[i], kbase);
        const uint32_t pos = start[d] + wh[d] + rank[i];
        s_keys[pos] = key[i];
        s_vals[pos] = val[i];
      }
    }
    __syncthreads();
    if (kPass < 2 || !last) {
#pragma unroll
      for (int it = 0; it < kItems; ++it) {
        const int j = tid + it * kBlock;
        if (j >= tile_n) break;
        const uint32_t k = s_keys[j];
        const uint32_t at = base[digit_of<kPass>(k, kbase)] + (uint32_t)j;
        vals_out[at] = s_vals[j];
        keys_out[at] = k;
      }
    } else {
      // kG rectangle gathers of a thread at a time, so that they are in flight together
      // (the stores below go to other arrays, but the compiler cannot know that)
#pragma unroll
      for (int i0 = 0; i0 < kItems; i0 += kG) {
        ushort4 rcs[kG];
#pragma unroll
        for (int it = 0; it < kG; ++it) {
          const int j = tid + (i0 + it) * kBlock;
          rcs[it] = j < tile_n ? epi.rect[s_vals[j]] : make_ushort4(0, 0, 0, 0);
        }
#pragma unroll
        for (int it = 0; it < kG; ++it) {
          const int j = tid + (i0 + it) * kBlock;
          if (j >= tile_n) break;
          const uint32_t at = base[digit_of<kPass>(s_keys[j], kbase)] + (uint32_t)j;
          vals_out[at] = s_vals[j];
          ushort4 rc = rcs[it];
          uint32_t c = 0;
          if (rc.x < rc.z && rc.y < rc.w) {
            if (rc.z <= tiles_x && rc.w <= tiles_y) c = (uint32_t)(rc.z - rc.x) * (uint32_t)(rc.w - rc.y);
            else atomicOr(epi.status, (uint32_t)GS_FLAG_BAD_RECORDS);
          }
          if (c == 0) rc = make_ushort4(0, 0, 0, 0);
          epi.out_rect[at] = rc;
          epi.out_cnt[at] = c;
        }
      }
    }
    __syncthreads();   // the next tile overwrites the staged keys, the bases and the counts
  }
}

constexpr size_t down_smem(int items) {
  return sizeof(uint32_t) * (2 * kBlock * items + kWarps * kPitch + 2 * kRadix + kWarps);
}

struct SortArgs {
  const uint32_t* seg;
  int n_seg, g;
  bool each;   // k_scan_hist_each
  uint32_t *pmap, *ctl, *hist, *tot;
  cudaStream_t st;
};

template <int kPass, int kItems>
cudaError_t sort_pass(const SortArgs& a, const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out,
                      uint32_t* vals_out, const SortRectEpilogue& epi) {
  const cudaError_t e = allow_smem<k_downsweep<kPass, kItems>>(down_smem(kItems));
  if (e != cudaSuccess) return e;
  launch(k_upsweep<kPass>, a.g, kBlock, 0, a.st, keys_in, a.seg, a.n_seg, a.pmap, a.ctl, a.hist);
  if (a.each)
    launch(k_scan_hist_each<kPass>, a.n_seg, kRadix, 0, a.st, a.hist, a.g, a.pmap, a.ctl, a.tot);
  else
    launch(k_scan_hist<kPass>, dim3(a.n_seg, kRadix / 32), 1024, 0, a.st, a.hist, a.g, a.pmap, a.ctl, a.tot);
  launch(k_downsweep<kPass, kItems>, a.g, kBlock, down_smem(kItems), a.st, keys_in, vals_in, a.seg, a.n_seg, a.pmap,
         a.ctl, keys_out, vals_out, a.hist, a.tot, epi);
  return cudaSuccess;
}

template <int kItems>
cudaError_t sort_passes(const SortArgs& a, const uint32_t* keys, const SortBufs& b, const SortRectEpilogue& epi) {
  cudaError_t e = sort_pass<0, kItems>(a, keys, nullptr, b.keys_b, b.vals_b, epi);
  if (e == cudaSuccess) e = sort_pass<1, kItems>(a, b.keys_b, b.vals_b, b.keys_a, b.vals_a, epi);
  if (e == cudaSuccess) e = sort_pass<2, kItems>(a, b.keys_a, b.vals_a, b.keys_b, b.vals_b, epi);
  if (e == cudaSuccess) e = sort_pass<3, kItems>(a, b.keys_b, b.vals_b, b.keys_a, b.vals_a, epi);
  return e;
}

}  // namespace

size_t record_sort_temp_bytes(int64_t n_cap, int n_seg) {
  const int64_t g = parts_for(n_cap, n_seg) + n_seg;
  return align_up(sizeof(uint32_t) * kRadix * g, 256) + align_up(sizeof(uint32_t) * kRadix * n_seg, 256) +
         align_up(sizeof(uint32_t) * (n_seg + 2), 256);
}

cudaError_t record_sort(const uint32_t* keys, SortBufs b, const uint32_t* n_dev, int64_t n_cap, const uint32_t* seg,
                        int n_seg, const SortRectEpilogue& epi, uint32_t* ctl, void* temp, cudaStream_t st,
                        SortedRecords* out) {
  SortArgs a;
  a.seg = seg;
  a.n_seg = n_seg;
  a.g = (int)(parts_for(n_cap, n_seg) + n_seg);
  a.each = n_seg >= kEachSegs && parts_for(n_cap, n_seg) / n_seg <= kEachParts;
  Carver c(temp);
  a.hist = c.take<uint32_t>((size_t)kRadix * a.g);
  a.tot = c.take<uint32_t>((size_t)kRadix * n_seg);
  a.pmap = c.take<uint32_t>(n_seg + 2);
  a.ctl = ctl;
  a.st = st;
  launch(k_part_map, 1, 1024, 0, st, seg, n_seg, n_dev, n_cap, a.g, tile_keys(n_cap, n_seg), a.pmap, ctl);
  const cudaError_t e = small_sort(n_cap, n_seg) ? sort_passes<kItemsSmall>(a, keys, b, epi) : sort_passes<kItemsLarge>(a, keys, b, epi);
  if (e != cudaSuccess) return e;
  *out = SortedRecords{b.vals_b, b.vals_a, ctl};
  return cudaGetLastError();
}

}  // namespace gs
