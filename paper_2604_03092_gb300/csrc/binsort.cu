// Tile binning and the device radix sorts.
//
// Binning (splat2d_bin_sort): every visible (view, surfel) record stands for
// one instance per tile of its tile rect, with key = (global tile) << 32 |
// FP32 depth bits and value = surfel index; the instances are ordered by key
// with ties in ascending surfel index (= record order within a view), i.e.
// exactly a stable sort of the keys in record order.  It is done as a radix
// sort whose most significant digit is the whole tile index (count, scan,
// scatter into per-tile buckets) followed by a least-significant-digit radix
// sort of each bucket's depth bits in shared memory.
//
// splat2d_sort_pairs: a general stable LSD radix sort of (u64 key, u32 value)
// pairs with 8-bit digits over the key bits in use.  Each pass is upsweep
// (per-block digit histograms) -> scan of the histograms -> downsweep (stable
// ranking of each 2048-key tile with warp-level match, then scatter); blocks
// own contiguous, ordered slices, so equal keys keep their input order.
#include <cuda_runtime.h>

#include "splat2d_internal.cuh"

namespace s2d {

// ---------------------------------------------------------------------------
// Binning by tile: count -> scan -> scatter -> per-tile sort
//
// The first radix digit of the (tile, depth) key is the whole tile index: a
// counting pass gives each tile's instance count (warp-aggregated atomics:
// neighbouring surfels of a keyframe land in the same tiles), an exclusive
// scan gives each tile's [start, end) range directly, and a scatter pass
// drops every instance into its tile's bucket as a 64-bit composite
// (depth bits << 32 | surfel index).  Then each tile's bucket is sorted on
// its own by an LSD radix sort of the depth bits in shared memory (in global
// memory for the rare buckets too large for shared memory), and equal depth
// bits are put in ascending surfel index.  The result is the (tile, depth)
// order with ties in surfel order -- the stable sort of the instance keys.
// ---------------------------------------------------------------------------
struct TileBinArgs {
  const uint4* bins;  // per record: depth bits, rect x0 | y0 << 16, rect x1 | y1 << 16, tile count

  const DView* views;
  int32_t V;
  int64_t R;
  int32_t tile_w_log2, tile_h_log2;
  uint32_t* counts;   // per tile: instances (count pass) / next free bucket slot (scatter, from the scan)
  unsigned long long* bucket;
  int64_t cap;        // instance capacity (bucket length)
  Header* hdr;
  // scatter pass: the tiles' size classes and work-order bins
  const uint2* ranges;
  int64_t T;
  uint32_t* class_list;   // [SORT_CLASSES][T]
  uint32_t* class_count;  // [SORT_CLASSES]
  uint32_t* order_count;  // [ORDER_BINS]
};

// Size classes of the per-tile bucket sorts (upper bounds, inclusive; longer
// buckets go with the last class).
constexpr int SORT_CLASSES = 6;
constexpr int SORT_CLASS_BOUND[SORT_CLASSES] = {256, 2048, 4096, 6144, 8192, 12288};

__device__ __forceinline__ int sort_class(uint32_t n) {
  static_assert(SORT_CLASSES == 6, "one comparison per class bound");
  constexpr uint32_t b0 = SORT_CLASS_BOUND[0], b1 = SORT_CLASS_BOUND[1], b2 = SORT_CLASS_BOUND[2],
                     b3 = SORT_CLASS_BOUND[3], b4 = SORT_CLASS_BOUND[4];
  return n == 0 ? -1
                : (n <= b0 ? 0 : (n <= b1 ? 1 : (n <= b2 ? 2 : (n <= b3 ? 3 : (n <= b4 ? 4 : 5)))));
}

// Work-order bin of a list of n entries: floor(log2(n)) + 1, longest first.
__device__ __forceinline__ int order_bin(uint32_t n) { return ORDER_BINS - 1 - (n ? 32 - __clz(n) : 0); }

// Lanes of the warp that hold the same small value; `leader` is the first.
__device__ __forceinline__ uint32_t same_value(int x, bool in, int& leader) {
  const uint32_t m = __match_any_sync(0xffffffffu, in ? x : -1);
  leader = __ffs(m) - 1;
  return m;
}

// Appends every non-empty tile to its size class's list and counts the work
// order's bins, a warp's tiles with one atomic per class and bin.  Runs ahead
// of the scatter, over the whole grid (in the one-block scan these appends
// were most of its time: 166 K tiles 260 us).
__device__ void classify_tiles(const uint2* __restrict__ ranges, int64_t T, uint32_t* __restrict__ class_list,
                               uint32_t* __restrict__ class_count, uint32_t* __restrict__ order_count) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < T; i0 += stride) {
    const int64_t i = i0 + lane;
    const uint2 r = i < T ? ranges[i] : make_uint2(0u, 0u);
    const int cls = sort_class(r.y - r.x);
    int lead;
    const uint32_t mb = same_value(order_bin(r.y - r.x), i < T, lead);
    if (i < T && lane == lead) atomicAdd(order_count + order_bin(r.y - r.x), (uint32_t)__popc(mb));
    const uint32_t mc = same_value(cls, cls >= 0, lead);
    uint32_t at = 0;
    if (cls >= 0 && lane == lead) at = atomicAdd(class_count + cls, (uint32_t)__popc(mc));
    at = __shfl_sync(0xffffffffu, at, lead);
    if (cls >= 0) class_list[(size_t)cls * T + at + __popc(mc & lt_mask)] = (uint32_t)i;
  }
}

// The work order of the persistent render kernels: tiles bucketed by
// floor(log2(list length)), longest first.  Runs ahead of the first bucket sort.
__device__ void order_tiles(const uint2* __restrict__ ranges, int64_t T, const uint32_t* __restrict__ order_count,
                            uint32_t* __restrict__ order_cursor, uint32_t* __restrict__ order) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt_mask = (1u << lane) - 1u;
  static_assert(ORDER_BINS <= 64, "two bins per lane");
  // each lane: the first position of bins 2 lane and 2 lane + 1
  const uint32_t c0 = 2 * lane < ORDER_BINS ? order_count[2 * lane] : 0u,
                 c1 = 2 * lane + 1 < ORDER_BINS ? order_count[2 * lane + 1] : 0u;
  uint32_t x = c0 + c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const uint32_t first0 = x - c0 - c1, first1 = x - c1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < T; i0 += stride) {
    const int64_t i = i0 + lane;
    const uint2 r = i < T ? ranges[i] : make_uint2(0u, 0u);
    const int b = order_bin(r.y - r.x);
    int lead;
    const uint32_t m = same_value(b, i < T, lead);
    uint32_t at = 0;
    if (i < T && lane == lead) at = atomicAdd(order_cursor + b, (uint32_t)__popc(m));
    at = __shfl_sync(0xffffffffu, at, lead);
    const uint32_t f0 = __shfl_sync(0xffffffffu, first0, b >> 1), f1 = __shfl_sync(0xffffffffu, first1, b >> 1);
    if (i < T) order[((b & 1) ? f1 : f0) + at + __popc(m & lt_mask)] = (uint32_t)i;
  }
}

// Visit every (record, tile) instance: the count pass adds them up per tile,
// the scatter pass puts each record's composite (depth bits << 32 | surfel)
// into its tiles' buckets.  Warp lanes hold consecutive records (neighbouring
// pixels of a keyframe) and walk their tile rects in step, so runs of lanes
// on one tile take one atomic.
// Steps of the scatter whose cursor atomics are in flight together.
constexpr int BIN_KB = 4;

template <bool SCATTER>
__global__ void __launch_bounds__(256) k_tile_bin(const TileBinArgs A) {
  chain_release();
  chain_wait();
  if (SCATTER && step_failed(A.hdr->status)) return;
  if (SCATTER) classify_tiles(A.ranges, A.T, A.class_list, A.class_count, A.order_count);
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // this thread's records only increase: follow the owning view forward
  int v = A.R > 0 ? find_view_by_record(A.views, A.V, min64((int64_t)blockIdx.x * blockDim.x + threadIdx.x, A.R - 1))
                  : 0;
  for (int64_t r0 = (int64_t)blockIdx.x * blockDim.x; r0 < A.R; r0 += stride) {
    const int64_t r = r0 + threadIdx.x;
    // 16 contiguous bytes per record (the records themselves are 80 bytes
    // apart: reading their rects pulled most of each record from DRAM)
    const uint4 e = r < A.R ? __ldg(A.bins + r) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t nt = e.w;
    if (!__any_sync(0xffffffffu, nt != 0)) continue;
    // the rect's tiles in row-major order: t walks a row, then jumps to the
    // next row's first tile (no division per step)
    uint32_t t = 0, wrap = 0;
    int left = 0, w = 1;
    uint64_t comp = 0;
    if (nt) {
      while (v + 1 < A.V && __ldg(&A.views[v + 1].rbase) <= r) v++;
      const DView& vw = A.views[v];
      const uint32_t q0 = e.y, q1 = e.z;
      const int tx0 = (int)(q0 & 0xffffu) >> A.tile_w_log2, ty0 = (int)(q0 >> 16) >> A.tile_h_log2;
      w = ((int)(q1 & 0xffffu) >> A.tile_w_log2) - tx0 + 1;
      t = (uint32_t)(vw.tile_base + ty0 * vw.tiles_x + tx0);
      wrap = (uint32_t)(vw.tiles_x - w + 1);
      left = w;
      comp = ((uint64_t)e.x << 32) | (uint64_t)(uint32_t)(vw.soff + (r - vw.rbase));
    }
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, nt);
    auto advance = [&]() {
      t += (--left == 0) ? wrap : 1u;
      left = left == 0 ? w : left;
    };
    if (!SCATTER) {
      for (uint32_t k = 0; k < kmax; k++, advance()) {
        const bool has = k < nt;
        const TileRun tr = tile_run(has ? t : 0xffffffffu, has, lane);
        if (tr.lead) atomicAdd(A.counts + t, tr.run);
      }
    } else {
      // the cursor atomics of BIN_KB steps are issued before any of their
      // results is used, so the warp waits on one L2 round trip per batch
      for (uint32_t k0 = 0; k0 < kmax; k0 += BIN_KB) {
        uint32_t base[BIN_KB];
        int leader[BIN_KB];
#pragma unroll
        for (int j = 0; j < BIN_KB; j++) {
          base[j] = 0u;
          leader[j] = -1;
          if (k0 + j < kmax) {
            const bool has = k0 + j < nt;
            const TileRun tr = tile_run(has ? t : 0xffffffffu, has, lane);
            if (tr.lead) base[j] = atomicAdd(A.counts + t, tr.run);
            leader[j] = has ? tr.leader : -1;
            advance();
          }
        }
#pragma unroll
        for (int j = 0; j < BIN_KB; j++) {
          if (k0 + j >= kmax) break;  // uniform across the warp
          const uint32_t b = __shfl_sync(0xffffffffu, base[j], leader[j] & 31);
          if (leader[j] >= 0 && s2d_check((int64_t)b + (lane - leader[j]) < A.cap, A.hdr))
            A.bucket[b + (uint32_t)(lane - leader[j])] = comp;
        }
      }
    }
  }
}

// One block: exclusive scan of the tile counts -> ranges, scatter cursors,
// total and the capacity check.  Each thread takes SCAN_ITEMS consecutive
// tiles per sweep, so a sweep covers 8192 tiles with one block-wide scan of
// the threads' sums, the next sweep's counts already on their way.  The
// counts are left zero for the next count pass, and the binning's small
// counters (`small`) for the passes that follow.
constexpr int SCAN_ITEMS = 8;

__global__ void __launch_bounds__(1024) k_tile_scan(uint32_t* __restrict__ counts, uint32_t* __restrict__ cursors,
                                                    uint2* __restrict__ ranges, int64_t T, Header* __restrict__ hdr,
                                                    int64_t cap, uint32_t* __restrict__ small, int n_small) {
  __shared__ unsigned long long s_w[32];
  __shared__ unsigned long long s_carry;
  chain_release();
  chain_wait();
  if (threadIdx.x == 0) s_carry = 0;
  for (int i = threadIdx.x; i < n_small; i += 1024) small[i] = 0u;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t next[SCAN_ITEMS];
  // (the arrays are 256-byte aligned and a thread's tiles start at a multiple of 8)
  auto load = [&](int64_t i0) {
    if (i0 + SCAN_ITEMS <= T) {
      const uint4 a = *reinterpret_cast<const uint4*>(counts + i0), b = *reinterpret_cast<const uint4*>(counts + i0 + 4);
      next[0] = a.x; next[1] = a.y; next[2] = a.z; next[3] = a.w;
      next[4] = b.x; next[5] = b.y; next[6] = b.z; next[7] = b.w;
    } else {
#pragma unroll
      for (int j = 0; j < SCAN_ITEMS; j++) next[j] = i0 + j < T ? counts[i0 + j] : 0u;
    }
  };
  load((int64_t)threadIdx.x * SCAN_ITEMS);
  __syncthreads();
  for (int64_t base = 0; base < T; base += 1024 * SCAN_ITEMS) {
    const int64_t i0 = base + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    unsigned long long sum = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
      v[j] = next[j];
      sum += v[j];
    }
    load(i0 + 1024 * SCAN_ITEMS);
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    // every warp scans the warps' sums
    unsigned long long w = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    const unsigned long long carry = s_carry, total = __shfl_sync(0xffffffffu, w, 31);
    const unsigned long long before = __shfl_sync(0xffffffffu, w, wid > 0 ? wid - 1 : 0);
    unsigned long long incl = carry + (wid > 0 ? before : 0ull) + x - sum;
    uint2 rg[SCAN_ITEMS];
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
      const unsigned long long start = incl;
      incl += v[j];
      rg[j] = incl <= (unsigned long long)cap ? make_uint2((uint32_t)start, (uint32_t)incl) : make_uint2(0u, 0u);
    }
    if (i0 + SCAN_ITEMS <= T) {
#pragma unroll
      for (int j = 0; j < SCAN_ITEMS; j += 2)
        *reinterpret_cast<uint4*>(ranges + i0 + j) = make_uint4(rg[j].x, rg[j].y, rg[j + 1].x, rg[j + 1].y);
#pragma unroll
      for (int j = 0; j < SCAN_ITEMS; j += 4) {
        *reinterpret_cast<uint4*>(cursors + i0 + j) = make_uint4(rg[j].x, rg[j + 1].x, rg[j + 2].x, rg[j + 3].x);
        *reinterpret_cast<uint4*>(counts + i0 + j) = make_uint4(0u, 0u, 0u, 0u);
      }
    } else {
#pragma unroll
      for (int j = 0; j < SCAN_ITEMS; j++)
        if (i0 + j < T) {
          ranges[i0 + j] = rg[j];
          cursors[i0 + j] = rg[j].x;
          counts[i0 + j] = 0u;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) s_carry = carry + total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const unsigned long long total = s_carry;
    hdr->needed = total;
    if ((int64_t)total > cap) {
      hdr->status = SPLAT2D_ERR_CAPACITY;
      hdr->n_inst = 0;
    } else {
      hdr->n_inst = total;
    }
  }
}

// Number of bits needed to represent v (0 for v == 0).
__device__ __forceinline__ int bits_of(uint32_t v) { return v ? 32 - __clz(v) : 0; }

// Stable LSD radix sort of n composite keys (depth bits << 32 | surfel index)
// in place in `a` (b: scratch of the same size), 8-bit digits of
// key_of(x) = ((x >> 32) - dmin) << ishift | ((x & 0xffffffff) - imin) over
// `nbits` bits (ishift < 0: the depth part alone, key_of(x) = (x >> 32) - dmin); generic pointers (shared or global memory); ranked per warp
// with match_any so that equal digits keep their order.  `cnt` holds
// (NWARPS + 1) * 256 counters.  Returns with the result in `a`.
template <int NWARPS>
__device__ void block_radix_any(unsigned long long* a, unsigned long long* b, int n, uint32_t* cnt, uint32_t dmin,
                            uint32_t imin, int ishift, int nbits) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int per = (((n + NWARPS - 1) / NWARPS) + 31) & ~31;  // elements per warp, whole rounds
  const int lo = min(wid * per, n), hi = min(lo + per, n);
  const int passes = (nbits + 7) >> 3;
  unsigned long long* src = a;
  unsigned long long* dst = b;
  auto digit = [&](unsigned long long x, int shift) -> uint32_t {
    const unsigned long long dk = (unsigned long long)((uint32_t)(x >> 32) - dmin);
    const unsigned long long k = ishift < 0 ? dk : ((dk << ishift) | (unsigned long long)((uint32_t)x - imin));
    return (uint32_t)(k >> shift) & 0xffu;
  };
  for (int pass = 0; pass < passes; pass++) {
    const int shift = 8 * pass;
    for (int i = threadIdx.x; i < NWARPS * 256; i += NWARPS * 32) cnt[i] = 0;
    __syncthreads();
    for (int base = lo; base < hi; base += 32) {
      const int i = base + lane;
      const uint32_t d = i < hi ? digit(src[i], shift) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      if (d < 256 && lane == __ffs(peers) - 1) cnt[wid * 256 + d] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      uint32_t acc = 0;
      for (int w = 0; w < NWARPS; w++) {
        const uint32_t c = cnt[w * 256 + threadIdx.x];
        cnt[w * 256 + threadIdx.x] = acc;
        acc += c;
      }
      cnt[NWARPS * 256 + threadIdx.x] = acc;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      uint32_t v[8], sum = 0;
      for (int k = 0; k < 8; k++) {
        v[k] = cnt[NWARPS * 256 + lane * 8 + k];
        sum += v[k];
      }
      uint32_t x = sum;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      uint32_t run = x - sum;
      for (int k = 0; k < 8; k++) {
        cnt[NWARPS * 256 + lane * 8 + k] = run;
        run += v[k];
      }
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      const uint32_t dbase = cnt[NWARPS * 256 + threadIdx.x];
      for (int w = 0; w < NWARPS; w++) cnt[w * 256 + threadIdx.x] += dbase;
    }
    __syncthreads();
    for (int base = lo; base < hi; base += 32) {
      const int i = base + lane;
      const unsigned long long key = i < hi ? src[i] : 0ull;
      const uint32_t d = i < hi ? digit(key, shift) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      uint32_t pos = 0;
      if (d < 256) pos = cnt[wid * 256 + d];
      __syncwarp();
      if (d < 256) {
        if (lane == __ffs(peers) - 1) cnt[wid * 256 + d] = pos + __popc(peers);
        dst[pos + __popc(peers & lt_mask)] = key;
      }
      __syncwarp();
    }
    __syncthreads();
    unsigned long long* tmp = src;
    src = dst;
    dst = tmp;
  }
  if (src != a) {
    for (int i = threadIdx.x; i < n; i += NWARPS * 32) a[i] = src[i];
    __syncthreads();
  }
}

// Sort one tile's bucket by (depth bits, surfel index).  The depth digits are
// taken relative to the bucket's smallest depth, so only the bits that vary
// are sorted; equal depths are then put in surfel order, and a bucket with a
// long run of equal depths is sorted once more on the full composite key.
template <int NWARPS>
__device__ void sort_bucket_any(unsigned long long* a, unsigned long long* b, int n, uint32_t* cnt, uint32_t* red) {
  // red[0..3]: min depth, max depth, min index, max index; red[4]: long-run flag
  if (threadIdx.x == 0) {
    red[0] = 0xffffffffu; red[1] = 0u; red[2] = 0xffffffffu; red[3] = 0u; red[4] = 0u;
  }
  __syncthreads();
  uint32_t dmn = 0xffffffffu, dmx = 0u, imn = 0xffffffffu, imx = 0u;
  for (int i = threadIdx.x; i < n; i += NWARPS * 32) {
    const unsigned long long x = a[i];
    const uint32_t d = (uint32_t)(x >> 32), s = (uint32_t)x;
    dmn = min(dmn, d); dmx = max(dmx, d); imn = min(imn, s); imx = max(imx, s);
  }
  dmn = __reduce_min_sync(0xffffffffu, dmn);
  dmx = __reduce_max_sync(0xffffffffu, dmx);
  imn = __reduce_min_sync(0xffffffffu, imn);
  imx = __reduce_max_sync(0xffffffffu, imx);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&red[0], dmn); atomicMax(&red[1], dmx); atomicMin(&red[2], imn); atomicMax(&red[3], imx);
  }
  __syncthreads();
  const uint32_t dmin = red[0], dbits = (uint32_t)bits_of(red[1] - red[0]);
  const uint32_t imin = red[2], ibits = (uint32_t)bits_of(red[3] - red[2]);
  block_radix_any<NWARPS>(a, b, n, cnt, dmin, 0u, -1, (int)dbits);
  // equal depth bits: ascending surfel index (short runs in place)
  for (int i = threadIdx.x; i < n; i += NWARPS * 32) {
    const uint32_t d = (uint32_t)(a[i] >> 32);
    const bool starts = (i == 0 || (uint32_t)(a[i - 1] >> 32) != d) && i + 1 < n && (uint32_t)(a[i + 1] >> 32) == d;
    if (!starts) continue;
    int e = i + 1;
    while (e + 1 < n && e - i < 64 && (uint32_t)(a[e + 1] >> 32) == d) e++;
    if (e + 1 < n && (uint32_t)(a[e + 1] >> 32) == d) {
      red[4] = 1u;  // a long run: handled below
      continue;
    }
    for (int x = i + 1; x <= e; x++) {
      const unsigned long long key = a[x];
      int y = x - 1;
      while (y >= i && a[y] > key) {
        a[y + 1] = a[y];
        y--;
      }
      a[y + 1] = key;
    }
  }
  __syncthreads();
  if (red[4]) block_radix_any<NWARPS>(a, b, n, cnt, dmin, imin, (int)ibits, (int)(dbits + ibits));
}

// Shared-memory radix sort of a bucket of at most NWARPS * 32 * ITEMS
// composites, the keys of each pass held in registers.  Warp w owns a
// contiguous slice of the array; per pass it ranks its keys round by round
// (a round = 32 consecutive keys) with a ballot multisplit: eight ballots, one
// per digit bit, give each lane the mask of lanes holding its digit, so the
// rank within the round is a population count, and the round's first lane of
// each digit advances the warp's 16-bit counter of that digit.  A block scan
// of the (digit, warp) counters in digit-major order turns them into output
// offsets, so equal digits keep their order (stable), and every key is then
// stored at its offset.  Digits are those of block_radix_any.  Returns the
// buffer holding the result (a or b).  a and b may be the same buffer: a
// pass loads all its keys into registers before a block barrier and
// scatters them after it.
template <int NWARPS>
struct RegSortSmem {
  static constexpr int CP = NWARPS + 2;  // padded counter row: conflict-free leader updates
  static constexpr size_t CNT_BYTES = sizeof(uint16_t) * 256 * CP;
  static constexpr size_t BYTES = ((CNT_BYTES + 15) & ~(size_t)15) + sizeof(uint32_t) * (32 + 8);
};

template <int NWARPS, int ITEMS>
__device__ unsigned long long* block_radix_reg(unsigned long long* a, unsigned long long* b, int n, uint16_t* cnt,
                                               uint32_t* tot, uint32_t dmin, uint32_t imin, int ishift, int nbits,
                                               int lsb = 0) {
  constexpr int NT = NWARPS * 32, CP = RegSortSmem<NWARPS>::CP;
  static_assert(NWARPS % 8 == 0, "the counter scan takes 8 counters per thread");
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int per = (((n + NWARPS - 1) / NWARPS) + 31) & ~31;
  const int lo = min(wid * per, n), hi = min(lo + per, n);
  const int nr = (hi - lo + 31) >> 5;  // rounds of this warp (<= ITEMS)
  const int passes = (nbits + 7) >> 3;
  unsigned long long* src = a;
  unsigned long long* dst = b;
  auto digit = [&](unsigned long long key, int shift) -> uint32_t {
    const uint32_t dk = (uint32_t)(key >> 32) - dmin;
    if (ishift < 0) return (dk >> (shift + lsb)) & 0xffu;  // the depth part: no 64-bit shifts
    const unsigned long long kk = ((unsigned long long)dk << ishift) | (unsigned long long)((uint32_t)key - imin);
    return (uint32_t)(kk >> (shift + lsb)) & 0xffu;
  };
  int first = 0;
  if (passes > 0) {
    // The first pass may leave equal digits in any order (the order it starts
    // from is arbitrary anyway): each key takes its slot within its digit from
    // one shared atomic on a 256-bin histogram, and only the 256 bins are
    // scanned.  The later passes keep the order of equal digits (below).
    uint32_t* hist = reinterpret_cast<uint32_t*>(cnt);  // 256 words of the counter space
    unsigned long long key[ITEMS];
    uint32_t off[ITEMS];
    for (int i = threadIdx.x; i < 256; i += NT) hist[i] = 0u;
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
      const int i = lo + k * 32 + lane;
      key[k] = (k < nr && i < hi) ? src[i] : 0ull;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
      if (k < nr && lo + k * 32 + lane < hi) {
        const uint32_t d = digit(key[k], 0);
        off[k] = (d << 16) | atomicAdd(&hist[d], 1u);
      }
    }
    __syncthreads();
    uint32_t v = 0, x = 0;
    if (threadIdx.x < 256) {
      v = hist[threadIdx.x];
      x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) tot[wid] = x;
    }
    __syncthreads();
    if (threadIdx.x < 256) {
      uint32_t before = 0;
      for (int w = 0; w < wid; w++) before += tot[w];
      hist[threadIdx.x] = before + x - v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; k++)
      if (k < nr && lo + k * 32 + lane < hi) dst[hist[off[k] >> 16] + (off[k] & 0xffffu)] = key[k];
    __syncthreads();
    unsigned long long* t = src;
    src = dst;
    dst = t;
    first = 1;
  }
  for (int pass = first; pass < passes; pass++) {
    const int shift = 8 * pass;
    unsigned long long key[ITEMS];
    uint32_t off[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
      const int i = lo + k * 32 + lane;
      key[k] = (k < nr && i < hi) ? src[i] : 0ull;
    }
    for (int i = threadIdx.x; i < 256 * CP / 2; i += NT) reinterpret_cast<uint32_t*>(cnt)[i] = 0u;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
      if (k < nr) {
        const bool valid = lo + k * 32 + lane < hi;
        const uint32_t d = valid ? digit(key[k], shift) : 0u;
        uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int bit = 0; bit < 8; bit++) {
          const bool on = (d >> bit) & 1u;
          const uint32_t bal = __ballot_sync(0xffffffffu, on);
          peers &= on ? bal : ~bal;
        }
        const int leader = __ffs(peers) - 1;
        uint32_t pre = 0;
        if (valid && lane == leader) {
          pre = cnt[d * CP + wid];
          cnt[d * CP + wid] = (uint16_t)(pre + __popc(peers));
        }
        pre = __shfl_sync(0xffffffffu, pre, leader & 31);
        off[k] = (d << 16) | (pre + __popc(peers & lt_mask));
        __syncwarp();
      }
    }
    __syncthreads();
    {
      // exclusive scan of the counters in (digit, warp) order, 8 per thread
      const int f0 = 8 * threadIdx.x, d = f0 / NWARPS, w0 = f0 % NWARPS;
      uint32_t c[8], sum = 0;
#pragma unroll
      for (int j = 0; j < 8; j++) {
        c[j] = cnt[d * CP + w0 + j];
        sum += c[j];
      }
      uint32_t x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) tot[wid] = x;
      __syncthreads();
      if (wid == 0) {
        uint32_t y = lane < NWARPS ? tot[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
          if (lane >= o) y += z;
        }
        if (lane < NWARPS) tot[lane] = y;
      }
      __syncthreads();
      uint32_t ex = x - sum + (wid > 0 ? tot[wid - 1] : 0u);
#pragma unroll
      for (int j = 0; j < 8; j++) {
        cnt[d * CP + w0 + j] = (uint16_t)ex;
        ex += c[j];
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
      if (k < nr && lo + k * 32 + lane < hi) {
        const uint32_t d = off[k] >> 16;
        dst[(uint32_t)cnt[d * CP + wid] + (off[k] & 0xffffu)] = key[k];
      }
    }
    __syncthreads();
    unsigned long long* t = src;
    src = dst;
    dst = t;
  }
  return src;
}

// Sort a bucket of at most NWARPS * 32 * ITEMS composites by (depth bits,
// surfel index) and write it out as (tile | depth bits) keys and surfel
// values: load it from global memory into shared memory (finding the
// bucket's depth and index ranges on the way), radix-sort the top 16 bits of
// the depth relative to the smallest depth (two passes where the depths span
// more), then write every entry out at its place: an entry that ties with no
// neighbour on those bits at its sorted position, an entry of a run of ties
// at the run's start plus the number of the run's composites below its own
// (the composites are distinct), so every run is put in (depth, surfel)
// order in parallel.  A run longer than 64 triggers one exact re-sort on the
// relative composite key instead, whose result is written over.
template <int NWARPS, int ITEMS>
__device__ void sort_bucket_reg(const unsigned long long* __restrict__ g, int n, unsigned long long* sa,
                                unsigned long long* sb, uint16_t* cnt, uint32_t* tot, uint32_t* red,
                                uint64_t tile, uint64_t* __restrict__ okeys, uint32_t* __restrict__ ovals) {
  constexpr int NT = NWARPS * 32;
  if (threadIdx.x == 0) {
    red[0] = 0xffffffffu; red[1] = 0u; red[2] = 0xffffffffu; red[3] = 0u; red[4] = 0u;
  }
  __syncthreads();
  uint32_t dmn = 0xffffffffu, dmx = 0u, imn = 0xffffffffu, imx = 0u;
  for (int i = threadIdx.x; i < n; i += NT) {
    const unsigned long long x = __ldcg(g + i);
    sa[i] = x;
    const uint32_t d = (uint32_t)(x >> 32), s = (uint32_t)x;
    dmn = min(dmn, d); dmx = max(dmx, d); imn = min(imn, s); imx = max(imx, s);
  }
  dmn = __reduce_min_sync(0xffffffffu, dmn);
  dmx = __reduce_max_sync(0xffffffffu, dmx);
  imn = __reduce_min_sync(0xffffffffu, imn);
  imx = __reduce_max_sync(0xffffffffu, imx);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&red[0], dmn); atomicMax(&red[1], dmx); atomicMin(&red[2], imn); atomicMax(&red[3], imx);
  }
  __syncthreads();
  const uint32_t dmin = red[0], dbits = (uint32_t)bits_of(red[1] - red[0]);
  const uint32_t imin = red[2], ibits = (uint32_t)bits_of(red[3] - red[2]);
  // radix passes over the top 16 bits of the relative depth only; entries
  // that tie there form runs, put in (depth, surfel) order as they are
  // written out below
  const int lsb = max((int)dbits - 16, 0);
  unsigned long long* r = block_radix_reg<NWARPS, ITEMS>(sa, sb, n, cnt, tot, dmin, 0u, -1, (int)dbits - lsb, lsb);
  const int lane = threadIdx.x & 31;
  auto top = [&](unsigned long long x) -> uint32_t { return ((uint32_t)(x >> 32) - dmin) >> lsb; };
  auto emit = [&](int p, unsigned long long key) {
    okeys[p] = tile | (key >> 32);
    ovals[p] = (uint32_t)key;
  };
  for (int i0 = 0; i0 < n; i0 += NT) {
    const int i = i0 + threadIdx.x;
    const bool in = i < n;
    const unsigned long long key = in ? r[i] : 0ull;
    const uint32_t d = top(key);
    // the neighbours' top bits: the adjacent lanes' entries, across warps a load
    uint32_t dp = __shfl_up_sync(0xffffffffu, d, 1), dn = __shfl_down_sync(0xffffffffu, d, 1);
    if (lane == 0 && in && i > 0) dp = top(r[i - 1]);
    if (lane == 31 && i + 1 < n) dn = top(r[i + 1]);
    if (!in) continue;
    if (!((i > 0 && dp == d) || (i + 1 < n && dn == d))) {
      emit(i, key);
      continue;
    }
    int s = i, e = i;
    while (s > 0 && i - s < 64 && top(r[s - 1]) == d) s--;
    while (e + 1 < n && e - i < 64 && top(r[e + 1]) == d) e++;
    if (e - s >= 64) {
      red[4] = 1u;
      continue;
    }
    int rank = 0;
    for (int y = s; y <= e; y++) rank += r[y] < key ? 1 : 0;
    emit(s + rank, key);
  }
  __syncthreads();
  if (red[4]) {
    const unsigned long long* x =
        block_radix_reg<NWARPS, ITEMS>(r, r == sa ? sb : sa, n, cnt, tot, dmin, imin, (int)ibits, (int)(dbits + ibits));
    for (int i = threadIdx.x; i < n; i += NT) emit(i, x[i]);
  }
}

// Per-tile bucket sorts in size classes, each a persistent launch over its
// class's tile list with shared memory sized for the class (so short buckets
// run several CTAs per SM); the last class also takes the buckets longer than
// its capacity and sorts those in global memory.
struct SegArgs {
  const uint2* ranges;
  unsigned long long* bucket;   // scattered composites (sorted in place for the oversized buckets)
  unsigned long long* scratch;  // ping-pong space for the oversized buckets (same indexing as bucket)
  uint64_t* keys;               // out: (tile << 32) | depth bits
  uint32_t* vals;               // out: surfel index
  Header* hdr;
  int64_t cap;                  // instance capacity
  const uint32_t* list;         // this class's tiles
  const uint32_t* list_count;   // their number
  uint32_t* queue;              // this class's work counter
  // first class: the work order of the render kernels
  int64_t T;
  const uint32_t* order_count;
  uint32_t* order_cursor;
  uint32_t* order;
};

// Short buckets (at most 32 * WS_ITEMS composites): one warp each, no block
// barriers (six CTAs per SM; at 9 warps per SM, without the register bound,
// latency-bound: 269 against 201 us for one keyframe x 8 views, preprocess and
// binning).  The same two radix passes as sort_bucket_reg: the keys go from
// global memory to registers, the first pass ranks them by shared atomics, the
// second (stable) by ballot multisplit against one counter per digit, each
// scan of the 256 counters taking 8 per lane.  Runs of ties are ranked in
// parallel as the bucket is written out; a run longer than 64 takes stable
// passes over the whole relative composite instead.  A 256-thread CTA per
// bucket spent most of a short one at its barriers: buckets of about 150
// entries (12 uneven submaps, 166 K tiles) 785 us.
constexpr int WS_ITEMS = 8;
constexpr int WS_WARPS = 4;  // buckets (warps) per CTA; they share nothing
struct WarpSortSmem {
  unsigned long long key[32 * WS_ITEMS];
  uint32_t cnt[256];
};

__device__ __forceinline__ void warp_scan256(uint32_t* cnt, int lane) {
  uint4 a = reinterpret_cast<uint4*>(cnt)[2 * lane], b = reinterpret_cast<uint4*>(cnt)[2 * lane + 1];
  const uint32_t sum = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
  uint32_t x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  uint32_t run = x - sum, t;
  t = a.x; a.x = run; run += t;
  t = a.y; a.y = run; run += t;
  t = a.z; a.z = run; run += t;
  t = a.w; a.w = run; run += t;
  t = b.x; b.x = run; run += t;
  t = b.y; b.y = run; run += t;
  t = b.z; b.z = run; run += t;
  b.w = run;
  reinterpret_cast<uint4*>(cnt)[2 * lane] = a;
  reinterpret_cast<uint4*>(cnt)[2 * lane + 1] = b;
  __syncwarp();
}

__device__ __forceinline__ void warp_clear256(uint32_t* cnt, int lane) {
  reinterpret_cast<uint4*>(cnt)[2 * lane] = make_uint4(0u, 0u, 0u, 0u);
  reinterpret_cast<uint4*>(cnt)[2 * lane + 1] = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
}

// One stable pass by the digit (composite's sort key >> shift) & 255 over S.key.
template <typename KeyOf>
__device__ __forceinline__ void warp_pass_stable(WarpSortSmem& S, int n, int shift, int lane, const KeyOf& key_of) {
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int nr = (n + 31) >> 5;
  unsigned long long key[WS_ITEMS];
  uint32_t off[WS_ITEMS];
  warp_clear256(S.cnt, lane);
#pragma unroll
  for (int k = 0; k < WS_ITEMS; k++) {
    if (k >= nr) break;
    const bool valid = k * 32 + lane < n;
    key[k] = valid ? S.key[k * 32 + lane] : 0ull;
    const uint32_t d = valid ? (uint32_t)(key_of(key[k]) >> shift) & 0xffu : 0u;
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int bit = 0; bit < 8; bit++) {
      const bool on = (d >> bit) & 1u;
      const uint32_t bal = __ballot_sync(0xffffffffu, on);
      peers &= on ? bal : ~bal;
    }
    const int leader = __ffs(peers) - 1;
    uint32_t pre = 0;
    if (valid && lane == leader) {
      pre = S.cnt[d];
      S.cnt[d] = pre + __popc(peers);
    }
    pre = __shfl_sync(0xffffffffu, pre, leader & 31);
    off[k] = (d << 16) | (pre + __popc(peers & lt_mask));
    __syncwarp();
  }
  warp_scan256(S.cnt, lane);
#pragma unroll
  for (int k = 0; k < WS_ITEMS; k++)
    if (k < nr && k * 32 + lane < n) S.key[S.cnt[off[k] >> 16] + (off[k] & 0xffffu)] = key[k];
  __syncwarp();
}

__device__ void warp_sort_bucket(const unsigned long long* __restrict__ g, int n, WarpSortSmem& S, int lane,
                                 uint64_t tile, uint64_t* __restrict__ okeys, uint32_t* __restrict__ ovals) {
  const int nr = (n + 31) >> 5;
  uint32_t dmin, dbits;
  int lsb;
  {
    unsigned long long key[WS_ITEMS];
    uint32_t dmn = 0xffffffffu, dmx = 0u;
#pragma unroll
    for (int k = 0; k < WS_ITEMS; k++)
      if (k < nr) key[k] = k * 32 + lane < n ? __ldg(g + k * 32 + lane) : 0ull;
    warp_clear256(S.cnt, lane);
#pragma unroll
    for (int k = 0; k < WS_ITEMS; k++)
      if (k < nr && k * 32 + lane < n) {
        const uint32_t d = (uint32_t)(key[k] >> 32);
        dmn = min(dmn, d);
        dmx = max(dmx, d);
      }
    dmin = __reduce_min_sync(0xffffffffu, dmn);
    dbits = (uint32_t)bits_of(__reduce_max_sync(0xffffffffu, dmx) - dmin);
    lsb = max((int)dbits - 16, 0);
    // first pass (the order of equal digits is free)
    uint32_t off[WS_ITEMS];
#pragma unroll
    for (int k = 0; k < WS_ITEMS; k++)
      if (k < nr && k * 32 + lane < n) {
        const uint32_t d = (((uint32_t)(key[k] >> 32) - dmin) >> lsb) & 0xffu;
        off[k] = (d << 16) | atomicAdd(&S.cnt[d], 1u);
      }
    __syncwarp();
    warp_scan256(S.cnt, lane);
#pragma unroll
    for (int k = 0; k < WS_ITEMS; k++)
      if (k < nr && k * 32 + lane < n) S.key[S.cnt[off[k] >> 16] + (off[k] & 0xffffu)] = key[k];
    __syncwarp();
  }
  if ((int)dbits - lsb > 8)
    warp_pass_stable(S, n, 8, lane, [&](unsigned long long x) { return ((uint32_t)(x >> 32) - dmin) >> lsb; });
  auto top = [&](unsigned long long x) -> uint32_t { return ((uint32_t)(x >> 32) - dmin) >> lsb; };
  auto emit = [&](int p, unsigned long long key) {
    okeys[p] = tile | (key >> 32);
    ovals[p] = (uint32_t)key;
  };
  bool long_run = false;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const bool in = i < n;
    const unsigned long long key = in ? S.key[i] : 0ull;
    const uint32_t d = top(key);
    // the neighbours' top bits: the adjacent lanes' entries, across rounds a load
    uint32_t dp = __shfl_up_sync(0xffffffffu, d, 1), dn = __shfl_down_sync(0xffffffffu, d, 1);
    if (lane == 0 && in && i > 0) dp = top(S.key[i - 1]);
    if (lane == 31 && i + 1 < n) dn = top(S.key[i + 1]);
    if (!in) continue;
    if (!((i > 0 && dp == d) || (i + 1 < n && dn == d))) {
      emit(i, key);
      continue;
    }
    int s = i, e = i;
    while (s > 0 && i - s < 64 && top(S.key[s - 1]) == d) s--;
    while (e + 1 < n && e - i < 64 && top(S.key[e + 1]) == d) e++;
    if (e - s >= 64) {
      long_run = true;
      continue;
    }
    int rank = 0;
    for (int y = s; y <= e; y++) rank += S.key[y] < key ? 1 : 0;
    emit(s + rank, key);
  }
  if (__any_sync(0xffffffffu, long_run)) {
    uint32_t imn = 0xffffffffu, imx = 0u;
    for (int i = lane; i < n; i += 32) {
      imn = min(imn, (uint32_t)S.key[i]);
      imx = max(imx, (uint32_t)S.key[i]);
    }
    const uint32_t imin = __reduce_min_sync(0xffffffffu, imn);
    const int ibits = bits_of(__reduce_max_sync(0xffffffffu, imx) - imin);
    for (int shift = 0; shift < (int)dbits + ibits; shift += 8)
      warp_pass_stable(S, n, shift, lane, [&](unsigned long long x) {
        return (unsigned long long)((uint32_t)(x >> 32) - dmin) << ibits | (unsigned long long)((uint32_t)x - imin);
      });
    for (int i = lane; i < n; i += 32) emit(i, S.key[i]);
  }
}

__global__ void __launch_bounds__(WS_WARPS * 32, 6) k_tile_sort_warp(const SegArgs A) {
  __shared__ __align__(16) WarpSortSmem s_sort[WS_WARPS];
  chain_wait();
  chain_release();  // after the wait: the next class starts without one (see k_tile_sort)
  if (step_failed(A.hdr->status)) return;
  order_tiles(A.ranges, A.T, A.order_count, A.order_cursor, A.order);
  const int lane = threadIdx.x & 31;
  WarpSortSmem& S = s_sort[threadIdx.x >> 5];
  const uint32_t n_tiles = *A.list_count;
  // buckets of one class are alike, so the warps take them in turn, and know
  // the next one's place while they sort this one
  const uint32_t step = gridDim.x * WS_WARPS;
  uint32_t q = blockIdx.x * WS_WARPS + (threadIdx.x >> 5);
  uint32_t t_next = q < n_tiles ? A.list[q] : 0u;
  uint2 r_next = q < n_tiles ? A.ranges[t_next] : make_uint2(0u, 0u);
  for (; q < n_tiles; q += step) {
    const uint32_t t = t_next;
    const uint2 rg = r_next;
    if (q + step < n_tiles) {
      t_next = A.list[q + step];
      r_next = A.ranges[t_next];
    }
    if (!s2d_check(rg.x <= rg.y && (int64_t)rg.y <= A.cap && rg.y - rg.x <= 32 * WS_ITEMS, A.hdr)) continue;
    warp_sort_bucket(A.bucket + rg.x, (int)(rg.y - rg.x), S, lane, (uint64_t)t << 32, A.keys + rg.x, A.vals + rg.x);
    __syncwarp();
  }
}

template <int NWARPS, int ITEMS>
struct SegClass {
  static constexpr int THREADS = NWARPS * 32;
  static constexpr int CAP = NWARPS * 32 * ITEMS;
  static constexpr size_t SMEM = sizeof(unsigned long long) * CAP + RegSortSmem<NWARPS>::BYTES;
};

template <int NWARPS, int ITEMS, bool LAST>
// The bucket is sorted in place in one shared buffer (each radix pass holds
// its keys in registers between its loads and its scatter, with block
// barriers in between).  Bound by issue and by the barriers, so more CTAs per
// SM pay even where their keys spill: the 257..2048 class (256 threads, 21 KB
// of shared memory) runs 8 with 32 registers a thread, the 2049..4096 class (512
// threads, 41 KB) 4 with 32, and the 4097..6144 and 6145..8192 classes (57 and
// 73 KB) 3 with 40, which their shared memory allows (with 32 as well: 24 x 24
// 5556 us).  Against 6 and 3 CTAs, and digits by 64-bit shifts: binning 840 ->
// 785 us (8 keyframes x 8 views), 5734 -> 5538 (24 x 24), 731 -> 724 (12 uneven
// submaps); 5 or 4 CTAs of the first class 861, 868.
__global__ void __launch_bounds__(NWARPS * 32, NWARPS == 16 ? (ITEMS == 8 ? 4 : 3) : (NWARPS == 8 ? 8 : 1)) k_tile_sort(const SegArgs A) {
  using C = SegClass<NWARPS, ITEMS>;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* sa = reinterpret_cast<unsigned long long*>(smem);
  unsigned long long* sb = sa;  // in place: every pass holds its keys in registers
  static_assert(!LAST || sizeof(unsigned long long) * C::CAP >= sizeof(uint32_t) * ((NWARPS + 1) * 256 + 8),
                "the oversized-bucket counters fit in the key buffer");
  uint16_t* cnt = reinterpret_cast<uint16_t*>(sa + C::CAP);
  uint32_t* tot = reinterpret_cast<uint32_t*>(smem + sizeof(unsigned long long) * C::CAP +
                                              ((RegSortSmem<NWARPS>::CNT_BYTES + 15) & ~(size_t)15));
  uint32_t* red = tot + 32;
  __shared__ uint32_t s_q;
  // The classes sort disjoint buckets, so a class runs beside the one before
  // it (8 keyframes x 8 views: 1215 -> 1150 us for preprocess and binning):
  // the scatter pass they depend on was complete before the first class let
  // them start, and the wait for the class before comes last.  Until then
  // what the scatter wrote is read through L2.
  chain_release();
  const uint32_t n_tiles = step_failed(__ldcg(&A.hdr->status)) ? 0u : __ldcg(A.list_count);
  for (;;) {
    if (threadIdx.x == 0) s_q = atomicAdd(A.queue, 1u);
    __syncthreads();
    const uint32_t q = s_q;
    __syncthreads();
    if (q >= n_tiles) break;
    const uint32_t t = __ldcg(A.list + q);
    const uint2 rg = __ldcg(A.ranges + t);
    if (!s2d_check(rg.x <= rg.y && (int64_t)rg.y <= A.cap, A.hdr)) continue;
    const int n = (int)(rg.y - rg.x);
    const uint64_t tile = (uint64_t)t << 32;
    if (!LAST || n <= C::CAP) {
      sort_bucket_reg<NWARPS, ITEMS>(A.bucket + rg.x, n, sa, sb, cnt, tot, red, tile, A.keys + rg.x, A.vals + rg.x);
    } else {
      uint32_t* c32 = reinterpret_cast<uint32_t*>(smem);
      chain_wait();
      sort_bucket_any<NWARPS>(A.bucket + rg.x, A.scratch + rg.x, n, c32, c32 + (NWARPS + 1) * 256);
      const unsigned long long* res = A.bucket + rg.x;
      for (int i = threadIdx.x; i < n; i += NWARPS * 32) {
        const unsigned long long key = res[i];
        A.keys[rg.x + i] = tile | (key >> 32);
        A.vals[rg.x + i] = (uint32_t)key;
      }
    }
    __syncthreads();
  }
  chain_wait();
}

template <int NWARPS, int ITEMS, bool LAST>
static cudaError_t launch_tile_sort_class(const SegArgs& S, cudaStream_t st) {
  using C = SegClass<NWARPS, ITEMS>;
  auto k = k_tile_sort<NWARPS, ITEMS, LAST>;
  static PerDevice resident;
  return launch_chained(k, resident_ctas(resident, k, C::THREADS, C::SMEM), C::THREADS, C::SMEM, st, S);
}

// Count, scan, scatter (which also lists the tiles by size class) and the
// classes' sorts (the first of which also writes the work order), each chained
// to the one before.  With separate passes for the order, a launch per class
// whatever the range sizes, memsets in between and unchained launches: one
// 128x96 view 85 -> 45 us, one 512x384 view of its keyframe 109 -> 69, 8 views
// of it 277 -> 156, 12 uneven submaps 1425 -> 745, 24 keyframes x 24 views
// 6220 -> 5870.
cudaError_t launch_bin_tiles(const Layout& L, const RastParams& P, char* ws, cudaStream_t st) {
  if (L.T <= 0) return cudaSuccess;
  Header* hdr = reinterpret_cast<Header*>(ws + L.header);
  uint32_t* counts = reinterpret_cast<uint32_t*>(ws + L.tile_count);
  uint32_t* cursors = reinterpret_cast<uint32_t*>(ws + L.tile_cursor);
  uint2* ranges = reinterpret_cast<uint2*>(ws + L.ranges);
  // small counters: work-order bins and cursors, per class its queue and list size
  uint32_t* small = reinterpret_cast<uint32_t*>(ws + L.tile_hist);
  uint32_t *order_count = small, *order_cursor = small + ORDER_BINS, *queues = small + 2 * ORDER_BINS;
  static_assert(2 * ORDER_BINS + 2 * SORT_CLASSES <= TILE_HIST_WORDS, "the small counters fit");
  TileBinArgs A;
  A.bins = reinterpret_cast<const uint4*>(ws + L.bins);
  A.views = reinterpret_cast<const DView*>(ws + L.views);
  A.V = L.V;
  A.R = L.R;
  A.tile_w_log2 = P.tile_w_log2;
  A.tile_h_log2 = P.tile_h_log2;
  A.counts = counts;
  A.bucket = reinterpret_cast<unsigned long long*>(ws + L.keys1);
  A.cap = L.cap;
  A.hdr = hdr;
  A.ranges = ranges;
  A.T = L.T;
  A.class_list = reinterpret_cast<uint32_t*>(ws + L.tile_class);
  A.class_count = queues + SORT_CLASSES;
  A.order_count = order_count;
  const int64_t work = L.R > L.T ? L.R : L.T;
  const int grid = (int)min64((work + 255) / 256, (int64_t)sm_count() * 16);
  cudaError_t e = cudaSuccess;
  // the counts are zero: cleared by the preprocess, and again by each scan
  if (L.R > 0) {
    e = launch_chained(k_tile_bin<false>, grid, 256, 0, st, A);
    if (e != cudaSuccess) return e;
  }
  e = launch_chained(k_tile_scan, 1, 1024, 0, st, counts, cursors, ranges, L.T, hdr, L.cap, small, TILE_HIST_WORDS);
  if (e != cudaSuccess) return e;
  A.counts = cursors;
  e = launch_chained(k_tile_bin<true>, grid, 256, 0, st, A);
  if (e != cudaSuccess) return e;
  SegArgs S;
  S.ranges = ranges;
  S.bucket = A.bucket;
  S.scratch = reinterpret_cast<unsigned long long*>(ws + L.keys0);
  S.keys = reinterpret_cast<uint64_t*>(ws + L.keys0);
  S.vals = reinterpret_cast<uint32_t*>(ws + L.vals0);
  S.hdr = hdr;
  S.cap = L.cap;
  S.T = L.T;
  S.order_count = order_count;
  S.order_cursor = order_cursor;
  S.order = reinterpret_cast<uint32_t*>(ws + L.tile_order);
  static_assert(32 * WS_ITEMS == SORT_CLASS_BOUND[0] && SegClass<8, 8>::CAP == SORT_CLASS_BOUND[1] &&
                    SegClass<16, 8>::CAP == SORT_CLASS_BOUND[2] && SegClass<16, 12>::CAP == SORT_CLASS_BOUND[3] &&
                    SegClass<16, 16>::CAP == SORT_CLASS_BOUND[4] && SegClass<32, 12>::CAP == SORT_CLASS_BOUND[5],
                "class capacities match the class bounds");
  for (int c = 0; c < SORT_CLASSES; c++) {
    // a surfel has one entry per tile, so no bucket is longer than a view's surfel range
    if (c > 0 && L.max_range <= SORT_CLASS_BOUND[c - 1]) break;
    S.list = A.class_list + (size_t)c * L.T;
    S.list_count = A.class_count + c;
    S.queue = queues + c;
    switch (c) {
      case 0: {
        static PerDevice resident;
        const int grid = persistent_grid(resident, k_tile_sort_warp, WS_WARPS * 32, 0, (L.T + WS_WARPS - 1) / WS_WARPS);
        e = launch_chained(k_tile_sort_warp, grid, WS_WARPS * 32, 0, st, S);
        break;
      }
      case 1: e = launch_tile_sort_class<8, 8, false>(S, st); break;
      case 2: e = launch_tile_sort_class<16, 8, false>(S, st); break;
      case 3: e = launch_tile_sort_class<16, 12, false>(S, st); break;
      case 4: e = launch_tile_sort_class<16, 16, false>(S, st); break;
      default: e = launch_tile_sort_class<32, 12, true>(S, st); break;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// LSD radix sort
// ---------------------------------------------------------------------------
// Contiguous slice of the n keys owned by block b: whole 2048-key tiles.
__device__ __forceinline__ void sort_slice(int64_t n, int nb, int b, int64_t& lo, int64_t& hi) {
  const int64_t tiles = (n + SORT_TILE - 1) / SORT_TILE;
  const int64_t per = (tiles + nb - 1) / nb;
  lo = min64((int64_t)b * per * SORT_TILE, n);
  hi = min64(lo + per * SORT_TILE, n);
}

__global__ void __launch_bounds__(SORT_THREADS) k_sort_upsweep(const uint64_t* __restrict__ keys,
                                                               const unsigned long long* __restrict__ n_dev,
                                                               int64_t n_static, int shift,
                                                               uint32_t* __restrict__ hist) {
  __shared__ uint32_t s_h[8][256];
  const int64_t n = n_dev ? (int64_t)*n_dev : n_static;
  const int wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < 8 * 256; i += SORT_THREADS) (&s_h[0][0])[i] = 0;
  __syncthreads();
  int64_t lo, hi;
  sort_slice(n, gridDim.x, blockIdx.x, lo, hi);
  for (int64_t i = lo + threadIdx.x; i < hi; i += SORT_THREADS) {
    const uint32_t d = (uint32_t)(__ldg(keys + i) >> shift) & 0xffu;
    atomicAdd(&s_h[wid][d], 1u);
  }
  __syncthreads();
  uint32_t* totals = hist + 256 * (size_t)gridDim.x;
  for (int d = threadIdx.x; d < 256; d += SORT_THREADS) {
    uint32_t t = 0;
#pragma unroll
    for (int w = 0; w < 8; w++) t += s_h[w][d];
    hist[(size_t)d * gridDim.x + blockIdx.x] = t;
    if (t) atomicAdd(totals + d, t);
  }
}

// Exclusive scan over the digit-major histogram (256 x nb): block d scans row
// d (nb <= 1024 block counts) and adds the number of keys with smaller digits.
__global__ void __launch_bounds__(1024) k_sort_scan(uint32_t* __restrict__ hist, int nb) {
  __shared__ uint32_t s_w[32];
  const int d = blockIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t* totals = hist + 256 * (size_t)nb;
  // keys with a smaller digit
  uint32_t below = (threadIdx.x < (unsigned)d) ? totals[threadIdx.x] : 0u;
  for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
  if (lane == 0) s_w[wid] = below;
  __syncthreads();
  uint32_t base = 0;
  for (int w = 0; w < 32; w++) base += s_w[w];
  __syncthreads();
  const int i = threadIdx.x;
  const uint32_t v = i < nb ? hist[(size_t)d * nb + i] : 0u;
  uint32_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[wid] = x;
  __syncthreads();
  uint32_t wpre = 0;
  for (int w = 0; w < wid; w++) wpre += s_w[w];
  if (i < nb) hist[(size_t)d * nb + i] = base + wpre + x - v;
}

// Stable scatter.  Warp w ranks keys [tile + 256 w, tile + 256 w + 256) in
// eight rounds of 32 (lane order within a round), so (warp, round, lane)
// order equals input order.
__global__ void __launch_bounds__(SORT_THREADS) k_sort_downsweep(
    const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint64_t* __restrict__ kout,
    uint32_t* __restrict__ vout, const unsigned long long* __restrict__ n_dev, int64_t n_static, int shift,
    uint32_t* __restrict__ hist) {
  __shared__ uint32_t s_wcnt[8][256];  // per-warp digit counts, then warp prefixes
  __shared__ uint32_t s_run[256];      // running output offset per digit for this block
  __shared__ uint32_t s_tcnt[256];
  const int64_t n = n_dev ? (int64_t)*n_dev : n_static;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t lt_mask = (1u << lane) - 1u;
  int64_t lo, hi;
  sort_slice(n, gridDim.x, blockIdx.x, lo, hi);
  for (int d = threadIdx.x; d < 256; d += SORT_THREADS) s_run[d] = hist[(size_t)d * gridDim.x + blockIdx.x];
  // the scan has consumed the digit totals: clear them for the next pass
  if (blockIdx.x == 0)
    for (int d = threadIdx.x; d < 256; d += SORT_THREADS) hist[256 * (size_t)gridDim.x + d] = 0u;
  for (int i = threadIdx.x; i < 8 * 256; i += SORT_THREADS) (&s_wcnt[0][0])[i] = 0;
  __syncthreads();
  for (int64_t tile = lo; tile < hi; tile += SORT_TILE) {
    uint64_t k[SORT_IPT];
    uint32_t val[SORT_IPT], dig[SORT_IPT], rank[SORT_IPT];
#pragma unroll
    for (int r = 0; r < SORT_IPT; r++) {
      const int64_t i = tile + wid * 256 + r * 32 + lane;
      const bool ok = i < hi;
      k[r] = ok ? kin[i] : 0ull;
      val[r] = ok ? vin[i] : 0u;
      dig[r] = ok ? (uint32_t)(k[r] >> shift) & 0xffu : 256u;
    }
#pragma unroll
    for (int r = 0; r < SORT_IPT; r++) {
      const uint32_t d = dig[r];
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t before = __popc(peers & lt_mask);
      const int leader = __ffs(peers) - 1;
      uint32_t base = 0;
      if (d < 256) base = s_wcnt[wid][d];
      __syncwarp();
      if (d < 256 && lane == leader) s_wcnt[wid][d] = base + __popc(peers);
      __syncwarp();
      rank[r] = base + before;
    }
    __syncthreads();
    // per digit: exclusive prefix over warps, and the tile total
    for (int d = threadIdx.x; d < 256; d += SORT_THREADS) {
      uint32_t acc = 0;
#pragma unroll
      for (int w = 0; w < 8; w++) {
        const uint32_t c = s_wcnt[w][d];
        s_wcnt[w][d] = acc;
        acc += c;
      }
      s_tcnt[d] = acc;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SORT_IPT; r++) {
      const uint32_t d = dig[r];
      if (d < 256) {
        const uint32_t pos = s_run[d] + s_wcnt[wid][d] + rank[r];
        kout[pos] = k[r];
        vout[pos] = val[r];
      }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += SORT_THREADS) {
      s_run[d] += s_tcnt[d];
#pragma unroll
      for (int w = 0; w < 8; w++) s_wcnt[w][d] = 0;
    }
    __syncthreads();
  }
}

cudaError_t launch_sort(uint64_t* keys0, uint32_t* vals0, uint64_t* keys1, uint32_t* vals1,
                        const unsigned long long* n_dev, int64_t n_max, int key_bits, uint32_t* hist,
                        int sort_blocks, int* final_buffer, cudaStream_t st) {
  *final_buffer = 0;
  if (n_max <= 0 || key_bits <= 0) return cudaSuccess;
  uint64_t* kb[2] = {keys0, keys1};
  uint32_t* vb[2] = {vals0, vals1};
  int cur = 0;
  for (int shift = 0; shift < key_bits; shift += 8) {
    k_sort_upsweep<<<sort_blocks, SORT_THREADS, 0, st>>>(kb[cur], n_dev, n_max, shift, hist);
    count_launches(1);
    k_sort_scan<<<256, 1024, 0, st>>>(hist, sort_blocks);
    count_launches(1);
    k_sort_downsweep<<<sort_blocks, SORT_THREADS, 0, st>>>(kb[cur], vb[cur], kb[cur ^ 1], vb[cur ^ 1], n_dev,
                                                           n_max, shift, hist);
    count_launches(1);
    cur ^= 1;
  }
  *final_buffer = cur;
  return cudaGetLastError();
}

}  // namespace s2d
