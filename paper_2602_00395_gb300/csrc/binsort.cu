// gs_bin_sort: tile binning and depth order of the tile-based rasteriser
// (Sec. 3.1 of arXiv 2602.00395).
//
// Every pair of one splat shares its depth, so the order (tile, depth, splat)
// is built in two stages instead of sorting 64-bit (tile, depth) pair keys:
//
//   records  per (view, splat): its tiles (the FP32 rectangle, narrowed row
//            by row to the footprint ellipse, see row_span_v); the V x n_pad
//            records are sorted by (view, depth bits) with a stable LSD radix
//            sort (record index order breaks ties)
//   scan     emission offsets in that order and the pair count P
//   emit     key = view * tiles + tile (32 bits), value = splat, written in
//            (view, depth, splat) order
//   sort     stable LSD radix sort of the pairs on those keys: the depth order
//            within a tile is the emission order, so no depth bits are moved
//   ranges   [start, end) of every tile
//
// A radix pass cuts its segment into one contiguous range per resident block: a
// kernel counts each range's digits, another turns the counts into first output
// positions (for many ranges), and the scatter walks its range tile by tile,
// ranks each tile's keys stably in shared memory and writes every digit's run
// contiguously, carrying the positions from tile to tile; no block waits on
// another.  The result is the total order (key, splat index).  Grids are sized
// for the chip and read P from device memory, so the call needs no host
// synchronisation (and can be captured in a graph).
#include "common.cuh"
#include "ranges.cuh"

namespace gs {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanChunk = kScanThreads * kScanItems;  // 2048
// A radix tile is kRadixThreads x ITEMS items.  ITEMS is 16 where digits are many
// and the input fills the chip (longer runs per digit; 2 resident blocks per SM),
// else 8 (3 blocks): 12.2M pairs, random low digits 87 against 102 us, high digits
// with few values per warp 69 against 58 us.
constexpr int kRadixThreads = 256;
__host__ __device__ constexpr int radix_tile(int items) { return kRadixThreads * items; }
__host__ __device__ constexpr int radix_blocks(int items) { return items == 16 ? 2 : 3; }
constexpr int kRadixWarps = kRadixThreads / 32;

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// The tile rows of record g (see foot_rows).
__device__ __forceinline__ FootRows record_rows(const float4* __restrict__ rec, size_t g, const gs_frame& fr, int Tx,
                                                int Ty, float& depth) {
  const float4 a = rec[3 * g + 0];
  const float4 b = rec[3 * g + 1];
  const float4 c = rec[3 * g + 2];
  depth = c.y;
  const int r = __float_as_int(c.z);
  FootRows f = foot_rows(a.x, a.y, a.z, a.w, b.x, r, __float_as_uint(c.w), fr.footprint_bins != 0, fr.tile_w,
                         fr.tile_h, Tx, Ty);
  if (r <= 0) f.x1 = f.x0;  // culled: no tiles
  return f;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t& total, uint32_t* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    uint32_t w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) s_warp[lane] = w;
  }
  __syncthreads();
  total = s_warp[(blockDim.x >> 5) - 1];
  const uint32_t before = warp > 0 ? s_warp[warp - 1] : 0;
  __syncthreads();
  return before + x - v;
}

// ------------------------------------------------------------------ records
// Per record g: rkeys[g] = bits(depth) (then sorted within each view's segment,
// the first pass taking g itself as the value); and its row table for the emit:
// one entry per row of its rectangle, (pairs in the rows above, first tile),
// allocated from `rows` by one atomic per block, and the header
// hdr[g] = (bits(depth), first row | rows << 16, table offset, pairs).  The
// table holds at most 2 empty rows per record beyond its pairs (non-empty rows
// are contiguous), so rows_cap = pair capacity + 2 x records overflows only with
// the pairs; then the record keeps no table and GS_FLAG_CAPACITY is raised.
// Bound by the latency of its loads and its uneven row loops: blocks of 128 let
// a finished warp's place be taken sooner (sort of 8 views of 1M: 1.39 ms against
// 1.40 with 256, 1.45 with 512).
constexpr int kRecThreads = 128;
__global__ void __launch_bounds__(kRecThreads) record_keys_kernel(
    const float4* __restrict__ rec, int n_pad, gs_frame fr, int Tx, int Ty, uint32_t* __restrict__ rkeys,
    uint4* __restrict__ hdr, uint2* __restrict__ rows, uint64_t rows_cap, uint32_t* __restrict__ rows_used,
    int32_t* __restrict__ status) {
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_base;
  const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = g < (size_t)fr.n_views * n_pad;
  float depth = 0.f;
  FootRows f{};
  uint32_t R = 0;
  if (in) {
    f = record_rows(rec, g, fr, Tx, Ty, depth);
    if (f.x1 > f.x0 && f.y1 > f.y0) R = (uint32_t)(f.y1 - f.y0);
  }
  uint32_t total;
  const uint32_t ex = block_exclusive_scan(R, total, s_warp);
  if (threadIdx.x == 0) s_base = total ? atomicAdd(rows_used, total) : 0u;
  __syncthreads();
  if (!in) return;
  const uint32_t off = s_base + ex;
  uint32_t cnt = 0;
  if (R && (uint64_t)off + R <= rows_cap) {
    float vlo = f.exact ? band_v(f, f.y0 * fr.tile_h) : 0.f;
    for (uint32_t k = 0; k < R; ++k) {
      int a, b;
      if (f.exact) {
        const float vhi = band_v(f, (f.y0 + (int)k + 1) * fr.tile_h);
        row_span_v(f, vlo, vhi, fr.tile_w, Tx, a, b);
        vlo = vhi;
      } else {
        a = f.x0;
        b = f.x1;
      }
      rows[(size_t)off + k] = make_uint2(cnt, (uint32_t)a);
      cnt += (uint32_t)(b - a);
    }
  } else if (R) {
    cnt = foot_count(f, fr.tile_w, fr.tile_h, Tx);
    R = 0;
    if (status) atomicOr(status, GS_FLAG_CAPACITY);
  }
  hdr[g] = make_uint4(__float_as_uint(depth), (uint32_t)f.y0 | (R << 16), off, cnt);
  rkeys[g] = __float_as_uint(depth);
}

// ------------------------------------------------------------------- scan
// scnt[p] = the pairs of the record at sorted position p, and the sum of each
// chunk of kScanChunk of them.
__global__ void __launch_bounds__(kScanThreads) gather_counts_kernel(const uint32_t* __restrict__ order,
                                                                     const uint4* __restrict__ hdr,
                                                                     uint32_t* __restrict__ scnt, size_t items,
                                                                     uint32_t* __restrict__ block_sums) {
  __shared__ uint32_t s_warp[32];
  const size_t base = (size_t)blockIdx.x * kScanChunk;
  uint32_t c[kScanItems], s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const size_t p = base + (size_t)k * kScanThreads + threadIdx.x;
    c[k] = p < items ? __ldg(&hdr[__ldg(order + p)].w) : 0u;
  }
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const size_t p = base + (size_t)k * kScanThreads + threadIdx.x;
    if (p < items) scnt[p] = c[k];
    s += c[k];
  }
  uint32_t total;
  block_exclusive_scan(s, total, s_warp);
  if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

// One block: exclusive scan of the block sums; the grand total goes to *total
// (GS_FLAG_CAPACITY is raised when it exceeds the capacity).
__global__ void __launch_bounds__(1024) scan_blocks_kernel(uint32_t* __restrict__ sums, int nb,
                                                           uint32_t* __restrict__ total, uint64_t capacity,
                                                           int32_t* __restrict__ status) {
  __shared__ uint32_t s_warp[32];
  uint32_t carry = 0;
  for (int base = 0; base < nb; base += (int)blockDim.x * kScanItems) {
    const int b = base + (int)threadIdx.x * kScanItems;
    uint32_t v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      v[k] = b + k < nb ? sums[b + k] : 0u;
      s += v[k];
    }
    uint32_t tot;
    uint32_t run = block_exclusive_scan(s, tot, s_warp) + carry;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      if (b + k < nb) sums[b + k] = run;
      run += v[k];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) {
    *total = carry;
    if ((uint64_t)carry > capacity && status) atomicOr(status, GS_FLAG_CAPACITY);
  }
}

// In place: the exclusive scan of n entries, given the scanned sums of its chunks.
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(uint32_t* __restrict__ v_all, size_t n,
                                                                  const uint32_t* __restrict__ block_sums) {
  __shared__ uint32_t s_warp[32];
  const size_t base = (size_t)blockIdx.x * kScanChunk + (size_t)threadIdx.x * kScanItems;
  const bool whole = base + kScanItems <= n;
  __align__(16) uint32_t v[kScanItems];
  if (whole) {
#pragma unroll
    for (int k = 0; k < kScanItems; k += 4)
      *reinterpret_cast<uint4*>(v + k) = *reinterpret_cast<const uint4*>(v_all + base + k);
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = (base + k < n) ? v_all[base + k] : 0u;
  }
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) s += v[k];
  uint32_t total;
  uint32_t run = block_exclusive_scan(s, total, s_warp) + block_sums[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const uint32_t c = v[k];
    v[k] = run;
    run += c;
  }
  if (whole) {
#pragma unroll
    for (int k = 0; k < kScanItems; k += 4)
      *reinterpret_cast<uint4*>(v_all + base + k) = *reinterpret_cast<const uint4*>(v + k);
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
      if (base + k < n) v_all[base + k] = v[k];
  }
}

// Gather, scan and total in one block, for up to kSmallScan records: one launch
// where three would each cost more than the work (the whole sort of 8192 records
// 101 against 103 us with three, of 12,288 the other way: 114 against 112, of
// 16,384 112 against 106).
constexpr size_t kSmallScan = 8192;
__global__ void __launch_bounds__(1024) small_offsets_kernel(const uint32_t* __restrict__ order,
                                                             const uint4* __restrict__ hdr, uint32_t* __restrict__ scnt,
                                                             int items, uint32_t* __restrict__ total, uint64_t capacity,
                                                             int32_t* __restrict__ status) {
  __shared__ uint32_t s_warp[32];
  uint32_t carry = 0;
  for (int base = 0; base < items; base += 1024 * kScanItems) {
    const int p = base + (int)threadIdx.x * kScanItems;
    uint32_t v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = p + k < items ? __ldg(&hdr[__ldg(order + p + k)].w) : 0u;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) s += v[k];
    uint32_t tot;
    uint32_t run = block_exclusive_scan(s, tot, s_warp) + carry;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      if (p + k < items) scnt[p + k] = run;
      run += v[k];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) {
    *total = carry;
    if ((uint64_t)carry > capacity && status) atomicOr(status, GS_FLAG_CAPACITY);
  }
}

inline int scan_blocks(size_t n) { return (int)((n + kScanChunk - 1) / kScanChunk); }

// ------------------------------------------------------------------- emit
// A warp writes the pairs [p0, p1) of the emission order that belong to 32
// records in (view, depth) order: lane L holds record L's first pair `start`
// (non-decreasing over the lanes), header h, first tile key of its view gkey0 and
// splat index.  Consecutive lanes write consecutive pairs; each finds the record
// that owns its pair by a binary search over the lanes and the pair's row by a
// binary search over that record's row table (see record_keys_kernel), N pairs
// per lane at once so that the searches' loads overlap.
template <int N>
__device__ __forceinline__ void emit_span(uint32_t p0, uint32_t p1, uint32_t start, uint4 h, uint32_t gkey0,
                                          uint32_t gsplat, const uint2* __restrict__ rows, int Tx, uint64_t capacity,
                                          uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int lane = threadIdx.x & 31;
  const uint32_t max_rows = __reduce_max_sync(0xffffffffu, h.y >> 16);
  const uint32_t n = p1 - p0;
  for (uint32_t done = 0; done < n; done = n - done > 32 * N ? done + 32 * N : n) {
    const uint32_t pr = p0 + done;
    int lo[N];
    uint32_t a[N], b[N], q[N], off[N];
    bool in[N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
      lo[u] = 0;
      in[u] = 32u * u + lane < n - done;
    }
    // owner = largest lane whose start <= p (lanes with no pairs never win over the next lane)
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const int cand = lo[u] + step;
        const uint32_t sc = __shfl_sync(0xffffffffu, start, cand & 31);
        if (cand < 32 && sc <= pr + 32 * u + lane) lo[u] = cand;
      }
    }
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const uint32_t R = __shfl_sync(0xffffffffu, h.y, lo[u]) >> 16;
      q[u] = pr + 32 * u + lane - __shfl_sync(0xffffffffu, start, lo[u]);
      off[u] = __shfl_sync(0xffffffffu, h.z, lo[u]);
      a[u] = 0;
      b[u] = R && in[u] ? R - 1 : 0;
    }
    // last row whose pairs above are <= q (empty rows repeat the count before them)
    for (uint32_t span = max_rows; span > 1; span = (span + 1) >> 1) {
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const uint32_t mid = (a[u] + b[u] + 1) >> 1;
        if (a[u] < b[u]) {
          if (__ldg(&rows[(size_t)off[u] + mid].x) <= q[u]) a[u] = mid; else b[u] = mid - 1;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const uint64_t at = (uint64_t)pr + 32 * u + lane;
      uint32_t tile = __shfl_sync(0xffffffffu, gkey0, lo[u]);
      const uint32_t osplat = __shfl_sync(0xffffffffu, gsplat, lo[u]);
      const uint32_t oyr = __shfl_sync(0xffffffffu, h.y, lo[u]);
      if (in[u] && at < capacity) {
        if (oyr >> 16) {
          const uint2 e = __ldg(&rows[(size_t)off[u] + a[u]]);
          // q - e.x < the row's pairs, so txx stays in the row; the clamp only
          // keeps every tile index inside the view if that ever failed
          const uint32_t txx = min(e.y + (q[u] - e.x), (uint32_t)(Tx - 1));
          tile += ((oyr & 0xffffu) + a[u]) * (uint32_t)Tx + txx;
        }
        // (no rows but pairs: the record's row table did not fit, which happens
        // only when the pairs exceed the capacity and GS_FLAG_CAPACITY is
        // raised; its slots still get a valid tile and splat so that every slot
        // below the capacity holds an in-range pair)
        keys[at] = tile;
        vals[at] = osplat;
      }
    }
  }
}

// The record at sorted position p (none past the items): its header, first tile
// key and splat index.  One division per record instead of one per pair
// (views x tiles < 2^32).
__device__ __forceinline__ void emit_record(size_t p, size_t items, const uint4* __restrict__ hdr,
                                            const uint32_t* __restrict__ order, int n_pad, uint32_t tiles, uint4& h,
                                            uint32_t& gkey0, uint32_t& gsplat) {
  h = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t g = p < items ? __ldg(order + p) : 0u;
  if (p < items) h = __ldg(hdr + g);
  const uint32_t gview = g / (uint32_t)n_pad;
  gkey0 = gview * tiles;
  gsplat = g - gview * (uint32_t)n_pad;
}

// Few pairs per record: a warp emits 32 consecutive records, two pairs per lane
// at once (8 blocks per SM; four at once on fewer: 286 against 246 us for 45M pairs
// of 8M records).  Bound by the latency of the searches.
__global__ void __launch_bounds__(256, 8) emit_kernel(const uint4* __restrict__ hdr, const uint2* __restrict__ rows,
                                                      int n_pad, size_t items, int Tx, uint32_t tiles,
                                                      const uint32_t* __restrict__ order,
                                                      const uint32_t* __restrict__ offsets, uint64_t capacity,
                                                      uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // sorted record position
  if (p - (threadIdx.x & 31) >= items) return;                     // whole warp
  uint4 h;
  uint32_t gkey0, gsplat;
  emit_record(p, items, hdr, order, n_pad, tiles, h, gkey0, gsplat);
  const uint32_t start = __ldg(offsets + min(p, items - 1)) + (p < items ? 0u : __ldg(&hdr[__ldg(order + items - 1)].w));
  emit_span<2>(__shfl_sync(0xffffffffu, start, 0), __shfl_sync(0xffffffffu, start + h.w, 31), start, h, gkey0, gsplat,
               rows, Tx, capacity, keys, vals);
}

// Many pairs per record: a warp emits a chunk of consecutive pairs (an equal share
// of them, from kEmitChunkMin to kEmitChunk), whose first record it finds by a
// 32-way search over the records' first pairs.  A warp per 32 records left the
// chip to the few warps with the largest splats: 61k records of 64 pairs on
// average 76 us, 30 us with chunks.  The caller takes it from a capacity of 16
// pairs per record on: below that a chunk spans many groups of 32 records and a
// warp per group has the same share (8M records of 6 pairs: 246 us so).  Where one
// record in 64 is eight times as wide, the whole sort takes with chunks and without
// 125 and 137 us (8000 records of 10 pairs), 160 and 194 (61,000 of 23), 298 and 316
// (300,000 of 23), 706 and 700 (1M of 23), 1352 and 1387 (1M of 54); where all are
// alike it is slower with them from about 150,000 records on, by 7 % at 1M of 15
// pairs and 12 % at 8M.  Records
// without pairs come in runs (the culled ones first in their view, with depth 0):
// a group that owns none of the chunk's pairs is followed by another search
// instead of the groups after it (3 views of 1M records, 3000 with pairs in each:
// the sort 17.4 ms with a walk, 0.31 so).
constexpr uint32_t kEmitChunk = 512, kEmitChunkMin = 64;
__global__ void __launch_bounds__(256) emit_chunk_kernel(const uint4* __restrict__ hdr, const uint2* __restrict__ rows,
                                                         int n_pad, size_t items, int Tx, uint32_t tiles,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ offsets,
                                                         const uint32_t* __restrict__ n_pairs, uint64_t capacity,
                                                         uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int lane = threadIdx.x & 31;
  const uint32_t total = *n_pairs, P = (uint32_t)min((uint64_t)total, capacity);
  const uint32_t warps = gridDim.x * (blockDim.x / 32);
  const uint32_t chunk = min(kEmitChunk, max(kEmitChunkMin, (P / warps + 32) & ~31u));
  for (uint64_t c0 = (uint64_t)(blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32) * chunk; c0 < P;
       c0 += (uint64_t)warps * chunk) {
    uint32_t p0 = (uint32_t)c0;
    const uint32_t p1 = (uint32_t)min((uint64_t)P, c0 + chunk);
    size_t r = 0;
    auto find = [&]() {  // r: from its value on, the last record that starts at or before p0
      size_t len = items - r;
      while (len > 1) {
        const size_t step = (len + 31) / 32, at = lane * step;
        const uint32_t ok = __ballot_sync(0xffffffffu, at < len && __ldg(offsets + r + at) <= p0);
        const size_t k = (size_t)(31 - __clz(ok)) * step;  // lane 0 always holds
        r += k;
        len = min(step, len - k);
      }
    };
    find();
    while (p0 < p1) {  // 32 records at a time
      uint4 h;
      uint32_t gkey0, gsplat;
      emit_record(r + lane, items, hdr, order, n_pad, tiles, h, gkey0, gsplat);
      const uint32_t start = r + lane < items ? __ldg(offsets + r + lane) : total;
      const uint32_t end = min(p1, __shfl_sync(0xffffffffu, start + h.w, 31));
      if (p0 < end) {
        emit_span<4>(p0, end, start, h, gkey0, gsplat, rows, Tx, capacity, keys, vals);
        p0 = end;
        r += 32;
        if (r >= items) break;
      } else {  // (the record that find() leaves owns p0, so the next group owns pairs)
        find();
      }
    }
  }
}

// ------------------------------------------------------------ radix passes
// A pass sorts nseg segments independently and stably on one 8-bit digit.
// Segment g holds items [g * stride, g * stride + len): the record sort has one
// segment per view (len = stride = n_pad), the pair sort one segment whose
// length is the pair count P in device memory.  A segment is cut into tiles (see
// radix_tile) and its tiles into bps contiguous ranges of equal length,
// one per block (g * bps + b).  hist[(g * bps + b) * 256 + d] counts digit d in a
// range; the first output position of a range's digit follows from the ranges
// before it and the totals of the smaller digits.  With one histogram per tile of
// 2048 instead, the histograms of the 45M pairs of 8 views of 1080p took a
// 22 MB scan of three kernels per pass.
struct Seg {
  const uint32_t* len_dev;  // device length of the single segment, or null
  uint64_t cap;             // clamp of *len_dev
  uint32_t len;             // host length of every segment (len_dev == null)
  uint32_t stride;          // items between segment starts
};

__device__ __forceinline__ uint32_t seg_len(const Seg& sg) {
  if (!sg.len_dev) return sg.len;
  const uint64_t p = *sg.len_dev;
  return (uint32_t)(p < sg.cap ? p : sg.cap);
}

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K key, int shift) {
  return (uint32_t)(key >> shift) & 255u;
}

__device__ __forceinline__ uint32_t digit_of(uint32_t key, int shift) { return (key >> shift) & 255u; }

// The lanes of the warp that hold the same digit (256: no item).  The match
// instruction takes longer the more distinct digits the warp holds; nine ballots
// take the same time always.  FEW: the digits of a warp are mostly alike.
template <bool FEW>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d) {
  if constexpr (FEW) return __match_any_sync(0xffffffffu, d);
  uint32_t m = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const bool one = (d >> b) & 1u;
    const uint32_t v = __ballot_sync(0xffffffffu, one);
    m &= one ? v : ~v;
  }
  return m;
}

// Digit counts of one range.  A thread counts ITEMS consecutive keys (read
// as 16-byte vectors) and adds each run of equal digits to its warp's counters
// with one shared atomic: a splat's pairs are adjacent and share their high tile
// digit, so runs are common.  Pos: the type of positions (see positions_wrap).
template <int ITEMS, class Pos>
__global__ void __launch_bounds__(kRadixThreads) radix_hist_kernel(const uint32_t* __restrict__ keys, Seg sg, int bps,
                                                                   int shift, uint32_t* __restrict__ hist) {
  __shared__ uint32_t s_cnt[kRadixWarps][256];
  const int g = blockIdx.x / bps, b = blockIdx.x - g * bps, tid = threadIdx.x, warp = tid >> 5;
  const Range<Pos> rg = range_of<Pos>(seg_len(sg), radix_tile(ITEMS), bps, b);
  const Pos begin = rg.begin, end = rg.end;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) s_cnt[w][tid] = 0;
  __syncthreads();
  const uint32_t* kin = keys + (size_t)g * sg.stride;
  uint32_t kk[ITEMS], next[ITEMS];  // the next tile's keys are on their way while this one is counted
  auto load = [&](Pos at) {
    if (at + ITEMS <= end) {
#pragma unroll
      for (int v = 0; v < ITEMS; v += 4) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(kin + at + v));
        next[v] = w.x; next[v + 1] = w.y; next[v + 2] = w.z; next[v + 3] = w.w;
      }
    } else {
#pragma unroll
      for (int k = 0; k < ITEMS; ++k) next[k] = at + k < end ? kin[at + k] : 0u;
    }
  };
  if (begin < end) load(begin + (uint32_t)tid * ITEMS);
  for (Pos base = begin; base < end; base += radix_tile(ITEMS)) {
    const Pos at = base + (uint32_t)tid * ITEMS;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) kk[k] = next[k];
    if (base + radix_tile(ITEMS) < end) load(at + radix_tile(ITEMS));
    uint32_t prev = 256u, run = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t d = at + k < end ? digit_of(kk[k], shift) : 256u;
      if (d != prev) {
        if (run) atomicAdd(&s_cnt[warp][prev], run);
        prev = d;
        run = 0;
      }
      run += d < 256u;
    }
    if (run) atomicAdd(&s_cnt[warp][prev], run);
  }
  __syncthreads();
  uint32_t c = 0;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) c += s_cnt[w][tid];
  hist[(size_t)blockIdx.x * 256 + tid] = c;
}

// For segments of many ranges: hist becomes, per digit, the exclusive prefix over
// the segment's ranges, and totals its digits' totals.  A block takes 32 digits
// of one segment, a warp every 32nd part of its ranges, a lane one digit.
__global__ void __launch_bounds__(1024) radix_prefix_kernel(uint32_t* __restrict__ hist, uint32_t* __restrict__ totals,
                                                            int bps) {
  __shared__ uint32_t s_sum[32][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = blockIdx.x * 32 + lane, g = blockIdx.y;
  uint32_t* h = hist + (size_t)g * bps * 256 + d;
  const int per = (bps + 31) / 32, b0 = min(warp * per, bps), b1 = min(b0 + per, bps);
  uint32_t s = 0;
#pragma unroll 4
  for (int b = b0; b < b1; ++b) s += h[(size_t)b * 256];
  s_sum[warp][lane] = s;
  __syncthreads();
  uint32_t run = 0;
  for (int w = 0; w < warp; ++w) run += s_sum[w][lane];
  if (warp == 31) totals[(size_t)g * 256 + d] = run + s;
#pragma unroll 4
  for (int b = b0; b < b1; ++b) {
    const uint32_t c = h[(size_t)b * 256];
    h[(size_t)b * 256] = run;
    run += c;
  }
}
// Up to this many ranges a scatter block sums the ranges' counts itself, which
// spares the kernel above (small inputs are bound by their launches: the sort of
// 65,536 records, 32 ranges a pass, 120 us against 128 with the kernel; of 98,304,
// 48 ranges, 140 against 133).
constexpr int kDirectRanges = 32;

// Stable scatter of one range, tile by tile.  Warp w owns a tile's items
// [w * 32 * ITEMS, (w + 1) * 32 * ITEMS), item k of lane L at
// offset k * 32 + L, so the warps' strips and the items within a strip are in
// input order.  Each warp ranks its strip against private digit counters (one
// match per item, no block barrier); the per-digit prefix over the warps and
// the tile's digit starts follow from one block scan; the keys are reordered by
// (digit, rank) in shared memory and each digit's run written contiguously.
// Measured on 12.2M pairs (2 views of 1080p): low digits 87 us, high digits 58 us;
// the chain of dependent steps per tile bounds it (the stores cost 30 us of it,
// loads are a tile ahead).  With a tile per block and a histogram per tile the
// whole sort of 8 views took 1.78 ms, 1.53 ms so (45M pairs, 8M records); a
// render of 61k large splats 0.50 -> 0.35 ms, a step of 1k Gaussians 0.27 -> 0.20.
// totals null: hist holds plain counts (see kDirectRanges).  vin null: the
// values are the items' positions.
template <bool FEW, int ITEMS, class Pos>
__global__ void __launch_bounds__(kRadixThreads, radix_blocks(ITEMS)) radix_scatter_kernel(
    const uint32_t* __restrict__ kin_all, const uint32_t* __restrict__ vin_all, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, Seg sg, int bps, int shift, const uint32_t* __restrict__ hist,
    const uint32_t* __restrict__ totals) {
  constexpr int kTile = radix_tile(ITEMS);
  __shared__ uint32_t s_keys[kTile];
  __shared__ uint32_t s_vals[kTile];
  __shared__ uint32_t s_wc[kRadixWarps][256];  // per-warp digit counts, then their first tile positions
  __shared__ uint32_t s_gofs[256];            // output position minus tile position, per digit
  __shared__ uint32_t s_warp[32];
  const int g = blockIdx.x / bps, b = blockIdx.x - g * bps;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Range<Pos> rg = range_of<Pos>(seg_len(sg), kTile, bps, b);
  const Pos begin = rg.begin, end = rg.end;
  if (begin >= end) return;
  const uint32_t lt = lanemask_lt();
  // first output position of digit tid in this range
  uint32_t next;
  {
    const uint32_t* h = hist + (size_t)g * bps * 256 + tid;
    uint32_t before = 0, all = 0, tot;
    if (totals) {
      before = h[(size_t)b * 256];
      all = totals[(size_t)g * 256 + tid];
    } else {
#pragma unroll 8
      for (int q = 0; q < bps; ++q) {
        const uint32_t c = h[(size_t)q * 256];
        if (q < b) before += c;
        all += c;
      }
    }
    next = block_exclusive_scan(all, tot, s_warp) + before + (uint32_t)g * sg.stride;
  }
  const uint32_t* kin = kin_all + (size_t)g * sg.stride;
  const uint32_t* vin = vin_all ? vin_all + (size_t)g * sg.stride : nullptr;
  // the next tile's items are loaded while this one is ranked
  uint32_t key[ITEMS], vv[ITEMS], nkey[ITEMS], nval[ITEMS];
  const uint32_t mine = (uint32_t)warp * 32 * ITEMS + lane;
  auto load = [&](Pos tile) {
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const Pos idx = tile + mine + (uint32_t)k * 32;
      nkey[k] = idx < end ? __ldg(kin + idx) : 0u;
      nval[k] = idx < end ? (vin ? __ldg(vin + idx) : (uint32_t)g * sg.stride + (uint32_t)idx) : 0u;
    }
  };
  load(begin);
  for (Pos tile = begin; tile < end; tile += kTile) {
    const Pos base = tile + mine;
    uint32_t rank[ITEMS], peers[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      key[k] = nkey[k];
      vv[k] = nval[k];
    }
    if (tile + kTile < end) load(tile + kTile);
    auto digit = [&](int k) { return base + (uint32_t)k * 32 < end ? digit_of(key[k], shift) : 256u; };
#pragma unroll
    for (int q = lane; q < 256; q += 32) s_wc[warp][q] = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) peers[k] = digit_peers<FEW>(digit(k));
    // the first lane of each digit takes the digit's next ranks for all its
    // peers; the items' atomics follow one another without waiting
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t d = digit(k);
      rank[k] = 0;
      if (d < 256u && (peers[k] & lt) == 0) rank[k] = atomicAdd(&s_wc[warp][d], (uint32_t)__popc(peers[k]));
      __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
      rank[k] = __shfl_sync(0xffffffffu, rank[k], __ffs(peers[k]) - 1) + (uint32_t)__popc(peers[k] & lt);
    __syncthreads();
    // digit tid: the tile's count, its start, and the warps' first positions
    uint32_t cw[kRadixWarps], count = 0;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) {
      cw[w] = s_wc[w][tid];
      count += cw[w];
    }
    uint32_t incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t start = incl - count;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) start += w < warp ? s_warp[w] : 0u;
    s_gofs[tid] = next - start;
    next += count;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) {
      s_wc[w][tid] = start;
      start += cw[w];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t d = digit(k);
      if (d < 256u) {
        const uint32_t pos = s_wc[warp][d] + rank[k];
        s_keys[pos] = key[k];
        s_vals[pos] = vv[k];
      }
    }
    __syncthreads();
    // (what is read below is written again only after two more barriers)
    const uint32_t tot = (uint32_t)min((Pos)kTile, end - tile);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const uint32_t p = (uint32_t)k * kRadixThreads + tid;
      if (p < tot) {
        const uint32_t kk = s_keys[p];
        const size_t at = (size_t)(s_gofs[digit_of(kk, shift)] + p);
        kout[at] = kk;
        vout[at] = s_vals[p];
      }
    }
  }
}

// All four passes of a segment of up to kSmallSort records in one block.  So few
// records are bound by the launches (twelve for the passes above): one step of 1k
// Gaussians 200 us with them, 155 us so.  Same ranking as above; the items stay in
// shared memory between the passes.  At most kSmallSort because the keys, places
// and counters of more do not fit 48 KB of shared memory.
constexpr int kSmallThreads = 512, kSmallItems = 8, kSmallSort = kSmallThreads * kSmallItems;
__global__ void __launch_bounds__(kSmallThreads) small_sort_kernel(const uint32_t* __restrict__ keys, uint32_t len,
                                                                   uint32_t* __restrict__ vout) {
  constexpr int kWarps = kSmallThreads / 32;
  __shared__ uint32_t s_keys[kSmallSort];
  __shared__ uint16_t s_vals[kSmallSort];
  __shared__ uint16_t s_wc[kWarps][256];  // per-warp digit counts, then their first positions
  __shared__ uint32_t s_warp[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt(), mine = (uint32_t)warp * 32 * kSmallItems + lane;
  const size_t first = (size_t)blockIdx.x * len;
  uint32_t key[kSmallItems], val[kSmallItems], rank[kSmallItems];
#pragma unroll
  for (int k = 0; k < kSmallItems; ++k) {
    val[k] = mine + (uint32_t)k * 32;
    key[k] = val[k] < len ? __ldg(keys + first + val[k]) : 0u;
  }
  for (int shift = 0; shift < 32; shift += 8) {
#pragma unroll
    for (int q = lane; q < 256; q += 32) s_wc[warp][q] = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k) {
      const uint32_t d = mine + (uint32_t)k * 32 < len ? digit_of(key[k], shift) : 256u;
      const uint32_t peers = digit_peers<false>(d);
      const uint32_t before = d < 256u ? s_wc[warp][d] : 0u;
      rank[k] = before + (uint32_t)__popc(peers & lt);
      __syncwarp();
      if (d < 256u && (peers & lt) == 0) s_wc[warp][d] = (uint16_t)(before + (uint32_t)__popc(peers));
      __syncwarp();
    }
    __syncthreads();
    uint32_t count = 0, total;
    if (tid < 256)
      for (int w = 0; w < kWarps; ++w) count += s_wc[w][tid];
    uint32_t at = block_exclusive_scan(count, total, s_warp);
    if (tid < 256)
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = s_wc[w][tid];
        s_wc[w][tid] = (uint16_t)at;
        at += c;
      }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k) {
      if (mine + (uint32_t)k * 32 < len) {
        const uint32_t pos = s_wc[warp][digit_of(key[k], shift)] + rank[k];
        s_keys[pos] = key[k];
        s_vals[pos] = (uint16_t)val[k];
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k) {
      const uint32_t p = mine + (uint32_t)k * 32;
      if (p < len) {
        key[k] = s_keys[p];
        val[k] = s_vals[p];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kSmallItems; ++k) {
    const uint32_t p = mine + (uint32_t)k * 32;
    if (p < len) vout[first + p] = (uint32_t)first + val[k];
  }
}

// ------------------------------------------------------------------ ranges
__device__ __forceinline__ uint32_t pairs_in_use(const uint32_t* n_pairs, uint64_t capacity) {
  const uint64_t p = *n_pairs;
  return (uint32_t)(p < capacity ? p : capacity);
}

// A thread looks at four consecutive keys (one 16-byte load) and the key after
// them; a tile starts where its key differs from the previous one and ends
// where it differs from the next.
__global__ void ranges_kernel(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ n_pairs,
                              uint64_t capacity, uint64_t n_tiles, uint32_t* __restrict__ ranges) {
  const uint32_t P = pairs_in_use(n_pairs, capacity);
  const size_t step = (size_t)gridDim.x * blockDim.x * 4;
  for (size_t p0 = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; p0 < P; p0 += step) {
    uint32_t tl[5];
    if (p0 + 4 <= P) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(keys + p0));
      tl[0] = a.x; tl[1] = a.y; tl[2] = a.z; tl[3] = a.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) tl[k] = p0 + k < P ? keys[p0 + k] : 0xffffffffu;
    }
    tl[4] = p0 + 4 < P ? keys[p0 + 4] : 0xffffffffu;
    uint32_t prev = p0 > 0 ? keys[p0 - 1] : 0xffffffffu;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const size_t p = p0 + k;
      if (p < P && tl[k] < n_tiles) {  // every emitted tile is below n_tiles; the test guards the writes
        if (tl[k] != prev) ranges[2 * (size_t)tl[k]] = (uint32_t)p;
        if (tl[k + 1] != tl[k]) ranges[2 * (size_t)tl[k] + 1] = (uint32_t)(p + 1);
      }
      prev = tl[k];
    }
  }
}

// ------------------------------------------------------------- tile order
// The blends run one block per tile; starting the longest lists first keeps a
// few heavy tiles from running alone at the end.  A tile's class is
// 8 * floor(log2 len) + the next 3 bits of len (256 classes, 0 for an empty
// list); the order is a counting sort by class, heaviest first.
__device__ __forceinline__ uint32_t tile_class(uint32_t len) {
  if (len == 0) return 0;
  const int e = 31 - __clz(len);
  const uint32_t m = e >= 3 ? (len >> (e - 3)) & 7u : (len << (3 - e)) & 7u;
  return min(255u, 1u + 8u * (uint32_t)e + m);
}

__global__ void tile_class_count_kernel(const uint32_t* __restrict__ ranges, uint32_t n_tiles,
                                        uint32_t* __restrict__ cls_count) {
  __shared__ uint32_t s_cnt[256];
  s_cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_tiles) atomicAdd(&s_cnt[tile_class(ranges[2 * t + 1] - ranges[2 * t])], 1u);
  __syncthreads();
  if (s_cnt[threadIdx.x]) atomicAdd(&cls_count[threadIdx.x], s_cnt[threadIdx.x]);
}

// cls_count -> the first slot of each class, heaviest class first (one block of 256)
__global__ void tile_class_starts_kernel(uint32_t* __restrict__ cls_count) {
  __shared__ uint32_t s_warp[32];
  const uint32_t c = cls_count[255 - threadIdx.x];  // thread k holds class 255 - k
  uint32_t total;
  const uint32_t ex = block_exclusive_scan(c, total, s_warp);
  cls_count[255 - threadIdx.x] = ex;
}

__global__ void tile_order_kernel(const uint32_t* __restrict__ ranges, uint32_t n_tiles,
                                  uint32_t* __restrict__ cls_next, uint32_t* __restrict__ order) {
  // one atomic per class present in the warp (most tiles share class 0, the
  // empty lists); a warp's tiles of one class keep their index order
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const uint32_t c = t < n_tiles ? tile_class(ranges[2 * t + 1] - ranges[2 * t]) : 0xffffffffu;
  const uint32_t peers = __match_any_sync(0xffffffffu, c);
  const int leader = __ffs(peers) - 1;
  uint32_t base = 0;
  if ((int)lane == leader && c != 0xffffffffu) base = atomicAdd(&cls_next[c], (uint32_t)__popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (c != 0xffffffffu) order[base + __popc(peers & ((1u << lane) - 1u))] = t;
}

// The whole order in one block, for few tiles: three launches and a memset less (the
// sort with 8160 tiles 116 against 121 us, with 14,400 122 against 123, with 32,400
// 136 against 122).
constexpr uint32_t kSmallOrder = 8192;
__global__ void __launch_bounds__(1024) small_tile_order_kernel(const uint32_t* __restrict__ ranges, uint32_t n_tiles,
                                                                uint32_t* __restrict__ order) {
  __shared__ uint32_t s_next[256], s_warp[32];
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  if (tid < 256) s_next[tid] = 0;
  __syncthreads();
  for (uint32_t t0 = 0; t0 < n_tiles; t0 += 1024) {
    const uint32_t t = t0 + tid;
    const uint32_t c = t < n_tiles ? tile_class(ranges[2 * t + 1] - ranges[2 * t]) : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, c);
    if (c < 256u && (peers & ((1u << lane) - 1u)) == 0) atomicAdd(&s_next[c], (uint32_t)__popc(peers));
  }
  __syncthreads();
  const uint32_t mine = tid < 256 ? s_next[255 - tid] : 0u;  // thread k holds class 255 - k
  uint32_t total;
  const uint32_t first = block_exclusive_scan(mine, total, s_warp);
  if (tid < 256) s_next[255 - tid] = first;
  __syncthreads();
  for (uint32_t t0 = 0; t0 < n_tiles; t0 += 1024) {
    const uint32_t t = t0 + tid;
    const uint32_t c = t < n_tiles ? tile_class(ranges[2 * t + 1] - ranges[2 * t]) : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, c);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if ((int)lane == leader && c < 256u) base = atomicAdd(&s_next[c], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (c < 256u) order[base + __popc(peers & ((1u << lane) - 1u))] = t;
  }
}

void fill_tile_order(const uint32_t* ranges, uint32_t n_tiles, uint32_t* cls, uint32_t* order, cudaStream_t st) {
  const unsigned tb = (n_tiles + 255) / 256;
  if (n_tiles <= kSmallOrder) {
    if (n_tiles) small_tile_order_kernel<<<1, 1024, 0, st>>>(ranges, n_tiles, order);
    return;
  }
  if (tb == 0 || cudaMemsetAsync(cls, 0, 256 * sizeof(uint32_t), st) != cudaSuccess) return;  // reported by the caller
  tile_class_count_kernel<<<tb, 256, 0, st>>>(ranges, n_tiles, cls);
  tile_class_starts_kernel<<<1, 256, 0, st>>>(cls);
  tile_order_kernel<<<tb, 256, 0, st>>>(ranges, n_tiles, cls, order);
}

// ---------------------------------------------------------------- planning
inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

struct SortPlan {
  int Tx, Ty, rec_pass, pair_pass;
  size_t n_items;  // views x n_pad
  size_t off_scnt, off_sums, off_rk0, off_rk1, off_rv0, off_rv1, off_keys, off_vals, off_hist, off_tot, off_hdr, off_rows,
      off_used, off_cls, total;
  uint64_t rows_cap;
};

inline int bits_for(uint64_t v) {  // smallest b with 2^b >= v
  int b = 0;
  while ((1ull << b) < v) ++b;
  return b;
}

// Items per thread of a pass over at most `len` items in each of nseg segments:
// 16 where the digits are many and there are two large tiles for every resident
// block.
inline int radix_items(uint64_t len, int nseg, bool few) {
  return !few && len * (uint64_t)nseg >= (uint64_t)2 * 152 * radix_blocks(16) * radix_tile(16) ? 16 : 8;
}
// Ranges (blocks) of a segment of at most `len` items when nseg segments share
// the chip: one per resident scatter block, at most one per tile.
inline int ranges_per_segment(uint64_t len, int nseg, int items) {
  const uint64_t tiles = std::max<uint64_t>(1, (len + radix_tile(items) - 1) / radix_tile(items));
  const uint64_t fair = (uint64_t)(152 * radix_blocks(items) + nseg - 1) / nseg;
  return (int)std::min<uint64_t>(tiles, std::max<uint64_t>(1, fair));
}

SortPlan plan_sort(int32_t n_pad, gs_frame fr, uint64_t capacity) {
  SortPlan p;
  p.Tx = (fr.width + fr.tile_w - 1) / fr.tile_w;
  p.Ty = (fr.height + fr.tile_h - 1) / fr.tile_h;
  const uint64_t tiles = (uint64_t)fr.n_views * p.Tx * p.Ty;
  p.pair_pass = std::max(1, (bits_for(tiles) + 7) / 8);
  p.rec_pass = 4;  // 32 depth bits within each view
  p.n_items = (size_t)fr.n_views * n_pad;
  // (a pass of 8 items per thread has the most ranges)
  const int rec_ranges = ranges_per_segment((uint64_t)n_pad, fr.n_views, 8);
  const size_t hist_n = (size_t)256 * std::max((size_t)ranges_per_segment(capacity, 1, 8), (size_t)fr.n_views * rec_ranges);
  const size_t sums_n = (size_t)scan_blocks(p.n_items) + 1;
  size_t o = 0;
  p.off_scnt = o;   o += align256(p.n_items * 4);
  p.off_sums = o;   o += align256(sums_n * 4);
  p.off_rk0 = o;    o += align256(p.n_items * 4);
  p.off_rk1 = o;    o += align256(p.n_items * 4);
  p.off_rv0 = o;    o += align256(p.n_items * 4);
  p.off_rv1 = o;    o += align256(p.n_items * 4);
  p.off_keys = o;   o += align256(capacity * 4);
  p.off_vals = o;   o += align256(capacity * 4);
  p.off_hist = o;   o += align256(hist_n * 4);
  p.off_tot = o;    o += rec_ranges > kDirectRanges ? align256((size_t)256 * fr.n_views * 4) : 0;
  p.rows_cap = std::min<uint64_t>(capacity + 2 * (uint64_t)p.n_items, 0xffffffffull);
  p.off_hdr = o;    o += align256(p.n_items * 16);
  p.off_rows = o;   o += align256(p.rows_cap * 8);
  p.off_used = o;   o += 256;
  p.off_cls = o;    o += 256 * 4;
  p.total = o;
  return p;
}

// One stable pass (see Seg) over at most len_max items per segment; vin null: the
// values are the items' positions.
template <bool FEW, int ITEMS, class Pos>
void radix_pass(const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout, int shift, Seg sg, int nseg,
                uint64_t len_max, uint32_t* hist, uint32_t* totals, cudaStream_t st) {
  const int bps = ranges_per_segment(len_max, nseg, ITEMS);
  const unsigned grid = (unsigned)((size_t)nseg * bps);
  const bool direct = bps <= kDirectRanges;
  radix_hist_kernel<ITEMS, Pos><<<grid, kRadixThreads, 0, st>>>(kin, sg, bps, shift, hist);
  if (!direct) radix_prefix_kernel<<<dim3(256 / 32, nseg), 1024, 0, st>>>(hist, totals, bps);
  radix_scatter_kernel<FEW, ITEMS, Pos><<<grid, kRadixThreads, 0, st>>>(kin, vin, kout, vout, sg, bps, shift, hist,
                                                                        direct ? nullptr : totals);
}

// Stable LSD passes over 8-bit digits from bit 0; the keys/values ping-pong
// between buffer 0 and 1 starting in `cur`, which is updated.  iota: the first
// pass's values are the items' positions instead of vbuf[cur].  The last digit
// (the exponents of the depths, the views and upper rows of the tiles) takes few
// values within a warp.
void radix_passes(uint32_t** kbuf, uint32_t** vbuf, int& cur, int npass, bool iota, Seg sg, int nseg, uint64_t len_max,
                  uint32_t* hist, uint32_t* totals, cudaStream_t st) {
  for (int pass = 0; pass < npass; ++pass) {
    const bool few = npass > 1 && pass + 1 == npass;
    const bool long_tiles = radix_items(len_max, nseg, few) == 16;
    auto* run = few ? radix_pass<true, 8, uint32_t>
                    : long_tiles ? radix_pass<false, 16, uint32_t> : radix_pass<false, 8, uint32_t>;
    if (positions_wrap(len_max, radix_tile(16)))  // (a segment so long has long tiles)
      run = few ? radix_pass<true, 8, uint64_t> : radix_pass<false, 16, uint64_t>;
    run(kbuf[cur], iota && pass == 0 ? nullptr : vbuf[cur], kbuf[cur ^ 1], vbuf[cur ^ 1], 8 * pass, sg, nseg, len_max,
        hist, totals, st);
    cur ^= 1;
  }
}

}  // namespace
}  // namespace gs

extern "C" size_t gs_bin_sort_workspace_size(int32_t n_pad, gs_frame frame, uint64_t capacity) {
  if (n_pad < 0 || !gs::frame_ok(frame)) return 0;
  return gs::plan_sort(n_pad, frame, capacity).total;
}

extern "C" gs_status gs_bin_sort(const gs_projected* proj, int32_t n_pad, gs_frame frame, void* workspace,
                                 size_t workspace_bytes, gs_sorted* out, int32_t* status, void* stream) {
  using namespace gs;
  GS_REQUIRE(proj && out && proj->rec, "gs_bin_sort: null argument");
  GS_REQUIRE(out->keys && out->vals && out->ranges && out->n_pairs, "gs_bin_sort: null output buffer");
  GS_REQUIRE(n_pad >= 0 && n_pad % 4 == 0, "gs_bin_sort: bad n_pad=%d", n_pad);
  GS_REQUIRE(frame_ok(frame), "gs_bin_sort: bad frame (tile %dx%d)", frame.tile_w, frame.tile_h);
  GS_REQUIRE(out->capacity > 0 && out->capacity < (1ull << 32), "gs_bin_sort: capacity must be in [1, 2^32)");
  const SortPlan p = plan_sort(n_pad, frame, out->capacity);
  GS_REQUIRE(p.Tx < 65536 && p.Ty < 65536, "gs_bin_sort: at most 65535 tiles per row and column");
  GS_REQUIRE((uint64_t)frame.n_views * p.Tx * p.Ty < 0xffffffffull, "gs_bin_sort: views x tiles must be below 2^32 - 1");
  GS_REQUIRE(workspace && workspace_bytes >= p.total, "gs_bin_sort: workspace needs %zu bytes, got %zu", p.total,
             workspace_bytes);
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  uint32_t* scnt = (uint32_t*)(ws + p.off_scnt);
  uint32_t* sums = (uint32_t*)(ws + p.off_sums);
  uint32_t* hist = (uint32_t*)(ws + p.off_hist);
  uint32_t* totals = (uint32_t*)(ws + p.off_tot);
  const float4* rec = reinterpret_cast<const float4*>(proj->rec);
  const uint64_t T = (uint64_t)p.Tx * p.Ty;

  uint4* hdr = (uint4*)(ws + p.off_hdr);
  uint2* rows = (uint2*)(ws + p.off_rows);
  uint32_t* rows_used = (uint32_t*)(ws + p.off_used);
  if (cudaMemsetAsync(out->ranges, 0, (size_t)frame.n_views * T * 2 * sizeof(uint32_t), st) != cudaSuccess ||
      (p.n_items == 0 && cudaMemsetAsync(out->n_pairs, 0, sizeof(uint32_t), st) != cudaSuccess) ||
      cudaMemsetAsync(rows_used, 0, sizeof(uint32_t), st) != cudaSuccess)
    return check_launch("gs_bin_sort: memset");
  if (p.n_items == 0) {  // no splats: every range is empty
    if (out->order) fill_tile_order(out->ranges, (uint32_t)(frame.n_views * T), (uint32_t*)(ws + p.off_cls), out->order, st);
    return check_launch("gs_bin_sort");
  }
  const int eb = (int)((p.n_items + 255) / 256);
  // records sorted by depth within each view's segment
  uint32_t* rk[2] = {(uint32_t*)(ws + p.off_rk0), (uint32_t*)(ws + p.off_rk1)};
  uint32_t* rv[2] = {(uint32_t*)(ws + p.off_rv0), (uint32_t*)(ws + p.off_rv1)};
  record_keys_kernel<<<(unsigned)((p.n_items + kRecThreads - 1) / kRecThreads), kRecThreads, 0, st>>>(
      rec, n_pad, frame, p.Tx, p.Ty, rk[0], hdr, rows, p.rows_cap, rows_used, status);
  int rcur = 0;
  const Seg rseg{nullptr, 0, (uint32_t)n_pad, (uint32_t)n_pad};
  if (n_pad <= kSmallSort)
    small_sort_kernel<<<frame.n_views, kSmallThreads, 0, st>>>(rk[0], (uint32_t)n_pad, rv[0]);
  else
    radix_passes(rk, rv, rcur, p.rec_pass, true, rseg, frame.n_views, (uint64_t)n_pad, hist, totals, st);
  // emission offsets in that order, and the pair count
  if (p.n_items <= kSmallScan) {
    small_offsets_kernel<<<1, 1024, 0, st>>>(rv[rcur], hdr, scnt, (int)p.n_items, out->n_pairs, out->capacity, status);
  } else {
    const int sb = scan_blocks(p.n_items);
    gather_counts_kernel<<<sb, kScanThreads, 0, st>>>(rv[rcur], hdr, scnt, p.n_items, sums);
    scan_blocks_kernel<<<1, 1024, 0, st>>>(sums, sb, out->n_pairs, out->capacity, status);
    scan_apply_kernel<<<sb, kScanThreads, 0, st>>>(scnt, p.n_items, sums);
  }
  // pairs in (view, depth, splat) order, then stable passes on their tile keys;
  // the last pass must land in the caller's arrays
  uint32_t* kbuf[2] = {out->keys, (uint32_t*)(ws + p.off_keys)};
  uint32_t* vbuf[2] = {out->vals, (uint32_t*)(ws + p.off_vals)};
  int cur = (p.pair_pass % 2 == 0) ? 0 : 1;
  if (out->capacity >= 16 * (uint64_t)p.n_items) {
    const unsigned cb = (unsigned)std::min<uint64_t>((out->capacity + 8 * kEmitChunkMin - 1) / (8 * kEmitChunkMin), 152 * 8);
    emit_chunk_kernel<<<cb, 256, 0, st>>>(hdr, rows, n_pad, p.n_items, p.Tx, (uint32_t)T, rv[rcur], scnt, out->n_pairs,
                                          out->capacity, kbuf[cur], vbuf[cur]);
  } else {
    emit_kernel<<<eb, 256, 0, st>>>(hdr, rows, n_pad, p.n_items, p.Tx, (uint32_t)T, rv[rcur], scnt, out->capacity,
                                    kbuf[cur], vbuf[cur]);
  }
  const Seg pseg{out->n_pairs, out->capacity, 0, 0};
  // (the digits' totals, of more than kDirectRanges ranges, in the row tables that the emit has read)
  radix_passes(kbuf, vbuf, cur, p.pair_pass, false, pseg, 1, out->capacity, hist, (uint32_t*)(ws + p.off_rows), st);
  const int rb = (int)std::min<uint64_t>((out->capacity + 255) / 256, 152 * 16);
  ranges_kernel<<<rb, 256, 0, st>>>(out->keys, out->n_pairs, out->capacity, (uint64_t)frame.n_views * T,
                                    out->ranges);
  if (out->order) fill_tile_order(out->ranges, (uint32_t)(frame.n_views * T), (uint32_t*)(ws + p.off_cls), out->order, st);
  return check_launch("gs_bin_sort");
}
