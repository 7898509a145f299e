// The tile lists of gs_bin_sort by counting: every view's records are sorted by depth, its
// depth-ordered records cut into chunks, the chunks' hits counted per tile, and from the
// scanned counts every hit is written once, straight to its place in its tile's list.
//
//   direct_units_kernel  in record order: the runs of tiles of every visible record (one per tile
//                        row, the declared decision of band_span_rn), stored behind a header;
//                        the histograms of the four depth digits of each view; M and the row count
//   direct_sort_kernel   four times: one stable 8-bit pass over each view's visible records in a
//                        single sweep (histogram known, prefixes by decoupled look-back)
//   direct_order_kernel  (frames of many records) the sorted records' rows, and chunks of equal work
//   direct_count_kernel  hits of each chunk per tile of its view
//   direct_scan_kernel   per tile: exclusive scan over the chunks; ranges, M, capacity check
//   direct_emit_kernel   each chunk's record ids to the lists
//
// Compared with emitting (tile, record) pairs into partial order and sorting them (the general
// path, for the frames that dir_plan refuses), a hit moves 4 bytes once
// instead of 8 bytes out, 8 in and 8 out again, the gathers in depth order touch one place per
// record (its header and runs) instead of four, no two warps claim work from one
// counter, and a frame takes 9 or 10 launches instead of 21. gs_bin_sort, that path -> this one,
// kernel times: 5M Gaussians in 4 views of 1600 x 1060 (72.8M entries) 6.03 -> 3.65 ms, 500k in
// 12 mixed views (34.7M) 1.46 -> 1.07 ms, 1.5M in one 1246 x 826 view (16.5M) 430 -> 416 us, 600k
// on 979 x 653 192 -> 185, 100k on 312 x 207 85 -> 65, 2k on 64 x 64 75 -> 38. The emission is half
// of it at the larger sizes; without its scattered 4-byte stores it takes 149 of 203 us (1.5M).
#pragma once

#include <algorithm>

#include "gs_common.cuh"
#include "scan.cuh"

namespace gs {

constexpr int kDirThreads = 256;
constexpr int kDirWarps = kDirThreads / 32;
constexpr int kDirItems = 8;
constexpr int kDirTile = kDirThreads * kDirItems;   // records per block of a sort pass
constexpr int kDirPasses = 4;                       // 8-bit digits of the depth's 32 bits
constexpr int kDirMaxTiles = 20000;                 // per view: 10 1/8 bytes of shared memory each in the emission
constexpr int kDirMaxViews = 1024;
constexpr int64_t kDirMatrix = 1 << 24;             // entries of the (chunk, tile) matrix, at most
constexpr int64_t kDirMostRecords = (1ll << 30) - 1;   // per view: the look-back words count in 30 bits
// the lines of dir_plan's rule: see there
constexpr int64_t kDirTilesFew = 65536, kDirTileRecords = 12, kDirUnequalRecords = 10000;
constexpr uint32_t kDirSpins = 1u << 20;            // polls of a look-back word before the frame is given up

// Device words shared by the kernels of a frame, zeroed before the first.
struct DirWords {
  unsigned long long alloc;        // units handed out: rows and headers
  unsigned long long rows, hits;   // rows of all visible records; M
  uint32_t ticket[kDirPasses];     // partitions started by each sort pass
  uint32_t scan_done;              // blocks of the scan that have finished
  uint32_t failed;                 // a look-back ran out of polls
};

struct DirArgs {
  gs_proj_t P;
  const gs_camera_t *cams;
  int n_views;
  int64_t n;              // records per view
  int tw, th;
  float inv_tw;
  uint64_t cap;           // list capacity (rows and hits)
  uint64_t unit_cap;      // units that the buffer holds (dir_unit_cap)
  uint32_t stretch;       // units that a warp draws at a time (0: what each batch needs)
  int parts;              // sort partitions per view
  int chunks;             // chunks per view
  int n_tiles;
  DirWords *words;
  uint32_t *nvis;         // [views] visible records (zeroed)
  uint32_t *hist;         // [views][4][256] depth digit counts (zeroed)
  uint32_t *state;        // [4][views * parts][256] look-back words (zeroed)
  uint2 *units;           // headers (record, rows << 16 | tiles of its rectangle, up to 65535), each followed by
                          // its rows' runs (first tile of the view, length)
  uint32_t *k0, *v0, *k1, *v1;   // depth keys and header positions; v1 first holds them in record order;
                          // at the end v1 has the order and, with `ordered`, k1 the record ids
  uint2 *ordered;         // (header position, rows) in depth order, over k0 and v0; null: chunks of equal counts
  uint32_t *weights;      // [views][groups] work of 256 depth-ordered records
  uint32_t *starts;       // [views][chunks + 1] first group of each chunk
  uint32_t *order_done;   // [views] blocks of direct_order_kernel that have finished (zeroed)
  int groups;             // groups of 256 records per view, if all were visible
  uint32_t share;         // without `ordered`: records per chunk
  uint32_t *matrix;       // [view][chunk][tile of the view]
  uint32_t *totals;       // [tiles]
  uint2 *ranges;
};

__device__ __forceinline__ bool dir_stopped(const DirArgs &a) {
  return a.words->rows > a.cap || a.words->hits > a.cap || a.words->failed != 0u;
}

// ------------------------------------------------------------------ runs of tiles
// A block takes a run of records view by view, its warps 32 records at a time in record order,
// each with the next 32 records' inputs on their way; a warp's rows are spread over its
// lanes (each finds its record by a search over the lanes' row prefix). On frames of more than a
// million records units come from a stretch of 1024 that the warp draws from the frame's counter when
// its last one is used up, so that neither a barrier nor the counter is on a batch's path: with one draw
// and five barriers per 256 records the kernel took 67 us at 1.5M records and 589 us at 20M, now 70
// and 560: issue (58% of the slots at 600k records, the exact roundings' square roots and divisions) is
// what is left.
// With fewer records a batch draws what it needs: the stretches' rests would be most of the workspace (100k
// records of 312 x 207 37.9 MB -> 10.2, 600k of 979 x 653 129 -> 66), for 0 to 3 us of the whole binning at 600k.
constexpr uint32_t kDirStretch = 1024;
constexpr int64_t kStretchRecords = 1 << 20;   // more of them: stretches
constexpr int kUnitBlocks = 5;            // per SM

inline uint32_t dir_stretch(int64_t R) { return R > kStretchRecords ? kDirStretch : 0u; }
// The units up to which a batch draws on the warp's stretch; a batch of more draws its own.
__host__ __device__ inline uint32_t own_draw(uint32_t stretch) { return stretch / 4; }

__device__ __forceinline__ uint32_t dir_header(uint32_t rows, uint32_t tiles) {
  return rows << 16 | min(tiles, 0xffffu);   // rows <= 65535: rect is 16-bit
}

// A warp's 32 records, field by field: lanes read different records' fields at once.
struct DirBatch {
  float u[32], v[32], beta[32], gamma[32], qb[32], dyr[32], inv_A[32];
  uint32_t x01[32], y0[32];
};

struct DirRec {
  int32_t radius;
  uint2 rect;
  float2 m;
  float4 co;
  float qmax;
  uint32_t key;
};

__global__ void __launch_bounds__(kDirThreads, kUnitBlocks) direct_units_kernel(const DirArgs a) {
  __shared__ DirBatch s_rec[kDirWarps];
  __shared__ uint32_t s_hist[kDirPasses * 256];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  DirBatch &rec = s_rec[warp];
  for (int i = t; i < kDirPasses * 256; i += kDirThreads) s_hist[i] = 0;
  __syncthreads();
  // batches of 32 records, numbered view by view; this block's are [b0, b1)
  const int64_t per_view = (a.n + 31) / 32, total = per_view * a.n_views;
  const int64_t b0 = total * blockIdx.x / gridDim.x, b1 = total * (blockIdx.x + 1) / gridDim.x;
  uint64_t rows = 0, hits = 0;
  uint64_t at = 0, at_end = 0;   // the warp's stretch of units
  const uint32_t own = own_draw(a.stretch);
  for (int64_t bv = b0; bv < b1;) {
    const int v = (int)(bv / per_view);
    const int64_t v0 = (int64_t)v * per_view, ve = min(b1, v0 + per_view);
    const gs_camera_t &cam = a.cams[v];
    const int64_t seg = (int64_t)v * a.n;
    uint32_t seen = 0;
    auto load = [&](int64_t b) -> DirRec {
      DirRec d;
      d.radius = 0;
      const int64_t i = (b - v0) * 32 + lane;
      if (b < ve && i < a.n) {
        const int64_t r = seg + i;
        d.radius = a.P.radius[r];
        d.rect = reinterpret_cast<const uint2 *>(a.P.rect)[r];
        d.m = reinterpret_cast<const float2 *>(a.P.mean2d)[r];
        d.co = reinterpret_cast<const float4 *>(a.P.conic_opacity)[r];
        d.qmax = reinterpret_cast<const float4 *>(a.P.rgb)[r].w;
        d.key = __float_as_uint(a.P.depth[r]);
      }
      return d;
    };
    int64_t b = bv + warp;
    DirRec next = load(b);
    for (; b < ve; b += kDirWarps) {
      const DirRec d = next;
      next = load(b + kDirWarps);
      const uint32_t r = (uint32_t)(seg + (b - v0) * 32 + lane);
      const bool vis = d.radius > 0;
      uint32_t nrow = 0, area = 0;
      if (vis) {
        // within the grid: the counters of later kernels are indexed by these tiles
        const uint32_t x0 = d.rect.x & 0xffffu, y0 = d.rect.x >> 16;
        const uint32_t x1 = min(d.rect.y & 0xffffu, (uint32_t)cam.grid_x), y1 = min(d.rect.y >> 16, (uint32_t)cam.grid_y);
        const float qb = __fmul_rn(d.qmax, kBinMargin);
        float dyr, inv_A;
        band_consts_rn(d.co.x, d.co.y, d.co.z, qb, dyr, inv_A);
        rec.u[lane] = d.m.x;
        rec.v[lane] = d.m.y;
        rec.beta[lane] = d.co.y;
        rec.gamma[lane] = d.co.z;
        rec.qb[lane] = qb;
        rec.dyr[lane] = dyr;
        rec.inv_A[lane] = inv_A;
        rec.x01[lane] = x0 | x1 << 16;
        rec.y0[lane] = y0;
        if (x1 > x0 && y1 > y0) {
          nrow = y1 - y0;
          area = nrow * (x1 - x0);
        }
#pragma unroll
        for (int p = 0; p < kDirPasses - 1; ++p) atomicAdd(&s_hist[p * 256 + ((d.key >> (8 * p)) & 255u)], 1u);
      }
      // the top digit takes a few values in all: one addition per value, not per lane
      for (uint32_t left = __ballot_sync(0xffffffffu, vis); left;) {
        const uint32_t top = __shfl_sync(0xffffffffu, d.key, __ffs(left) - 1) >> 24;
        const uint32_t same = __ballot_sync(0xffffffffu, vis && d.key >> 24 == top);
        if (lane == 0) atomicAdd(&s_hist[(kDirPasses - 1) * 256 + top], __popc(same));
        left &= ~same;
      }
      const uint32_t vm = __ballot_sync(0xffffffffu, vis);
      const uint32_t n_vis = __popc(vm);
      seen += n_vis;
      uint32_t incl = nrow;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t rexcl = incl - nrow;
      const uint32_t n_units = __shfl_sync(0xffffffffu, incl, 31);
      rows += n_units;
      const uint32_t need = n_units + n_vis;
      uint64_t from = at;
      if (need > own || at + need > at_end) {
        const uint32_t draw = need > own ? need : a.stretch;
        unsigned long long got = 0;
        if (lane == 0) got = atomicAdd(&a.words->alloc, (unsigned long long)draw);
        from = __shfl_sync(0xffffffffu, got, 0);
        if (need <= own) {
          at = from;
          at_end = from + draw;
        }
      }
      if (need <= own) at += need;
      const bool keep = from + need <= a.unit_cap;   // else the row count ends the frame (dir_unit_cap)
      const uint32_t off = (uint32_t)from + rexcl + __popc(vm & lanemask_lt());
      if (vis && keep) {
        a.units[off] = make_uint2(r, dir_header(nrow, area));
        a.v1[r] = off;
      }
      __syncwarp();
      for (uint32_t u0 = 0; u0 < n_units; u0 += 32) {
        const uint32_t u = u0 + lane;
        int j = 0;   // the last record whose rows start at or before u
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
          const uint32_t e = __shfl_sync(0xffffffffu, rexcl, j + step);
          if (j + step < 32 && e <= u) j += step;
        }
        const uint32_t row = u - __shfl_sync(0xffffffffu, rexcl, j);
        const uint32_t off_j = __shfl_sync(0xffffffffu, off, j);
        if (u < n_units) {
          const int ty = (int)(rec.y0[j] + row);
          const uint32_t x01 = rec.x01[j];
          const float Y0 = (float)(ty * a.th) + 0.5f, Y1 = (float)min((ty + 1) * a.th, cam.height) - 0.5f;
          float xl, xr;
          int lo = 0;
          uint32_t run = 0;
          if (band_span_rn(rec.u[j], rec.v[j], rec.beta[j], rec.gamma[j], rec.qb[j], rec.dyr[j], rec.inv_A[j], Y0, Y1, xl, xr))
            run = band_columns(xl, xr, (int)(x01 & 0xffffu), (int)(x01 >> 16), a.tw, a.inv_tw, cam.width, lo);
          if (keep && GS_CHECK((uint64_t)off_j + 1 + row < a.unit_cap, 4, off_j))
            a.units[off_j + 1 + row] = make_uint2((uint32_t)(ty * cam.grid_x + lo), run);
          hits += run;
        }
      }
      __syncwarp();   // the next batch rewrites the warp's records
    }
    if (lane == 0 && seen) atomicAdd(&a.nvis[v], seen);
    __syncthreads();
    for (int i = t; i < kDirPasses * 256; i += kDirThreads)
      if (s_hist[i]) {
        atomicAdd(&a.hist[v * kDirPasses * 256 + i], s_hist[i]);
        s_hist[i] = 0;
      }
    __syncthreads();
    bv = ve;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hits += __shfl_xor_sync(0xffffffffu, hits, o);
  if (lane == 0 && rows) {   // rows is the same in every lane
    atomicAdd(&a.words->rows, (unsigned long long)rows);
    atomicAdd(&a.words->hits, (unsigned long long)hits);
  }
}

// ------------------------------------------------------------------ depth sort
// One stable pass by the digit (key >> 8 PASS) & 255 over every view's visible records: blocks
// take partitions of 2048 in order (a ticket, so that whoever a block waits for has
// started), rank their keys by one ballot per digit bit (as rs_downsweep_kernel does), publish
// their digit counts and add up those before them, back to the last partition whose prefix is
// known. Reads and writes each key and value once; the passes it replaces read the keys
// twice and took three launches. A look-back that stays unanswered gives the frame up
// (GS_ERR_TIMEOUT) instead of waiting on.
constexpr uint32_t kSeenSum = 1u << 30, kSeenPrefix = 2u << 30, kSeenMask = 3u << 30;

template <int PASS>
__global__ void __launch_bounds__(kDirThreads, 4) direct_sort_kernel(const DirArgs a) {
  constexpr bool FIRST = PASS == 0, LAST = PASS == kDirPasses - 1;
  constexpr int shift = 8 * PASS;
  __shared__ uint32_t s_keys[kDirTile];
  __shared__ uint32_t s_vals[kDirTile];
  __shared__ uint32_t s_whist[kDirWarps][257];
  __shared__ uint32_t s_goff[256];
  __shared__ uint32_t s_tstart[257];
  __shared__ uint32_t s_ticket;
  __shared__ bool s_stop;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) {
    s_ticket = atomicAdd(&a.words->ticket[PASS], 1u);
    s_stop = dir_stopped(a);   // one read for the block: another block may be giving up now
  }
  for (int d = lane; d < 257; d += 32) s_whist[warp][d] = 0;
  __syncthreads();
  if (s_stop) return;
  const int v = (int)(s_ticket / (uint32_t)a.parts), p = (int)(s_ticket - (uint32_t)v * a.parts);
  const uint32_t count = FIRST ? (uint32_t)a.n : a.nvis[v];
  const uint32_t begin = (uint32_t)p * kDirTile;
  if (begin >= count) return;
  const uint32_t tile_n = min((uint32_t)kDirTile, count - begin);
  const int64_t seg = (int64_t)v * a.n;
  const uint32_t *ki = PASS == 1 || PASS == 3 ? a.k0 : a.k1, *vi = FIRST ? a.v1 : (PASS == 1 || PASS == 3 ? a.v0 : a.v1);
  uint32_t *ko = PASS == 0 || PASS == 2 ? a.k0 : a.k1, *vo = PASS == 0 || PASS == 2 ? a.v0 : a.v1;
  uint32_t k[kDirItems], val[kDirItems], dig[kDirItems], rank[kDirItems];
#pragma unroll
  for (int j = 0; j < kDirItems; ++j) {
    const uint32_t li = warp * (32 * kDirItems) + j * 32 + lane;
    bool valid = li < tile_n;
    const int64_t at = seg + begin + li;
    if (FIRST) {
      const int32_t rad = valid ? a.P.radius[at] : 0;
      k[j] = valid ? __float_as_uint(a.P.depth[at]) : 0u;
      val[j] = valid ? vi[at] : 0u;   // not written for invisible records, and not used
      valid = rad > 0;
    } else {
      k[j] = valid ? ki[at] : 0u;
      val[j] = valid ? vi[at] : 0u;
    }
    dig[j] = valid ? (k[j] >> shift) & 255u : 256u;
  }
  // the digit's base: its place among the view's digits
  const uint32_t hcount = a.hist[(v * kDirPasses + PASS) * 256 + t];
  const uint32_t lt = lanemask_lt();
  const bool sentinels = FIRST || tile_n < (uint32_t)kDirTile;
#pragma unroll
  for (int j = 0; j < kDirItems; ++j) {
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const uint32_t bit = (dig[j] >> b) & 1u;
      peers &= __ballot_sync(0xffffffffu, bit) ^ (bit - 1u);
    }
    if (sentinels) {
      const uint32_t sb = dig[j] >> 8;
      peers &= __ballot_sync(0xffffffffu, sb) ^ (sb - 1u);
    }
    const uint32_t before = __popc(peers & lt);
    const uint32_t base = s_whist[warp][dig[j]];
    __syncwarp();
    rank[j] = base + before;
    if (before == 0) s_whist[warp][dig[j]] = base + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // thread d: the warps' exclusive offsets of digit d and the partition's count
  uint32_t tot = 0;
#pragma unroll
  for (int w = 0; w < kDirWarps; ++w) {
    const uint32_t c = s_whist[w][t];
    s_whist[w][t] = tot;
    tot += c;
  }
  if (t == 0) {
    uint32_t run = 0;   // the sentinels' offsets
    for (int w = 0; w < kDirWarps; ++w) {
      const uint32_t c = s_whist[w][256];
      s_whist[w][256] = run;
      run += c;
    }
  }
  volatile uint32_t *state = a.state + ((size_t)PASS * a.n_views + v) * a.parts * 256 + t;
  state[(size_t)p * 256] = (p == 0 ? kSeenPrefix : kSeenSum) | tot;
  uint32_t all, all_h;
  const uint32_t start = block_exclusive_scan<uint32_t>(tot, &all);
  const uint32_t digit_base = block_exclusive_scan<uint32_t>(hcount, &all_h);
  s_tstart[t] = start;
  if (t == 0) s_tstart[256] = all;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kDirItems; ++j) {
    const uint32_t pos = s_tstart[dig[j]] + s_whist[warp][dig[j]] + rank[j];
    s_keys[pos] = k[j];
    s_vals[pos] = val[j];
  }
  uint32_t prefix = 0;
  bool ok = true;
  if (p > 0) {
    uint32_t polls = 0;
    for (int q = p - 1; q >= 0;) {
      const uint32_t s = state[(size_t)q * 256];
      if ((s & kSeenMask) == 0u) {
        if (++polls >= kDirSpins || ((polls & 1023u) == 0u && *(volatile uint32_t *)&a.words->failed)) {
          ok = false;
          break;
        }
        continue;
      }
      prefix += s & ~kSeenMask;
      if ((s & kSeenMask) == kSeenPrefix) break;
      --q;
    }
    if (ok) state[(size_t)p * 256] = kSeenPrefix | (prefix + tot);
  }
  if (!ok) atomicOr(&a.words->failed, 1u);
  s_goff[t] = digit_base + prefix - start;   // place of the partition's first key of the digit, less its slot
  if (__syncthreads_or(!ok)) return;
  for (uint32_t i = t; i < all; i += kDirThreads) {
    const uint32_t key = s_keys[i];
    const int64_t to = seg + (uint32_t)(s_goff[(key >> shift) & 255u] + i);
    if (!LAST) ko[to] = key;
    vo[to] = s_vals[i];
  }
}

// ------------------------------------------------------------------ counts and ranges
// The records in depth order, as (header position, rows), and the chunks' bounds. A record's
// cost to the kernels that follow is about that of the tiles of its rectangle plus a
// constant, and the nearest records can have hundreds of tiles, the farthest one: chunks of
// equal record counts left the emission's last blocks behind (12 views: 766 -> 645 us). So
// the groups of 256 records get weights, and the last block of a view to finish cuts them
// into chunks of equal weight.
constexpr uint32_t kRecordWeight = 16;

__global__ void __launch_bounds__(kDirThreads) direct_order_kernel(const DirArgs a, int blocks_per_view) {
  __shared__ bool s_last;
  if (dir_stopped(a)) return;
  const int v = blockIdx.x / blocks_per_view, b = blockIdx.x - v * blocks_per_view;
  const uint32_t nv = a.nvis[v];
  const uint32_t ng = (nv + kDirThreads - 1) / kDirThreads;
  const int64_t seg = (int64_t)v * a.n;
  uint32_t *weights = a.weights + (int64_t)v * a.groups;
  const int t = threadIdx.x;
  // four groups a turn: a record's header is a gather from a random place, and with one group the
  // block waited out a round trip per record (20M records, 15M of them visible: 319 -> 289 us; 12 views
  // 73 -> 58)
  constexpr int kTurn = 4;
  __shared__ uint32_t s_w[kTurn][kDirWarps];
  for (uint32_t g = kTurn * b; g < ng; g += kTurn * blocks_per_view) {
    uint32_t off[kTurn];
    uint2 h[kTurn];
#pragma unroll
    for (int i = 0; i < kTurn; ++i) {
      const uint32_t k = (g + i) * kDirThreads + t;
      off[i] = k < nv ? a.v1[seg + k] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kTurn; ++i) {
      const bool on = (g + i) * kDirThreads + t < nv;
      h[i] = on && GS_CHECK(off[i] < a.unit_cap, 4, off[i]) ? a.units[off[i]] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kTurn; ++i) {
      const uint32_t k = (g + i) * kDirThreads + t;
      uint32_t w = 0;
      if (k < nv) {
        a.ordered[seg + k] = make_uint2(off[i], h[i].y >> 16);
        a.k1[seg + k] = h[i].x;
        w = (h[i].y & 0xffffu) + kRecordWeight;
      }
      w = __reduce_add_sync(0xffffffffu, w);
      if ((t & 31) == 0) s_w[i][t >> 5] = w;
    }
    __syncthreads();
    if (t < kTurn && g + t < ng) {
      uint32_t sum = 0;
#pragma unroll
      for (int i = 0; i < kDirWarps; ++i) sum += s_w[t][i];
      weights[g + t] = sum;
    }
    __syncthreads();
  }
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = atomicAdd(&a.order_done[v], 1u) == (uint32_t)blocks_per_view - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // thread t takes groups [g0, g1): their weight, the weight before them, and the chunks that
  // start among them. Group g belongs to chunk floor(P_g C / W), P_g the weight before it.
  const uint32_t per = (ng + kDirThreads - 1) / kDirThreads;
  const uint32_t g0 = min(ng, t * per), g1 = min(ng, g0 + per);
  uint64_t own = 0, W;
#pragma unroll 8
  for (uint32_t g = g0; g < g1; ++g) own += __ldcg(weights + g);
  uint64_t P = block_exclusive_scan<uint64_t>(own, &W);
  uint32_t *starts = a.starts + (int64_t)v * (a.chunks + 1);
  const uint64_t C = (uint64_t)a.chunks;
  int64_t before = g0 == 0 ? -1 : (int64_t)((P - (g0 < ng ? __ldcg(weights + g0 - 1) : 0u)) * C / (W ? W : 1));
  // chunk before + 1 starts at the first P_g C that reaches this (a 64-bit division per group took
  // as long as their loads: 28 -> 22 us at 1.5M records)
  uint64_t bound = (uint64_t)(before + 1) * W;
  for (uint32_t gb = g0; gb < g1; gb += 8) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = gb + i < g1 ? __ldcg(weights + gb + i) : 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (gb + i >= g1) break;
      for (; bound <= P * C; bound += W) starts[++before] = gb + i;
      P += w[i];
    }
  }
  if (g1 == ng && g0 < g1)
    for (int64_t q = before + 1; q <= (int64_t)C; ++q) starts[q] = ng;
  if (ng == 0)
    for (int64_t i = t; i <= (int64_t)C; i += kDirThreads) starts[i] = 0;
}

// Depth-ordered records [begin, end) of chunk c of view v.
__device__ __forceinline__ void chunk_records(const DirArgs &a, int v, int c, uint32_t &begin, uint32_t &end) {
  const uint32_t nv = a.nvis[v];
  if (a.ordered) {
    const uint32_t *starts = a.starts + (int64_t)v * (a.chunks + 1) + c;
    begin = min(nv, starts[0] * kDirThreads);
    end = min(nv, starts[1] * kDirThreads);
  } else {
    begin = min(nv, (uint32_t)c * a.share);
    end = min(nv, begin + a.share);
  }
}

// The view's k-th record in depth order: header position, rows, record id.
struct OrderedRec {
  uint32_t off, rows, rec;
};
__device__ __forceinline__ OrderedRec ordered_record(const DirArgs &a, int64_t seg, uint32_t k) {
  if (a.ordered) {
    const uint2 o = a.ordered[seg + k];
    return OrderedRec{o.x, o.y, a.k1[seg + k]};
  }
  const uint32_t off = a.v1[seg + k];
  const uint2 h = GS_CHECK(off < a.unit_cap, 4, off) ? a.units[off] : make_uint2(0u, 0u);
  return OrderedRec{off, h.y >> 16, h.x};
}

// Block (view, chunk): hits per tile. A warp takes 32 records at a time and spreads their
// rows over its lanes, two rows a lane; the counters are in shared memory, in no order.
__global__ void __launch_bounds__(kDirThreads) direct_count_kernel(const DirArgs a) {
  extern __shared__ uint32_t s_cnt[];
  if (dir_stopped(a)) return;
  const int v = blockIdx.x / a.chunks, c = blockIdx.x - v * a.chunks;
  const int tiles = a.cams[v].grid_x * a.cams[v].grid_y;
  for (int i = threadIdx.x; i < tiles; i += kDirThreads) s_cnt[i] = 0;
  __syncthreads();
  uint32_t begin, end;
  chunk_records(a, v, c, begin, end);
  const int64_t seg = (int64_t)v * a.n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t k0 = begin + warp * 32;
  OrderedRec next = k0 + lane < end ? ordered_record(a, seg, k0 + lane) : OrderedRec{0u, 0u, 0u};
  for (; k0 < end; k0 += kDirThreads) {
    const uint32_t off = next.off, nrow = next.rows;
    const uint32_t kn = k0 + kDirThreads + lane;
    next = kn < end ? ordered_record(a, seg, kn) : OrderedRec{0u, 0u, 0u};
    uint32_t incl = nrow;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t rexcl = incl - nrow;
    const uint32_t n_units = __shfl_sync(0xffffffffu, incl, 31);
    for (uint32_t u0 = 0; u0 < n_units; u0 += 64) {
      uint2 run[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t u = u0 + 32 * i + lane;
        int j = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
          const uint32_t e = __shfl_sync(0xffffffffu, rexcl, j + step);
          if (j + step < 32 && e <= u) j += step;
        }
        const uint32_t row = u - __shfl_sync(0xffffffffu, rexcl, j);
        const uint32_t off_j = __shfl_sync(0xffffffffu, off, j);
        run[i] = u < n_units ? a.units[off_j + 1 + row] : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        for (uint32_t q = 0; q < run[i].y; ++q) atomicAdd(&s_cnt[run[i].x + q], 1u);
    }
  }
  __syncthreads();
  uint32_t *row = a.matrix + (int64_t)a.chunks * a.cams[v].tile_offset + (int64_t)c * tiles;
  for (int i = threadIdx.x; i < tiles; i += kDirThreads) row[i] = s_cnt[i];
}

// kScanCols tiles a block, the chunks spread over the block's other threads: every tile's counts
// turned into offsets within its list, chunk after chunk; the last block scans the tiles'
// totals into the ranges. With few tiles eight a block (whole 32-byte sectors of the matrix's
// rows), so that there are blocks enough: 16 -> 11 us at 260 tiles; with more, 32 (4056 tiles:
// 24 -> 17 us).
constexpr int kDirScanThreads = 512;

template <int kScanCols>
__global__ void __launch_bounds__(kDirScanThreads) direct_scan_kernel(const DirArgs a, int64_t *d_count,
                                                                      int32_t *d_error) {
  constexpr int kScanGroups = kDirScanThreads / kScanCols;
  __shared__ uint32_t s_sum[kScanGroups][kScanCols];
  __shared__ bool s_last;
  const int t = threadIdx.x, col = t & (kScanCols - 1), grp = t / kScanCols;
  const bool stopped = dir_stopped(a);
  if (!stopped) {
    const int tile = blockIdx.x * kScanCols + col;
    const bool on = tile < a.n_tiles;
    const int v = view_of_tile(a.cams, a.n_views, min(tile, a.n_tiles - 1));
    const int toff = a.cams[v].tile_offset, tiles = a.cams[v].grid_x * a.cams[v].grid_y;
    const int per = (a.chunks + kScanGroups - 1) / kScanGroups;
    const int c0 = min(a.chunks, grp * per), c1 = min(a.chunks, c0 + per);
    uint32_t *m = a.matrix + (int64_t)a.chunks * toff + (tile - toff);
    uint32_t sum = 0;
    if (on)
#pragma unroll 8
      for (int c = c0; c < c1; ++c) sum += m[(int64_t)c * tiles];
    s_sum[grp][col] = sum;
    __syncthreads();
    uint32_t run = 0, all = 0;
#pragma unroll 16
    for (int g = 0; g < kScanGroups; ++g) {
      const uint32_t x = s_sum[g][col];
      if (g < grp) run += x;
      all += x;
    }
    if (on) {
      for (int c = c0; c < c1; c += 8) {
        uint32_t x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = c + i < c1 ? m[(int64_t)(c + i) * tiles] : 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (c + i < c1) {
            m[(int64_t)(c + i) * tiles] = run;
            run += x[i];
          }
      }
      if (grp == 0) a.totals[tile] = all;
    }
    __threadfence();
  }
  __syncthreads();
  if (t == 0) s_last = atomicAdd(&a.words->scan_done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (stopped) {
    for (int i = t; i < a.n_tiles; i += kDirScanThreads) a.ranges[i] = make_uint2(0u, 0u);
  } else {
    constexpr int kPer = 8;
    __shared__ uint32_t s_warp[kDirScanThreads / 32];
    uint32_t run = 0;
    for (int b = 0; b < a.n_tiles; b += kDirScanThreads * kPer) {
      uint32_t x[kPer], local = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int tile = b + t * kPer + i;
        x[i] = tile < a.n_tiles ? __ldcg(a.totals + tile) : 0u;
        local += x[i];
      }
      uint32_t incl = local;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((t & 31) >= o) incl += y;
      }
      if ((t & 31) == 31) s_warp[t >> 5] = incl;
      __syncthreads();
      uint32_t pre = run + incl - local;
#pragma unroll
      for (int w = 0; w < kDirScanThreads / 32; ++w) {
        if (w < (t >> 5)) pre += s_warp[w];
        run += s_warp[w];
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int tile = b + t * kPer + i;
        if (tile < a.n_tiles) a.ranges[tile] = make_uint2(pre, pre + x[i]);
        pre += x[i];
      }
      __syncthreads();
    }
  }
  if (t == 0) {
    const uint64_t m = a.words->hits, rows = a.words->rows;
    const bool over = m > a.cap || rows > a.cap;
    // on overflow: a capacity that holds both the entries and the rows
    *d_count = (int64_t)(over && rows > m ? rows : m);
    if (d_error) {
      if (over) atomicOr(d_error, (int32_t)GS_ERR_CAPACITY);
      if (a.words->failed) atomicOr(d_error, (int32_t)GS_ERR_TIMEOUT);
    }
  }
}

// ------------------------------------------------------------------ emission
// Block (view, chunk), 32 W depth-ordered records (a group) at a time. A record hits a tile at
// most once, so a group's hits of a tile are a mask of 32 W bits, and its list entries
// the records of the set bits in order: the threads set the bits of their units (a record's run
// of tiles in one tile row) and note the tiles that had none yet; then each noted tile's
// thread writes its records after the tile's cursor and clears the mask. Two barriers a group.
// Bound by the latency of a group's shared-memory steps (34% of issue slots at 600k records, stalls on
// barriers and shared memory). At 1.5M records / 20M in 4 views: this form 203 / 1690 us; every hit ranked by
// a population count of the bits below it, with a third barrier for the cursors, 210 / 1967,
// and with the hits spread evenly over the lanes first, 242 / 1849; groups of 32, 64 or 128
// records, 256 or 512 threads 203 to 216 / 1650 to 2130; a warp writing a tile's entries together
// where there are more than 4 or 8, 273 and 237 / 2513 and 2221. One warp per chunk with cursors
// of its own and no barriers: a record's rectangle over the lanes, record after record, 345 / 4198; the
// hits spread over the lanes, those of a tile ranked by match.any, 234 / 1809.
// W words of mask per tile: 4 W + 4 + 2 1/8 bytes of shared memory per tile of the view.
// T threads a block: 256, and with one word of mask (more than 7,250 tiles a view, of which one or
// two blocks fit an SM) 512: 5M-class frames of 10,736 tiles 3.56 -> 3.25 ms (1.5M in 4 views), of 16,224
// 4.45 -> 4.00, 300k on 13,110 313 -> 290 us.

inline size_t emit_smem(int words, int tiles) {
  return (4 * (size_t)words + 4 + 2) * tiles + 4 * (((size_t)tiles + 31) / 32) + 16;
}

// A tile's mask, left clear.
template <int W>
__device__ __forceinline__ void take_mask(uint32_t *s, uint32_t m[W]) {
  if constexpr (W == 2) {
    const uint2 x = *reinterpret_cast<uint2 *>(s);
    *reinterpret_cast<uint2 *>(s) = make_uint2(0u, 0u);
    m[0] = x.x; m[1] = x.y;
  } else {
    m[0] = *s;
    *s = 0u;
  }
}

template <int W, int T>
__global__ void __launch_bounds__(T, 1024 / T) direct_emit_kernel(const DirArgs a, uint32_t *__restrict__ vals) {
  constexpr int kEmitThreads = T, kGroup = 32 * W, kGroups = kEmitThreads / kGroup;
  constexpr uint32_t kEmitStage = 3 * kEmitThreads;   // units staged at a time, three loads a thread in flight
  extern __shared__ uint4 s_raw4[];
  __shared__ uint32_t s_pre[kEmitThreads + 1], s_off[kEmitThreads], s_rid[kEmitThreads];
  __shared__ uint32_t s_warp[kEmitThreads / 32];
  __shared__ uint32_t s_cnt[2];
  __shared__ uint2 s_unit[kEmitStage];
  if (dir_stopped(a)) return;
  const int v = blockIdx.x / a.chunks, c = blockIdx.x - v * a.chunks;
  uint32_t begin, end;
  chunk_records(a, v, c, begin, end);
  if (begin >= end) return;
  const gs_camera_t &cam = a.cams[v];
  const int tiles = cam.grid_x * cam.grid_y, words = (tiles + 31) / 32;
  uint32_t *s_mask = reinterpret_cast<uint32_t *>(s_raw4);   // [tiles][W]
  uint32_t *s_cur = s_mask + W * tiles;                      // next place of each tile
  uint32_t *s_touch = s_cur + tiles;                         // bit per tile: in the list
  uint16_t *s_list = reinterpret_cast<uint16_t *>(s_touch + words);
  const uint32_t *row = a.matrix + (int64_t)a.chunks * cam.tile_offset + (int64_t)c * tiles;
  const uint2 *ranges = a.ranges + cam.tile_offset;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < W * tiles; i += kEmitThreads) s_mask[i] = 0u;
  for (int i = t; i < words; i += kEmitThreads) s_touch[i] = 0u;
  for (int i = t; i < tiles; i += kEmitThreads) s_cur[i] = ranges[i].x + row[i];
  if (t < 2) s_cnt[t] = 0u;
  const int64_t seg = (int64_t)v * a.n;
  OrderedRec next = begin + t < end ? ordered_record(a, seg, begin + t) : OrderedRec{0u, 0u, 0u};
  uint32_t turn = 0;
  for (uint32_t k0 = begin; k0 < end; k0 += kEmitThreads) {
    // the block's next records (one a thread) and the prefix of their rows
    const OrderedRec rec = next;
    const uint32_t kn = k0 + kEmitThreads + t;
    next = kn < end ? ordered_record(a, seg, kn) : OrderedRec{0u, 0u, 0u};
    uint32_t incl = rec.rows;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    s_off[t] = rec.off;
    s_rid[t] = rec.rec;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kEmitThreads / 32; ++w) {
      const uint32_t x = s_warp[w];
      if (w < warp) before += x;
      all += x;
    }
    s_pre[t] = before + incl - rec.rows;
    if (t == 0) s_pre[kEmitThreads] = all;
    __syncthreads();
    uint32_t sb = 0, se = 0;   // the units in s_unit
    const int ng = (int)min((uint32_t)kGroups, (end - k0 + kGroup - 1) / kGroup);
    for (int g = 0; g < ng; ++g) {
      const uint32_t u0 = s_pre[g * kGroup], u1 = s_pre[(g + 1) * kGroup];
      if (u0 == u1) continue;
      uint32_t *cnt = &s_cnt[turn & 1];
      for (uint32_t from = u0; from < u1;) {
        if (from >= se || (u1 > se && from == u0)) {
          // units from here on: each the last record whose rows start at or before it, and its
          // run there, as (tile | length << 16, record of the block's)
          sb = from;
          se = min(all, sb + kEmitStage);
          __syncthreads();   // the previous units have been read
          uint32_t j[kEmitStage / kEmitThreads];
          uint2 x[kEmitStage / kEmitThreads];
#pragma unroll
          for (int i = 0; i < (int)(kEmitStage / kEmitThreads); ++i) {
            const uint32_t u = sb + t + i * kEmitThreads;
            if (u < se) {
              j[i] = 0;
#pragma unroll
              for (int step = kEmitThreads / 2; step > 0; step >>= 1)
                if (s_pre[j[i] + step] <= u) j[i] += step;
              x[i] = a.units[s_off[j[i]] + 1u + (u - s_pre[j[i]])];
            }
          }
#pragma unroll
          for (int i = 0; i < (int)(kEmitStage / kEmitThreads); ++i)
            if (sb + t + i * kEmitThreads < se)
              s_unit[t + i * kEmitThreads] = make_uint2(x[i].x | x[i].y << 16, j[i]);
          __syncthreads();
        }
        const uint32_t to = min(u1, se);
        for (uint32_t u = from + t; u < to; u += kEmitThreads) {
          const uint2 un = s_unit[u - sb];
          const uint32_t tile = un.x & 0xffffu, len = un.x >> 16, j = un.y - g * kGroup;
          if (len == 0) continue;
          uint32_t *m = s_mask + W * tile + (j >> 5);
          const uint32_t bit = 1u << (j & 31u);
          for (uint32_t q = 0; q < len; ++q) atomicOr(m + W * q, bit);
          const uint32_t last = tile + len - 1u;
          for (uint32_t w = tile >> 5; w <= last >> 5; ++w) {
            const uint32_t lo = w == tile >> 5 ? tile & 31u : 0u, hi = w == last >> 5 ? last & 31u : 31u;
            const uint32_t bits = (0xffffffffu << lo) & (0xffffffffu >> (31u - hi));
            uint32_t fresh = bits & ~s_touch[w];   // (a look first: most tiles of a dense group are noted)
            if (fresh) fresh &= ~atomicOr(&s_touch[w], fresh);
            if (fresh) {
              uint32_t at = atomicAdd(cnt, (uint32_t)__popc(fresh));
              do {
                s_list[at++] = (uint16_t)(32u * w + __ffs(fresh) - 1u);
                fresh &= fresh - 1u;
              } while (fresh);
            }
          }
        }
        from = to;
      }
      __syncthreads();
      const uint32_t n_list = *cnt;
      const uint32_t *rid = s_rid + g * kGroup;
      for (uint32_t i = t; i < n_list; i += kEmitThreads) {
        const uint32_t tile = s_list[i];
        uint32_t m[W], cur = s_cur[tile];
        take_mask<W>(s_mask + W * tile, m);
        s_touch[tile >> 5] = 0u;   // every tile noted in this word is in the list
#pragma unroll
        for (int w = 0; w < W; ++w)
          while (m[w]) {
            const uint32_t id = rid[32 * w + __ffs(m[w]) - 1];
            m[w] &= m[w] - 1u;
            if (GS_CHECK(cur < a.cap, 4, cur)) vals[cur] = id;
            ++cur;
          }
        s_cur[tile] = cur;
      }
      ++turn;
      if (t == 0) s_cnt[turn & 1] = 0u;
      __syncthreads();
    }
  }
}

// keys[i] = tile << 32 | depth bits of list entry i: a warp per tile.
__global__ void direct_keys_kernel(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ vals,
                                   const float *__restrict__ depth, int n_tiles, uint64_t *__restrict__ keys) {
  const int warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
  for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < n_tiles; t += warps) {
    const uint2 rg = ranges[t];
    for (uint32_t i = rg.x + lane; i < rg.y; i += 32) keys[i] = ((uint64_t)t << 32) | __float_as_uint(depth[vals[i]]);
  }
}

// ------------------------------------------------------------------ host side
struct DirPlan {
  int chunks, parts, max_tiles, groups, unit_grid;
  int most_chunks;        // of any frame like this one with fewer records too
  uint32_t share;
  bool ordered, ok;
};

// Units that the buffer holds: the lists' capacity in rows and a header per record, with stretches
// times 4/3 (a warp gives up at most own_draw units of each one) and each warp's last. Frames
// whose rows fit the capacity fit this.
inline uint64_t dir_unit_cap(int64_t R, int64_t cap, int64_t unit_grid) {
  const uint64_t used = (uint64_t)cap + (uint64_t)R, stretch = dir_stretch(R);
  static_assert(kDirStretch % 4 == 0, "at least 3/4 of a stretch is used");
  return (stretch ? used * 4 / 3 + (uint64_t)unit_grid * kDirWarps * stretch : used) + 1;
}

// Entries of the (chunk, tile) matrix, at most: in proportion to what is sorted, up to a bound.
inline int64_t dir_matrix_cap(int64_t R, int64_t cap) {
  return std::min<int64_t>(kDirMatrix, 4 * (R + cap) + (1 << 18));
}

// Whether a frame takes this path, and its chunks: eight blocks per SM in all,
// sixteen with several views, whose sizes may differ (12 views of a quarter to full size: 1165
// us for the whole binning with eight, 1086 with sixteen; one view of 4056 tiles 426 and 447,
// the matrix being longer to scan), of at least 64 records, 128 where a view has more than 10,000 tiles
// and 4096 records (20k records in 4 views of 13,110 tiles 220 -> 184 us), and a matrix within its bound. Refused:
//  - views of more tiles than the emission has shared memory for, sizes beyond the counters', less
//    than a record a view, and frames whose layout gs_frame_init has not written (a view's tables in
//    shared memory are sized by the largest view: max_width and max_height have to cover every view's);
//  - more than 65,536 tiles in all and fewer than 12 records to each: what a chunk costs in tables and
//    in the matrix goes by the tiles (general path -> this one: 2k records in each of 32 views of 4056 tiles
//    127 -> 219 us, 20k 277 -> 364, 50k, 12.3 a tile, 564 -> 561; 20k in 12 views of 6700 203 -> 254, 100k 572 -> 551);
//  - views of unequal sizes, the largest of more than 10,000 tiles, of 10k records and more: the small
//    views' blocks hold as much shared memory as the large one's and have as many hits on few tiles
//    (3 views of 10,736 tiles, a quarter and a sixteenth of that: 20k 136 -> 109 us, 100k 188 -> 250, 500k 503 -> 713;
//    12 such views 20k 207 -> 247, 100k 519 -> 639; where the largest has 8475, 3 views 455 -> 505 at 500k, 12
//    views 485 -> 455 at 100k, 2330 -> 1717 at 500k).
inline DirPlan dir_plan(const gs_frame_t *f, int64_t R, int64_t cap) {
  DirPlan p{};
  if (f->n_views < 1 || f->n_views > kDirMaxViews || R < f->n_views || f->n_tiles < 1) return p;
  if (f->tile_w < 1 || f->tile_h < 1 || f->max_width < 1 || f->max_height < 1) return p;
  const int64_t n = R / f->n_views;
  const int64_t gx = ((int64_t)f->max_width + f->tile_w - 1) / f->tile_w;
  const int64_t gy = ((int64_t)f->max_height + f->tile_h - 1) / f->tile_h;
  if (gx * gy > kDirMaxTiles || gx * gy * f->n_views < f->n_tiles || n > kDirMostRecords) return p;
  if (f->n_tiles > kDirTilesFew && R < kDirTileRecords * f->n_tiles) return p;
  const bool large = gx * gy > 10000;
  if (large && 4 * (int64_t)f->n_tiles < 3 * gx * gy * f->n_views && n >= kDirUnequalRecords) return p;
  p.max_tiles = (int)(gx * gy);
  int64_t chunks = ((f->n_views > 1 ? 16ll : 8ll) * num_sms() + f->n_views - 1) / f->n_views;
  const int64_t groups = (n + kDirThreads - 1) / kDirThreads, by_matrix = dir_matrix_cap(R, cap) / f->n_tiles;
  if (chunks > by_matrix) chunks = by_matrix;
  if (chunks < 1) return p;
  p.most_chunks = (int)std::min<int64_t>(chunks, (n + 63) / 64);
  p.groups = (int)groups;
  p.ordered = chunks < groups;
  if (!p.ordered) {   // few records: equal shares of whole 64s, as many as fill the chunks
    p.share = (uint32_t)std::max<int64_t>(((n + chunks - 1) / chunks + 63) / 64 * 64, large && n >= 4096 ? 128 : 64);
    chunks = (n + p.share - 1) / p.share;
  }
  const int64_t batches = (n + 31) / 32 * f->n_views, grid = (batches + kDirWarps - 1) / kDirWarps;
  p.unit_grid = (int)(grid < (int64_t)kUnitBlocks * num_sms() ? grid : (int64_t)kUnitBlocks * num_sms());
  p.chunks = (int)chunks;
  p.parts = (int)((n + kDirTile - 1) / kDirTile);
  p.ok = dir_unit_cap(R, cap, p.unit_grid) < (1ull << 32);   // header positions are 32-bit
  return p;
}

struct DirWs {
  void *zero;
  size_t zero_bytes;
  DirArgs a;
  size_t bytes;
};

// Workspace: the zeroed words first, then the buffers. n_tiles and views of the frame. Its size
// does not fall with more records or a larger capacity (chunks of whole 64s make their number do so).
inline DirWs dir_layout(void *base, int64_t R, int64_t cap, int64_t views, int64_t n_tiles, const DirPlan &plan) {
  DirWs w{};
  char *p = static_cast<char *>(base);
  size_t off = 0;
  auto take = [&](size_t bytes) -> void * {
    void *q = p ? p + off : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return q;
  };
  w.zero = p;
  w.a.words = (DirWords *)take(sizeof(DirWords));
  w.a.nvis = (uint32_t *)take(4 * (size_t)views);
  w.a.order_done = (uint32_t *)take(4 * (size_t)views);
  w.a.hist = (uint32_t *)take(4 * (size_t)views * kDirPasses * 256);
  w.a.state = (uint32_t *)take(4 * (size_t)kDirPasses * views * plan.parts * 256);
  w.zero_bytes = off;
  w.a.units = (uint2 *)take(8 * (size_t)dir_unit_cap(R, cap, plan.unit_grid));
  w.a.k0 = (uint32_t *)take(8 * (size_t)R);   // k0 | v0, and once they are done with, `ordered`
  w.a.v0 = w.a.k0 + R;
  w.a.k1 = (uint32_t *)take(4 * (size_t)R);
  w.a.v1 = (uint32_t *)take(4 * (size_t)R);
  w.a.ordered = plan.ordered ? reinterpret_cast<uint2 *>(w.a.k0) : nullptr;
  w.a.weights = (uint32_t *)take(4 * (size_t)views * plan.groups);
  w.a.starts = (uint32_t *)take(4 * (size_t)views * (plan.most_chunks + 1));
  w.a.matrix = (uint32_t *)take(4 * (size_t)plan.most_chunks * n_tiles);
  w.a.totals = (uint32_t *)take(4 * (size_t)n_tiles);
  w.bytes = off;
  return w;
}

inline size_t dir_ws_size(const gs_frame_t *f, int64_t R, int64_t cap, const DirPlan &p) {
  return dir_layout(nullptr, R, cap, f->n_views, f->n_tiles, p).bytes;
}

// The most any frame on this path needs for R records: as many views as there may be, a
// partition, a group and two chunks more per view than the records fill, the matrix at its bound, and the
// tiles at theirs.
inline size_t dir_ws_bound(int64_t R, int64_t cap) {
  DirPlan p{};
  const int64_t views = std::min<int64_t>(kDirMaxViews, std::max<int64_t>(R, 1));
  p.unit_grid = kUnitBlocks * num_sms();
  const DirWs w = dir_layout(nullptr, R, cap, views, std::max<int64_t>(kDirTilesFew, R / kDirTileRecords), p);
  return w.bytes + 4 * (size_t)dir_matrix_cap(R, cap) + 4 * (size_t)kDirPasses * 256 * ((size_t)R / kDirTile + views + 1) +
         4 * ((size_t)R / kDirThreads + 16 * (size_t)num_sms() + 4 * views) + 1024;
}

inline gs_status_t dir_bin_sort(const gs_proj_t *proj, const gs_frame_t *f, gs_bins_t *bins, void *ws, size_t ws_bytes,
                                const DirPlan &plan, int32_t *d_error, cudaStream_t s) {
  const int64_t R = proj->n_records;
  DirWs layout = dir_layout(ws, R, bins->capacity, f->n_views, f->n_tiles, plan);
  if (ws_bytes < layout.bytes) return GS_ERR_INVALID_ARG;
  DirArgs &a = layout.a;
  a.P = *proj;
  a.cams = f->cams_dev;
  a.n_views = f->n_views;
  a.n = R / f->n_views;
  a.tw = f->tile_w;
  a.th = f->tile_h;
  a.inv_tw = 1.f / (float)f->tile_w;
  a.cap = (uint64_t)bins->capacity;
  a.unit_cap = dir_unit_cap(R, bins->capacity, plan.unit_grid);
  a.stretch = dir_stretch(R);
  a.groups = plan.groups;
  a.share = plan.share;
  a.parts = plan.parts;
  a.chunks = plan.chunks;
  a.n_tiles = f->n_tiles;
  a.ranges = reinterpret_cast<uint2 *>(bins->ranges);
  GS_CUDA_TRY(cudaMemsetAsync(layout.zero, 0, layout.zero_bytes, s));
  direct_units_kernel<<<plan.unit_grid, kDirThreads, 0, s>>>(a);
  GS_LAUNCH_CHECK();
  const int sg = plan.parts * f->n_views;
  direct_sort_kernel<0><<<sg, kDirThreads, 0, s>>>(a);
  GS_LAUNCH_CHECK();
  direct_sort_kernel<1><<<sg, kDirThreads, 0, s>>>(a);
  GS_LAUNCH_CHECK();
  direct_sort_kernel<2><<<sg, kDirThreads, 0, s>>>(a);
  GS_LAUNCH_CHECK();
  direct_sort_kernel<3><<<sg, kDirThreads, 0, s>>>(a);
  GS_LAUNCH_CHECK();
  if (plan.ordered) {
    const int per_view = (8 * num_sms() + f->n_views - 1) / f->n_views;
    direct_order_kernel<<<per_view * f->n_views, kDirThreads, 0, s>>>(a, per_view);
    GS_LAUNCH_CHECK();
  }
  const int cg = plan.chunks * f->n_views;
  const size_t smem_c = 4 * (size_t)plan.max_tiles;
  // the attributes are set to the same values by every caller
  GS_CUDA_TRY(cudaFuncSetAttribute(direct_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kDirMaxTiles));
  // two words where two blocks or more fit an SM
  const int w = emit_smem(2, plan.max_tiles) <= 100 * 1024 ? 2 : 1;
  const size_t smem_e = emit_smem(w, plan.max_tiles);
  const int et = w == 2 ? 256 : 512;
  auto emit = w == 2 ? direct_emit_kernel<2, 256> : direct_emit_kernel<1, 512>;
  GS_CUDA_TRY(cudaFuncSetAttribute(emit, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)emit_smem(1, kDirMaxTiles)));
  direct_count_kernel<<<cg, kDirThreads, smem_c, s>>>(a);
  GS_LAUNCH_CHECK();
  if (f->n_tiles <= 1024)
    direct_scan_kernel<8><<<(f->n_tiles + 7) / 8, kDirScanThreads, 0, s>>>(a, bins->d_count, d_error);
  else
    direct_scan_kernel<32><<<(f->n_tiles + 31) / 32, kDirScanThreads, 0, s>>>(a, bins->d_count, d_error);
  GS_LAUNCH_CHECK();
  emit<<<cg, et, smem_e, s>>>(a, bins->vals);
  GS_LAUNCH_CHECK();
  if (bins->keys) {
    direct_keys_kernel<<<num_sms() * 8, 256, 0, s>>>(a.ranges, bins->vals, proj->depth, f->n_tiles, bins->keys);
    GS_LAUNCH_CHECK();
  }
  return GS_OK;
}

}  // namespace gs
