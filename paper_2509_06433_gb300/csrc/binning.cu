// Tile binning of the projected Gaussians by global radix sorts (grids of fewer tiles than
// multiprocessors; larger ones take tile_sort.cu, which shares k_tile_scan), after the
// (view, Gaussian) items have been stably sorted by camera depth:
//   k_sorted_counts   tiles emitted per item in depth order, per-block totals
//   k_scan_blocks     exclusive scan of the block totals, pair count, capacity check
//   k_item_offsets    per item (depth order): first pair index, rectangle, ids
//   k_tile_scan       row-wise prefix sum of each view's span grid = pairs per tile, then the
//                     tile ranges [start, end) and the digit histograms of the pair sort
//   k_emit_pairs      one (key, value) pair per emitted (view, Gaussian, tile), 1024 pairs per block
//
// An item emits, row by row through its tile rectangle, the tiles of each row's span that
// its widened alpha >= 1/255 ellipse meets (row_span).
// key   = ((k * Tx * Ty + ty * Tx + tx) << 32) | g
// value = the pair's emission index (its slot in the per-pair gradient buffer).
// Pairs are emitted item by item in (depth bits, k*N + g) order. The pair sort then orders
// the tile bits only (stable), which leaves every tile's pairs in (depth bits, k*N + g)
// order: the order of a stable sort of ((tile << 32) | depth bits) keys emitted in (k, g)
// order. Because the sort orders by tile, the ranges are the exclusive scan of the per-tile
// pair counts.
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kScanThreads = 1024;
constexpr int kEmitThreads = 256;

// Tiles touched by each live item in depth order, and per-chunk totals for the scan (chunks of
// kProjBlock items; the blocks stride over the chunks of the n_live live items). Block 0 also
// resets what the tile scan accumulates into: the pair sort's digit histograms, the slabs'
// look-back status and the slab counter.
__global__ void __launch_bounds__(kProjBlock) k_sorted_counts(Layout L, uint8_t* __restrict__ ws) {
  pdl_begin();
  Status* st = at<Status>(ws, L.status);
  if (blockIdx.x == 0) {
    uint32_t* hist = at<uint32_t>(ws, L.hist);
    for (int i = threadIdx.x; i < 4 * 256; i += kProjBlock) hist[i] = 0;
    uint64_t* vlb = at<uint64_t>(ws, L.view_lb);
    for (int i = threadIdx.x; i < L.K * L.scan_slabs; i += kProjBlock) vlb[i] = 0;
    if (threadIdx.x == 0) st->view_ctr = 0;
  }
  const int64_t n_live = st->n_live;
  const int64_t chunks = (n_live + kProjBlock - 1) / kProjBlock;
  __shared__ uint32_t warp_sums[kProjBlock / 32];
  for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
    const int64_t s = c * kProjBlock + threadIdx.x;
    uint32_t cnt = 0;
    if (s < n_live) cnt = at<uint32_t>(ws, L.live_count)[at<uint32_t>(ws, L.item_vals[0])[s]];
    at<uint32_t>(ws, L.sorted_counts)[s] = cnt;
    uint32_t v = cnt;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tot = 0;
      for (int w = 0; w < kProjBlock / 32; ++w) tot += warp_sums[w];
      at<uint32_t>(ws, L.block_sums)[c] = tot;
    }
    __syncthreads();
  }
}

// Inclusive scan of x over a 1024-thread block; tmp: 32 words. Returns the inclusive value;
// *total receives the block total.
__device__ __forceinline__ uint64_t block_inclusive_scan1024(uint64_t x, uint64_t* tmp, uint64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint64_t w = tmp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    tmp[lane] = w;
  }
  __syncthreads();
  const uint64_t r = (warp ? tmp[warp - 1] : 0) + incl;
  *total = tmp[31];
  __syncthreads();
  return r;
}

// Exclusive scan of the per-block pair totals; total pair count, capacity check; clears the
// pair sort's tile counters.
__global__ void __launch_bounds__(kScanThreads) k_scan_blocks(Layout L, uint8_t* __restrict__ ws) {
  pdl_begin();
  const uint32_t* sums = at<uint32_t>(ws, L.block_sums);
  uint64_t* offs = at<uint64_t>(ws, L.block_offsets);
  Status* st = at<Status>(ws, L.status);
  const int64_t chunks = (static_cast<int64_t>(st->n_live) + kProjBlock - 1) / kProjBlock;
  __shared__ uint64_t tmp[32];
  // each thread sums a run of consecutive totals, one block-wide scan of the runs' sums gives
  // every run its start, and the thread then writes its run's offsets (one barrier round, not
  // one per 1024 totals)
  const int64_t per = (chunks + kScanThreads - 1) / kScanThreads;
  const int64_t b0 = threadIdx.x * per, b1 = b0 + per < chunks ? b0 + per : chunks;
  uint64_t run = 0;
  for (int64_t i = b0; i < b1; ++i) run += sums[i];
  uint64_t carry;
  uint64_t start = block_inclusive_scan1024(run, tmp, &carry) - run;
  for (int64_t i = b0; i < b1; ++i) {
    offs[i] = start;
    start += sums[i];
  }
  if (threadIdx.x == 0) {
    st->total_pairs = carry;
    st->num_pairs = static_cast<uint32_t>(carry < static_cast<uint64_t>(L.cap) ? carry : L.cap);
    if (carry > static_cast<uint64_t>(L.cap)) atomicOr(&st->err, GS_DEVERR_PAIR_OVERFLOW);
  }
  if (threadIdx.x < 4) st->tile_ctr[4 + threadIdx.x] = 0;
}

// Per live item in depth order: its first pair index (clamped to the capacity), and the compact
// record the pair-parallel emission reads. Also stores the offset with the projection record
// (the backward pass finds a pair's gradient slot from it). The blocks stride over the chunks.
__global__ void __launch_bounds__(kProjBlock) k_item_offsets(Layout L, uint8_t* __restrict__ ws) {
  pdl_begin();
  __shared__ uint32_t s_warp[kProjBlock / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const Status* st = at<Status>(ws, L.status);
  const int64_t n_live = st->n_live;
  const int64_t chunks = (n_live + kProjBlock - 1) / kProjBlock;
  const uint64_t cap = static_cast<uint64_t>(L.cap);
  const uint64_t n = st->num_pairs;
  uint32_t* offsets = at<uint32_t>(ws, L.item_offsets);
  if (blockIdx.x == 0 && t == 0 && n_live == 0) offsets[0] = 0;
  for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
    const int64_t s = c * kProjBlock + t;
    const uint32_t cnt = at<uint32_t>(ws, L.sorted_counts)[s];
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t wo = 0;
#pragma unroll
    for (int w = 0; w < kProjBlock / 32; ++w) wo += (w < warp) ? s_warp[w] : 0u;
    __syncthreads();
    const uint64_t off = at<uint64_t>(ws, L.block_offsets)[c] + wo + incl - cnt;
    if (s < n_live && cnt) {
      // the emission blocks (kEmitPairs pairs each) whose first or last pair is one of this item's
      // pairs learn here which item that is (the block's window of items)
      const uint64_t lo = off, hi = off + cnt < n ? off + cnt : n;
      uint32_t* first_item = at<uint32_t>(ws, L.emit_first);
      uint32_t* last_item = at<uint32_t>(ws, L.emit_last);
      for (uint64_t b = lo / kEmitPairs; b * kEmitPairs < hi; ++b) {
        const uint64_t b0 = b * kEmitPairs;
        const uint64_t b1 = (b0 + kEmitPairs < n ? b0 + kEmitPairs : n) - 1;
        if (b0 >= lo) first_item[b] = static_cast<uint32_t>(s);
        if (b1 < hi) last_item[b] = static_cast<uint32_t>(s);
      }
    }
    if (s < n_live) {
      offsets[s] = static_cast<uint32_t>(off < cap ? off : cap);
      if (s == n_live - 1) offsets[n_live] = static_cast<uint32_t>(off + cnt < cap ? off + cnt : cap);
      const uint32_t pos = at<uint32_t>(ws, L.item_vals[0])[s];
      const uint32_t kg = at<uint32_t>(ws, L.live_kg)[pos];
      at<uint32_t>(ws, L.live_off)[pos] = static_cast<uint32_t>(off < cap ? off : cap);
      const uint32_t k = static_cast<uint32_t>(kg / static_cast<uint64_t>(L.N));
      const uint2 rows = at<uint2>(ws, L.live_rows)[pos];
      at<int4>(ws, L.item_rect)[s] = make_int4(static_cast<int>(rows.x), static_cast<int>(rows.y), 0, 0);
      at<uint2>(ws, L.item_kg)[s] = make_uint2(k, kg - k * static_cast<uint32_t>(L.N));
    }
  }
}

// Per-tile pair counts, ranges and what the next stage starts from. One block per slab of kScanRows
// tile rows of a view (slabs numbered in block start order): the row-wise prefix sums of the slab's
// part of the view's span grids (one warp per row) are the copies' pairs of every tile, kept in
// shared memory; the exclusive scan over the slab's tiles starts from the slab's pair offset (decoupled
// look-back over the lower-numbered slabs). Writes the ranges (clamped to the pairs actually emitted;
// [0, 0) for an empty tile), and for the tile-sort binning the cursors of each tile's sub-lists
// (one per copy of the span grid) and the list of tiles with more than kTileSortShort pairs, else
// the digit histograms of the pair sort. Bound by latency (a few dependent round trips); slabs keep
// the serial part short: one view of 3600 tiles took 28 us in one block of 1024 threads with four
// grid copies, 12 us with one.
constexpr int kTileScanThreads = 256;

__global__ void __launch_bounds__(kTileScanThreads) k_tile_scan(Layout L, uint8_t* __restrict__ ws) {
  pdl_begin();
  extern __shared__ uint32_t s_count[];  // [diff_copies][kScanRows * Tx]
  constexpr int kWarps = kTileScanThreads / 32;
  __shared__ uint64_t s_warp[kWarps];
  __shared__ uint32_t s_hist[4 * 256];
  __shared__ uint32_t s_slab;
  __shared__ uint64_t s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Status* st = at<Status>(ws, L.status);
  if (threadIdx.x == 0) s_slab = atomicAdd(&st->view_ctr, 1u);
  if (!L.tile_sort)
    for (int i = threadIdx.x; i < 4 * 256; i += kTileScanThreads) s_hist[i] = 0;
  __syncthreads();
  const int slab = static_cast<int>(s_slab);
  if (slab >= L.K * L.scan_slabs) return;
  const int k = slab / L.scan_slabs, ty0 = (slab - k * L.scan_slabs) * kScanRows;
  const int rows = L.Ty - ty0 < kScanRows ? L.Ty - ty0 : kScanRows;
  const int tiles = rows * L.Tx, copies = L.diff_copies;
  // after a capacity overflow the pair sort does not run: leave every tile empty
  const uint64_t n = st->total_pairs > static_cast<uint64_t>(L.cap) ? 0 : st->total_pairs;
  const int stride = L.Tx + 1;
  const int64_t cells = static_cast<int64_t>(stride) * (L.Ty + 1);
  const int32_t* grid = at<int32_t>(ws, L.tile_diff) + static_cast<int64_t>(k) * copies * cells;
  // (one warp per row: the copies' loads and the next 32 columns' are in flight together)
  static_assert(kWarps == kScanRows, "one warp per tile row of the slab");
  if (warp < rows) {
    const int32_t* row = grid + static_cast<int64_t>(ty0 + warp) * stride;
    uint32_t* out = s_count + warp * L.Tx;
    int32_t carry[kTileSubLists] = {}, next[kTileSubLists];
#pragma unroll
    for (int c = 0; c < kTileSubLists; ++c) next[c] = c < copies && lane < L.Tx ? row[c * cells + lane] : 0;
    for (int x = lane; x < L.Tx + lane; x += 32) {
      int32_t v[kTileSubLists];
#pragma unroll
      for (int c = 0; c < kTileSubLists; ++c) {
        v[c] = next[c];
        next[c] = c < copies && x + 32 < L.Tx ? row[c * cells + x + 32] : 0;
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int c = 0; c < kTileSubLists; ++c) {
          const int32_t u = __shfl_up_sync(0xffffffffu, v[c], o);
          if (lane >= o) v[c] += u;
        }
      }
#pragma unroll
      for (int c = 0; c < kTileSubLists; ++c) {
        if (c < copies && x < L.Tx) out[c * kScanRows * L.Tx + x] = static_cast<uint32_t>(carry[c] + v[c]);
        carry[c] += __shfl_sync(0xffffffffu, v[c], 31);
      }
    }
  }
  __syncthreads();
  // a run of consecutive tiles per thread: its pairs, the exclusive scan of the runs, then its tiles
  const int per = (tiles + kTileScanThreads - 1) / kTileScanThreads;
  const int r0 = static_cast<int>(threadIdx.x) * per < tiles ? static_cast<int>(threadIdx.x) * per : tiles;
  const int r1 = r0 + per < tiles ? r0 + per : tiles;
  uint64_t mine = 0;
  for (int c = 0; c < copies; ++c)
    for (int r = r0; r < r1; ++r) mine += s_count[c * kScanRows * L.Tx + r];
  uint64_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint64_t before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    before += w < warp ? s_warp[w] : 0u;
    total += s_warp[w];
  }
  if (warp == 0) {
    const uint64_t base = lb_exclusive_warp(at<uint64_t>(ws, L.view_lb), static_cast<uint32_t>(slab), total, &st->err);
    if (lane == 0) s_base = base;
  }
  __syncthreads();
  uint64_t start = s_base + before + incl - mine;
  const int64_t tile0 = static_cast<int64_t>(k) * L.Tx * L.Ty + static_cast<int64_t>(ty0) * L.Tx;
  for (int r = r0; r < r1; ++r) {
    const int64_t tg = tile0 + r;
    uint64_t end = start;
    for (int c = 0; c < copies; ++c) {
      if (L.tile_sort)
        at<uint32_t>(ws, L.tile_cursor)[(c * L.n_tiles + tg) * kCursorStride] = static_cast<uint32_t>(end < n ? end : n);
      end += s_count[c * kScanRows * L.Tx + r];
    }
    const bool any = end > start;
    at<uint2>(ws, L.ranges)[tg] = make_uint2(any ? static_cast<uint32_t>(start < n ? start : n) : 0u,
                                             any ? static_cast<uint32_t>(end < n ? end : n) : 0u);
    if (L.tile_sort) {
      if (end - start > static_cast<uint64_t>(kTileSortShort) && n) {
        at<uint32_t>(ws, L.long_tiles)[atomicAdd(&st->n_long_next, 1u)] = static_cast<uint32_t>(tg);
        if (end - start > static_cast<uint64_t>(kTileSortGiant)) st->giant = 1;
      }
    } else if (any) {
      for (int p = 0; p < L.passes; ++p)
        atomicAdd(&s_hist[p * 256 + ((static_cast<uint32_t>(tg) >> (8 * p)) & 0xffu)], static_cast<uint32_t>(end - start));
    }
    start = end;
  }
  if (L.tile_sort) return;
  __syncthreads();
  uint32_t* hist = at<uint32_t>(ws, L.hist);
  for (int i = threadIdx.x; i < L.passes * 256; i += kTileScanThreads)
    if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
}

// Pairs [b * kEmitPairs, (b + 1) * kEmitPairs) of the emission order (window b; the blocks
// stride over the windows). The block stages its window of items (pair offsets, row-table ranges, view and Gaussian ids) and, when they fit,
// the window items' row-span entries in shared memory; each pair then finds its item and its
// row by binary searches in shared memory.
constexpr int kEmitRows = 1024;  // row-span entries staged per block (else read from the table)

__global__ void __launch_bounds__(kEmitThreads) k_emit_pairs(Layout L, uint8_t* __restrict__ ws) {
  pdl_wait();
  constexpr int kPerThread = (kEmitPairs + 1 + kEmitThreads - 1) / kEmitThreads;  // items per thread in the scan
  __shared__ uint32_t s_off[kEmitPairs + 2];
  __shared__ uint32_t s_rt[kEmitPairs + 1];    // first row-table entry of each window item
  __shared__ uint32_t s_nk[kEmitPairs + 1];    // entries | view << 16
  __shared__ uint32_t s_g[kEmitPairs + 1];     // Gaussian id
  __shared__ uint32_t s_rbase[kEmitPairs + 1];  // first staged entry of each window item
  __shared__ int2 s_rows[kEmitRows];
  __shared__ uint32_t s_warp[kEmitThreads / 32];
  __shared__ int64_t s_lo, s_hi;
  const uint64_t n = at<Status>(ws, L.status)->num_pairs;
  // clear the pair sort's look-back status (grid-stride over the tiles in use)
  {
    const uint64_t used = static_cast<uint64_t>(sort_tiles(static_cast<int64_t>(n), L.pair_sort_items)) * 256;
    const uint64_t gsize = static_cast<uint64_t>(gridDim.x) * kEmitThreads;
    uint32_t* sstat = at<uint32_t>(ws, L.sort_status);
    for (int p = 0; p < L.passes; ++p)
      for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * kEmitThreads + threadIdx.x; i < used; i += gsize)
        sstat[static_cast<uint64_t>(p) * L.max_sort_tiles * 256 + i] = 0;
    // and the per-pair record bits of the backward pass
    uint32_t* valid = at<uint32_t>(ws, L.pair_valid);
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * kEmitThreads + threadIdx.x; i < (n + 31) / 32; i += gsize)
      valid[i] = 0;
  }
  // the blocks stride over the windows of kEmitPairs pairs that hold emitted pairs
  const uint64_t n_windows = (n + kEmitPairs - 1) / kEmitPairs;
  for (uint64_t win_id = blockIdx.x; win_id < n_windows; win_id += gridDim.x) {
  __syncthreads();  // the previous window's shared staging is no longer read
  const uint64_t start = win_id * kEmitPairs;
  const uint64_t end = start + kEmitPairs < n ? start + kEmitPairs : n;
  const uint32_t* offsets = at<uint32_t>(ws, L.item_offsets);
  if (threadIdx.x == 0) {  // the items holding the window's first and last pairs (k_item_offsets)
    s_lo = at<uint32_t>(ws, L.emit_first)[win_id];
    s_hi = at<uint32_t>(ws, L.emit_last)[win_id];
  }
  __syncthreads();
  const int64_t lo = s_lo;
  // every item of the window emits (items that emit nothing sort last), so win <= kEmitPairs
  const int win = static_cast<int>(s_hi - lo + 1);
  const int4* rects = at<int4>(ws, L.item_rect);
  const uint2* kgs = at<uint2>(ws, L.item_kg);
  const int2* rowtab = at<int2>(ws, L.row_table);
  for (int i = threadIdx.x; i <= win; i += kEmitThreads) s_off[i] = offsets[lo + i];
  for (int i = threadIdx.x; i < win; i += kEmitThreads) {
    const int4 rc = rects[lo + i];  // (first row-table entry, entries)
    const uint2 kg = kgs[lo + i];
    s_rt[i] = static_cast<uint32_t>(rc.x);
    s_nk[i] = static_cast<uint32_t>(rc.y) | (kg.x << 16);
    s_g[i] = kg.y;
  }
  __syncthreads();
  // exclusive scan of the window items' entry counts (kPerThread consecutive items per thread)
  uint32_t loc[kPerThread], sum = 0;
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    const int i = threadIdx.x * kPerThread + q;
    loc[q] = i < win ? (s_nk[i] & 0xffffu) : 0u;
    sum += loc[q];
  }
  {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t base = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kEmitThreads / 32; ++w) {
      base += w < warp ? s_warp[w] : 0u;
      total += s_warp[w];
    }
    base += incl - sum;
#pragma unroll
    for (int q = 0; q < kPerThread; ++q) {
      const int i = threadIdx.x * kPerThread + q;
      if (i < win) s_rbase[i] = base;
      base += loc[q];
    }
    __syncthreads();
    if (total <= static_cast<uint32_t>(kEmitRows)) {
      for (int i = threadIdx.x; i < win; i += kEmitThreads) {
        const uint32_t nr = s_nk[i] & 0xffffu, b = s_rbase[i], rt = s_rt[i];
        for (uint32_t r = 0; r < nr; ++r) s_rows[b + r] = rowtab[rt + r];
      }
    } else if (threadIdx.x == 0) {
      s_warp[0] = 0xffffffffu;  // marker: entries stay in global memory
    }
    __syncthreads();
  }
  const bool staged = s_warp[0] != 0xffffffffu;
  uint64_t* keys = at<uint64_t>(ws, L.keys[0]);
  uint32_t* vals = at<uint32_t>(ws, L.vals[0]);
  const uint64_t tiles_per_view = static_cast<uint64_t>(L.Tx) * L.Ty;
  for (uint64_t j = start + threadIdx.x; j < end; j += kEmitThreads) {
    const uint32_t jj = static_cast<uint32_t>(j);
    int a = 0, b = win;  // s_off[a] <= j < s_off[b]
    while (b - a > 1) {
      const int mid = (a + b) >> 1;
      if (s_off[mid] <= jj) a = mid; else b = mid;
    }
    const uint32_t nk = s_nk[a];
    const int nrows = static_cast<int>(nk & 0xffffu);
    // the pair's tile: its row is the last entry whose earlier-row pair count is <= r
    const int r = static_cast<int>(jj - s_off[a]);
    int tx = 0, ty = 0;
    if (nrows > 0) {
      const int2* tab = staged ? s_rows + s_rbase[a] : rowtab + s_rt[a];
      int p = 0, q = nrows;  // tab[p].x <= r, and r < tab[q].x or q = entries
      while (q - p > 1) {
        const int mid = (p + q) >> 1;
        if (tab[mid].x <= r) p = mid; else q = mid;
      }
      const int2 e = tab[p];
      tx = (e.y & 0xffff) + (r - e.x);
      ty = static_cast<int>(static_cast<uint32_t>(e.y) >> 16);
    }
    const uint64_t tid = static_cast<uint64_t>(nk >> 16) * tiles_per_view + static_cast<uint64_t>(ty) * L.Tx + tx;
    if (!GS_INDEX_OK(tid < static_cast<uint64_t>(L.n_tiles) && tx < L.Tx && ty < L.Ty && j < static_cast<uint64_t>(L.cap),
                     &at<Status>(ws, L.status)->err))
      continue;
    keys[j] = (tid << 32) | s_g[a];
    vals[j] = jj;
  }
  }  // windows
  pdl_trigger();
}

}  // namespace

cudaError_t launch_tile_scan(const Layout& L, void* ws, cudaStream_t s) {
  const size_t smem = static_cast<size_t>(L.diff_copies) * kScanRows * L.Tx * 4;  // <= 128 KB (Tx <= 1024)
  if (smem > 32 * 1024) {  // (images wider than 4096 pixels)
    const cudaError_t e = cudaFuncSetAttribute(k_tile_scan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kTileSubLists * kScanRows * 1024 * 4);
    if (e != cudaSuccess) {
      cudaGetLastError();  // returned here: not to be found again by the process's next call
      return e;
    }
  }
  launch(k_tile_scan, static_cast<unsigned>(L.K * L.scan_slabs), kTileScanThreads, smem, s, L, static_cast<uint8_t*>(ws));
  return cudaGetLastError();
}

cudaError_t launch_bin(const Layout& L, void* ws, cudaStream_t s) {
  auto* w = static_cast<uint8_t*>(ws);
  // the live items are counted on the device: the per-item kernels stride over their chunks
  const int64_t resident = static_cast<int64_t>(device_sms()) * (2048 / kProjBlock);
  const unsigned item_grid = static_cast<unsigned>(L.n_proj_blocks < resident ? L.n_proj_blocks : resident);
  launch(k_sorted_counts, item_grid, kProjBlock, 0, s, L, w);
  launch(k_scan_blocks, 1, kScanThreads, 0, s, L, w);
  launch(k_item_offsets, item_grid, kProjBlock, 0, s, L, w);
  const cudaError_t e = launch_tile_scan(L, ws, s);
  if (e != cudaSuccess) return e;  // (the emission would read item offsets and ranges that nobody wrote)
  // the emission's blocks stride over the windows of emitted pairs (their number is on the device);
  // enough blocks that a typical count takes one window per block (a block looping over several
  // windows serialises their latency-bound searches), few enough that surplus blocks cost little
  const int64_t emit_resident = static_cast<int64_t>(device_sms()) * 128;
  launch(k_emit_pairs, static_cast<unsigned>(L.n_emit_blocks < emit_resident ? L.n_emit_blocks : emit_resident),
         kEmitThreads, 0, s, L, w);
  return cudaGetLastError();
}

}  // namespace gs
