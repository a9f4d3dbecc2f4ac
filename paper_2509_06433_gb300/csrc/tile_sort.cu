// Tile-sort binning: the pairs of the live items go straight to their tile's list, and every list
// is sorted by (depth bits, item) on its own, one block per tile.
//   k_tile_scan (binning.cu)  per-tile pair counts -> ranges, sub-lists, long tiles
//   k_tile_emit               compaction of the live items; one unsorted record per pair
//   k_tile_sort               lists of up to kTileSortShort pairs, in shared memory
//   k_tile_sort_long          longer lists, cut by depth into pieces that fit in shared memory; the
//                             longest by many blocks at once
//
// Order: a tile's list in (depth bits, k N + g) order, as a stable sort of ((tile << 32) | depth)
// keys emitted in (k, g) order leaves it. A pair's slot (emission index) is its item's first pair
// plus the pair's number in the item, the items taken in increasing k N + g order, so within a
// tile equal depths are ordered by slot: the sort key is the 64-bit (depth bits, slot), unique, and
// the result does not depend on the order in which the emission's atomic cursors filled the list.
//
// Why: the lists are short (tens to a few thousand pairs) and independent, so a tile's whole sort
// fits in one block's shared memory: one read and one write of the pairs, where the global radix
// sorts take four passes over the items, three scans and ceil(tile bits / 8) passes over the pairs,
// each a dependent launch. Grids of fewer tiles than multiprocessors keep the global sorts (a block
// per tile would leave the GPU idle and make the lists long).
//
// The sort of a list: one distribution pass into at most n + 256 buckets for n pairs, then each pair
// counts the smaller keys of its own bucket. The buckets adapt to the depths' distribution: 256
// equal slices of the list's depth range are counted first, and a slice of n pairs is cut into the
// largest power of two <= n buckets (a wall seen next to a near object would otherwise fall into a
// few buckets). Where all depths are equal (a floor seen straight from above), the buckets are taken
// from the slots instead. A list that still has a bucket of more than kMaxBucket pairs (many equal
// or almost equal depths beside others) is sorted by a bitonic network.
#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kEmitThreads = 256;
constexpr int kShortThreads = 256;
constexpr int kLongThreads = 512;
constexpr int kLongBlocks = 3;    // resident per SM (75 KB of shared memory each)
constexpr int kLongShared = 4608;  // longest list sorted in one piece
constexpr int kLongSlices = 2048;  // depth slices a longer one is cut into
constexpr uint32_t kMaxBucket = 64;
constexpr int kSlices = 256;

// Most tasks that the long lists of so many pairs give out (see kChunk).
__device__ __forceinline__ uint32_t task_bound(const Layout& L, uint64_t pairs) {
  return min(L.max_tasks, static_cast<uint32_t>(pairs / 32 + 64));
}

// One block per projection block: compacts its live items (in item order) and writes one record
// (depth bits, slot, Gaussian id) per pair at the next free place of its tile's sub-list: the tile
// scan has split every list between the projection blocks b with the same b % kTileSubLists. The
// rate is set by the cursors' atomics, about one warp's per 30 cycles on one address and fewer when the
// cursors of neighbouring tiles share a 32-byte sector, so that the fullest tile decides: one sector
// per cursor and four cursors per tile. The rows of a warp's items are numbered consecutively and
// examined one per lane (row_span gives the same tiles as in the projection), then the pairs of those
// 32 rows are numbered consecutively and written one per lane, four rounds in flight, so that tall
// or wide items do not idle the warp. (One atomic per tile and warp where a view crowds into few tiles saves
// 0.3 of 8 ms at 2M pairs of one tile and costs 10 of 108 us of binning at 2M spread over 3600: not built.)
__global__ void __launch_bounds__(kEmitThreads, 4) k_tile_emit(Layout L, uint8_t* __restrict__ ws, int64_t block0) {
  pdl_wait();
  constexpr int kWarps = kEmitThreads / 32;
  const int64_t b = block0 + blockIdx.x, first = b * L.proj_items;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  Status* st = at<Status>(ws, L.status);
  __shared__ uint32_t s_cnt[2][kWarps], s_live[kWarps];
  __shared__ uint64_t s_pairs[kWarps];
  __shared__ uint32_t s_w0;
  __shared__ uint32_t s_lv[2][kWarps];
  __shared__ uint8_t s_row[kWarps][32], s_item[kWarps][32];
  const uint32_t cnt = at<uint32_t>(ws, L.surv_blocks)[b];  // staged survivors, live or not
  const uint64_t cap = static_cast<uint64_t>(L.cap), total_pairs = st->total_pairs;
  const bool overflow = total_pairs > cap;  // every tile's range is empty
  // the block's first live item and first pair: the sums over 256 blocks before it, then over blocks
  uint32_t base = 0, total_live = 0;
  uint64_t pairs = 0;
  {
    const int64_t super = b / 256, n_super = (L.n_proj_groups + 255) / 256;
    for (int64_t i = threadIdx.x; i < n_super; i += kEmitThreads) {
      const uint32_t l = at<uint32_t>(ws, L.super_live)[i];
      total_live += l;
      if (i < super) {
        base += l;
        pairs += at<uint64_t>(ws, L.super_pairs)[i];
      }
    }
    const int64_t i = super * 256 + threadIdx.x;
    static_assert(kEmitThreads == 256, "one block of the group per thread");
    if (i < b) {
      base += at<uint32_t>(ws, L.live_blocks)[i];
      pairs += at<uint32_t>(ws, L.block_pairs)[i];
    }
    base = __reduce_add_sync(0xffffffffu, base);
    total_live = __reduce_add_sync(0xffffffffu, total_live);
    pairs = warp_sum_u64(pairs);
    if (lane == 0) {
      s_live[wib] = base;
      s_pairs[wib] = pairs;
      s_cnt[1][wib] = total_live;
    }
    __syncthreads();
    base = 0, pairs = 0, total_live = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      base += s_live[w];
      pairs += s_pairs[w];
      total_live += s_cnt[1][w];
    }
  }
  if (b == 0 && threadIdx.x == 0) {
    st->n_live = total_live;
    st->num_pairs = static_cast<uint32_t>(overflow ? cap : total_pairs);
    if (overflow) atomicOr(&st->err, GS_DEVERR_PAIR_OVERFLOW);
    // the tile scan is over: what it counted with starts at zero again for a repeated gs_bin_sort
    st->n_long = st->n_long_next;
    st->n_long_next = 0;
    st->view_ctr = 0;
    st->task_next = st->task_end = 0;
    st->task_left = 0;
  }
  if (b == 0)
    for (int i = threadIdx.x; i < L.K * L.scan_slabs; i += kEmitThreads) at<uint64_t>(ws, L.view_lb)[i] = 0;
  if (st->giant) {  // no task of the long lists is written yet: this block's share
    const int64_t n = task_bound(L, total_pairs);
    for (int64_t i = n * b / L.n_proj_groups + threadIdx.x; i < n * (b + 1) / L.n_proj_groups; i += kEmitThreads)
      at<uint4>(ws, L.tasks)[i].x = 0u;  // (kNoTask)
  }
  // the record bits of the backward pass: this block's share
  {
    const int64_t words = (static_cast<int64_t>(overflow ? cap : total_pairs) + 31) / 32;
    uint32_t* valid = at<uint32_t>(ws, L.pair_valid);
    for (int64_t i = words * b / L.n_proj_groups + threadIdx.x; i < words * (b + 1) / L.n_proj_groups; i += kEmitThreads)
      valid[i] = 0;
  }
  // rank bases of the block's live-mask words (warps 0-1: up to 64 words)
  if (threadIdx.x < 64) {
    const int64_t w = first / 32 + threadIdx.x;
    const bool in = threadIdx.x < L.proj_items / 32 && w < (L.KN + 31) / 32;
    const uint32_t c = in ? __popc(at<uint32_t>(ws, L.live_mask)[w]) : 0u;
    int total;
    const uint32_t excl = static_cast<uint32_t>(warp_exclusive_scan(static_cast<int>(c), total));
    if (threadIdx.x == 0) s_w0 = static_cast<uint32_t>(total);
    asm volatile("bar.sync 1, 64;" ::: "memory");  // the two warps of the mask words
    if (in) at<uint32_t>(ws, L.live_wpre)[w] = base + excl + (threadIdx.x >= 32 ? s_w0 : 0u);
  }
  const int64_t per_view = static_cast<int64_t>(L.Tx) * L.Ty;
  uint32_t* cursor = at<uint32_t>(ws, L.tile_cursor) + (b & (kTileSubLists - 1)) * L.n_tiles * kCursorStride;
  uint4* rec = at<uint4>(ws, L.pair_grads);
  int buf = 0;  // (s_cnt[1] is read before the first round's barrier, written after it)
  for (uint32_t j0 = 0; j0 < cnt; j0 += kEmitThreads, buf ^= 1) {
    // an equal share of the round's items for every warp
    const uint32_t share = (min(cnt - j0, static_cast<uint32_t>(kEmitThreads)) + kWarps - 1) / kWarps;
    const uint32_t j = j0 + wib * share + lane;
    const bool valid = lane < static_cast<int>(share) && j < cnt;
    Ellipse E{};
    uint4 meta = make_uint4(0, 0, 0, 0);
    const uint32_t n = valid ? at<uint32_t>(ws, L.sorted_counts)[first + j] : 0u;
    const bool live = n > 0;
    if (live) {
      const float4 a = at<float4>(ws, L.stage_ell)[2 * (first + j)], c = at<float4>(ws, L.stage_ell)[2 * (first + j) + 1];
      E = Ellipse{a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
      meta = at<uint4>(ws, L.stage_meta)[first + j];
    }
    int wtotal;
    const uint32_t excl = static_cast<uint32_t>(warp_exclusive_scan(static_cast<int>(n), wtotal));
    const uint32_t lives = __ballot_sync(0xffffffffu, live), rank = __popc(lives & ((1u << lane) - 1u));
    if (lane == 0) {
      s_cnt[buf][wib] = static_cast<uint32_t>(wtotal);
      s_lv[buf][wib] = __popc(lives);
    }
    __syncthreads();
    uint64_t wbase = pairs;  // the warp's first pair and first live item
    uint32_t lbase = base;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = s_cnt[buf][w], l = s_lv[buf][w];
      wbase += w < wib ? c : 0u;
      lbase += w < wib ? l : 0u;
      pairs += c;
      base += l;
    }
    uint32_t g = 0, tile0 = 0;
    if (live) {
      const uint64_t off = wbase + excl;
      at<uint32_t>(ws, L.live_kg)[lbase + rank] = meta.y;
      at<uint32_t>(ws, L.live_count)[lbase + rank] = n;
      at<uint32_t>(ws, L.live_off)[lbase + rank] = static_cast<uint32_t>(off < cap ? off : cap);
      const uint32_t k = meta.y / static_cast<uint32_t>(L.N);
      g = meta.y - k * static_cast<uint32_t>(L.N);
      tile0 = static_cast<uint32_t>(k * per_view);
    }
    if (overflow) continue;
    const int x0 = static_cast<int>(meta.z & 0xffffu), x1 = static_cast<int>(meta.z >> 16);
    int2 rows = make_int2(0, 0);
    if (live) rows = ellipse_rows(E, static_cast<int>(meta.w & 0xffffu), static_cast<int>(meta.w >> 16));
    int nrows;
    const int rst = warp_exclusive_scan(rows.y - rows.x, nrows);
    const bool any_rows = rows.y > rows.x;  // (every live item has rows)
    if (any_rows) s_item[wib][rank] = static_cast<uint8_t>(lane);
    __syncwarp();
    uint32_t slot0 = static_cast<uint32_t>(wbase);  // first pair of the next 32 rows (total <= cap < 2^30)
    for (int rb = 0; rb < nrows; rb += 32) {
      const int r = rb + lane;
      const int o = s_item[wib][warp_owner_rank(rst, any_rows, rb)];
      const Ellipse eo = shfl_ellipse(E, o);
      const int ox0 = __shfl_sync(0xffffffffu, x0, o), ox1 = __shfl_sync(0xffffffffu, x1, o);
      const int ty = __shfl_sync(0xffffffffu, rows.x, o) + (r - __shfl_sync(0xffffffffu, rst, o));
      const uint32_t row_depth = __shfl_sync(0xffffffffu, meta.x, o), row_g = __shfl_sync(0xffffffffu, g, o);
      const uint32_t row_tile0 = __shfl_sync(0xffffffffu, tile0, o);
      int len = 0;
      uint32_t tile = 0;
      if (r < nrows) {
        const int2 sp = row_span(eo, ty, ox0, ox1);
        len = sp.x <= sp.y ? sp.y - sp.x + 1 : 0;
        tile = row_tile0 + static_cast<uint32_t>(ty * L.Tx + sp.x);
      }
      int total;
      const int pst = warp_exclusive_scan(len, total);
      // the rows with tiles, in order (all of them but for gaps between tiles' pixel centres)
      const uint32_t full = __ballot_sync(0xffffffffu, len > 0);
      if (len > 0) s_row[wib][__popc(full & ((1u << lane) - 1u))] = static_cast<uint8_t>(lane);
      __syncwarp();
      for (int pb = 0; pb < total; pb += 128) {
        uint32_t pos[4], dep[4], gid[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int p = pb + 32 * q + lane;
          pos[q] = 0xffffffffu;
          if (pb + 32 * q >= total) continue;  // (warp-uniform)
          const int ro = s_row[wib][warp_owner_rank(pst, len > 0, pb + 32 * q)];
          const size_t t = __shfl_sync(0xffffffffu, tile, ro) + static_cast<uint32_t>(p - __shfl_sync(0xffffffffu, pst, ro));
          dep[q] = __shfl_sync(0xffffffffu, row_depth, ro);
          gid[q] = __shfl_sync(0xffffffffu, row_g, ro);
          if (p < total && GS_INDEX_OK(t < static_cast<uint64_t>(L.n_tiles), &st->err))
            pos[q] = atomicAdd(&cursor[t * kCursorStride], 1u);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (pos[q] == 0xffffffffu) continue;
          if (!GS_INDEX_OK(pos[q] < cap, &st->err)) continue;
          rec[pos[q]] = make_uint4(dep[q], slot0 + static_cast<uint32_t>(pb + 32 * q + lane), gid[q], 0u);
        }
      }
      slot0 += static_cast<uint32_t>(total);
      __syncwarp();  // s_row is read before the next 32 rows overwrite it
    }
  }
  pdl_trigger();
}

// Working arrays of one list's sort, in shared memory: keys, their Gaussian ids (first the digits that
// the buckets are taken from), the buckets' counts / ends (two 16-bit buckets per word).
struct SortArrays {
  uint64_t* key;
  uint32_t* gid;
  uint32_t* fine;
};
// Words of the bucket counts of n pairs: at most n + kSlices buckets.
__host__ __device__ constexpr uint32_t bucket_words(uint32_t n) { return (n + kSlices + 1) / 2; }
struct SortShared {
  uint32_t slice[kSlices];     // pairs of each slice, then its first bucket << 5 | bucket bits
  uint32_t warp[3][32];
  uint32_t n_fine, max_bucket;
};

// One more pair in bucket f; returns the bucket's count before.
__device__ __forceinline__ uint32_t bucket_add(uint32_t* fine, uint32_t f) {
  const uint32_t sh = 16 * (f & 1u);
  return (atomicAdd(&fine[f >> 1], 1u << sh) >> sh) & 0xffffu;
}
__device__ __forceinline__ uint32_t bucket_get(const uint32_t* fine, uint32_t f) {
  return reinterpret_cast<const uint16_t*>(fine)[f];
}

// Exclusive prefix of x over the block's threads; *total: the block's sum. tmp: 32 words, not
// written by anyone else before the next barrier.
template <int THREADS>
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t* tmp, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int wtotal;
  const uint32_t excl = static_cast<uint32_t>(warp_exclusive_scan(static_cast<int>(x), wtotal));
  if (lane == 0) tmp[warp] = static_cast<uint32_t>(wtotal);
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) {
    const uint32_t c = tmp[w];
    before += w < warp ? c : 0u;
    all += c;
  }
  *total = all;
  return before + excl;
}

// The digits of a record that its bucket is taken from, their least and largest, and all of them in A.gid.
struct DigitRange {
  uint32_t lo, hi;
};
template <int THREADS, bool SLOTS>
__device__ __forceinline__ DigitRange list_digits(const uint4* rec, uint32_t n, SortArrays A, SortShared& S) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t lo = 0xffffffffu, hi = 0;
  for (uint32_t i = t; i < n; i += THREADS) {
    const uint32_t d = SLOTS ? rec[i].y : rec[i].x;
    A.gid[i] = d;
    lo = min(lo, d);
    hi = max(hi, d);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    S.warp[0][warp] = lo;
    S.warp[1][warp] = hi;
  }
  if (t < kSlices) S.slice[t] = 0;
  if (t == 0) S.max_bucket = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) {
    lo = min(lo, S.warp[0][w]);
    hi = max(hi, S.warp[1][w]);
  }
  return {lo, hi};
}

// Sorts the n records rec[0, n) of tile `tile` by their digits (the depths, or with SLOTS the slots); writes
// keys_out[i] = (tile << 32) | Gaussian id and vals_out[i] = slot. All threads of the block call it.
template <int THREADS, bool SLOTS>
__device__ __forceinline__ void sort_digits(const uint4* rec, uint32_t n, DigitRange range, SortArrays A, SortShared& S,
                                            uint64_t tile, uint64_t* __restrict__ keys_out,
                                            uint32_t* __restrict__ vals_out) {
  const int t = threadIdx.x, lane = t & 31;
  const uint32_t lo = range.lo, hi = range.hi;
  const int bits = 32 - __clz(hi - lo), shift = bits > 8 ? bits - 8 : 0;
  // pairs per slice, buckets per slice
  for (uint32_t i = t; i < n; i += THREADS) atomicAdd(&S.slice[(A.gid[i] - lo) >> shift], 1u);
  __syncthreads();
  uint32_t fbits = 0, nf = 0;
  if (t < kSlices) {
    const uint32_t c = S.slice[t];
    fbits = c > 1 ? min(shift, 31 - __clz(c)) : 0;
    nf = 1u << fbits;
  }
  uint32_t n_fine;
  const uint32_t f0 = block_scan<THREADS>(nf, S.warp[2], &n_fine);
  if (t < kSlices) S.slice[t] = (f0 << 5) | fbits;
  const uint32_t words = (n_fine + 1) / 2;
  for (uint32_t i = t; i < words; i += THREADS) A.fine[i] = 0;
  __syncthreads();
  const uint32_t rest = (1u << shift) - 1u;  // (shift <= 24)
  auto bucket = [&](uint32_t d) {
    const uint32_t s = S.slice[(d - lo) >> shift];
    return (s >> 5) + (((d - lo) & rest) >> (shift - (s & 31u)));
  };
  for (uint32_t i = t; i < n; i += THREADS) bucket_add(A.fine, bucket(A.gid[i]));
  __syncthreads();
  // exclusive prefix of the bucket counts (a run of consecutive words per thread)
  {
    const uint32_t per = ((words + THREADS - 1) / THREADS) | 1u;  // odd: the runs start in different banks
    const uint32_t i0 = min(t * per, words), i1 = min(i0 + per, words);
    uint32_t sum = 0, most = 0;
    for (uint32_t i = i0; i < i1; ++i) {
      const uint32_t c0 = A.fine[i] & 0xffffu, c1 = A.fine[i] >> 16;
      sum += c0 + c1;
      most = max(most, max(c0, c1));
    }
    uint32_t all;
    uint32_t at0 = block_scan<THREADS>(sum, S.warp[0], &all);
    for (uint32_t i = i0; i < i1; ++i) {
      const uint32_t c0 = A.fine[i] & 0xffffu, c1 = A.fine[i] >> 16;
      A.fine[i] = at0 | ((at0 + c0) << 16);
      at0 += c0 + c1;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0 && most > kMaxBucket) S.max_bucket = most;  // (any of them: only whether there is one)
  }
  __syncthreads();
  // into the buckets; afterwards fine[f] is bucket f's end
  for (uint32_t i = t; i < n; i += THREADS) {
    const uint4 r = rec[i];
    const uint32_t pos = bucket_add(A.fine, bucket(SLOTS ? r.y : r.x));
    A.key[pos] = (static_cast<uint64_t>(r.x) << 32) | r.y;
    A.gid[pos] = r.z;
  }
  __syncthreads();
  const uint64_t hi_word = tile << 32;
  if (S.max_bucket == 0) {
    for (uint32_t i = t; i < n; i += THREADS) {
      const uint64_t key = A.key[i];
      const uint32_t f = bucket(static_cast<uint32_t>(SLOTS ? key : key >> 32));
      const uint32_t s = f ? bucket_get(A.fine, f - 1) : 0u, e = bucket_get(A.fine, f);
      uint32_t rank = s;
      for (uint32_t j = s; j < e; ++j) rank += A.key[j] < key ? 1u : 0u;
      keys_out[rank] = hi_word | A.gid[i];
      vals_out[rank] = static_cast<uint32_t>(key);
    }
    return;
  }
  // bitonic network over the next power of two (absent keys compare as the largest)
  const int levels = 32 - __clz(n - 1);  // (n > kMaxBucket here)
  for (int k = 0; k < levels; ++k) {
    for (int j = k; j >= 0; --j) {
      for (uint32_t q = t; q < 1u << (levels - 1); q += THREADS) {
        // the first step of a merge compares mirrored positions, so every comparison is ascending
        const uint32_t r = q & ((1u << j) - 1u), a = ((q >> j) << (j + 1)) + r;
        const uint32_t c = j == k ? a + (2u << j) - 1u - 2u * r : a + (1u << j);
        if (c < n) {
          const uint64_t ka = A.key[a], kc = A.key[c];
          if (kc < ka) {
            A.key[a] = kc;
            A.key[c] = ka;
            const uint32_t ga = A.gid[a];
            A.gid[a] = A.gid[c];
            A.gid[c] = ga;
          }
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t i = t; i < n; i += THREADS) {
    keys_out[i] = hi_word | A.gid[i];
    vals_out[i] = static_cast<uint32_t>(A.key[i]);
  }
}

// (A call of its own: with both digits in one loop the common lists took 1 to 2 us longer.)
template <int THREADS>
__device__ __noinline__ void sort_by_slot(const uint4* rec, uint32_t n, SortArrays A, SortShared& S, uint64_t tile,
                                          uint64_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out) {
  const DigitRange slots = list_digits<THREADS, true>(rec, n, A, S);
  sort_digits<THREADS, true>(rec, n, slots, A, S, tile, keys_out, vals_out);
}

// Sorts the n records rec[0, n): by depth, or by slot where all depths are equal.
template <int THREADS>
__device__ __forceinline__ void sort_list(const uint4* rec, uint32_t n, SortArrays A, SortShared& S, uint64_t tile,
                                          uint64_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out) {
  const DigitRange depths = list_digits<THREADS, false>(rec, n, A, S);
  if (depths.lo != depths.hi) {
    sort_digits<THREADS, false>(rec, n, depths, A, S, tile, keys_out, vals_out);
  } else {
    __syncthreads();  // the warps' ranges are read
    sort_by_slot<THREADS>(rec, n, A, S, tile, keys_out, vals_out);
  }
}

template <int CAP>
struct ListSmem {
  uint64_t key[CAP];
  uint32_t gid[CAP];
  uint32_t fine[bucket_words(CAP)];
  SortShared S;
};

__global__ void __launch_bounds__(kShortThreads) k_tile_sort(Layout L, uint8_t* __restrict__ ws, int64_t tile0) {
  pdl_wait();
  extern __shared__ __align__(16) uint8_t smem_raw[];
  ListSmem<kTileSortShort>& M = *reinterpret_cast<ListSmem<kTileSortShort>*>(smem_raw);
  const int64_t tile = tile0 + blockIdx.x;
  const uint2 rg = at<uint2>(ws, L.ranges)[tile];
  const uint32_t n = rg.y - rg.x;
  if (n > 0 && n <= static_cast<uint32_t>(kTileSortShort))
    sort_list<kShortThreads>(at<uint4>(ws, L.pair_grads) + rg.x, n, SortArrays{M.key, M.gid, M.fine}, M.S,
                                    static_cast<uint64_t>(tile), at<uint64_t>(ws, L.keys[0]) + rg.x,
                                    at<uint32_t>(ws, L.vals[0]) + rg.x);
  pdl_trigger();
}

// The lists longer than kTileSortShort, taken from the tile scan's list by a grid of resident blocks.
// A list of more than kLongShared pairs is first cut: its records go to the other record buffer in the order
// of kLongSlices equal slices of its depth range, and runs of slices that fit are sorted in shared memory
// one after another. A slice that does not fit (a wall among scattered depths) is cut again on its own, from
// that buffer to the first. A segment of fewer different depths than slices is cut by depths and slots
// written as one number, ((depth - least depth) << slot bits) | (slot - least slot). Either range loses 11
// bits each time, so no list is cut more than seven times (32 and 30 bits). The record buffers are the 16
// bytes per pair of pair_grads from byte 0 and from byte 16 capacity on; the third 16 bytes hold the slices
// still to be cut. Projection and binning of 12,000 pairs of one tile, and of 200,000 by one block (the many of
// run_tasks take 134 to 225), us: all depths equal 78 and 742 (932 and 18,311 when such slices went through a
// network of compare-exchanges in global memory), half of them equal 110 and 1003 (484 and 8954), all different
// 82 and 784.
struct LongSmem {
  ListSmem<kLongShared> list;
  uint32_t slice[kLongSlices];
  uint32_t lo[2][kLongThreads / 32], hi[2][kLongThreads / 32];
  uint4 task;
  uint32_t word;  // one value for the whole block
};
struct Segment {  // records [start, start + n) of buffer src
  uint32_t start, n, src;
};
constexpr int kSliceBits = 11;
static_assert(kLongSlices == 1 << kSliceBits, "slices of a power-of-two width");

// Least and largest word `w` (0 depth, 1 slot) of the records.
__device__ __forceinline__ DigitRange word_range(const uint4* rec, uint32_t n, int w, LongSmem& M) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t lo = 0xffffffffu, hi = 0;
  for (uint32_t j = t; j < n; j += kLongThreads) {
    const uint32_t d = reinterpret_cast<const uint32_t*>(&rec[j])[w];
    lo = min(lo, d);
    hi = max(hi, d);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    M.lo[w][warp] = lo;
    M.hi[w][warp] = hi;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < kLongThreads / 32; ++v) {
    lo = min(lo, M.lo[w][v]);
    hi = max(hi, M.hi[w][v]);
  }
  return {lo, hi};
}

// The slice of a record: of its depth, or of depth and slot as one number.
struct Slicing {
  uint32_t depth0, slot0;
  int slot_bits, shift;
  __device__ __forceinline__ uint32_t operator()(const uint4& r) const {
    uint64_t v = static_cast<uint64_t>(r.x - depth0) << slot_bits;
    if (slot_bits) v |= r.y - slot0;
    return static_cast<uint32_t>(v >> shift);
  }
};
__device__ __forceinline__ int depth_bits(DigitRange d) { return 32 - __clz(d.hi - d.lo); }
__device__ __forceinline__ Slicing depth_slices(DigitRange d) { return {d.lo, 0u, 0, depth_bits(d) - kSliceBits}; }
__device__ __forceinline__ Slicing depth_slot_slices(DigitRange d, DigitRange s) {
  const int sbits = 32 - __clz(s.hi - s.lo);
  return {d.lo, s.lo, sbits, max(depth_bits(d) + sbits - kSliceBits, 0)};
}

// Exclusive prefix of M.slice.
__device__ __forceinline__ void scan_slices(LongSmem& M) {
  constexpr int kPer = kLongSlices / kLongThreads;
  const int t = threadIdx.x;
  uint32_t c[kPer], sum = 0, all;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    c[q] = M.slice[t * kPer + q];
    sum += c[q];
  }
  uint32_t at0 = block_scan<kLongThreads>(sum, M.list.S.warp[0], &all);
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    M.slice[t * kPer + q] = at0;
    at0 += c[q];
  }
}
__device__ __forceinline__ void clear_slices(LongSmem& M) {
  for (int s = threadIdx.x; s < kLongSlices; s += kLongThreads) M.slice[s] = 0;
}

// Moves the n records to `cut` in the order of their slices; M.slice (zero before) then holds the slices' ends.
template <class Slice>
__device__ __forceinline__ void cut_by(const uint4* rec, uint4* cut, uint32_t n, LongSmem& M, Slice slice) {
  const int t = threadIdx.x;
  for (uint32_t j = t; j < n; j += kLongThreads) atomicAdd(&M.slice[slice(rec[j])], 1u);
  __syncthreads();
  scan_slices(M);
  __syncthreads();
  for (uint32_t j = t; j < n; j += kLongThreads) {
    const uint4 r = rec[j];
    cut[atomicAdd(&M.slice[slice(r)], 1u)] = r;
  }
  __syncthreads();
}
__device__ __forceinline__ void cut_segment(const uint4* rec, uint4* cut, uint32_t n, LongSmem& M) {
  clear_slices(M);
  const DigitRange d = word_range(rec, n, 0, M);
  if (depth_bits(d) >= kSliceBits) {
    const int shift = depth_bits(d) - kSliceBits;  // (written out: it is the common one)
    cut_by(rec, cut, n, M, [=](const uint4& r) { return (r.x - d.lo) >> shift; });
  } else {
    cut_by(rec, cut, n, M, depth_slot_slices(d, word_range(rec, n, 1, M)));
  }
}

// Sorts the segment of `tile`'s list by the whole block.
__device__ __forceinline__ void sort_segment(const Layout& L, uint8_t* __restrict__ ws, uint32_t tile, Segment seg,
                                             LongSmem& M) {
  uint4* const buf = at<uint4>(ws, L.pair_grads);
  uint4* const left = buf + 2 * L.cap + seg.start;  // the slices still to be cut
  const SortArrays shared{M.list.key, M.list.gid, M.list.fine};
  auto in_shared = [&](uint32_t src, uint32_t start, uint32_t n) {
    sort_list<kLongThreads>(buf + src * L.cap + start, n, shared, M.list.S, tile, at<uint64_t>(ws, L.keys[0]) + start,
                            at<uint32_t>(ws, L.vals[0]) + start);
    __syncthreads();  // the next piece reuses the arrays
  };
  if (seg.n <= static_cast<uint32_t>(kLongShared)) {
    in_shared(seg.src, seg.start, seg.n);
    return;
  }
  for (int n_left = 0;;) {
    const uint32_t other = seg.src ^ 1u;
    cut_segment(buf + seg.src * L.cap + seg.start, buf + other * L.cap + seg.start, seg.n, M);
    uint32_t start = 0;
    for (int s0 = 0; s0 < kLongSlices && start < seg.n;) {
      int a = s0, b = kLongSlices;  // the most slices [s0, a) whose records fit
      while (a < b) {
        const int mid = (a + b + 1) / 2;
        if (M.slice[mid - 1] - start <= static_cast<uint32_t>(kLongShared)) a = mid; else b = mid - 1;
      }
      const bool fits = a > s0;
      a = fits ? a : s0 + 1;
      const uint32_t m = M.slice[a - 1] - start;
      if (fits && m > 0) in_shared(other, seg.start + start, m);
      if (!fits) {
        if (threadIdx.x == 0) left[n_left] = make_uint4(seg.start + start, m, other, 0u);
        ++n_left;
      }
      start += m;
      s0 = a;
    }
    __syncthreads();  // the last slices and the list of those left are read and written
    if (n_left == 0) return;
    const uint4 next = left[--n_left];
    seg = Segment{next.x, next.y, next.z};
  }
}

// Segments of more than kTileSortGiant records (a map seen from afar, all of it in a few tiles) are cut by many
// blocks: in chunks of kChunk records they take the ranges, count the slices and move the records, one phase
// after the other, and what comes out are segments again. All of it goes through one list of tasks that the
// blocks take in turn. The last block to finish a phase gives out the next one's tasks, so no block waits for
// work that another has yet to start, whichever of them are resident; a block without a task waits until there
// is one or none is left. Tasks: per level 3 n / kChunk + 3 chunks and 2 (2 n / kLongShared + 1) segments of a
// segment of n > kTileSortGiant, at most 0.0022 n, and at most seven levels: less than capacity / 32.
// Projection and binning, us, by one block per list / by many (by the global radix sorts): all pairs in one tile
// 50k 222 / 97 (81), 200k 784 / 135 (119), 800k 3147 / 284 (227), 2M 8113 / 627 (435; the cursors' atomics are
// 0.3 ms of it); 2M in 16 tiles 829 / 348 (483). Lists of 16k are as fast either way: 64 of them 215 / 223,
// one of 12k 80 / 83; chunks of 8192 records 90 and 229.
constexpr int kChunk = 4096;
constexpr int kPieceStep = kLongShared / 2;
enum TaskKind : uint32_t { kNoTask, kSegmentTask, kRangeTask, kCountTask, kMoveTask };
// A task: kind | source buffer << 8, tile, the segment's start, its records (kSegmentTask) or the chunk's number.
__device__ __forceinline__ uint4 make_task(TaskKind kind, uint32_t src, uint32_t tile, uint32_t start, uint32_t n) {
  return make_uint4(kind | src << 8, tile, start, n);
}
// What the blocks that cut a giant segment share, in the third record buffer from the segment's start on.
struct Giant {
  uint32_t n, lo[2], hi[2], done[3];
  uint32_t slice[kLongSlices];
};
static_assert(sizeof(Giant) <= 16 * kTileSortGiant, "fits in the segment's part of the third buffer");

__device__ __forceinline__ uint32_t load_relaxed(const uint32_t* p) { return *const_cast<const volatile uint32_t*>(p); }

// Gives out the threads' tasks (at most two each, the first n of own). All threads of the block call it; what they
// wrote before is seen by whoever takes a task. A task's first word, its kind, is written last and by itself.
__device__ __forceinline__ void give_out(const Layout& L, uint8_t* __restrict__ ws, const uint4 (&own)[2], uint32_t n,
                                         LongSmem& M) {
  Status* st = at<Status>(ws, L.status);
  uint32_t total;
  const uint32_t mine = block_scan<kLongThreads>(n, M.list.S.warp[1], &total);
  __threadfence();
  if (threadIdx.x == 0) {
    atomicAdd(&st->task_left, static_cast<int32_t>(total));
    M.word = atomicAdd(&st->task_end, total);
  }
  __syncthreads();
  const uint32_t first = M.word + mine;
  if (n && first + n <= task_bound(L, st->total_pairs)) {
    uint4* task = at<uint4>(ws, L.tasks) + first;
    for (uint32_t i = 0; i < n; ++i) {
      task[i].y = own[i].y;
      task[i].z = own[i].z;
      task[i].w = own[i].w;
    }
    __threadfence();
    for (uint32_t i = 0; i < n; ++i) *const_cast<volatile uint32_t*>(&task[i].x) = own[i].x;
  } else if (n) {  // (never, by the bound; whoever waits for it gives up too)
    atomicOr(&st->err, GS_DEVERR_TIMEOUT);
  }
  __syncthreads();
}
__device__ __forceinline__ void give_out_chunks(const Layout& L, uint8_t* __restrict__ ws, TaskKind kind, uint32_t src,
                                                uint32_t tile, uint32_t start, uint32_t n, LongSmem& M) {
  const uint32_t chunks = (n + kChunk - 1) / kChunk;
  for (uint32_t c0 = 0; c0 < chunks; c0 += kLongThreads) {
    const uint32_t c = c0 + threadIdx.x;
    const uint4 own[2] = {make_task(kind, src, tile, start, c), make_uint4(0, 0, 0, 0)};
    give_out(L, ws, own, c < chunks ? 1u : 0u, M);
  }
}

// Whether this block is the last to finish `done`'s phase; it then sees what the others wrote.
__device__ __forceinline__ bool last_of(uint32_t* done, uint32_t chunks, LongSmem& M) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    M.word = atomicAdd(done, 1u) == chunks - 1 ? 1u : 0u;
    __threadfence();
  }
  __syncthreads();
  const bool last = M.word != 0;
  __syncthreads();
  return last;
}

__device__ __forceinline__ void run_task(const Layout& L, uint8_t* __restrict__ ws, uint4 task, LongSmem& M) {
  const int t = threadIdx.x;
  const uint32_t kind = task.x & 0xffu, src = task.x >> 8, tile = task.y, start = task.z;
  uint4* const buf = at<uint4>(ws, L.pair_grads);
  Giant* const G = reinterpret_cast<Giant*>(buf + 2 * L.cap + start);
  if (kind == kSegmentTask) {
    const uint32_t n = task.w;
    if (n <= static_cast<uint32_t>(kTileSortGiant)) {
      sort_segment(L, ws, tile, Segment{start, n, src}, M);
      return;
    }
    for (int s = t; s < kLongSlices; s += kLongThreads) G->slice[s] = 0;
    if (t < 3) G->done[t] = 0;
    if (t < 2) {
      G->lo[t] = 0xffffffffu;
      G->hi[t] = 0;
    }
    if (t == 0) G->n = n;
    give_out_chunks(L, ws, kRangeTask, src, tile, start, n, M);
    return;
  }
  const uint32_t n = __ldcg(&G->n), chunks = (n + kChunk - 1) / kChunk, first = task.w * kChunk;
  const uint32_t m = min(n - first, static_cast<uint32_t>(kChunk));
  const uint4* rec = buf + src * L.cap + start + first;
  if (kind == kRangeTask) {
    for (int w = 0; w < 2; ++w) {
      const DigitRange r = word_range(rec, m, w, M);
      if (t == 0) {
        atomicMin(&G->lo[w], r.lo);
        atomicMax(&G->hi[w], r.hi);
      }
    }
    if (last_of(&G->done[0], chunks, M)) give_out_chunks(L, ws, kCountTask, src, tile, start, n, M);
    return;
  }
  const DigitRange d{__ldcg(&G->lo[0]), __ldcg(&G->hi[0])};
  const Slicing slice = depth_bits(d) >= kSliceBits ? depth_slices(d)
                                                    : depth_slot_slices(d, DigitRange{__ldcg(&G->lo[1]), __ldcg(&G->hi[1])});
  clear_slices(M);
  __syncthreads();
  for (uint32_t j = t; j < m; j += kLongThreads) atomicAdd(&M.slice[slice(rec[j])], 1u);
  __syncthreads();
  if (kind == kCountTask) {
    for (int s = t; s < kLongSlices; s += kLongThreads)
      if (M.slice[s]) atomicAdd(&G->slice[s], M.slice[s]);
    if (!last_of(&G->done[1], chunks, M)) return;
    for (int s = t; s < kLongSlices; s += kLongThreads) M.slice[s] = __ldcg(&G->slice[s]);
    __syncthreads();
    scan_slices(M);
    __syncthreads();
    for (int s = t; s < kLongSlices; s += kLongThreads) G->slice[s] = M.slice[s];
    give_out_chunks(L, ws, kMoveTask, src, tile, start, n, M);
    return;
  }
  // kMoveTask: places for the chunk's records of each slice, then the records
  uint4* cut = buf + (src ^ 1u) * L.cap + start;
  for (int s = t; s < kLongSlices; s += kLongThreads)
    if (M.slice[s]) M.slice[s] = atomicAdd(&G->slice[s], M.slice[s]);
  __syncthreads();
  for (uint32_t j = t; j < m; j += kLongThreads) {
    const uint4 r = rec[j];
    cut[atomicAdd(&M.slice[slice(r)], 1u)] = r;
  }
  if (!last_of(&G->done[2], chunks, M)) return;
  // the slices' ends; piece j is the run of slices that begin in [j, j + 1) kPieceStep, its last slice on its own
  // when the run does not fit in shared memory
  for (int s = t; s < kLongSlices; s += kLongThreads) M.slice[s] = __ldcg(&G->slice[s]);
  __syncthreads();
  auto begin = [&](int s) { return s ? M.slice[s - 1] : 0u; };
  auto first_from = [&](uint32_t x) {  // the first slice that begins at x or later, kLongSlices if none does
    int a = 0, b = kLongSlices;
    while (a < b) {
      const int mid = (a + b) / 2;
      if (begin(mid) >= x) b = mid; else a = mid + 1;
    }
    return a;
  };
  for (uint32_t j0 = 0; j0 * kPieceStep < n; j0 += kLongThreads) {
    const uint32_t x = (j0 + t) * kPieceStep;
    uint4 own[2];
    uint32_t n_own = 0;
    if (x < n) {
      const int a = first_from(x), b = first_from(x + kPieceStep);
      const uint32_t p0 = begin(a), p1 = begin(b), last = b > a ? begin(b - 1) : p0;
      const bool fits = p1 - p0 <= static_cast<uint32_t>(kLongShared);
      const uint32_t mid = fits ? p1 : last;
      if (mid > p0) own[n_own++] = make_task(kSegmentTask, src ^ 1u, tile, start + p0, mid - p0);
      if (p1 > mid) own[n_own++] = make_task(kSegmentTask, src ^ 1u, tile, start + mid, p1 - mid);
    }
    give_out(L, ws, own, n_own, M);
  }
}

// The lists as the first tasks, then those given out on the way.
__device__ __noinline__ void run_tasks(const Layout& L, uint8_t* __restrict__ ws, LongSmem& M) {
  Status* st = at<Status>(ws, L.status);
  const uint32_t n_long = st->n_long;
  for (;;) {
    if (threadIdx.x == 0) {
      const uint32_t k = atomicAdd(&st->task_next, 1u);
      uint4 task = make_uint4(kNoTask, 0, 0, 0);
      if (k < n_long) {
        const uint32_t tile = at<uint32_t>(ws, L.long_tiles)[k];
        const uint2 rg = at<uint2>(ws, L.ranges)[tile];
        task = make_task(kSegmentTask, 0, tile, rg.x, rg.y - rg.x);
      } else {
        const uint32_t i = k - n_long;
        const uint4* given = at<uint4>(ws, L.tasks) + i;
        const bool exists = i < task_bound(L, st->total_pairs);
        // (no fence while waiting: it would empty the L1 of the blocks that work on the same multiprocessor)
        for (uint32_t spins = 0;; ++spins) {
          uint32_t x = exists ? load_relaxed(&given->x) : 0u;
          const bool over = !x && n_long + load_relaxed(reinterpret_cast<const uint32_t*>(&st->task_left)) == 0;
          if (over) {  // tasks that were given out before the last one was done are seen now
            __threadfence();
            x = exists ? load_relaxed(&given->x) : 0u;
          }
          if (x) {
            __threadfence();
            task = make_uint4(x, __ldcg(&given->y), __ldcg(&given->z), __ldcg(&given->w));
          }
          if (x || over) break;
          if (spins == kSpinLimit / 4) {
            atomicOr(&st->err, GS_DEVERR_TIMEOUT);
            break;
          }
          __nanosleep(min(100u << min(spins, 4u), 1000u));
        }
      }
      M.task = task;
    }
    __syncthreads();
    const uint4 task = M.task;
    if ((task.x & 0xffu) == kNoTask) return;
    run_task(L, ws, task, M);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(&st->task_left, -1);
  }
}

__global__ void __launch_bounds__(kLongThreads, kLongBlocks) k_tile_sort_long(Layout L, uint8_t* __restrict__ ws) {
  pdl_wait();
  extern __shared__ __align__(16) uint8_t smem_raw[];
  LongSmem& M = *reinterpret_cast<LongSmem*>(smem_raw);
  const Status* st = at<Status>(ws, L.status);
  if (st->giant) {
    run_tasks(L, ws, M);
  } else {
    const uint32_t n_long = st->n_long;
    for (uint32_t i = blockIdx.x; i < n_long; i += gridDim.x) {
      const uint32_t tile = at<uint32_t>(ws, L.long_tiles)[i];
      const uint2 rg = at<uint2>(ws, L.ranges)[tile];
      sort_segment(L, ws, tile, Segment{rg.x, rg.y - rg.x, 0u}, M);
    }
  }
  pdl_trigger();
}
static_assert(kLongShared < 65536, "16-bit bucket counts in shared memory");
static_assert(kPairGradStride * sizeof(float) >= 48, "pair_grads holds both record buffers and the list of slices");

}  // namespace

cudaError_t launch_tile_bin(const Layout& L, void* ws, cudaStream_t s) {
  auto* w = static_cast<uint8_t*>(ws);
  // dynamic shared memory limits, raised once per device (idempotent: threads may race here)
  static bool ready[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!ready[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(ListSmem<kTileSortShort>)));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tile_sort_long, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(sizeof(LongSmem)));
    if (e != cudaSuccess) {
      cudaGetLastError();
      return e;
    }
    ready[dev] = true;
  }
  const cudaError_t e = launch_tile_scan(L, ws, s);
  if (e != cudaSuccess) return e;  // (the emission would write at cursors that nobody set)
  const int64_t sms = device_sms();
  // groups of whole views: a group's emission covers every projection block holding its items
  const int64_t per_view = static_cast<int64_t>(L.Tx) * L.Ty;
  int64_t b0 = 0;
  for (int i = 0; i < L.sort_groups; ++i) {
    const int64_t k0 = static_cast<int64_t>(L.K) * i / L.sort_groups, k1 = static_cast<int64_t>(L.K) * (i + 1) / L.sort_groups;
    const int64_t b1 = i + 1 == L.sort_groups ? L.n_proj_groups : (k1 * L.N + L.proj_items - 1) / L.proj_items;
    if (b1 > b0) launch(k_tile_emit, static_cast<unsigned>(b1 - b0), kEmitThreads, 0, s, L, w, b0);
    b0 = b1;
    launch(k_tile_sort, static_cast<unsigned>((k1 - k0) * per_view), kShortThreads, sizeof(ListSmem<kTileSortShort>), s,
           L, w, k0 * per_view);
  }
  launch(k_tile_sort_long, static_cast<unsigned>(L.n_tiles < kLongBlocks * sms ? L.n_tiles : kLongBlocks * sms), kLongThreads,
         sizeof(LongSmem), s, L, w);
  return cudaGetLastError();
}

}  // namespace gs
