// Internal declarations of the sm_103a rasterizer library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "../../include/gs.h"

namespace gs {

constexpr int kTile = 16;             // tile side (pixels)
constexpr int kTilePixels = kTile * kTile;
constexpr int kProjBlock = 256;       // (view, Gaussian) items per scan chunk of the binning
constexpr int kProjItemsMax = 2048;   // (view, Gaussian) items per projection block: 256 to
                                      // this, a power of two, so that there are >= kProjTargetBlocks
constexpr int kProjTargetBlocks = 1216;
constexpr int kProjThreads = 256;     // threads of a projection block
constexpr int kProjViews = 4;         // views whose cameras a projection block keeps in shared memory
constexpr int kEmitPairs = 1024;      // pairs emitted per emission block
constexpr int kProjGridCells = 6144;  // largest (Tx+1)(Ty+1) difference grid kept in shared memory
constexpr int kSortThreads = 256;     // onesweep block
constexpr int kSortItems = 15;        // keys per thread per onesweep tile (default; 8 also built)
constexpr int kSortTileKeys = kSortThreads * kSortItems;
constexpr int kMaxSortPasses = 8;
constexpr int kPairGradStride = 12;   // floats per pair gradient record (10 used)
constexpr int kPoseBlock = 128;       // Gaussians / live items per projection-backward block
// Tile-sort binning (tile_sort.cu): each tile's list sorted by its own block.
constexpr int kTileSortMinTiles = 152;  // fewer tiles than SMs: the global radix sorts instead
constexpr int kScanRows = 8;            // tile rows per block of the tile scan
constexpr int kTileSubLists = 4;        // cursors per tile: projection block b emits into sub-list b % 4
constexpr int kCursorStride = 8;        // u32 between two cursors: one 32-byte sector each
constexpr int kTileSortMaxDensity = 800;  // Gaussians per tile of a view (see make_layout)
constexpr int64_t kTileSortMaxItems = 1 << 25;  // most Gaussians (so list entries; 27-bit bucket numbers)
constexpr int kTileSortShort = 2048;    // longest list sorted by a short-list block
constexpr int kTileSortGiant = 16384;   // longest list that one block cuts
constexpr int kTileSortGroupItems = 6400000;  // (view, Gaussian) items per emission / sort launch
constexpr uint32_t kSpinLimit = 1u << 21;  // bounded decoupled look-back (about a second of polling)

// Workspace status block (first 256 bytes of the workspace).
struct Status {
  uint32_t err;
  uint32_t num_pairs;       // min(total pairs, capacity)
  uint64_t total_pairs;     // unclamped
  uint64_t evals;           // Gaussian-pixel evaluations of the last forward raster
  uint32_t tile_ctr[kMaxSortPasses];  // onesweep dynamic tile counters: [0,4) item sort, [4,8) pair sort
  uint64_t composited;      // evaluations of the last forward raster that blended a splat
  uint32_t row_ctr;         // entries of the row-span table handed out by the projection
  uint32_t loss_ctr;        // blocks of the loss-fused forward done (reset by the last one)
  uint32_t n_live;          // live items: (view, Gaussian) items that emit at least one pair
  uint32_t view_ctr;        // tile-scan blocks started
  uint32_t proj_done;       // projection blocks finished (the last one scans their live counts)
  uint32_t n_long;          // tiles whose list is longer than kTileSortShort (tile-sort binning)
  uint32_t n_long_next;     // the same while the tile scan counts them
  uint32_t giant;           // whether a list is longer than kTileSortGiant
  uint32_t task_next, task_end;  // the long lists' tasks: taken, given out
  int32_t task_left;        // tasks given out and not done, less the done lists
};
static_assert(sizeof(Status) <= 256, "status block");

// Everything a kernel needs to find its buffers; built on the host from gs_config_t.
struct Layout {
  int64_t N, KN, cap;
  int K, W, H, Tx, Ty;
  int64_t n_tiles;          // K * Tx * Ty
  int tile_bits, key_bits;
  int passes;               // pair-sort passes over the tile bits: ceil(tile_bits / 8)
  int item_sort_items, pair_sort_items;  // keys per thread of the onesweep tiles of the two sorts
  int64_t max_item_tiles;   // onesweep tiles of the per-item depth sort
  float near_plane, lambda_depth;
  int fwd_px, bwd_px;       // pixels per thread of the compositing kernels (0 = default)
  int fwd_chunk, bwd_chunk; // splats staged per chunk of the compositing kernels (0 = default)
  int raster_bps;           // cap on resident compositing blocks per SM (0 = none)
  int color_mode, sh_degree, sh_coeffs;  // gs_color_mode_t; SH degree and (degree + 1)^2
  int64_t color_stride;     // index of (view k, Gaussian g) in color_opacity = k * color_stride + g
  int64_t n_proj_blocks;    // ceil(KN / kProjBlock)
  int64_t n_proj_groups;    // ceil(KN / proj_items): projection blocks
  int proj_items;           // items per projection block
  int64_t max_sort_tiles;   // onesweep tiles of the pair sort at capacity
  int64_t n_pose_blocks;    // ceil(N / kPoseBlock)
  int64_t n_item_chunks;    // ceil(KN / kPoseBlock): chunks of live items of the projection backward
  int64_t n_loss_blocks;
  // byte offsets into the workspace
  size_t status, proj_uv, proj_conic, proj_tiles, proj_depth_key, proj_radius, color_opacity, block_sums,
      block_offsets, keys[2], vals[2], ranges, hist, sort_status, pair_grads, pose_partials, loss_partials;
  // per-item depth sort (u32 depth key, u32 item index), its histograms and look-back status,
  // and the tiles touched by each item in depth order
  size_t item_keys[2], item_vals[2], item_hist, item_status, sorted_counts;
  // in depth order: exclusive pair offset of each item (KN + 1 entries), its row-span
  // table entries (int4: first entry, number of entries, -, -), its (view, Gaussian id)
  size_t item_offsets, item_rect, item_kg;
  // row-span table: per live item, its rows from the first to the last non-empty one, each an
  // int2 (pairs of the item in earlier rows, first column | row << 16). Entries are handed out by
  // an atomic counter; at most pair_capacity of them (more is reported as a pair overflow).
  size_t row_table;
  // one bit per pair slot: set by gs_raster_bwd for every record it writes (pairs in front of
  // every pixel's last contributor of their tile); the other records are never written, their
  // gradient is zero. Cleared by the emission.
  size_t pair_valid;
  size_t tile_loss;         // float [n_tiles]: per-tile loss partials of the loss-fused forward
  // per view a (Ty+1) x (Tx+1) grid: +1 / -1 at the first / one-past-last tile of every
  // emitted row span; its row-wise prefix sum is the number of pairs of each tile (diff_copies
  // grids per view: projection block b adds to copy b % diff_copies)
  size_t tile_diff;
  int diff_copies;          // kTileSubLists with the tile-sort binning, else 1
  int64_t n_emit_blocks;    // ceil(cap / kEmitPairs)
  size_t emit_first, emit_last;  // u32 [n_emit_blocks]: items holding each emission block's first / last pair
  // Live items (those that emit at least one pair) and their compaction. Only live items get
  // projection records (proj_uv, proj_conic, proj_tiles, proj_depth_key, proj_radius);
  // the others are marked dead and nothing reads their records. A live item's position among
  // the live items (in increasing k N + g order) is its rank in live_mask: live_wpre[i / 32] +
  // the set bits of word i / 32 below bit i & 31 (live_rank).
  //   live_mask  u32 [ceil(KN / 32)]: bit (i & 31) of word i / 32 set when item i = k N + g is live
  //   live_wpre  u32 [ceil(KN / 32)]: live items before word i / 32
  //   live_kg    u32 [KN]: the live items in increasing k N + g order (valid prefix n_live)
  //   live_count u32 [KN]: tiles emitted by each of them
  //   live_rows  uint2 [KN]: their row-span table entries (first entry, number of entries)
  //   live_off   u32 [KN]: their first pair index (emission order), clamped to the capacity
  //   live_blocks, live_bases  u32 [n_proj_groups]: live items of each projection block, and (radix sorts)
  //              the block's first position among all live items (scanned by the last block)
  //   view_lb    u64 [K * scan_slabs]: look-back status of the tile scan's blocks
  //   item_partials float [KN][16]: the projection backward's per-live-item partial gradients
  size_t live_mask, live_wpre, live_kg, live_count, live_rows, live_off, live_blocks, live_bases, view_lb,
      item_partials;
  // Tile-sort binning (tile_sort = true): the pairs go straight to their tile's list (atomic
  // cursors) and every list is sorted by (depth, item) on its own; the buffers of the item
  // depth sort, the row-span table and the second key / value buffers are then not allocated.
  //   stage_ell   float4 [KN][2]: ellipse of each live item, in its projection block's segment of
  //              survivors of the cull (surv_blocks u32 [n_proj_groups]: their number)
  //   stage_meta  uint4 [KN]: its depth key, item id, rectangle x0|x1<<16, y0|y1<<16
  //   (every survivor's tiles emitted, 0 when it is not live: sorted_counts)
  //   block_pairs u32 [n_proj_groups], super_pairs u64, super_live u32 [ceil(n_proj_groups / 256)]:
  //              pairs of each projection block's live items; pairs and live items of 256 blocks
  //   tile_cursor u32 [kTileSubLists][n_tiles][kCursorStride]: next free pair of each tile's
  //              sub-lists (entry 0)
  //   long_tiles  u32 [n_tiles]: the tiles with lists longer than kTileSortShort
  //   tasks       uint4 [max_tasks]: what the blocks of k_tile_sort_long give one another to do
  // The unsorted lists are uint4 (depth bits, slot, Gaussian id, -) in the first 16 pair_capacity
  // bytes of pair_grads, which holds nothing before the backward; the rest of it is scratch of
  // the long lists' sorts.
  bool tile_sort;
  int sort_groups;          // launches the views are split over (emission, sort)
  int sorted;               // buffer (keys[], vals[]) holding the sorted pairs
  size_t zero_bytes;        // the buffers from `status` on that start at zero, cleared together
  int scan_slabs;           // blocks per view of the tile scan (kScanRows tile rows each)
  size_t stage_ell, stage_meta, surv_blocks, block_pairs, super_pairs, super_live, tile_cursor, long_tiles, tasks;
  uint32_t max_tasks;
  size_t total;
};

// Decoupled look-back over a sequence of blocks numbered in their start order (Merrill &
// Garland, "Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016), on 64-bit
// status words: the top two bits flag an aggregate (1) or an inclusive prefix (2), the low 62
// bits hold the value; 0 = not published yet. Called by all 32 lanes of one warp of block
// `id`, which first publishes the block's aggregate; the lanes then read kLbWindows * 32
// predecessors per round (independent loads), consume the aggregates in front of the nearest
// inclusive prefix (or in front of the nearest unpublished block, which is read again next
// round), and return to every lane the sum of the
// aggregates of blocks [0, id), after publishing the block's inclusive prefix. The wait for an
// unpublished predecessor is bounded: after kSpinLimit polls without progress it sets
// GS_DEVERR_TIMEOUT in *err and returns what it has.
constexpr uint64_t kLbAggregate = 1ull << 62;
constexpr uint64_t kLbPrefix = 2ull << 62;
constexpr uint64_t kLbValue = (1ull << 62) - 1;
__device__ __forceinline__ uint64_t lb_load(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void lb_store(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
constexpr int kLbWindows = 8;  // 32-block windows read per round (loads in flight together)
__device__ __forceinline__ uint64_t lb_exclusive_warp(uint64_t* status, uint32_t id, uint64_t aggregate,
                                                      uint32_t* err) {
  const int lane = threadIdx.x & 31;
  if (id == 0) {
    if (lane == 0) lb_store(&status[0], kLbPrefix | aggregate);
    return 0;
  }
  if (lane == 0) lb_store(&status[id], kLbAggregate | aggregate);
  uint64_t excl = 0;
  uint32_t spins = 0;
  int64_t j = static_cast<int64_t>(id) - 1;  // window q, lane l: block j - 32 q - l
  bool done = false;
  while (!done) {
    uint64_t v[kLbWindows];
#pragma unroll
    for (int q = 0; q < kLbWindows; ++q) {
      const int64_t jj = j - 32 * q - lane;
      v[q] = jj >= 0 ? lb_load(&status[jj]) : kLbPrefix;  // before block 0: a zero prefix
    }
    int64_t consumed = 0;
#pragma unroll
    for (int q = 0; q < kLbWindows; ++q) {
      if (done) break;
      const uint64_t f = v[q] & ~kLbValue;
      const uint32_t pref = __ballot_sync(0xffffffffu, f == kLbPrefix);
      const uint32_t blocked = __ballot_sync(0xffffffffu, f == 0);
      const int p = pref ? __ffs(pref) - 1 : 32, b = blocked ? __ffs(blocked) - 1 : 32;
      if (p < b) {  // every block in front of the nearest prefix has published: done
        excl += warp_sum_u64(lane <= p ? (v[q] & kLbValue) : 0);
        done = true;
        break;
      }
      excl += warp_sum_u64(lane < b ? (v[q] & kLbValue) : 0);  // the aggregates in front of the gap
      consumed += b;
      if (b < 32) break;  // an unpublished block: read again from it
    }
    if (done) break;
    j -= consumed;
    if (consumed == 0 && ++spins > kSpinLimit) {
      if (lane == 0) atomicOr(err, GS_DEVERR_TIMEOUT);
      break;
    }
  }
  if (lane == 0) lb_store(&status[id], kLbPrefix | (excl + aggregate));
  return excl;
}

// Whether item kg is live (emits pairs); its projection records exist only then.
__device__ __forceinline__ bool item_live(const uint32_t* live_mask, int64_t kg) {
  return (live_mask[kg >> 5] >> (kg & 31)) & 1u;
}
// Position of live item kg among the live items.
__device__ __forceinline__ uint32_t live_rank(const uint32_t* live_mask, const uint32_t* live_wpre, int64_t kg) {
  return live_wpre[kg >> 5] + __popc(live_mask[kg >> 5] & ((1u << (kg & 31)) - 1u));
}

// The lanes of a warp hold consecutive numbers, lane l the numbers [st, next lane's st) (none when !any).
// Returns, for the number r0 + lane, the rank of its owner among the lanes with any (0, 1, ...); r0 and
// the lanes' numbers cover the asked ones. One warp-wide OR and a ballot instead of a binary search
// by shuffles (five dependent ones).
__device__ __forceinline__ int warp_owner_rank(int st, bool any, int r0) {
  const int local = st - r0;
  const uint32_t heads = __reduce_or_sync(0xffffffffu, (any && local > 0 && local < 32) ? 1u << local : 0u);
  const int before = __popc(__ballot_sync(0xffffffffu, any && local <= 0));
  return before - 1 + __popc(heads & (0xffffffffu >> (31 - (threadIdx.x & 31))));
}
__device__ __forceinline__ int warp_exclusive_scan(int x, int& total) {
  const int lane = threadIdx.x & 31;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - x;
}

bool make_layout(const gs_config_t* cfg, Layout* L);

template <class T>
__host__ __device__ inline T* at(void* ws, size_t off) {
  return reinterpret_cast<T*>(static_cast<uint8_t*>(ws) + off);
}
template <class T>
__host__ __device__ inline const T* at(const void* ws, size_t off) {
  return reinterpret_cast<const T*>(static_cast<const uint8_t*>(ws) + off);
}

struct GaussPtrs {
  const void* means;
  const void* log_scales;
  const void* quats;
  const void* logits;
  const void* rgb;
  int dtype, means_dtype;
};

// Debug builds (-DGS_DEBUG) check the data-dependent indices of gathers and scatters: a failed
// check sets GS_DEVERR_BOUNDS in the error word and the access is skipped (no trap). Release
// builds compile the checks away.
#ifdef GS_DEBUG
#define GS_INDEX_OK(cond, err) ((cond) ? true : (atomicOr((err), GS_DEVERR_BOUNDS), false))
#else
#define GS_INDEX_OK(cond, err) true
#endif

// ---------------------------------------------------------------------------- launches
// Programmatic dependent launch: every kernel of the library begins with pdl_begin(), which
// waits until the preceding grid of the stream has completed (its writes are then visible)
// and lets the following grid start launching. Kernels are launched with the programmatic
// stream-serialization attribute, so the launch latency of each kernel overlaps the tail of
// the previous one. Outside such launches the two instructions are no-ops.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// For the long compositing kernels: wait at entry, but let the following grid launch only
// once this block's main loop is done (pdl_trigger), so its blocks do not sit on the SMs for
// the whole kernel.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Dynamic shared memory that caps `kernel` at `bps` resident blocks per multiprocessor (0: no
// cap, none added): the multiprocessor's shared memory divided by bps, less the kernel's static
// shared memory and the per-block reserve, rounded down to 128 bytes (0 when the cap is above
// what fits anyway). Raises the kernel's dynamic shared memory limit when the padding needs it.
template <typename... KArgs>
inline size_t cap_smem(void (*kernel)(KArgs...), int bps) {
  if (bps <= 0) return 0;
  int dev = 0, per_sm = 0, reserve = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserve, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return 0;
  long pad = static_cast<long>(per_sm) / bps - static_cast<long>(fa.sharedSizeBytes) - reserve;
  const long room = static_cast<long>(optin) - static_cast<long>(fa.sharedSizeBytes);
  pad = (pad < room ? pad : room) / 128 * 128;
  if (pad <= 0) return 0;
  if (pad > fa.maxDynamicSharedSizeBytes &&
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pad)) != cudaSuccess)
    return 0;
  return static_cast<size_t>(pad);
}

// ---------------------------------------------------------------------------- device helpers
__device__ __forceinline__ float load_attr(const void* p, int64_t i, int dtype) {
  if (dtype == GS_F32) return static_cast<const float*>(p)[i];
  if (dtype == GS_BF16) return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
  return __half2float(static_cast<const __half*>(p)[i]);
}

// ---------------------------------------------------------------------------- pair culling
// The widened ellipse of a projected Gaussian inside which its opacity can reach 1/255, as
// the discrete projection evaluates it in binary32: E = {d : d^T Sigma2^-1 d <= kap} with
// kap = 2 (ln(255 o) + 0.02 |ln(255 o)| + 1.5e-4), o = 1 / (1 + exp(-logit)). Stored: the
// mean (u, v), Sigma2's off-diagonal b, 1 / c (c: Sigma2's yy entry), sqrt(det Sigma2), the
// half-extents hx = sqrt(kap a), hy = sqrt(kap c), and kxy = b / a (the y offset, per unit
// x offset, of E's leftmost / rightmost points).
struct Ellipse {
  float u, v, b, inv_c, sdet, hx, hy, kxy;
};

// Tile columns [xa, xb] (returned as x, y; xa > xb: none) of tile row ty whose square of
// pixel centres, widened by 0.05 px + 0.2% of the half-extent, meets E; clamped to [x0, x1).
// E's part inside the row's strip is convex, so its x-extent ends at E's leftmost /
// rightmost point when that lies inside the strip, else where E's boundary crosses the
// strip edge on that point's side. Every step is one binary32 rounding in a fixed order,
// so the projection (counts) and the emission (tiles) reproduce each other bit for bit.
__device__ __forceinline__ float ellipse_cross(const Ellipse& E, float Ye, float sgn) {
  const float dye = __fsub_rn(Ye, E.v);
  const float ad = fabsf(dye);
  const float w = __fsqrt_rn(fmaxf(__fmul_rn(__fsub_rn(E.hy, ad), __fadd_rn(E.hy, ad)), 0.0f));
  return __fadd_rn(E.u, __fmul_rn(__fmaf_rn(__fmul_rn(sgn, E.sdet), w, __fmul_rn(E.b, dye)), E.inv_c));
}
__device__ __forceinline__ int2 row_span(const Ellipse& E, int ty, int x0, int x1) {
  const int2 none = make_int2(1, 0);
  const float tf = static_cast<float>(kTile);
  const float mgx = __fmaf_rn(0.002f, E.hx, 0.05f);
  const float mgy = __fmaf_rn(0.002f, E.hy, 0.05f);
  const float y_lo = __fmul_rn(static_cast<float>(ty), tf);
  const float Y0 = __fsub_rn(__fadd_rn(y_lo, 0.5f), mgy);
  const float Y1 = __fadd_rn(__fadd_rn(y_lo, __fsub_rn(tf, 0.5f)), mgy);
  if (__fadd_rn(E.v, E.hy) < Y0 || __fsub_rn(E.v, E.hy) > Y1) return none;
  const float yR = __fmaf_rn(E.kxy, E.hx, E.v);
  const float yL = __fmaf_rn(-E.kxy, E.hx, E.v);
  const float xr = (yR >= Y0 && yR <= Y1) ? __fadd_rn(E.u, E.hx)
                                          : (yR > Y1 ? ellipse_cross(E, Y1, 1.0f) : ellipse_cross(E, Y0, 1.0f));
  const float xl = (yL >= Y0 && yL <= Y1) ? __fsub_rn(E.u, E.hx)
                                          : (yL > Y1 ? ellipse_cross(E, Y1, -1.0f) : ellipse_cross(E, Y0, -1.0f));
  const float inv_t = 1.0f / tf;
  float fa = ceilf(__fmul_rn(__fsub_rn(__fsub_rn(xl, mgx), __fsub_rn(tf, 0.5f)), inv_t));
  float fb = floorf(__fmul_rn(__fsub_rn(__fadd_rn(xr, mgx), 0.5f), inv_t));
  fa = fmaxf(fa, static_cast<float>(x0));
  fb = fminf(fb, static_cast<float>(x1 - 1));
  if (!(fa <= fb)) return none;
  return make_int2(static_cast<int>(fa), static_cast<int>(fb));
}

__device__ __forceinline__ Ellipse shfl_ellipse(const Ellipse& E, int o) {
  Ellipse e;
  e.u = __shfl_sync(0xffffffffu, E.u, o);
  e.v = __shfl_sync(0xffffffffu, E.v, o);
  e.b = __shfl_sync(0xffffffffu, E.b, o);
  e.inv_c = __shfl_sync(0xffffffffu, E.inv_c, o);
  e.sdet = __shfl_sync(0xffffffffu, E.sdet, o);
  e.hx = __shfl_sync(0xffffffffu, E.hx, o);
  e.hy = __shfl_sync(0xffffffffu, E.hy, o);
  e.kxy = __shfl_sync(0xffffffffu, E.kxy, o);
  return e;
}

// The rows of [y0, y1) that can hold a non-empty row_span: those whose widened strip of pixel
// centres meets E's vertical extent, with 0.02 rows + 1e-6 (|v| + hy) of slack for the rounding of
// row_span's own test. A NaN bound leaves its side at the rectangle's edge.
__device__ __forceinline__ int2 ellipse_rows(const Ellipse& E, int y0, int y1) {
  const float mgy = 0.002f * E.hy + 0.05f;
  const float slack = 0.02f + 1e-6f * (fabsf(E.v) + E.hy);
  const float inv_t = 1.0f / static_cast<float>(kTile);
  const float lo = ceilf((E.v - E.hy - mgy - (static_cast<float>(kTile) - 0.5f)) * inv_t - slack);
  const float hi = floorf((E.v + E.hy + mgy - 0.5f) * inv_t + slack);
  const int a = static_cast<int>(fmaxf(lo, static_cast<float>(y0)));
  const int b = static_cast<int>(fminf(hi, static_cast<float>(y1 - 1))) + 1;
  return make_int2(a, b > a ? b : a);
}

// Launchers (each defined in its own translation unit). All return cudaGetLastError().
cudaError_t launch_project(const Layout& L, const GaussPtrs& g, const gs_camera_t* cams, void* ws, cudaStream_t s);
cudaError_t launch_bin(const Layout& L, void* ws, cudaStream_t s);
cudaError_t launch_tile_scan(const Layout& L, void* ws, cudaStream_t s);
cudaError_t launch_tile_bin(const Layout& L, void* ws, cudaStream_t s);  // the tile-sort binning
cudaError_t launch_item_sort(const Layout& L, void* ws, cudaStream_t s);
cudaError_t launch_sort_passes(const Layout& L, void* ws, cudaStream_t s);

struct FusedLossArgs {
  const float* rgb_t;
  const float* depth_t;
  float* g_rgb;
  float* g_depth;
  float* d_loss;
};
cudaError_t launch_raster_fwd(const Layout& L, void* ws, float* rgb, float* depth, float* T_final, int32_t* last,
                              bool stats, const FusedLossArgs* loss, cudaStream_t s, const float* ext_depth = nullptr,
                              const float* ext_rgb = nullptr);
// the loss-fused forward continuing, block by block, into the backward pass (dL_dT = 0)
cudaError_t launch_raster_fwd_l1_bwd(const Layout& L, void* ws, float* rgb, float* depth, float* T_final, int32_t* last,
                                     const FusedLossArgs& loss, cudaStream_t s);
cudaError_t launch_raster_bwd(const Layout& L, void* ws, const float* rgb, const float* depth, const float* T_final,
                              const int32_t* last, const float* dL_drgb, const float* dL_ddepth, const float* dL_dT,
                              cudaStream_t s);
cudaError_t launch_loss(const Layout& L, const float* rgb, const float* depth, const float* rgb_t,
                        const float* depth_t, float* g_rgb, float* g_depth, float* d_loss, void* ws, cudaStream_t s);
cudaError_t launch_project_bwd(const Layout& L, const GaussPtrs& g, const gs_camera_t* cams, void* ws,
                               const gs_grads_t& out, cudaStream_t s);
cudaError_t launch_screen_grads(const Layout& L, const void* ws, float* d_mean2d, float* d_conic, float* d_depth,
                                float* d_opacity, float* d_rgb, cudaStream_t s);

// Generic stable onesweep sort of (key, u32 value) pairs: u64 keys for the (tile, depth) pairs
// and gs_sort_pairs, u32 keys for the per-item depth sort of gs_bin_sort.
template <class KeyT>
struct SortArgsT {
  KeyT* keys[2];
  uint32_t* vals[2];
  const uint32_t* n_dev;  // device pair count (nullptr: use n_host)
  int64_t n_host;         // host pair count or capacity bound
  uint32_t* hist;         // [passes][256] global digit counts (filled before the passes)
  uint32_t* tile_status;  // [passes][max_tiles][256]
  uint32_t* tile_ctr;     // [passes]
  uint32_t* err;
  int64_t max_tiles;
  int passes;
  int key_bits;   // the last pass only looks at the bits below key_bits
  int first_bit;  // pass p sorts on bits [first_bit + 8p, first_bit + 8p + 8)
  const uint64_t* total_dev;  // if set and *total_dev > n_host (capacity overflow), do nothing
  uint32_t first_tile;        // diagnostic: 1 withholds tile 0, so its successors' waits run out
  int items;                  // keys per thread per tile: 8 or 15 (0: kSortItems)
};
__host__ __device__ inline int sort_items(int items) { return (items == 4 || items == 8) ? items : kSortItems; }
// onesweep tiles of n keys at `items` keys per thread
__host__ __device__ inline int64_t sort_tiles(int64_t n, int items) {
  const int64_t tk = static_cast<int64_t>(kSortThreads) * sort_items(items);
  return n > 0 ? (n + tk - 1) / tk : 1;
}
// Keys per thread for a sort of up to n keys: small sorts take short tiles, so that enough
// blocks share the work.
// keys per thread: small sorts take small tiles (more blocks, shorter per-tile latency)
// (gs_sort_pairs also runs in scratch that only longer tiles fit)
constexpr int kSortItemsMid = 8;
inline int pick_sort_items(int64_t n) { return n <= 200000 ? 4 : (n <= 1000000 ? kSortItemsMid : kSortItems); }
// The depth sort of the items has 32-bit keys and four passes: long tiles from 600k items on. Binning by the radix
// sorts, us with 8 / 15 keys per thread for the items: 700k 126.2 / 128.0, 800k 138.7 / 134.1, 850k 148.2 / 142.3,
// 990k 163.8 / 153.3 (the pairs' sort as above: 8 keys for 868k pairs 117.8, 15 keys 118.5).
inline int pick_item_sort_items(int64_t n) { return n <= 200000 ? 4 : (n <= 600000 ? kSortItemsMid : kSortItems); }
using SortArgs = SortArgsT<uint64_t>;
using SortArgs32 = SortArgsT<uint32_t>;
cudaError_t launch_onesweep(const SortArgs& a, cudaStream_t s);
cudaError_t launch_onesweep(const SortArgs32& a, cudaStream_t s);
cudaError_t launch_sort_prepare(const SortArgs& a, cudaStream_t s);  // zero status, build histogram
int bin_sort_launch_count(const Layout& L);  // kernels one gs_bin_sort launches
int device_sms();  // multiprocessors of the current device (cached per device)

}  // namespace gs
