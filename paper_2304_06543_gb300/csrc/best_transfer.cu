// Best-transfer table from scratch: the data-parallel replacement of the
// paper's Gamma-DS heap maintenance (Section 3.4 "Allotment subspace
// multi-graph implementation", Section 3.5.2), which took 74% of ASRAL's time
// in the paper's measurements (Section 5).
//
//   T[u][v] = lexmin over d with assign[d] == u of (CM(d,v) - CM(d,u), d)
//
// Pipeline (all device-side, one stream):
//   1. bt_count: units per center.  kTiles CTAs, each a contiguous range of
//      units, count in shared memory; one returned atomic per (tile, center)
//      adds the tile's count to the center's total and gives the tile its
//      block inside the center's segment;
//   2. bt_plan (one CTA): segment offsets from the totals, and work items of
//      at most `chunk` rows of one center, `chunk` chosen so that every SM
//      gets about kItemsPerSm items;
//   3. bt_place: each tile writes its units into its blocks (shared-memory
//      cursors; the order inside a block is arbitrary);
//   4. bt_sort_items: the unit ids of every item in ascending order (bitonic:
//      shuffles below a stride of 32, shared memory above), so that inside
//      an item a lower row index is a lower d; the packed table is set to its
//      identity in the same launch;
//   5. the scan: CM rows are streamed and every 16-byte column group keeps a
//      running lexicographic minimum; at the end of an item (or of a CTA's
//      share of one) the partial minima are folded in shared memory and
//      merged into a packed (cost, d) 64-bit table with atomicMin
//      (bt_scan_bulk: every CTA an equal contiguous share of the grouped
//      rows, staged whole by bulk copies);
//   6. bt_unpack: the (tc, td) int32 pair.
// Step 5 reads every CM byte of the allotted rows once and is the HBM-bound
// kernel; the other steps move O(n + k*k) bytes.
//
// Tables of 256 to 512 centers take a shorter path with no grouping (rows of
// 512 bytes to 2 KB gather poorly): bt_own, then bt_scan_stream reads the CM
// in row order, one narrow column slice and one row range per CTA, keeping
// the minima in shared memory, and bt_merge_ranges combines the ranges into
// (tc, td).  Fewer than 256 centers: the whole table of a row range fits
// shared memory, one kernel in row order and at most one merge
// (bt_scan_table).
#include <atomic>
#include <algorithm>

#include "lbdd_device.cuh"

namespace lbdd {

constexpr int kChunkMax = 512;          // rows per work item, at most (16-bit row index)
constexpr int kChunkMin = 64;           // rows per work item, at least (bounds the item count)
constexpr int kItemsPerSm = 8;          // work items per SM the plan aims for
constexpr int kTiles = 64;              // unit ranges of bt_count / bt_place
constexpr int kTileThreads = 1024;
constexpr int kTileUnroll = 8;          // assign loads in flight per thread

// ctl words (int32): error flag, item count, chunk, allotted rows
enum { BT_ERR = 0, BT_ITEMS, BT_CHUNK, BT_ROWS, BT_CTL_WORDS = 8 };

struct BtWorkspace {
  int* ctl;                     // BT_CTL_WORDS control words
  int32_t* cnt;                 // k + 1: units per center, then segment starts (cnt[k] = rows)
  int32_t* tile_rel;            // kTiles x k: a tile's block offset inside a center's segment
  int32_t* perm;                // n (+ 4 readable): allotted units grouped by center
  int4* items;                  // n / kChunkMin + k + 1 items {center, first row, rows, 0}
  unsigned long long* t64;      // k x k packed ((cost + 2^31) << 32) | d
  uint32_t* part;               // row-order path: one k x k key table per row range
  size_t bytes;
};

// Row-order path (bt_scan_stream): centers in [kStreamMinK, kStreamMaxK];
// int16: at most kStreamMaxRanges row ranges of at most kStreamRowSpan rows,
// int32: at most kStreamMaxRanges / 2 ranges (twice as wide keys, the same
// bytes of partial tables).
constexpr int kStreamMinK = 256, kStreamMaxK = 512;
constexpr int kStreamMaxRanges = 32;
constexpr int64_t kStreamRowSpan = 65536;  // the 16-bit row offset of a key

static size_t stream_part_bytes(int32_t n, int32_t k) {
  if (k < kStreamMinK || k > kStreamMaxK) return 0;
  return 4ull * k * k * (size_t)std::min<int32_t>(kStreamMaxRanges, n);
}

static inline size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

static BtWorkspace carve(void* base, int32_t n, int32_t k) {
  BtWorkspace W;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* p = static_cast<char*>(base) + o;
    o = al256(o + bytes);
    return p;
  };
  // ctl then cnt: one memset clears both
  W.ctl = reinterpret_cast<int*>(take(4 * BT_CTL_WORDS + 4ull * (k + 1)));
  W.cnt = W.ctl + BT_CTL_WORDS;
  W.tile_rel = reinterpret_cast<int32_t*>(take(4ull * kTiles * k));
  W.perm = reinterpret_cast<int32_t*>(take(4ull * n + 16));   // id windows round up to 16 bytes
  W.items = reinterpret_cast<int4*>(take(16ull * ((size_t)n / kChunkMin + (size_t)k + 1)));
  W.t64 = reinterpret_cast<unsigned long long*>(take(8ull * k * k));
  W.part = reinterpret_cast<uint32_t*>(take(stream_part_bytes(n, k)));
  W.bytes = o;
  return W;
}

static size_t table_part_bytes(int32_t n, int32_t k);
static size_t long_part_bytes(int32_t n, int32_t k);

// The least a call accepts, and what it makes full use of: the packed tables of
// short rows take the place of everything else, as many as there is room for.
size_t bt_workspace_min(int32_t n, int32_t k) {
  return n < 1 || k < 1 ? 0 : carve(nullptr, n, k).bytes + 256;
}
size_t bt_workspace_bytes(int32_t n, int32_t k) {
  return n < 1 || k < 1 ? 0
                        : std::max({bt_workspace_min(n, k), table_part_bytes(n, k) + 256,
                                    long_part_bytes(n, k) + 256});
}

// ------------------------------------------------------------- grouping ---

// Units of this CTA's tile: [t * per, min(n, (t + 1) * per)).
__device__ __forceinline__ void tile_range(int32_t n, int64_t* lo, int64_t* hi) {
  const int64_t per = ((int64_t)n + kTiles - 1) / kTiles;
  *lo = min((int64_t)n, (int64_t)blockIdx.x * per);
  *hi = min((int64_t)n, *lo + per);
}

// Units per center and per (tile, center).  Entries of assign outside
// [0, k) are not counted.
__global__ void __launch_bounds__(kTileThreads) bt_count(const int32_t* __restrict__ assign,
                                                         int32_t n, int32_t k, int32_t* cnt,
                                                         int32_t* tile_rel) {
  extern __shared__ int32_t h[];   // k counters
  const int tid = threadIdx.x;
  for (int i = tid; i < k; i += kTileThreads) h[i] = 0;
  __syncthreads();
  int64_t lo, hi;
  tile_range(n, &lo, &hi);
  for (int64_t b = lo; b < hi; b += (int64_t)kTileThreads * kTileUnroll) {
    int32_t a[kTileUnroll];
#pragma unroll
    for (int u = 0; u < kTileUnroll; ++u) {
      const int64_t i = b + u * kTileThreads + tid;
      a[u] = i < hi ? assign[i] : -1;
    }
#pragma unroll
    for (int u = 0; u < kTileUnroll; ++u)
      if (a[u] >= 0 && a[u] < k) atomicAdd(&h[a[u]], 1);
  }
  __syncthreads();
  for (int i = tid; i < k; i += kTileThreads)
    if (h[i]) tile_rel[(int64_t)blockIdx.x * k + i] = atomicAdd(&cnt[i], h[i]);
}

// Block-wide exclusive scan of one value per thread; returns this thread's
// prefix and writes the block total to *total.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t* s_warp,
                                                        int32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int32_t w = lane < kWarps ? s_warp[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    if (lane < kWarps) s_warp[lane] = w;   // inclusive warp prefixes
  }
  __syncthreads();
  const int32_t before = warp > 0 ? s_warp[warp - 1] : 0;
  *total = s_warp[kWarps - 1];
  return before + x - v;
}

// One CTA of kThreads: segment starts (exclusive prefix of the counts,
// centers in index order) into cnt[0..k), the allotted total into cnt[k],
// and the work items.  Records the item count, the
// chunk and the allotted rows in ctl.
__global__ void __launch_bounds__(kThreads) bt_plan(int32_t* cnt, int32_t k, int num_sms,
                                                    int4* items, int* ctl) {
  __shared__ int32_t s_warp[kWarps];
  const int tid = threadIdx.x;
  const int per = (k + kThreads - 1) / kThreads;
  const int c0 = min(k, tid * per), c1 = min(k, c0 + per);
  int32_t rows = 0;
  for (int c = c0; c < c1; ++c) rows += cnt[c];
  int32_t total;
  int32_t r = block_exclusive_scan(rows, s_warp, &total);
  const int64_t want = (int64_t)num_sms * kItemsPerSm;
  const int64_t even = ((int64_t)total + want - 1) / want;
  const int32_t chunk = (int32_t)(even < kChunkMin ? kChunkMin : even > kChunkMax ? kChunkMax : even);
  int32_t its = 0;
  for (int c = c0; c < c1; ++c) its += (cnt[c] + chunk - 1) / chunk;
  __syncthreads();                       // s_warp is reused
  int32_t nitems;
  int32_t it = block_exclusive_scan(its, s_warp, &nitems);
  for (int c = c0; c < c1; ++c) {
    const int32_t m = cnt[c];
    for (int32_t j = 0; j < m; j += chunk) items[it++] = make_int4(c, r + j, min(chunk, m - j), 0);
    cnt[c] = r;
    r += m;
  }
  if (tid == 0) {
    cnt[k] = total;
    ctl[BT_ITEMS] = nitems;
    ctl[BT_CHUNK] = chunk;
    ctl[BT_ROWS] = total;
  }
}

// Each tile's units into its blocks: cursor of center c = segment start +
// the tile's offset, advanced by shared-memory atomics.
__global__ void __launch_bounds__(kTileThreads) bt_place(const int32_t* __restrict__ assign,
                                                         int32_t n, int32_t k,
                                                         const int32_t* __restrict__ seg,
                                                         const int32_t* __restrict__ tile_rel,
                                                         int32_t* perm) {
  extern __shared__ int32_t cur[];   // k cursors (entries of centers absent from the tile unused)
  const int tid = threadIdx.x;
  for (int i = tid; i < k; i += kTileThreads)
    cur[i] = (int32_t)((uint32_t)seg[i] + (uint32_t)tile_rel[(int64_t)blockIdx.x * k + i]);
  __syncthreads();
  int64_t lo, hi;
  tile_range(n, &lo, &hi);
  for (int64_t b = lo; b < hi; b += (int64_t)kTileThreads * kTileUnroll) {
    int32_t a[kTileUnroll];
#pragma unroll
    for (int u = 0; u < kTileUnroll; ++u) {
      const int64_t i = b + u * kTileThreads + tid;
      a[u] = i < hi ? assign[i] : -1;
    }
#pragma unroll
    for (int u = 0; u < kTileUnroll; ++u)
      if (a[u] >= 0 && a[u] < k)
        perm[atomicAdd(&cur[a[u]], 1)] = (int32_t)(b + u * kTileThreads + tid);
  }
}

// The unit ids of each item in ascending order, one item per CTA at a time:
// thread i holds element i; compare-exchange partners at a stride below 32
// are reached by shuffles, the others through a double-buffered shared
// array (one barrier per step).  Also sets the packed table to ~0.
__global__ void __launch_bounds__(kThreads) bt_sort_items(const int4* __restrict__ items,
                                                          const int* __restrict__ ctl,
                                                          int32_t* perm, int32_t k,
                                                          unsigned long long* t64) {
  __shared__ int32_t xs[2][kChunkMax];
  const int tid = threadIdx.x;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + tid; i < (int64_t)k * k;
       i += (int64_t)gridDim.x * kThreads)
    t64[i] = ~0ull;
  const int total = ctl[BT_ITEMS];
  int buf = 0;     // kept across items: consecutive shared steps alternate buffers
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int4 desc = items[it];
    const int32_t r0 = desc.y, m = desc.z;
    if (m <= 1) continue;
    int P = 2;
    while (P < m) P <<= 1;
    int32_t v = tid < m ? perm[r0 + tid] : INT32_MAX;
    for (int size = 2; size <= P; size <<= 1) {
      const bool up = (tid & size) == 0;
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        int32_t w;
        if (stride >= 32) {
          xs[buf][tid] = v;
          __syncthreads();
          w = xs[buf][tid ^ stride];
          buf ^= 1;
        } else {
          w = __shfl_xor_sync(0xffffffffu, v, stride);
        }
        v = (((tid & stride) == 0) == up) ? min(v, w) : max(v, w);
      }
    }
    if (tid < m) perm[r0 + tid] = v;
  }
}

// ------------------------------------------------------------------ scan ---
//
// Keys of the int16 scan: one 32-bit key per column, ((t + 32768) << 16) |
// row of the item, so the lexicographic (t, d) minimum is one unsigned min
// (rows of an item are in increasing d; t fits 16 bits because costs are
// positive int16).  The int32 scan keeps (t, row) pairs with a strict '<':
// a thread sees the rows of an item in increasing order.

// ---------------------------------------------------- bulk-copy row scan ---
//
// CTA b scans the grouped rows
// [b * rows / G, (b + 1) * rows / G) of perm: equal bytes per CTA, no work
// queue.  Warp kWarps (the producer) walks that range: the segment starts
// (all k + 1 of them, copied into shared memory at start) give the center
// and the item boundaries of every position, the unit ids arrive in windows
// of kIdsWin by bulk copy one window ahead, and every CM row is copied whole
// global -> shared by one bulk copy (cp.async.bulk) into a ring of NS stages
// of at most RS rows of one item; a stage's barrier `full` completes once all
// of its bytes have landed.  The kWarps consumer warps scan the staged rows
// (one 16-byte column group per thread, R row groups; a row's own cost
// CM(d, c) is read from the staged row itself) and release the stage on its
// barrier `empty`.  At the end of an item, or of the part of it in this
// CTA's range, the consumers fold their partial minima (barrier `fold`,
// double-buffered) while the producer goes on filling stages.  Every wait is
// bounded: past kScanWaitLimitNs the waiter sets ctl[BT_ERR] and leaves (the
// producer first waits, bounded, for its copies in flight), and bt_unpack
// then marks the whole table.
constexpr int kBulkMinRowBytes = 512;
constexpr int kStageBytes = 32768;       // target bytes per stage (the producer's cost is per stage)
constexpr int kSmemLimit = 232448;       // dynamic shared memory of one CTA (227 KB)
constexpr int kMaxStages = 16;
constexpr int kIdsWin = 1024;            // unit ids per window (two windows in shared memory)
constexpr int kRedBytes = kThreads * 32; // one fold buffer: R*S*VPL keys (int16) or pairs (int32)
constexpr int kBulkThreads = kThreads + 32;
constexpr int kFoldCols = 8;             // columns per consumer thread in a fold (k <= 4096)
constexpr uint64_t kScanWaitLimitNs = 1000000000ull;
constexpr uint32_t kScanSleepNs = 1000000;

struct StageMeta {
  int32_t c;      // center of the rows
  int32_t r0;     // position in perm of the first row of the fold unit
  int32_t j;      // position of the stage's first row inside the fold unit
  int32_t rows;   // rows in the stage; -1 marks the end of the work
  int32_t last;   // the stage ends its fold unit
  int32_t pad0, pad1, pad2;
};

struct BulkShape {
  int S, R, RS, NS, row_bytes, stage_bytes;
};

__host__ __device__ inline size_t seg_smem_bytes(int32_t k) { return ((4 * (size_t)(k + 1)) + 15) & ~(size_t)15; }

// Shared memory besides the stages (fold buffers, id windows, segment
// starts, stage descriptors and barriers, the latter two at their largest).
static size_t bulk_fixed_bytes(int32_t k) {
  return 2 * (size_t)kRedBytes + 8 * (size_t)kIdsWin + seg_smem_bytes(k) +
         (size_t)kMaxStages * sizeof(StageMeta) + (2 * (size_t)kMaxStages + 3) * 8;
}

static BulkShape bulk_shape(int32_t k, int elem) {
  BulkShape p;
  const int VPL = 16 / elem;
  p.S = (k + VPL - 1) / VPL;
  p.R = kThreads / p.S;
  p.row_bytes = p.S * 16;
  const int per = std::max(1, kStageBytes / p.row_bytes);
  p.RS = std::min(32, std::max(p.R, per / p.R * p.R));
  p.stage_bytes = p.RS * p.row_bytes;
  p.NS = std::max(2, std::min<int>(kMaxStages, (int)((kSmemLimit - bulk_fixed_bytes(k)) / p.stage_bytes)));
  return p;
}

static size_t bulk_smem_bytes(const BulkShape& p, int32_t k) {
  return (size_t)p.NS * p.stage_bytes + 2 * (size_t)kRedBytes + 8 * (size_t)kIdsWin +
         seg_smem_bytes(k) + (size_t)p.NS * sizeof(StageMeta) + (2 * (size_t)p.NS + 3) * 8;
}

// Largest dynamic shared memory any shape needs (the attribute set once).
static size_t bulk_smem_max() { return kSmemLimit; }

__device__ __forceinline__ bool scan_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = gtimer_ns();
  while (!mbar_try_wait(bar, parity, kScanSleepNs))
    if (gtimer_ns() - t0 > kScanWaitLimitNs) return false;
  return true;
}

template <typename T>
__global__ void __launch_bounds__(kBulkThreads, 1)
bt_scan_bulk(const T* __restrict__ cm, int64_t ld, int32_t k, const int32_t* __restrict__ perm,
             const int32_t* __restrict__ seg, unsigned long long* t64, int* ctl, BulkShape p) {
  constexpr int VPL = 16 / (int)sizeof(T);
  extern __shared__ __align__(128) unsigned char dsm[];
  const int NS = p.NS, SB = p.stage_bytes, RB = p.row_bytes;
  unsigned char* stages = dsm;
  unsigned char* redb = dsm + (size_t)NS * SB;
  int32_t* s_ids = reinterpret_cast<int32_t*>(redb + 2 * kRedBytes);       // 2 windows
  int32_t* s_seg = s_ids + 2 * kIdsWin;                                    // k + 1
  StageMeta* meta = reinterpret_cast<StageMeta*>(reinterpret_cast<unsigned char*>(s_seg) +
                                                 seg_smem_bytes(k));
  uint64_t* full = reinterpret_cast<uint64_t*>(meta + NS);
  uint64_t* empty = full + NS;
  uint64_t* fold = empty + NS;
  uint64_t* idsbar = fold + 1;                                             // 2
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int32_t rows_total = ctl[BT_ROWS], chunk = ctl[BT_CHUNK];
  const int32_t P0 = (int32_t)((int64_t)blockIdx.x * rows_total / gridDim.x);
  const int32_t P1 = (int32_t)((int64_t)(blockIdx.x + 1) * rows_total / gridDim.x);
  if (tid < NS) {
    mbar_init(&full[tid], 1);
    mbar_init(&empty[tid], kWarps);
  }
  if (tid == 0) {
    mbar_init(fold, kWarps);
    mbar_init(&idsbar[0], 1);
    mbar_init(&idsbar[1], 1);
    mbar_fence_init();
  }
  for (int i = tid; i <= k; i += kBulkThreads) s_seg[i] = seg[i];
  __syncthreads();

  if (warp == kWarps) {
    // ---------------------------------------------------------- producer
    const int32_t A = P0 & ~3;                        // 16-byte aligned start of the id windows
    const int nwin = P1 > P0 ? (P1 - A + kIdsWin - 1) / kIdsWin : 0;
    int issued = -1, ready = -1;                      // id windows copied / waited for
    int s = 0, fills = 0;
    uint32_t eph = 0;                                 // slot s is free once phase eph ^ 1 completed
    bool ok = true;
    // center of P0: the largest c with seg[c] <= P0 (it is not empty)
    int c = 0;
    if (P0 < P1) {
      int lo = 0, hi = k - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_seg[mid] <= P0) lo = mid; else hi = mid - 1;
      }
      c = lo;
    }
    int32_t sb = s_seg[c], se = s_seg[c + 1];
    int32_t win_end = A;                              // ids below this position have landed
    int32_t pos = P0;
    // one fold unit per pass: the part of an item inside [P0, P1)
    while (ok && pos < P1) {
      while (se <= pos) { ++c; sb = s_seg[c]; se = s_seg[c + 1]; }
      const int32_t u0 = pos;
      const int32_t len = min(min(se, sb + ((pos - sb) / chunk + 1) * chunk), P1) - u0;
      for (int32_t j = 0; j < len; j += p.RS) {
        const int rows = min(p.RS, len - j);
        const int32_t q = u0 + j;
        if (q + rows > win_end || (issued < nwin - 1 && q >= A + issued * kIdsWin)) {
          // the window after q's goes out as soon as q enters q's window (its
          // buffer held the window before q's, whose rows are all issued);
          // then wait for the windows this stage reads
          const int wlast = min((q - A) / kIdsWin + 1, nwin - 1);
          while (issued < wlast) {
            ++issued;
            if (lane == 0) {
              const int32_t first = A + issued * kIdsWin;
              const uint32_t bytes = ((uint32_t)min(kIdsWin, P1 - first) * 4u + 15u) & ~15u;
              fence_proxy_async_smem();
              mbar_arrive_expect(&idsbar[issued & 1], bytes);
              bulk_load_smem(smem_u32(s_ids + (issued & 1) * kIdsWin), perm + first, bytes,
                             smem_u32(&idsbar[issued & 1]));
            }
          }
          const int wneed = (q + rows - 1 - A) / kIdsWin;
          while (ok && ready < wneed) {
            ++ready;
            ok = scan_wait(&idsbar[ready & 1], (ready >> 1) & 1);
          }
          win_end = A + (ready + 1) * kIdsWin;
          if (!ok) break;
        }
        if (!scan_wait(&empty[s], eph ^ 1)) { ok = false; break; }
        if (lane == 0) {
          StageMeta m;
          m.c = c; m.r0 = u0; m.j = j; m.rows = rows; m.last = j + p.RS >= len;
          m.pad0 = m.pad1 = m.pad2 = 0;
          meta[s] = m;
          mbar_arrive_expect(&full[s], (uint32_t)(rows * RB));
        }
        __syncwarp();
        const uint32_t dst = smem_u32(stages + (size_t)s * SB);
        for (int i = lane; i < rows; i += 32) {
          const int32_t d = s_ids[(q + i - A) & (2 * kIdsWin - 1)];
          bulk_load_smem(dst + (uint32_t)(i * RB), cm + (int64_t)d * ld, (uint32_t)RB,
                         smem_u32(&full[s]));
        }
        ++fills;
        if (++s == NS) { s = 0; eph ^= 1; }
      }
      pos = u0 + len;
    }
    if (ok) {
      if (scan_wait(&empty[s], eph ^ 1)) {
        if (lane == 0) {
          meta[s].rows = -1;     // end of the work
          mbar_arrive(&full[s]);
        }
      } else {
        ok = false;
      }
    }
    if (!ok) {
      if (lane == 0) atomicExch(&ctl[BT_ERR], 1);
      // copies still in flight: the last NS stage fills and unwaited id windows
      for (int f = max(0, fills - NS); f < fills; ++f) scan_wait(&full[f % NS], (f / NS) & 1);
      for (int w = ready + 1; w <= issued; ++w) scan_wait(&idsbar[w & 1], (w >> 1) & 1);
    }
    return;
  }

  // ------------------------------------------------------------ consumers
  const int S = p.S, R = p.R;
  const int slot = tid % S, g = tid / S;
  const bool act = g < R;
  int s = 0, rb = 0;
  uint32_t fph = 0, cph = 0;
  uint32_t key[VPL];
  int32_t bt[VPL], br[VPL];
#pragma unroll
  for (int q = 0; q < VPL; ++q) { key[q] = 0xffffffffu; bt[q] = kTInf; br[q] = -1; }
  for (;;) {
    if (!scan_wait(&full[s], fph)) {
      if (lane == 0) atomicExch(&ctl[BT_ERR], 1);
      break;
    }
    const StageMeta m = meta[s];
    if (m.rows < 0) break;
    if (act) {
      const unsigned char* sbase = stages + (size_t)s * SB;
      for (int i = g; i < m.rows; i += R) {
        const T* row = reinterpret_cast<const T*>(sbase + (size_t)i * RB);
        const int32_t own = (int32_t)row[m.c];
        const uint4 wv = reinterpret_cast<const uint4*>(row)[slot];
        const int32_t ri = m.j + i;
        if constexpr (sizeof(T) == 2) {
          const uint32_t crow = ((uint32_t)(32768 - own) << 16) | (uint32_t)ri;
          const uint32_t w4[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            key[2 * h] = min(key[2 * h], (w4[h] << 16) + crow);
            key[2 * h + 1] = min(key[2 * h + 1], (w4[h] & 0xffff0000u) + crow);
          }
        } else {
          const int32_t w4[4] = {(int32_t)wv.x, (int32_t)wv.y, (int32_t)wv.z, (int32_t)wv.w};
#pragma unroll
          for (int q = 0; q < VPL; ++q) {
            const int32_t t = w4[q] - own;
            if (t < bt[q]) { bt[q] = t; br[q] = ri; }
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++s == NS) { s = 0; fph ^= 1; }
    if (!m.last) continue;
    // end of a fold unit: fold the row groups, merge into the table
    unsigned char* red = redb + (size_t)rb * kRedBytes;
    if (act) {
#pragma unroll
      for (int q = 0; q < VPL; ++q) {
        const int at = g * S * VPL + slot * VPL + q;
        if constexpr (sizeof(T) == 2) reinterpret_cast<uint32_t*>(red)[at] = key[q];
        else reinterpret_cast<int2*>(red)[at] = make_int2(bt[q], br[q]);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(fold);
    if (!scan_wait(fold, cph)) {
      if (lane == 0) atomicExch(&ctl[BT_ERR], 1);
      break;
    }
    cph ^= 1;
    int32_t ft[kFoldCols], fr[kFoldCols];
#pragma unroll
    for (int q = 0; q < kFoldCols; ++q) {
      const int col = tid + q * kThreads;
      ft[q] = kTInf;
      fr[q] = -1;
      if (col < k) {
        if constexpr (sizeof(T) == 2) {
          uint32_t b = 0xffffffffu;
          for (int gg = 0; gg < R; ++gg)
            b = min(b, reinterpret_cast<const uint32_t*>(red)[gg * S * VPL + col]);
          if (b != 0xffffffffu) { ft[q] = (int32_t)(b >> 16) - 32768; fr[q] = (int32_t)(b & 0xffffu); }
        } else {
          for (int gg = 0; gg < R; ++gg) {
            const int2 e = reinterpret_cast<const int2*>(red)[gg * S * VPL + col];
            if (e.y >= 0 && (fr[q] < 0 || e.x < ft[q] || (e.x == ft[q] && e.y < fr[q]))) {
              ft[q] = e.x;
              fr[q] = e.y;
            }
          }
        }
      }
    }
    int32_t fd[kFoldCols];
#pragma unroll
    for (int q = 0; q < kFoldCols; ++q) fd[q] = fr[q] >= 0 ? perm[m.r0 + fr[q]] : -1;
#pragma unroll
    for (int q = 0; q < kFoldCols; ++q) {
      const int col = tid + q * kThreads;
      if (fr[q] >= 0 && col != m.c) {
        const unsigned long long pk =
            ((unsigned long long)(uint32_t)(ft[q] + (int64_t)2147483648LL) << 32) | (uint32_t)fd[q];
        atomicMin(&t64[(int64_t)m.c * k + col], pk);
      }
    }
    rb ^= 1;
#pragma unroll
    for (int q = 0; q < VPL; ++q) { key[q] = 0xffffffffu; bt[q] = kTInf; br[q] = -1; }
  }
}

__global__ void __launch_bounds__(kThreads) bt_unpack(const unsigned long long* __restrict__ t64,
                                                      int32_t k, int32_t* tc, int32_t* td,
                                                      const int* ctl) {
  const bool bad = ctl[BT_ERR] != 0;   // a scan wait ran out: the whole table is marked
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < (int64_t)k * k;
       i += (int64_t)gridDim.x * kThreads) {
    const unsigned long long e = t64[i];
    if (bad) {
      tc[i] = kTInf;
      td[i] = -2;
    } else if (e == ~0ull) {
      tc[i] = kTInf;
      td[i] = -1;
    } else {
      tc[i] = (int32_t)((int64_t)(e >> 32) - 2147483648LL);
      td[i] = (int32_t)(e & 0xffffffffu);
    }
  }
}

// ------------------------------------------------------------ row order ---
//
// Rows of kStreamMinK..kStreamMaxK centers (512 bytes to 2 KB) are short for
// row gathers, so this path reads the CM in row order instead and needs no
// grouping.  CTA (j, r) owns the column slice j (32 or 64 columns of int16, 32
// of int32 costs: stream_cols) and the row range r, and keeps in shared memory one key per
// (center, column of the slice): ((t + 32768) << 16) | (d - first row of the
// range) in 32 bits for int16, ((t + 2^31) << 32) | (d - first row) in 64
// bits for int32, so the smaller key is the lexicographically smaller (t, d)
// inside the range.  A thread
// owns 16 bytes of every 256th (128th) row; each is copied into the
// thread's own shared slot by cp.async kStreamStages rows ahead (the bytes in
// flight are bounded by shared memory, not registers), then the thread
// compares its keys with the table and lowers an entry with a shared atomicMin only where its
// key is smaller (entries only decrease, so a stale read never hides a
// smaller key).  A table row is laid out as two halves: the first half of
// every thread's keys, then the other half, so that the 128-bit shared loads
// of 8 threads cover 32 banks.  bt_own gathers CM(d, assign[d]) first (int16:
// together with the center, in one word); bt_merge_ranges takes, for every (u, v), the
// smallest t over the ranges in range order (ranges ascend in d, so the first
// range that attains it holds the smallest d) and writes tc/td.
//
// What bounds it is shared memory (staging, table reads and minima take about
// 40 cycles of its pipe per 512 bytes), then the partial tables.  Slices of
// 64 bytes instead of 128 with int16 costs halve the ranges, their tables and
// the share of keys that lower an entry: 200,000 x 500 int16 64.0 -> 62.1 us
// per call on inputs that were read before; on inputs new to L2 no difference.
// From about 400,000 rows on the wider slices are the faster ones.
constexpr int kStreamThreads = 1024;    // 4 or 8 threads per row slice, 256 or 128 rows at a time
constexpr int kStreamStages = 5;        // rows in flight per thread (cp.async stages)

__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Shared minimum at address `at`, where `key` is smaller than `cur`: one
// predicated reduction instead of a branch around an atomic.
__device__ __forceinline__ void red_min_if_less(uint32_t at, uint32_t key, uint32_t cur) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p red.shared.min.u32 [%0], %1;\n\t}"
               ::"r"(at), "r"(key), "r"(cur) : "memory");
}
// The same for a signed minimum; also voids the word at `unit`.
__device__ __forceinline__ void red_min_void_if_less(uint32_t at, int32_t t, int32_t cur,
                                                     uint32_t unit) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %1, %2;\n\t@p red.shared.min.s32 [%0], %1;\n\t"
      "@p st.shared.u32 [%3], %4;\n\t}" ::"r"(at), "r"(t), "r"(cur), "r"(unit), "r"(~0u) : "memory");
}
__device__ __forceinline__ void red_min_if_equal(uint32_t at, uint32_t d, int32_t t, int32_t cur) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.s32 p, %2, %3;\n\t@p red.shared.min.u32 [%0], %1;\n\t}"
               ::"r"(at), "r"(d), "r"(t), "r"(cur) : "memory");
}

// Per cost type: the key, and the key's split into cost and row offset.
template <typename T> struct StreamKey;
template <> struct StreamKey<int16_t> {
  using K = uint32_t;                    // ((t + 32768) << 16) | row offset
  static __device__ __forceinline__ int32_t cost(K key) { return (int32_t)(key >> 16) - 32768; }
  static __device__ __forceinline__ uint32_t offset(K key) { return key & 0xffffu; }
};
template <> struct StreamKey<int32_t> {
  using K = unsigned long long;          // ((t + 2^31) << 32) | row offset
  static __device__ __forceinline__ int32_t cost(K key) {
    return (int32_t)((int64_t)(key >> 32) - 2147483648LL);
  }
  static __device__ __forceinline__ uint32_t offset(K key) { return (uint32_t)key; }
};

// Programmatic dependent launch: a kernel launched with the attribute may
// start while its predecessor on the stream still runs; it waits here until
// the predecessor's results are visible (a no-op for an ordinary launch).
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel on the stream start launching.
__device__ __forceinline__ void release_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Dynamic shared memory of bt_scan_stream: the key table, then the stages.
template <typename T, int COLS>
static size_t stream_smem_bytes(int32_t k) {
  return (size_t)COLS * sizeof(typename StreamKey<T>::K) * (size_t)k +
         (size_t)kStreamStages * kStreamThreads * 16;
}

// Row ranges of the row-order path on `num_sms` SMs, 0 if it does not apply.
// int16 keys hold a 16-bit row offset (ranges of at most kStreamRowSpan
// rows); int32 keys are twice as wide, so at most half as many ranges fit the
// partial tables' bytes.
static int stream_ranges(int32_t n, int32_t k, int elem, int cols, int num_sms) {
  if (k < kStreamMinK || k > kStreamMaxK) return 0;
  const int64_t need = elem == 2 ? ((int64_t)n + kStreamRowSpan - 1) / kStreamRowSpan : 1;
  const int64_t cap = elem == 2 ? std::min<int64_t>(kStreamMaxRanges, n)
                                : std::min<int64_t>(kStreamMaxRanges / 2, n / 2);
  if (cap < 1 || need > cap) return 0;
  const int nslice = (k + cols - 1) / cols;
  return (int)std::min<int64_t>(cap, std::max<int64_t>(need, num_sms / nslice));
}

// Columns per slice: int32 32 (128 bytes), int16 32 or 64 (64 or 128 bytes).  A
// scan takes its waves times the rows of a range times the columns; slices of
// 64 columns fill the SMs better or worse, need fewer waves where the 65,536
// rows of a range force many ranges, and write and merge more tables.  They are
// taken where the time they save, in bytes of the CM, outweighs the tables (us
// per call, 32 / 64 columns: 200,000 x 500 62.8 / 63.6, 400,000 x 500 104.7 /
// 100.9, 1,000,000 x 500 265 / 214, 1,000,000 x 300 246 / 147, 1,000,000 x 256
// 124 / 137, 2,000,000 x 400 402 / 454).
static int stream_cols(int32_t n, int32_t k, int elem, int num_sms) {
  if (elem == 4) return 32;
  const int r32 = stream_ranges(n, k, 2, 32, num_sms), r64 = stream_ranges(n, k, 2, 64, num_sms);
  if (r32 < 1 || r64 < 1) return 32;
  auto time = [&](int cols, int ranges) {
    const int64_t ctas = (int64_t)((k + cols - 1) / cols) * ranges;
    return (double)((ctas + num_sms - 1) / num_sms) * cols / ranges;
  };
  const double saved = 2.0 * n * k * (1.0 - time(64, r64) / time(32, r32));
  return saved >= 8.0 * k * k * (r64 - r32) ? 64 : 32;
}

template <typename T>
__global__ void __launch_bounds__(kThreads) bt_own(const int32_t* __restrict__ assign, int32_t n,
                                                   int32_t k, const T* __restrict__ cm,
                                                   int64_t ld, int32_t* own) {
  release_successor();
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kThreads) {
    const int32_t a = assign[i];
    if constexpr (sizeof(T) == 2)   // center + 1 and own cost in one word, 0 = no center
      own[i] = (a >= 0 && a < k) ? ((a + 1) << 16) | (uint16_t)cm[i * ld + a] : 0;
    else
      own[i] = (a >= 0 && a < k) ? (int32_t)cm[i * ld + a] : 0;
  }
}

template <typename T, int COLS>
__global__ void __launch_bounds__(kStreamThreads, 1)
bt_scan_stream(const T* __restrict__ cm, int64_t ld, int32_t n, int32_t k,
               const int32_t* __restrict__ assign, const int32_t* __restrict__ own, int nslice,
               int nranges, typename StreamKey<T>::K* part) {
  using K = typename StreamKey<T>::K;
  constexpr int VPL = 16 / (int)sizeof(T);   // columns per thread (16 bytes)
  constexpr int HALF = VPL / 2;              // keys per 16-byte half
  constexpr int P = kStreamStages;
  extern __shared__ __align__(16) unsigned char stream_smem[];
  K* acc = reinterpret_cast<K*>(stream_smem);   // k rows of COLS keys, then the stages
  constexpr int TPR = COLS / VPL;              // threads per row slice
  constexpr int RPS = kStreamThreads / TPR;    // rows at a time
  constexpr int KB = COLS * (int)sizeof(K);    // bytes of a key row
  const int tid = threadIdx.x, cg = tid % TPR, rl = tid / TPR;
  const int j = blockIdx.x % nslice, r = blockIdx.x / nslice;
  const int64_t R0 = (int64_t)r * n / nranges, R1 = (int64_t)(r + 1) * n / nranges;
  const int c0 = j * COLS;
  const int w = min(COLS, k - c0);
  const bool act = cg * VPL < w;
  const uint4 none = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
  for (int i = tid; i < k * (KB / 16); i += kStreamThreads) reinterpret_cast<uint4*>(acc)[i] = none;
  __syncthreads();
  wait_predecessor();   // own[] comes from bt_own
  const T* colp = cm + c0 + cg * VPL;
  // rows of this thread: R0 + rl + RPS i, i < M; row i's 16 bytes go to
  // stage i % P of the thread's own shared slots P rows ahead (cp.async: a
  // thread waits only for its own copies, no barrier), its center and own
  // cost to a register ring P rows ahead
  const int64_t span = R1 - R0;
  const int32_t M = act && rl < span ? (int32_t)((span - rl + RPS - 1) / RPS) : 0;
  uint4* stage = reinterpret_cast<uint4*>(stream_smem + KB * (size_t)k);   // [P][kStreamThreads]
  // int16: one word per row holds both (bt_own)
  constexpr bool kPacked = sizeof(T) == 2;
  int32_t ra[P], ro[P];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    const int64_t d = R0 + rl + RPS * q;
    ra[q] = kPacked ? 0 : -1;
    ro[q] = 0;
    if (q < M) {
      cp_async16(&stage[q * kStreamThreads + tid], colp + d * ld);
      if (kPacked) {
        ra[q] = __ldg(own + d);
      } else {
        ra[q] = __ldg(assign + d);
        ro[q] = __ldg(own + d);
      }
    }
    cp_async_commit();
  }
  // rows advance by RPS: the addresses of row i + P (int16; with int32 costs
  // three running pointers measured slower than addresses from i: 45 against
  // 44 us, 60,000 x 400)
  const T* nx_cm = colp + (R0 + rl + RPS * (int64_t)P) * ld;
  const int32_t* nx_own = own + R0 + rl + RPS * P;
  const int64_t cm_step = RPS * ld;
  for (int32_t m = 0; m < M; m += P) {
#pragma unroll
    for (int q = 0; q < P; ++q) {
      cp_async_wait<P - 1>();                      // row m + q has landed
      const int32_t a = kPacked ? (ra[q] >> 16) - 1 : ra[q];
      const int32_t o = kPacked ? (int16_t)ra[q] : ro[q];
      const int32_t i = m + q;
      if (i < M && (kPacked ? ra[q] != 0 : a >= 0 && a < k)) {
        const uint4 x = stage[q * kStreamThreads + tid];
        const uint32_t off = (uint32_t)(rl + RPS * i);
        // the thread's first HALF keys sit in the first half of the key row,
        // the others in the second
        K* lo_p = acc + a * COLS + HALF * cg;
        K* hi_p = lo_p + COLS / 2;
        K key[VPL];
        if constexpr (sizeof(T) == 2) {
          const uint32_t crow = ((uint32_t)(32768 - o) << 16) | off;
          const uint32_t w4[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            key[2 * h] = (w4[h] << 16) + crow;
            key[2 * h + 1] = (w4[h] & 0xffff0000u) + crow;
          }
        } else {
          const int32_t w4[4] = {(int32_t)x.x, (int32_t)x.y, (int32_t)x.z, (int32_t)x.w};
#pragma unroll
          for (int h = 0; h < 4; ++h)
            key[h] = ((K)(uint32_t)((int64_t)w4[h] - o + 2147483648LL) << 32) | off;
        }
        if constexpr (sizeof(T) == 2) {
          // with 32 columns a key row's halves lie in the two halves of the
          // banks: odd rows of a warp take theirs in the other order
          const bool odd = COLS == 32 && (rl & 1);
          const uint32_t la = smem_u32(odd ? hi_p : lo_p), lb = smem_u32(odd ? lo_p : hi_p);
          const uint4 ca = *reinterpret_cast<const uint4*>(odd ? hi_p : lo_p);
          const uint4 cb = *reinterpret_cast<const uint4*>(odd ? lo_p : hi_p);
          red_min_if_less(la, odd ? key[4] : key[0], ca.x);
          red_min_if_less(la + 4, odd ? key[5] : key[1], ca.y);
          red_min_if_less(la + 8, odd ? key[6] : key[2], ca.z);
          red_min_if_less(la + 12, odd ? key[7] : key[3], ca.w);
          red_min_if_less(lb, odd ? key[0] : key[4], cb.x);
          red_min_if_less(lb + 4, odd ? key[1] : key[5], cb.y);
          red_min_if_less(lb + 8, odd ? key[2] : key[6], cb.z);
          red_min_if_less(lb + 12, odd ? key[3] : key[7], cb.w);
        } else {
          const uint4 lo = *reinterpret_cast<const uint4*>(lo_p);
          const uint4 hi = *reinterpret_cast<const uint4*>(hi_p);
          const K* cl = reinterpret_cast<const K*>(&lo);
          const K* ch = reinterpret_cast<const K*>(&hi);
#pragma unroll
          for (int h = 0; h < HALF; ++h) {
            if (key[h] < cl[h]) atomicMin(lo_p + h, key[h]);
            if (key[HALF + h] < ch[h]) atomicMin(hi_p + h, key[HALF + h]);
          }
        }
      }
      // stage q now takes row i + P
      ra[q] = kPacked ? 0 : -1;
      if (i + P < M) {
        if (kPacked) {
          cp_async16(&stage[q * kStreamThreads + tid], nx_cm);
          ra[q] = __ldg(nx_own);
        } else {
          const int64_t d = R0 + rl + RPS * (int64_t)(i + P);
          cp_async16(&stage[q * kStreamThreads + tid], colp + d * ld);
          ra[q] = __ldg(assign + d);
          ro[q] = __ldg(own + d);
        }
      }
      nx_cm += cm_step;
      nx_own += RPS;
      cp_async_commit();
    }
  }
  cp_async_wait<0>();
  release_successor();
  __syncthreads();
  K* out = part + (int64_t)r * k * k;
  for (int i = tid; i < k * COLS; i += kStreamThreads) {
    const int u = i / COLS, pc = i % COLS;   // pc: key slot in the row; its column:
    const int hh = pc / (COLS / 2), rest = pc % (COLS / 2);
    const int col = (rest / HALF) * VPL + hh * HALF + rest % HALF;
    if (col < w) out[(int64_t)u * k + c0 + col] = acc[i];
  }
}

template <typename K, typename T>
__global__ void __launch_bounds__(kThreads) bt_merge_ranges(const K* __restrict__ part,
                                                            int nranges, int32_t n, int32_t k,
                                                            int32_t* tc, int32_t* td) {
  wait_predecessor();   // the partial tables come from bt_scan_stream
  const int64_t kk = (int64_t)k * k;
  const K none = ~(K)0;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < kk;
       i += (int64_t)gridDim.x * kThreads) {
    K best = none;
    int br = -1;
    if constexpr (sizeof(K) == 8) {   // (eight in flight: 1 us slower at 400 and 500 centers)
      for (int r = 0; r < nranges; ++r) {
        const K key = part[r * kk + i];
        if (key != none && (br < 0 || StreamKey<T>::cost(key) < StreamKey<T>::cost(best))) {
          best = key;
          br = r;
        }
      }
    } else {
      constexpr int U = 8;   // tables in flight
      for (int r0 = 0; r0 < nranges; r0 += U) {
        K key[U];
#pragma unroll
        for (int u = 0; u < U; ++u) key[u] = r0 + u < nranges ? __ldcg(part + (r0 + u) * kk + i) : none;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (key[u] != none && (br < 0 || StreamKey<T>::cost(key[u]) < StreamKey<T>::cost(best))) {
            best = key[u];
            br = r0 + u;
          }
      }
    }
    const int32_t u = (int32_t)(i / k), v = (int32_t)(i % k);
    if (br < 0 || u == v) {
      tc[i] = kTInf;
      td[i] = -1;
    } else {
      tc[i] = StreamKey<T>::cost(best);
      td[i] = (int32_t)((int64_t)br * n / nranges + StreamKey<T>::offset(best));
    }
  }
}

// own: n words; part: nranges tables of k x k keys.
template <typename T, int COLS>
static cudaError_t stream_run(const T* cm, int64_t ld, int32_t n, int32_t k, const int32_t* assign,
                              int32_t* tc, int32_t* td, int32_t* own, void* parts, int nranges,
                              cudaStream_t st, int num_sms) {
  using K = typename StreamKey<T>::K;
  static std::atomic<uint64_t> attr_set{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!(attr_set.load() & (1ull << dev))) {
    e = cudaFuncSetAttribute(bt_scan_stream<T, COLS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)stream_smem_bytes<T, COLS>(kStreamMaxK));
    if (e != cudaSuccess) return e;
    attr_set.fetch_or(1ull << dev);
  }
  const int nslice = (k + COLS - 1) / COLS;
  K* part = static_cast<K*>(parts);
  bt_own<T><<<num_sms * 4, kThreads, 0, st>>>(assign, n, k, cm, ld, own);
  // the next two kernels may launch before their predecessor ends; each waits
  // for it (wait_predecessor) before reading its results
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(nslice * nranges);
  cfg.blockDim = dim3(kStreamThreads);
  cfg.dynamicSmemBytes = stream_smem_bytes<T, COLS>(k);
  e = cudaLaunchKernelEx(&cfg, bt_scan_stream<T, COLS>, cm, ld, n, k, assign, (const int32_t*)own,
                         nslice, nranges, part);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(num_sms * 4);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = 0;
  e = cudaLaunchKernelEx(&cfg, bt_merge_ranges<K, T>, (const K*)part, nranges, n, k, tc, td);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// ------------------------------------------------------------ short rows ---
//
// Fewer than kStreamMinK centers: a row is at most 1 KB and the whole table
// fits the shared memory of a CTA (or a few slices of its columns do), so
// one pass in row order needs no grouping, no work list and no packed table
// in global memory.  CTA (slice, range) reads its rows' 16-byte vectors in
// address order (every lane of a warp the next one: whole sectors whatever the
// row length), gets the row's center and own cost CM(d, c) by two small loads
// that hit the lines in flight, and lowers the entries of row c of its key
// table with shared minima, only where its key is smaller.  The CTAs of a
// cluster then reduce their tables through distributed shared memory, a share
// of the entries each.
//
// Up to kTableOneClusterK centers and kTableOneCluster entries one cluster does
// it all and writes tc/td itself: one launch, which is what such a call costs.
// Otherwise clusters of kTableCluster CTAs fill the chip, write one packed
// table each and bt_merge_tables (a dependent launch) takes the minimum over
// them.  Room for few tables (small workspaces, or up to kTablesInWorkspace
// bytes of int32 costs, where that is all the workspace holds) makes clusters of
// up to 8 CTAs and more slices; room for one table needs no merge, so such a
// call is one launch too.
//
// Where the one cluster ends, measured (us per call, one cluster against many):
// 40 centers int16 512 KB of costs 12.4 / 13.3, 768 KB 13.1 / 12.9, 1 MB 14.4 /
// 12.1, int32 1 MB 12.3 / 12.2, 2 MB 16.4 / 11.8.  The time of its reduction
// grows with k^2: 512 KB of int16 costs of 64, 100, 126 and 200 centers 12.4 /
// 13.2, 14.4 / 12.0, 14.4 / 11.3 and 22.5 / 10.4 (with one cluster up to 4 MB,
// calls of 200 centers took longer than the seven launches: 32 KB 32.7 against
// 28.7, 3.6 MB 34.0 against 32.3).
//
// The other limits, us per call (50,001 x 126, 200,000 x 126 and 30,000 x 200
// int32 unless said): clusters of 2, 4, 8 CTAs 24.6, 24.6, 28.8; 110.5, 66.8,
// 77.9; 26.7, 28.8, 37.2.  kTableReuse 4, 16, 64: 26.1, 24.6, 24.6; 70.6, 66.8,
// 70.6; 24.7, 28.8, 28.8 (400,000 x 64 int16 32.8, 32.8, 41.0).  kTableMinSlice 2,
// 4, 8, 16: 20,011 x 255 32.9, 24.6, 24.6, 24.7, int16 22.6, 22.6, 22.6, 26.7.
// kWideThreads 512, 640, 768, 1,024: 24.7, 24.6, 24.6, 24.7; 74.0, 66.8, 63.5,
// 63.6; 30.8, 28.8, 28.7, 30.7; 1,000,000 x 20 49.2, 45.2, 45.1, 47.7.
//
// Measured per call, before (seven launches: count, plan, place, sort, scan,
// unpack and a memset) and after: 2,000 x 20 int32 29.3 -> 10.1 to 12 us, 50,001 x
// 126 int32 52 -> 24.6 us (28.7 without the next batch in flight).
//
// int16 costs and ranges of at most 65,536 rows: one 32-bit key per entry,
// ((t + 32768) << 16 | d - first row), one pass, native shared minima.
// Otherwise t and d need 32 bits each, and a 64-bit shared minimum is a
// compare-and-swap loop that every improvement pays for (with a few rows per
// center and range, most keys improve).  So those entries are two words and a
// batch of rows, held in registers, goes through twice: first t takes the
// minimum (native; whoever lowers it voids the unit), then, after a barrier,
// the keys that equal it put their unit in the minimum.  Rows ascend from
// batch to batch, so a later equal t never replaces the unit.
constexpr int kTableThreads = 1024;         // 32-bit keys: short batches, many warps
constexpr int kTableUnroll = 4;             // vectors in flight per thread
constexpr int kWideThreads = 640;           // two words: two batches of 4 in registers
constexpr int kWideUnroll = 4;
constexpr int kTableCluster = 4;
constexpr int kTableOneClusterK = 64;       // centers and ...
constexpr int64_t kTableOneCluster = 384 << 10;   // ... entries up to which one cluster runs
constexpr int64_t kTablesInWorkspace = 4 << 20;   // bytes of int32 costs from which they count
constexpr size_t kTableSmem = 200 * 1024;
constexpr int kTableMaxClusters = 40;       // packed tables of a call, at most
constexpr int kTableReuse = 16;             // rows per center and range to aim for ...
constexpr int kTableMinSlice = 4;           // ... with slices of no less than 64 bytes

struct TableShape {
  int C, ncl, nslice, gs;   // cluster size, clusters per slice, slices, vectors per slice of a row
  bool wide;                // 64-bit keys
  size_t smem;
};

// `clusters`: clusters of kTableCluster CTAs that run at a time; `tables`:
// packed tables that the workspace holds.  With room for few of them, larger
// clusters and more slices keep the SMs busy.
static TableShape table_shape(int32_t n, int32_t k, int elem, int clusters, int tables) {
  TableShape p;
  const int vpl = 16 / elem;
  const int G = (k + vpl - 1) / vpl;
  const int64_t vecs = (int64_t)n * G;
  const bool one = k <= kTableOneClusterK && vecs * vpl <= kTableOneCluster;
  if (one)
    for (p.C = 1; p.C < 16 && vecs > (int64_t)p.C * 2 * kTableThreads;) p.C <<= 1;
  for (p.nslice = 1;; ++p.nslice) {
    p.gs = (G + p.nslice - 1) / p.nslice;
    p.ncl = one ? 1 : std::max(1, std::min({kTableMaxClusters, tables, clusters / p.nslice}));
    if (!one)   // (clusters of 8 leave some SMs of a GPC unused)
      for (p.C = kTableCluster; p.C < 8 && 2 * p.C * p.ncl * p.nslice <= 3 * clusters;) p.C <<= 1;
    if (!one && p.gs > kTableMinSlice && 2 * p.C * p.ncl * p.nslice <= kTableCluster * clusters)
      continue;
    // few rows per center and range: nearly every key would be a new minimum
    // and the tables would outweigh the costs; narrower slices of more rows
    if (!one && p.gs > kTableMinSlice && p.ncl > 1 &&
        (int64_t)n < (int64_t)kTableReuse * k * p.ncl * p.C)
      continue;
    p.wide = elem == 4 || ((int64_t)n + (int64_t)p.ncl * p.C - 1) / ((int64_t)p.ncl * p.C) > 65536;
    p.smem = (size_t)k * p.gs * vpl * (p.wide ? 8 : 4);
    if (p.smem <= kTableSmem) break;
  }
  p.nslice = (G + p.gs - 1) / p.gs;   // no empty slice
  return p;
}

// Packed tables of the largest call of this size (any cost width); fewer costs
// make do with those that the grouped scan's workspace has room for.
static bool tables_in_workspace(int32_t n, int32_t k) {
  return k < kStreamMinK && (int64_t)n * k * 4 + 16ll * n > kTablesInWorkspace;
}
static size_t table_part_bytes(int32_t n, int32_t k) {
  if (!tables_in_workspace(n, k)) return 0;
  return 8ull * k * k * kTableMaxClusters;
}

// Long tables of int32 costs, from kLongK centers and kLongBytes of costs on: the
// two-word table scan goes through every batch twice, the row-order scan of 256
// centers and more (64-bit keys) once, at the price of bt_own and more partial
// tables, which is why it does not pay below (us per call, table / row order:
// 200,000 x 64 35.2 / 42.0, 400,000 x 64 64.6 / 54.1, 200,000 x 100 49.8 / 39.9,
// 400,000 x 40 39.3 / 41.4, 1,000,000 x 255 544 / 211).  The seven launches took
// 187 us at 1,000,000 x 100 and 337 at 1,000,000 x 255, the table scan 217 and 544.
// A workspace without room for half the row ranges goes the grouped way, where
// its rows are long enough for bulk copies.
constexpr int kLongK = 64;
constexpr int64_t kLongBytes = 64 << 20;
static bool long_table(int32_t n, int32_t k) {
  return k >= kLongK && k < kStreamMinK && (int64_t)n * k * 4 >= kLongBytes;
}
static size_t long_part_bytes(int32_t n, int32_t k) {   // (152 SMs)
  return long_table(n, k) ? al256(4ull * n) + 8ull * k * k * (size_t)(152 / ((k + 31) / 32)) : 0;
}

// What CTA (slice, range) of a table scan reads.
template <typename T>
struct TablePart {
  static constexpr int VPL = 16 / (int)sizeof(T);
  int cr, range, ranges, c0, kp, gw;
  int64_t R0, R1;
  __device__ __forceinline__ TablePart(const TableShape& p, int32_t n, int32_t k) {
    const int cl = blockIdx.x / p.C, slice = cl % p.nslice;
    cr = cl / p.nslice;
    ranges = p.ncl * p.C;
    range = cr * p.C + (int)cluster_rank();
    R0 = first(range, n);
    R1 = first(range + 1, n);
    kp = p.gs * VPL;
    c0 = slice * kp;
    gw = min(p.gs, (k - c0 + VPL - 1) / VPL);   // vectors of this slice in a row
  }
  __device__ __forceinline__ int64_t first(int range_, int32_t n) const {
    return (int64_t)range_ * n / ranges;
  }
  // Column of entry e of a center's row of the table: entries are stored by
  // element of the vector, then by vector, so that the lanes of a warp, which
  // hold neighbouring vectors, touch neighbouring words.
  __device__ __forceinline__ int column(int e, int gs) const {
    const int h = e / gs;
    return c0 + (e - h * gs) * VPL + h;
  }
};

__device__ __forceinline__ void put_table(int32_t* tc, int32_t* td, int64_t at,
                                          unsigned long long best, bool diagonal) {
  const bool none = best == ~0ull || diagonal;
  tc[at] = none ? kTInf : (int32_t)((int64_t)(best >> 32) - 2147483648LL);
  td[at] = none ? -1 : (int32_t)(uint32_t)best;
}

// int16 costs, 32-bit keys.
__global__ void __launch_bounds__(kTableThreads, 1)
bt_scan_table(const int16_t* __restrict__ cm, int64_t ld, int32_t n, int32_t k,
              const int32_t* __restrict__ assign, TableShape p, unsigned long long* part,
              int32_t* tc, int32_t* td) {
  constexpr int VPL = 8, U = kTableUnroll;
  extern __shared__ __align__(16) unsigned char table_smem[];
  uint32_t* acc = reinterpret_cast<uint32_t*>(table_smem);   // [k][kp]
  const int tid = threadIdx.x;
  const TablePart<int16_t> P(p, n, k);
  const int gs = p.gs, kp = P.kp, gw = P.gw;
  const int64_t R0 = P.R0, R1 = P.R1;
  for (int i = tid; i < k * kp / 4; i += kTableThreads)
    reinterpret_cast<uint4*>(acc)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  __syncthreads();
  // vector i of the range: row i / gw, vector i % gw; a thread steps by the
  // CTA's threads
  const int dr = kTableThreads / gw, dg = kTableThreads - dr * gw;
  int64_t r = R0 + tid / gw;
  int g = tid % gw;
  while (r < R1) {
    uint4 x[U];
    int32_t a[U], own[U], gg[U];
    int64_t rr[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rr[u] = r;
      gg[u] = g;
      a[u] = -1;
      if (r < R1) {
        x[u] = __ldg(reinterpret_cast<const uint4*>(cm + r * ld + P.c0) + g);
        a[u] = __ldg(assign + r);
      }
      r += dr;
      g += dg;
      if (g >= gw) { g -= gw; ++r; }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      own[u] = 0;
      if ((uint32_t)a[u] < (uint32_t)k) own[u] = (int32_t)__ldg(cm + rr[u] * ld + a[u]);
      else a[u] = -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (a[u] < 0) continue;
      const uint32_t* e = acc + a[u] * kp + gg[u];
      const uint32_t w4[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
      const uint32_t crow = ((uint32_t)(32768 - own[u]) << 16) | (uint32_t)(rr[u] - R0);
      // entries only fall, so a stale read never hides a smaller key
#pragma unroll
      for (int h = 0; h < VPL; ++h) {
        const uint32_t key = ((h & 1) ? (w4[h / 2] & 0xffff0000u) : (w4[h / 2] << 16)) + crow;
        red_min_if_less(smem_u32(e + h * gs), key, e[h * gs]);
      }
    }
  }
  __syncthreads();
  cluster_sync_all();
  release_successor();
  // a share of the entries per CTA, over all tables of the cluster
  const int C = p.C, rank = P.range - P.cr * C;
  const int E = k * kp;
  const int e1 = (int)((int64_t)(rank + 1) * E / C);
  for (int e = (int)((int64_t)rank * E / C) + tid; e < e1; e += kTableThreads) {
    const int u = e / kp, v = P.column(e - u * kp, gs);
    if (v >= k) continue;
    unsigned long long best = ~0ull;
    for (int q = 0; q < C; ++q) {
      const uint32_t key = (uint32_t)dsmem_ld32(dsmem_addr(acc + e, (uint32_t)q));
      // ranges ascend in d: an equal cost keeps the earlier range's unit
      if (key != ~0u)
        best = min(best, ((unsigned long long)((key >> 16) + 0x7fff8000u) << 32) |
                             (uint32_t)(P.first(P.cr * C + q, n) + (key & 0xffffu)));
    }
    const int64_t at = (int64_t)u * k + v;
    if (p.ncl > 1) part[(int64_t)P.cr * k * k + at] = best;
    else put_table(tc, td, at, best, u == v);
  }
  cluster_sync_all();   // a table stays until every CTA has read it
}

// Two words per entry: t (kTInf: none) and d.
template <typename T>
__global__ void __launch_bounds__(kWideThreads, 1)
bt_scan_table_wide(const T* __restrict__ cm, int64_t ld, int32_t n, int32_t k,
                   const int32_t* __restrict__ assign, TableShape p, unsigned long long* part,
                   int32_t* tc, int32_t* td) {
  constexpr int VPL = 16 / (int)sizeof(T), U = kWideUnroll;
  extern __shared__ __align__(16) unsigned char table_smem[];
  const int tid = threadIdx.x;
  const TablePart<T> P(p, n, k);
  const int gs = p.gs, kp = P.kp, gw = P.gw;
  int32_t* at_t = reinterpret_cast<int32_t*>(table_smem);          // [k][kp]
  uint32_t* at_d = reinterpret_cast<uint32_t*>(at_t + k * kp);     // [k][kp]
  for (int i = tid; i < k * kp / 4; i += kWideThreads) {
    reinterpret_cast<int4*>(at_t)[i] = make_int4(kTInf, kTInf, kTInf, kTInf);
    reinterpret_cast<uint4*>(at_d)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  }
  __syncthreads();
  const int dr = kWideThreads / gw, dg = kWideThreads - dr * gw;
  int64_t r = P.R0 + tid / gw;
  int g = tid % gw;
  const int64_t vecs = (P.R1 - P.R0) * gw;
  const int64_t batches = (vecs + (int64_t)U * kWideThreads - 1) / ((int64_t)U * kWideThreads);
  auto cost = [](const uint4& x, int h) -> int32_t {
    const uint32_t w = (&x.x)[sizeof(T) == 4 ? h : h / 2];
    return sizeof(T) == 4 ? (int32_t)w : (h & 1) ? (int32_t)w >> 16 : (int32_t)(int16_t)w;
  };
  uint4 xn[U];          // the next batch, in flight while this one goes through
  int32_t an[U], gn[U];
  uint32_t rn[U];
  auto fetch = [&]() {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rn[u] = (uint32_t)r;
      gn[u] = g;
      an[u] = -1;
      if (r < P.R1) {
        xn[u] = __ldg(reinterpret_cast<const uint4*>(cm + r * ld + P.c0) + g);
        an[u] = __ldg(assign + r);
      }
      r += dr;
      g += dg;
      if (g >= gw) { g -= gw; ++r; }
    }
  };
  fetch();
  for (int64_t b = 0; b < batches; ++b) {
    uint4 x[U];
    int32_t a[U], own[U], at[U];
    uint32_t rr[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      x[u] = xn[u];
      a[u] = an[u];
      at[u] = gn[u];
      rr[u] = rn[u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      own[u] = 0;
      if ((uint32_t)a[u] < (uint32_t)k) {
        own[u] = (int32_t)__ldg(cm + (int64_t)rr[u] * ld + a[u]);
        at[u] += a[u] * kp;
      } else {
        at[u] = -1;
      }
    }
    fetch();
    uint32_t maybe = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (at[u] < 0) continue;
#pragma unroll
      for (int h = 0; h < VPL; ++h) {
        const int32_t t = cost(x[u], h) - own[u];
        const int e = at[u] + h * gs;
        const int32_t cur = at_t[e];
        red_min_void_if_less(smem_u32(at_t + e), t, cur, smem_u32(at_d + e));
        if (t <= cur) maybe |= 1u << u;   // the others are no minimum
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!(maybe >> u & 1)) continue;
#pragma unroll
      for (int h = 0; h < VPL; ++h) {
        const int32_t t = cost(x[u], h) - own[u];
        const int e = at[u] + h * gs;
        red_min_if_equal(smem_u32(at_d + e), rr[u], t, at_t[e]);
      }
    }
    __syncthreads();
  }
  cluster_sync_all();
  release_successor();
  const int C = p.C, rank = P.range - P.cr * C;
  const int E = k * kp;
  const int e1 = (int)((int64_t)(rank + 1) * E / C);
  for (int e = (int)((int64_t)rank * E / C) + tid; e < e1; e += kWideThreads) {
    const int u = e / kp, v = P.column(e - u * kp, gs);
    if (v >= k) continue;
    unsigned long long best = ~0ull;
    for (int q = 0; q < C; ++q) {
      const uint32_t t = (uint32_t)dsmem_ld32(dsmem_addr(at_t + e, (uint32_t)q));
      const uint32_t d = (uint32_t)dsmem_ld32(dsmem_addr(at_d + e, (uint32_t)q));
      if (d != ~0u) best = min(best, ((unsigned long long)(t ^ 0x80000000u) << 32) | d);
    }
    const int64_t out = (int64_t)u * k + v;
    if (p.ncl > 1) part[(int64_t)P.cr * k * k + out] = best;
    else put_table(tc, td, out, best, u == v);
  }
  cluster_sync_all();
}

__global__ void __launch_bounds__(kThreads) bt_merge_tables(const unsigned long long* __restrict__ part,
                                                            int ntab, int32_t k, int32_t* tc,
                                                            int32_t* td) {
  wait_predecessor();
  const int64_t kk = (int64_t)k * k;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < kk;
       i += (int64_t)gridDim.x * kThreads) {
    unsigned long long best = ~0ull;
#pragma unroll 4
    for (int t = 0; t < ntab; ++t) best = min(best, part[t * kk + i]);
    put_table(tc, td, i, best, i / k == i % k);
  }
}

// The scan kernel of a cost type and key width, and its threads.
template <typename T, bool WIDE>
static auto table_kernel() {
  if constexpr (WIDE) return bt_scan_table_wide<T>;
  else return bt_scan_table;
}
template <bool WIDE>
static constexpr int table_threads() { return WIDE ? kWideThreads : kTableThreads; }

// Sets the kernel's attributes once per device and returns how many of its
// clusters run at a time (GPCs whose SMs are no multiple of kTableCluster
// hold fewer than the SM count suggests).
template <typename T, bool WIDE>
static cudaError_t table_setup(int* clusters) {
  static std::atomic<int> known[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if ((*clusters = known[dev].load()) > 0) return cudaSuccess;
  auto kern = table_kernel<T, WIDE>();
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTableSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kTableCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kTableCluster);
  cfg.blockDim = dim3(table_threads<WIDE>());
  cfg.dynamicSmemBytes = kTableSmem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
  if (e != cudaSuccess) return e;
  *clusters = std::max(1, *clusters);
  known[dev].store(*clusters);
  return cudaSuccess;
}

template <typename T, bool WIDE>
static cudaError_t table_run(const T* cm, int64_t ld, int32_t n, int32_t k, const int32_t* assign,
                             int32_t* tc, int32_t* td, void* ws, const TableShape& p,
                             cudaStream_t st) {
  unsigned long long* part = static_cast<unsigned long long*>(ws);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)(p.C * p.ncl * p.nslice));
  cfg.blockDim = dim3(table_threads<WIDE>());
  cfg.dynamicSmemBytes = p.smem;
  cudaError_t e =
      cudaLaunchKernelEx(&cfg, table_kernel<T, WIDE>(), cm, ld, n, k, assign, p, part, tc, td);
  if (e != cudaSuccess || p.ncl == 1) return e;
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl;
  cfg.gridDim = dim3((unsigned)std::min<int64_t>(((int64_t)k * k + kThreads - 1) / kThreads, 608));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, bt_merge_tables, (const unsigned long long*)part, p.ncl, k, tc,
                            td);
}

template <typename T>
static cudaError_t table_call(const T* cm, int64_t ld, int32_t n, int32_t k, const int32_t* assign,
                              int32_t* tc, int32_t* td, void* ws, size_t ws_bytes,
                              cudaStream_t st) {
  int clusters = 0;
  // (the same route whatever a caller's workspace has beyond the size asked for)
  const size_t room = tables_in_workspace(n, k)
                          ? ws_bytes : std::min(ws_bytes, bt_workspace_min(n, k) - 256);
  const int tables = (int)std::min<size_t>(kTableMaxClusters, room / (8ull * k * k));
  cudaError_t e;
  if constexpr (sizeof(T) == 2) {
    if ((e = table_setup<T, false>(&clusters)) != cudaSuccess) return e;
    const TableShape p = table_shape(n, k, 2, clusters, tables);
    if (!p.wide) return table_run<T, false>(cm, ld, n, k, assign, tc, td, ws, p, st);
  }
  if ((e = table_setup<T, true>(&clusters)) != cudaSuccess) return e;
  const TableShape p = table_shape(n, k, (int)sizeof(T), clusters, tables);
  return table_run<T, true>(cm, ld, n, k, assign, tc, td, ws, p, st);
}

int bt_max_k(int elem_bytes) { return kThreads * (16 / elem_bytes); }

// Sets the bulk scan's dynamic shared memory limit once per device.
template <typename T>
static cudaError_t bulk_attr() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!(done.load() & (1ull << dev))) {
    e = cudaFuncSetAttribute(bt_scan_bulk<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bulk_smem_max());
    if (e != cudaSuccess) return e;
    done.fetch_or(1ull << dev);
  }
  return cudaSuccess;
}

template <typename T>
static cudaError_t scan_launch(const T* cm, int64_t ld, int32_t k, const BtWorkspace& W,
                               cudaStream_t st, int num_sms) {
  const BulkShape p = bulk_shape(k, (int)sizeof(T));
  const cudaError_t e = bulk_attr<T>();
  if (e != cudaSuccess) return e;
  bt_scan_bulk<T><<<num_sms, kBulkThreads, bulk_smem_bytes(p, k), st>>>(cm, ld, k, W.perm, W.cnt,
                                                                         W.t64, W.ctl, p);
  return cudaSuccess;
}

// Returns a cudaError_t (cudaSuccess on success); argument checks are done
// by the caller.
cudaError_t best_transfer_run(int32_t n, int32_t k, const void* cm, int elem_bytes, int64_t ld,
                              const int32_t* assign, int32_t* tc, int32_t* td, void* ws,
                              size_t ws_bytes, cudaStream_t st, int num_sms) {
  void* base = reinterpret_cast<void*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
  const BtWorkspace W = carve(base, n, k);
  const size_t room = ws_bytes - (size_t)(static_cast<char*>(base) - static_cast<char*>(ws));
  bool grouped = false;   // the row gathers below 256 centers
  if (elem_bytes == 4 && long_table(n, k)) {
    const int nslice = (k + 31) / 32;
    const size_t own = al256(4ull * n);
    const int ranges =
        (int)std::min<size_t>(num_sms / nslice, room > own ? (room - own) / (8ull * k * k) : 0);
    if (2 * ranges * nslice > num_sms)
      return stream_run<int32_t, 32>(static_cast<const int32_t*>(cm), ld, n, k, assign, tc, td,
                                     static_cast<int32_t*>(base), static_cast<char*>(base) + own,
                                     ranges, st, num_sms);
    grouped = 4 * k >= kBulkMinRowBytes;
  }
  if (k < kStreamMinK && !grouped)
    return elem_bytes == 2
               ? table_call(static_cast<const int16_t*>(cm), ld, n, k, assign, tc, td, base, room, st)
               : table_call(static_cast<const int32_t*>(cm), ld, n, k, assign, tc, td, base, room, st);
  const int cols = stream_cols(n, k, elem_bytes, num_sms);
  const int nranges = stream_ranges(n, k, elem_bytes, cols, num_sms);
  if (nranges > 0) {
    auto run = [&](auto* c, auto width) {
      return stream_run<std::remove_const_t<std::remove_pointer_t<decltype(c)>>, width.value>(
          c, ld, n, k, assign, tc, td, W.perm, W.part, nranges, st, num_sms);
    };
    const int16_t* c16 = static_cast<const int16_t*>(cm);
    return elem_bytes == 4 ? run(static_cast<const int32_t*>(cm), std::integral_constant<int, 32>())
           : cols == 32    ? run(c16, std::integral_constant<int, 32>())
                           : run(c16, std::integral_constant<int, 64>());
  }
  cudaError_t e = cudaMemsetAsync(W.ctl, 0, 4 * BT_CTL_WORDS + 4ull * (k + 1), st);
  if (e != cudaSuccess) return e;
  bt_count<<<kTiles, kTileThreads, 4 * (size_t)k, st>>>(assign, n, k, W.cnt, W.tile_rel);
  bt_plan<<<1, kThreads, 0, st>>>(W.cnt, k, num_sms, W.items, W.ctl);
  bt_place<<<kTiles, kTileThreads, 4 * (size_t)k, st>>>(assign, n, k, W.cnt, W.tile_rel, W.perm);
  bt_sort_items<<<num_sms * 4, kThreads, 0, st>>>(W.items, W.ctl, W.perm, k, W.t64);
  e = elem_bytes == 2
          ? scan_launch(static_cast<const int16_t*>(cm), ld, k, W, st, num_sms)
          : scan_launch(static_cast<const int32_t*>(cm), ld, k, W, st, num_sms);
  if (e != cudaSuccess) return e;
  bt_unpack<<<num_sms * 4, kThreads, 0, st>>>(W.t64, k, tc, td, W.ctl);
  return cudaGetLastError();
}

}  // namespace lbdd
