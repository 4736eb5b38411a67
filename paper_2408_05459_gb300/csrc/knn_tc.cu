// tcgen05 BF16 / FP8-e4m3 candidate search for the cosine KNN of Section 3.1.
//
// Two kernels share one scheme.  k_knn_pair sweeps all keys with CTA pairs
// (every sweep of the rows over themselves); k_knn_tc, one CTA at a time, takes
// the sweeps of listed key tiles, of the inverted lists' centroids, of a sample
// of the tiles and of keys above a threshold.
//
// Persistent CTAs (one per SM) share the (query block, 256-row key tile)
// pairs in equal contiguous runs (stream-K), so no wave tail is left idle.
// In each CTA of k_knn_tc:
//   warp 0     TMA producer: the current query block A (128 x dp, 128-byte
//              swizzle) when the run enters it, then key tiles B (256 rows x
//              128 bytes of features per stage: 64 BF16 or 128 FP8) through
//              an nstages-deep ring (mbarrier full/empty);
//   warp 1     MMA issuer: allocates 512 TMEM columns, issues
//              tcgen05.mma.cta_group::1.kind::f16 (BF16, K=16) with M=128,
//              N=256 (the pair: also kind::f8f6f4, E4M3, K=32) into two
//              ping-pong FP32 accumulators, commits stage releases,
//              accumulator-ready signals and the release of A at the end of
//              each query block;
//   warps 4-11 epilogue: two warps per TMEM lane quarter, each owning half of
//              every tile's 256 columns; tcgen05.ld (32x32b) of the thread's
//              accumulator row (TMEM lane = query row), threshold test and
//              insert into a register-resident list of its 16 best scores.
//              Row i thus leaves two 16-entry lists (one per column half),
//              kCandC = 32 candidates in total; a query block split between
//              two CTAs leaves partial lists that k_merge_lists combines.
// The MMA of tile t+1 overlaps the epilogue of tile t.  n x n scores never
// leave the SM.  Every mbarrier wait is bounded: on expiry the kernel records
// an error code, stops all roles, drains its own copies and MMAs (bounded),
// frees TMEM and returns.
//
// The producer and the MMA issuer run their loops as whole warps and elect a
// lane for the copies, MMAs and commits alone.  With the loops inside one
// lane's branch the MMAs, whose operands want uniform registers, took 167
// cycles each and a stage's hand-off another 160; warp-uniform they take 130,
// the tensor pipe's own rate (M = 256 over a pair, N = 256, K = 16).
#include <algorithm>
#include <atomic>

#include "tc_common.cuh"

namespace ancka {

namespace {

constexpr int kTM = 128;                 // query rows per CTA = TMEM lanes
constexpr int kTN = 256;                 // key rows per tile = accumulator columns
constexpr int kLists = 2;                // lists per row = column slices of every tile
constexpr int kEpiWarps = 4 * kLists;    // one warp per (TMEM lane quarter, column slice)
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kListC = kCandC / kLists;  // entries of each list
// Three warpgroups: the producer, the MMA issuer and two idle warps, then the
// eight epilogue warps.  What decides whether the MMAs wait is how soon an
// accumulator comes back, so the epilogue takes all 128 columns of its slice
// into registers before it looks at them; the first warpgroup gives up its
// registers for that (setmaxnreg: 128 x 64 + 256 x 216 = 63,488 of the
// 384 x 168 = 64,512 the block is launched with).
constexpr int kTcThreads = 128 + 32 * kEpiWarps;
constexpr int kRegsLow = 64, kRegsHigh = 216;
constexpr int kSliceN = kTN / kLists;    // columns of a tile per slice
constexpr int kABytes = kTM * kTKB;      // 16 KB per 128-byte block of A
constexpr int kBBytes = kTN * kTKB;      // 32 KB per stage of B
constexpr int kMmaPerStage = 4;          // 32 bytes of K per MMA: 16 BF16 or 32 FP8
constexpr int kMaxStages = 8;
// 227 KB opt-in dynamic shared memory; every kernel's limit is set to it,
// whatever the call needs, since the limit is the process's and another
// thread's call may need more
constexpr int kMaxSmem = 232448;
constexpr uint32_t kTmemCols = 512;      // two 256-column FP32 accumulators

// instruction descriptors: D = F32 (bits 4-5 = 1), both operands K-major,
// N >> 3 at bits 17-22, M >> 4 at bits 24-28; kind::f16 with A = B = BF16
// (format 1 at bits 7-9 and 10-12); kind::f8f6f4 with A = B = E4M3 (format 0)
constexpr uint32_t kIdescBF16 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTN >> 3) << 17) |
                                ((uint32_t)(kTM >> 4) << 24);
constexpr uint32_t kIdescE4M3 = (1u << 4) | ((uint32_t)(kTN >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);

struct __align__(8) Bars {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t a_full;
  uint64_t a_empty;
  uint64_t tfull[2];
  uint64_t tempty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int rot[2];  // key rotation of the current and the previous segment (written by the producer)
};

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          tmem_d),
      "l"(da), "l"(db), "r"(kIdescBF16), "r"(accum)
      : "memory");
}
// Row lists are kept sorted in descending score order, lv[0] >= ... >=
// lv[C-1], so the threshold is lv[C-1] and an insert is C independent
// select pairs (two levels deep) instead of a C-long minimum scan.  A score
// equal to an entry goes after it: among equal scores the earlier key stays.
template <int C>
__device__ __forceinline__ void sorted_insert(float (&lv)[C], int32_t (&li)[C], float s, int32_t j) {
#pragma unroll
  for (int c = C - 1; c >= 1; --c) {
    const bool at_or_before = s > lv[c];
    const bool before_prev = s > lv[c - 1];
    lv[c] = at_or_before ? (before_prev ? lv[c - 1] : s) : lv[c];
    li[c] = at_or_before ? (before_prev ? li[c - 1] : j) : li[c];
  }
  if (s > lv[0]) {
    lv[0] = s;
    li[0] = j;
  }
}

// r[e] for a lane-dependent e in 0..31: a five-level select tree
__device__ __forceinline__ float pick32(const uint32_t (&r)[32], int e) {
  float v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = __uint_as_float((e & 16) ? r[q + 16] : r[q]);
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
    for (int q = 0; q < w; ++q) v[q] = (e & w) ? v[q + w] : v[q];
  return v[0];
}
// the same over 16
__device__ __forceinline__ float pick16(const uint32_t (&r)[16], int e) {
  float v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = __uint_as_float((e & 8) ? r[q + 8] : r[q]);
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1)
#pragma unroll
    for (int q = 0; q < w; ++q) v[q] = (e & w) ? v[q + w] : v[q];
  return v[0];
}

// A row's list, and a 16-key chunk with a key above the threshold that has
// not been looked into yet (pj == kNoChunk: none).  Finding and inserting a
// key costs the whole warp ~150 dependent instructions however few lanes need
// it, so a lane that meets such a chunk sets it aside, 16 moves, and the warp
// goes through its lanes' chunks together once some lane has a second one
// (after about seven).  The threshold lags by the chunk, which only lets more
// keys through to the insert's own test: the list is the same.
constexpr uint32_t kNoChunk = 0xffffffffu;
template <int C>
struct RowList {
  float lv[C];
  int32_t li[C];
  uint32_t pr[16];  // the chunk's scores
  uint32_t pj;      // its first key
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      lv[c] = -INFINITY;
      li[c] = -1;
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) pr[e] = 0;
    pj = kNoChunk;
  }
  // the warp's chunks into its lists; n keys, i: the key this row excludes
  // (itself), or -1
  __device__ __forceinline__ void flush(uint32_t n, uint32_t i) {
    // pass mask against the threshold now (it only rises, so the mask is a
    // superset), in four chains; padding keys and the row itself removed
    const float thr = lv[C - 1];
    uint32_t q[4] = {0, 0, 0, 0};
#pragma unroll
    for (int e = 0; e < 16; ++e) q[e & 3] |= (__uint_as_float(pr[e]) > thr ? 1u : 0u) << e;
    uint32_t pm = pj == kNoChunk ? 0u : (q[0] | q[1]) | (q[2] | q[3]);
    if (pj < n && n - pj < 16) pm &= (1u << (n - pj)) - 1u;
    if (pj >= n) pm = 0;
    if (i - pj < 16) pm &= ~(1u << (i - pj));
    // one key per lane and round; lanes without keys idle
    while (__any_sync(0xffffffffu, pm != 0)) {
      const int e = __ffs(pm) - 1;
      const float v = pick16(pr, e);
      if (pm != 0 && v > lv[C - 1]) sorted_insert<C>(lv, li, v, (int32_t)(pj + e));
      pm &= pm - 1;
    }
    pj = kNoChunk;
  }
  // set aside the chunk r (keys j0 ..) in the lanes whose maximum of it passes
  __device__ __forceinline__ void push(const uint32_t (&r)[16], float mx, uint32_t j0, uint32_t n, uint32_t i) {
    if (__any_sync(0xffffffffu, mx > lv[C - 1] && pj != kNoChunk)) flush(n, i);
    if (mx > lv[C - 1]) {
#pragma unroll
      for (int e = 0; e < 16; ++e) pr[e] = r[e];
      pj = j0;
    }
  }
};

// Collect mode: append every key whose score reaches the row's fixed
// threshold t to the row's buffer (cap entries; the counter keeps counting
// past cap so the caller can see an overflow).  One atomic reserves a chunk's
// places: with one per key, a row whose keys nearly all pass waited for 32 of
// them in turn at every chunk, long after its buffer was full (a call at
// n = 8000, d = 500, K = 13 with a quarter of the rows near-parallel: 2.19 ->
// 1.91 ms).
__device__ __forceinline__ void collect_chunk(const uint32_t (&r)[32], float mx, int64_t j0, int64_t n, int64_t i,
                                              float t, int64_t ra, int32_t* __restrict__ cnt,
                                              int32_t* __restrict__ buf, int cap) {
  if (!__any_sync(0xffffffffu, mx >= t)) return;
  uint32_t pm = 0;
#pragma unroll
  for (int e = 0; e < 32; ++e) pm |= (__uint_as_float(r[e]) >= t ? 1u : 0u) << e;
  if (j0 + 32 > n) pm &= (j0 >= n) ? 0u : ((1u << (uint32_t)(n - j0)) - 1u);
  if (i >= j0 && i < j0 + 32) pm &= ~(1u << (uint32_t)(i - j0));
  if (!pm) return;
  for (int pos = atomicAdd(&cnt[ra], __popc(pm)); pm && pos < cap; ++pos) {
    buf[ra * (int64_t)cap + pos] = (int32_t)(j0 + __ffs(pm) - 1);
    pm &= pm - 1;
  }
}

// Fold one tile's column slice (kSliceN accumulator columns from TMEM address
// tb, keys jb ...) into the row's list: eight 16-column loads with the
// hardware's maximum of each behind one wait, release() to hand the
// accumulator back before any list work, then eight independent votes that say
// which chunks hold a key above some lane's threshold (about one a tile at
// n = 600,000).
template <int C, class Release>
__device__ __forceinline__ void fold_slice(uint32_t tb, uint32_t jb, uint32_t n, uint32_t i, RowList<C>& L,
                                           Release&& release) {
  constexpr int kChunks = kSliceN / 16;
  uint32_t r[kChunks][16];
  float mx[kChunks];
#pragma unroll
  for (int c = 0; c < kChunks; ++c) tmem_ld16_max_issue(tb + (uint32_t)(c * 16), r[c], mx[c]);
  tmem_wait();
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    pin(r[c]);
    pin1(mx[c]);
  }
  release();
  const float thr = L.lv[C - 1];
  float top = mx[0];
#pragma unroll
  for (int c = 1; c < kChunks; ++c) top = fmaxf(top, mx[c]);
  if (!__any_sync(0xffffffffu, top > thr)) return;  // more than half of the slices of a large sweep
  uint32_t hit = 0;
#pragma unroll
  for (int c = 0; c < kChunks; ++c) hit |= (__any_sync(0xffffffffu, mx[c] > thr) ? 1u : 0u) << c;
#pragma unroll
  for (int c = 0; c < kChunks; ++c)
    if (hit & (1u << c)) L.push(r[c], mx[c], jb + (uint32_t)(c * 16), n, i);
}

struct CollectArgs {
  const int32_t* a_rows;  // global row of each compact query row (null: A holds rows 0..n-1)
  int64_t n_a;            // compact query rows (0: as many as keys)
  const float* thr;       // collect mode: per compact row threshold
  int32_t* cnt;           // collect mode: per compact row counter
  int32_t* buf;           // collect mode: n_a x cap keys
  int cap;
  // tile-list mode (null: every block sweeps every key tile): query block qb
  // sweeps the key tiles blk_tiles[blk_ptr[qb] .. blk_ptr[qb + 1])
  const int64_t* blk_ptr = nullptr;
  const int32_t* blk_tiles = nullptr;
  int64_t blk_work = 0;   // blk_ptr[qblocks]
  int no_self = 0;        // the keys are another set (no row excludes "itself")
};

// The segment of query block qb that a run [w, w_end) covers from w:
// positions [t0, t1) of the block's len key tiles.
struct Seg {
  int64_t qb;
  int t0, t1, len;
  int64_t base;  // tile-list mode: offset of the block's tiles
};
__device__ __forceinline__ Seg segment_at(int64_t w, int64_t w_end, int n_tiles, int64_t qblocks,
                                          const CollectArgs& ca) {
  Seg sg;
  if (ca.blk_ptr) {
    int64_t lo = 0, hi = qblocks;  // the last qb with blk_ptr[qb] <= w
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (ca.blk_ptr[mid] <= w) lo = mid; else hi = mid;
    }
    sg.qb = lo;
    sg.base = ca.blk_ptr[lo];
    sg.len = (int)(ca.blk_ptr[lo + 1] - sg.base);
  } else {
    sg.qb = w / n_tiles;
    sg.base = sg.qb * n_tiles;
    sg.len = n_tiles;
  }
  sg.t0 = (int)(w - sg.base);
  sg.t1 = (int)(w_end - w < (int64_t)(sg.len - sg.t0) ? sg.t0 + (w_end - w) : sg.len);
  return sg;
}

// Work split (stream-K): the (query block, key tile) pairs, numbered
// qb * n_tiles + t, are cut into gridDim.x equal contiguous ranges, one per
// persistent CTA.  A CTA's range is a sequence of segments, one per query
// block it touches; only its first and its last segment can miss part of a
// block's key tiles.  Such a partial segment leaves its lists in slot 0
// (first segment) or 1 (last) of the CTA's partial area, and k_merge_lists
// combines the pieces of every split block.
__device__ __forceinline__ int64_t range_begin(int64_t c, int64_t work, int64_t ctas) { return c * work / ctas; }

// Position t of query block qb sweeps key tile (t + key_rotation(qb)) mod
// n_tiles.  The rotation puts the block's first tile at the time its owner
// CTA (the one whose run holds position 0) reaches it, modulo n_tiles, so at
// any moment the CTAs read the same key tile and each tile comes from DRAM
// about once per sweep (only a run's first, split segment is out of step).
__device__ __forceinline__ int key_rotation(int64_t qb, int n_tiles, int64_t work, int64_t ctas) {
  const int64_t x0 = qb * n_tiles;
  const int64_t c0 = ((x0 + 1) * ctas + work - 1) / work - 1;
  const int64_t lag = x0 - range_begin(c0, work, ctas);  // owner's time at position 0
  return (int)(lag % n_tiles);
}

// kCollect: collect mode (keys above a per-row threshold) instead of list
// mode (two 16-entry lists per row).
// key_stride > 1: only every key_stride-th key tile is swept (the sampled
// pass of the symmetric contraction).  k_last: MMAs issued for the last
// 128-byte block of features (those past the last one holding a feature of
// X are zero padding and are skipped).
template <bool kCollect>
__global__ void __launch_bounds__(kTcThreads, 1)
k_knn_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int64_t n,
         int64_t n_pad, int64_t qblocks, int kb_count, int k_last, int nstages, int key_stride,
         float* __restrict__ cand_val,
         int32_t* __restrict__ cand_idx, float* __restrict__ part_val,
         int32_t* __restrict__ part_idx, CollectArgs ca, unsigned long long* __restrict__ tick,
         int* __restrict__ err) {
  constexpr int kTK = 64;  // features per stage
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kb_count * kABytes;
  Bars* bars = reinterpret_cast<Bars*>(sB + nstages * kBBytes);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  const int n_tiles = (int)ceil_div(ceil_div(n_pad, kTN), key_stride);
  const int64_t work = ca.blk_ptr ? ca.blk_work : qblocks * n_tiles;
  const int64_t w_begin = range_begin(blockIdx.x, work, gridDim.x);
  const int64_t w_end = range_begin((int64_t)blockIdx.x + 1, work, gridDim.x);
  volatile int* abort = &bars->abort;

  if (threadIdx.x == 0) {
    for (int s = 0; s < nstages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    mbar_init(&bars->a_full, 1);
    mbar_init(&bars->a_empty, 1);
    mbar_init(&bars->tfull[0], 1);
    mbar_init(&bars->tfull[1], 1);
    mbar_init(&bars->tempty[0], kEpiWarps);
    mbar_init(&bars->tempty[1], kEpiWarps);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  if (warp < 4) {
    if constexpr (!kCollect) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLow));
    if (warp == 0) {
      bool pending[kMaxStages];
      uint32_t pend_par[kMaxStages];
      for (int s = 0; s < kMaxStages; ++s) pending[s] = false;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int seg = 0;
      uint32_t tiles_issued = 0;
      const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
      for (int64_t w = w_begin; w < w_end && ok; ++seg) {
        const Seg sg = segment_at(w, w_end, n_tiles, qblocks, ca);
        const int64_t qb = sg.qb;
        const int t0 = sg.t0, t1 = sg.t1;
        int rot = ca.blk_ptr ? 0 : key_rotation(qb, n_tiles, work, gridDim.x);
        w += t1 - t0;
        // the previous block of A stays in use until its last MMA completes
        if (seg > 0 && !mbar_wait_warp(&bars->a_empty, (uint32_t)((seg - 1) & 1), abort, err, 6)) {
          ok = false;
          break;
        }
        // Collect mode: a block this CTA sweeps whole starts at the key tile
        // the CTAs are reading now (tiles issued by all CTAs / CTAs), so that
        // CTAs whose rates drift apart re-align at every block and keep
        // sharing the key tiles in L2; a split block keeps the static rotation
        // both of its CTAs can compute.  (Not for lists, whose callers want the
        // same ones on every call: a key order that moves with timing resolves
        // exact score ties differently.)
        if (kCollect && t0 == 0 && t1 == n_tiles)
          rot = (int)((*reinterpret_cast<volatile unsigned long long*>(tick) / gridDim.x) % (uint64_t)n_tiles);
        rot = __shfl_sync(0xffffffffu, rot, 0);
        if (elect_one()) {
          bars->rot[seg & 1] = rot;
          __threadfence_block();
          mbar_expect_tx(&bars->a_full, (uint32_t)(kb_count * kABytes));
          for (int kb = 0; kb < kb_count; ++kb)
            tma_load_2d(sA0 + kb * kABytes, &tmA, kb * kTK, (int)(qb * kTM), &bars->a_full);
        }
        __syncwarp();
        for (int t = t0; t < t1 && ok; ++t) {
          const int kt = ca.blk_ptr ? ca.blk_tiles[sg.base + t]
                                    : (t + rot < n_tiles ? t + rot : t + rot - n_tiles) * key_stride;
          for (int kb = 0; kb < kb_count; ++kb) {
            if (!mbar_wait_warp(&bars->empty[stage], phase ^ 1, abort, err, 1)) {
              ok = false;
              break;
            }
            if (elect_one()) {
              mbar_expect_tx(&bars->full[stage], (uint32_t)kBBytes);
              tma_load_2d(sB0 + stage * kBBytes, &tmB, kb * kTK, kt * kTN, &bars->full[stage]);
            }
            __syncwarp();
            pending[stage] = true;
            pend_par[stage] = phase;
            if (++stage == nstages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (kCollect && ((++tiles_issued) & 15) == 0 && lane == 0) atomicAdd(tick, 16ull);
        }
      }
      if (!ok) {  // drain this warp's copies still in flight (bounded)
        if (seg > 0) mbar_wait(&bars->a_full, (uint32_t)((seg - 1) & 1), nullptr, nullptr, 0);
        for (int s = 0; s < nstages; ++s)
          if (pending[s]) mbar_wait(&bars->full[s], pend_par[s], nullptr, nullptr, 0);
      }
    } else if (warp == 1) {
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0;
      bool issued = false;
      int64_t g = 0;  // accumulator tiles so far (ping-pong over two)
      int seg = 0;
      const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
      for (int64_t w = w_begin; w < w_end && ok; ++seg) {
        const Seg sg = segment_at(w, w_end, n_tiles, qblocks, ca);
        const int t0 = sg.t0, t1 = sg.t1;
        w += t1 - t0;
        if (!mbar_wait_warp(&bars->a_full, (uint32_t)(seg & 1), abort, err, 2)) {
          ok = false;
          break;
        }
        for (int t = t0; t < t1; ++t, ++g) {
          const int b = (int)(g & 1);
          const uint32_t use = (uint32_t)(g >> 1);
          if (!mbar_wait_warp(&bars->tempty[b], (use & 1) ^ 1, abort, err, 3)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(b * kTN);
          for (int kb = 0; kb < kb_count; ++kb) {
            if (!mbar_wait_warp(&bars->full[stage], phase, abort, err, 4)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t a0 = sw128_desc(sA0 + kb * kABytes);
            const uint64_t b0 = sw128_desc(sB0 + stage * kBBytes);
            const int kmax = kb == kb_count - 1 ? k_last : kMmaPerStage;
            if (elect_one()) {
              // the next 32 bytes of K: 2 more in the descriptors' 16-byte units
  #pragma unroll
              for (int kk = 0; kk < kMmaPerStage; ++kk)
                if (kk < kmax) umma_bf16(d, a0 + kk * 2, b0 + kk * 2, (kb | kk) != 0 ? 1u : 0u);
              umma_commit(&bars->empty[stage]);
              if (kb == kb_count - 1) umma_commit(&bars->tfull[b]);
            }
            __syncwarp();
            issued = true;
            if (++stage == nstages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
        }
        if (ok && elect_one()) umma_commit(&bars->a_empty);  // A may be replaced once these MMAs complete
        __syncwarp();
      }
      if (!ok && issued) {  // wait for the MMAs issued before TMEM is freed (bounded)
        if (elect_one()) umma_commit(&bars->drain);
        __syncwarp();
        mbar_wait(&bars->drain, 0, nullptr, nullptr, 0);
      }
    }
  } else {
    if constexpr (!kCollect) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsHigh));
    const int ew = warp - 4;   // epilogue warp 0..7
    const int q = warp & 3;    // TMEM lane quarter this warp may access
    const int h = ew >> 2;     // column slice of every tile
    const int r = q * 32 + lane;
    constexpr int C = kListC;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    int64_t g = 0;
    int seg = 0;
    bool ok = true;
    for (int64_t w = w_begin; w < w_end && ok; ++seg) {
      const Seg sg = segment_at(w, w_end, n_tiles, qblocks, ca);
      const int64_t qb = sg.qb;
      const int t0 = sg.t0, t1 = sg.t1;
      int rot = 0;
      w += t1 - t0;
      // A row ra is query row ra, or compact row ra -> global row a_rows[ra]
      const int64_t ra = qb * kTM + r;
      const bool row_ok = ra < (ca.n_a > 0 ? ca.n_a : n);
      const int64_t i = ca.a_rows ? (row_ok ? (int64_t)ca.a_rows[ra] : -1) : ra;
      const int64_t i_self = ca.no_self ? -1 : i;  // the key index this row excludes
      const float t_row = kCollect && row_ok ? ca.thr[ra] : INFINITY;
      RowList<C> L;
      L.clear();
      for (int t = t0; t < t1; ++t, ++g) {
        const int b = (int)(g & 1);
        const uint32_t use = (uint32_t)(g >> 1);
        const bool got = mbar_wait(&bars->tfull[b], use & 1, abort, err, 5);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // the producer wrote the segment's rotation before loading its block
        // of A, which the first accumulator of the segment waited for
        if (t == t0) rot = *reinterpret_cast<volatile int*>(&bars->rot[seg & 1]);
        const int kt = ca.blk_ptr ? ca.blk_tiles[sg.base + t]
                                  : (t + rot < n_tiles ? t + rot : t + rot - n_tiles) * key_stride;
        const int64_t jb = (int64_t)kt * kTN + h * kSliceN;
        const uint32_t tb = lane_base + (uint32_t)(b * kTN + h * kSliceN);
        // the hardware's maximum over each load settles most chunks with one
        // compare and one vote
        auto release = [&] {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->tempty[b]);
        };
        if constexpr (kCollect) {
#pragma unroll 1
          for (int c = 0; c < kSliceN / 32; ++c) {
            uint32_t rv[32];
            float mx;
            tmem_ld32_max_issue(tb + (uint32_t)(c * 32), rv, mx);
            tmem_wait();
            pin(rv);
            pin1(mx);
            collect_chunk(rv, mx, jb + c * 32, n, i_self, t_row, ra, ca.cnt, ca.buf, ca.cap);
          }
          release();
        } else {
          fold_slice<C>(tb, (uint32_t)jb, (uint32_t)n, (uint32_t)i_self, L, release);
        }
      }
      if (!kCollect && ok) {
        float* ov;
        int32_t* oi;
        L.flush((uint32_t)n, (uint32_t)i_self);
        if (t0 == 0 && t1 == sg.len) {  // whole block: final lists
          if (!row_ok) continue;
          ov = cand_val + i * kCandC;
          oi = cand_idx + i * kCandC;
        } else {
          const int64_t slot = ((int64_t)blockIdx.x * 2 + (seg == 0 ? 0 : 1)) * kTM + r;
          ov = part_val + slot * kCandC;
          oi = part_idx + slot * kCandC;
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          ov[h * C + c] = L.lv[c];
          oi[h * C + c] = L.li[c];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------
// Full sweep on CTA pairs.
//
// A CTA that sweeps alone reads 12 KB of shared memory per 128 x 256 x 16 MMA
// and writes 8 KB (9 KB at d = 100) of key tiles for it, more than the 128
// bytes a cycle its shared memory gives in the 128 cycles that MMA takes.  Two
// CTAs of a cluster (the two SMs of a TPC) therefore share one M = 256,
// N = 256 accumulator pair (tcgen05 cta_group::2): each holds its own 128
// query rows and half (128) of a tile's keys, so that per MMA an SM reads
// 8 KB and writes 4 KB, and the key bytes that come from L2 halve.
//
// Measured (the contraction with its row preparation; one CTA a sweep before,
// the pair now): 72 -> 46 ms at n = 600,000, d = 100 (about 1240 cycles a tile
// for 907 of MMAs: the epilogue's list work; 41 ms without it, the clock then
// lower under power); 6.9 -> 5.2 ms at n = 100,000, d = 500 (MMA bound: 4150
// cycles a tile for 32 MMAs, SM clock 1.8 GHz under power); E4M3 3.4 -> 2.5 ms
// at n = 100,003, d = 256 (list work: 1.7 ms without it).
//
// Roles as in k_knn_tc, in both CTAs, except that the even CTA (the leader)
// alone issues the MMAs.  Each CTA's producer loads its own half and signals
// the leader's barrier (cta_group::2 copies), which expects the bytes of
// both; the commits of the leader's MMAs arrive in both CTAs (multicast), and
// the epilogue warps of both release an accumulator at the leader's barrier.
// The unit of work is 256 query rows x 256 keys, split stream-K over the
// pairs.  The leader picks a block's key rotation and hands it to its peer.
// ---------------------------------------------------------------------------
constexpr int kPairRows = 2 * kTM;             // query rows of a pair's block
constexpr int kPairBBytes = kTN / 2 * kTKB;    // 16 KB of keys per stage and CTA
constexpr int kPairMaxStages = 12;
struct __align__(8) PairBars {
  uint64_t full[kPairMaxStages];   // leader: both CTAs' halves of the stage have landed
  uint64_t empty[kPairMaxStages];  // each CTA: the MMAs that read the stage have completed
  uint64_t a_full;                 // leader: both CTAs' query rows have landed
  uint64_t a_empty;                // each CTA
  uint64_t tfull[2];               // each CTA
  uint64_t tempty[2];              // leader: released by the epilogue warps of both
  uint64_t rot_full;               // peer: the leader has written rot
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
  int rot[2];  // key rotation of the current and the previous segment
};

// M = 256 over the pair
constexpr uint32_t kIdescPairBF16 = (kIdescBF16 & ~(0x1fu << 24)) | ((uint32_t)(kPairRows >> 4) << 24);
constexpr uint32_t kIdescPairE4M3 = (kIdescE4M3 & ~(0x1fu << 24)) | ((uint32_t)(kPairRows >> 4) << 24);

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
  __syncwarp();
}
// this CTA's shared address as CTA `rank`'s address at the same offset
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
__device__ __forceinline__ void pair_tma_load(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
template <bool kE4M3>
__device__ __forceinline__ void pair_umma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t accum) {
  if constexpr (kE4M3)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, "
        "p;\n}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(kIdescPairE4M3), "r"(accum)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
            tmem_d),
        "l"(da), "l"(db), "r"(kIdescPairBF16), "r"(accum)
        : "memory");
}
// arrives at the barrier's offset in both CTAs once this thread's MMAs complete
__device__ __forceinline__ void pair_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void pair_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// One CTA of the pair; grid = 2 x pairs.  Arguments as for k_knn_tc; part_*
// hold two slots of kPairRows rows per pair.  With shares > 1 each block of
// rows is swept once per share of the key tiles (tiles share, share + shares,
// ...; past the last one the keys are padding), and row i leaves two lists per
// share, at (i * shares + share) * kCandC; qblocks counts (block, share) pairs.
// kShared: shares may exceed 1 (as a run-time value everywhere its arithmetic
// in the roles' loops cost 9% at d = 100: 194 against 178 ms at n = 1,200,000).
template <bool kE4M3, bool kShared>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1)
k_knn_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int64_t n,
           int64_t n_pad, int64_t qblocks, int kb_count, int k_last, int nstages, float* __restrict__ cand_val,
           int32_t* __restrict__ cand_idx, const float* __restrict__ out_scale, float* __restrict__ part_val,
           int32_t* __restrict__ part_idx, const int32_t* __restrict__ a_rows, int64_t n_rows, int share_count,
           unsigned long long* __restrict__ tick, int* __restrict__ err) {
  constexpr int kTK = kE4M3 ? 128 : 64;  // features per stage
  const int shares = kShared ? share_count : 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kb_count * kABytes;
  PairBars* bars = reinterpret_cast<PairBars*>(sB + nstages * kPairBBytes);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int64_t pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int n_tiles = (int)ceil_div(ceil_div(n_pad, kTN), shares);
  const int64_t work = qblocks * n_tiles;
  const int64_t w_begin = range_begin(pair, work, pairs);
  const int64_t w_end = range_begin(pair + 1, work, pairs);
  const CollectArgs none{};
  volatile int* abort = &bars->abort;

  if (threadIdx.x == 0) {
    for (int s = 0; s < nstages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    mbar_init(&bars->a_full, 1);
    mbar_init(&bars->a_empty, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->tfull[b], 1);
      mbar_init(&bars->tempty[b], 2 * kEpiWarps);
    }
    mbar_init(&bars->rot_full, 1);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers and TMEM are ready
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLow));
    if (warp == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int seg = 0;
      uint32_t tiles_issued = 0;
      const uint32_t a_full = peer_addr(smem_u32(&bars->a_full), 0);
      const uint32_t full0 = peer_addr(smem_u32(&bars->full[0]), 0);
      const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
      for (int64_t w = w_begin; w < w_end && ok; ++seg) {
        const Seg sg = segment_at(w, w_end, n_tiles, qblocks, none);
        const int share = (int)(sg.qb % shares);
        w += sg.t1 - sg.t0;
        // the previous query rows stay in use until their last MMA completes
        if (seg > 0 && !mbar_wait_warp(&bars->a_empty, (uint32_t)((seg - 1) & 1), abort, err, 6)) {
          ok = false;
          break;
        }
        // Key order: as in k_knn_tc, a block the pair sweeps whole starts at
        // the tile the pairs are reading now, a split block at the static
        // rotation both of its pairs compute.
        int rot;
        if (leader) {
          rot = key_rotation(sg.qb, n_tiles, work, pairs);
          if (sg.t0 == 0 && sg.t1 == n_tiles)
            rot = (int)((*reinterpret_cast<volatile unsigned long long*>(tick) / pairs) % (uint64_t)n_tiles);
          rot = __shfl_sync(0xffffffffu, rot, 0);
          if (elect_one()) {
            bars->rot[seg & 1] = rot;
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(smem_u32(&bars->rot[seg & 1]), 1)), "r"(rot)
                         : "memory");
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                             peer_addr(smem_u32(&bars->rot_full), 1))
                         : "memory");
          }
        } else {
          if (!mbar_wait_warp(&bars->rot_full, (uint32_t)(seg & 1), abort, err, 7)) {
            ok = false;
            break;
          }
          asm volatile("fence.acq_rel.cluster;" ::: "memory");
          rot = *reinterpret_cast<volatile int*>(&bars->rot[seg & 1]);
          rot = __shfl_sync(0xffffffffu, rot, 0);
        }
        if (elect_one()) {
          if (leader) mbar_expect_tx(&bars->a_full, (uint32_t)(2 * kb_count * kABytes));
          for (int kb = 0; kb < kb_count; ++kb)
            pair_tma_load(sA0 + kb * kABytes, &tmA, kb * kTK, (int)(sg.qb / shares * kPairRows + rank * kTM), a_full);
        }
        __syncwarp();
        for (int t = sg.t0; t < sg.t1 && ok; ++t) {
          const int kt = (t + rot < n_tiles ? t + rot : t + rot - n_tiles) * shares + share;
          for (int kb = 0; kb < kb_count; ++kb) {
            if (!mbar_wait_warp(&bars->empty[stage], phase ^ 1, abort, err, 1)) {
              ok = false;
              break;
            }
            if (elect_one()) {
              if (leader) mbar_expect_tx(&bars->full[stage], (uint32_t)(2 * kPairBBytes));
              pair_tma_load(sB0 + stage * kPairBBytes, &tmB, kb * kTK, (int)(kt * kTN + rank * (kTN / 2)),
                            full0 + (uint32_t)(stage * sizeof(uint64_t)));
            }
            __syncwarp();
            if (++stage == nstages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (leader && ((++tiles_issued) & 15) == 0 && lane == 0) atomicAdd(tick, 16ull);
        }
      }
      // on an abort, let this CTA's copies in flight land before the CTA may
      // exit: they report to the leader's barriers, so a fixed time (~1 ms,
      // several hundred times a copy's latency) stands in for a wait on them
      if (!ok)
        for (const long long t0 = clock64(); clock64() - t0 < 2000000;) {
        }
    } else if (warp == 1) {
      if (leader) {
        bool ok = true;
        int stage = 0;
        uint32_t phase = 0;
        bool issued = false;
        int64_t g = 0;  // accumulator tiles so far (ping-pong over two)
        int seg = 0;
        const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
        for (int64_t w = w_begin; w < w_end && ok; ++seg) {
          const Seg sg = segment_at(w, w_end, n_tiles, qblocks, none);
          w += sg.t1 - sg.t0;
          if (!mbar_wait_warp(&bars->a_full, (uint32_t)(seg & 1), abort, err, 2)) {
            ok = false;
            break;
          }
          for (int t = sg.t0; t < sg.t1; ++t, ++g) {
            const int b = (int)(g & 1);
            const uint32_t use = (uint32_t)(g >> 1);
            if (!mbar_wait_warp(&bars->tempty[b], (use & 1) ^ 1, abort, err, 3)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(b * kTN);
            for (int kb = 0; kb < kb_count; ++kb) {
              if (!mbar_wait_warp(&bars->full[stage], phase, abort, err, 4)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint64_t a0 = sw128_desc(sA0 + kb * kABytes);
              const uint64_t b0 = sw128_desc(sB0 + stage * kPairBBytes);
              const int kmax = kb == kb_count - 1 ? k_last : kMmaPerStage;
              if (elect_one()) {
                // the next 32 bytes of K: 2 more in the descriptors' 16-byte units
  #pragma unroll
                for (int kk = 0; kk < kMmaPerStage; ++kk)
                  if (kk < kmax) pair_umma<kE4M3>(d, a0 + kk * 2, b0 + kk * 2, (kb | kk) != 0 ? 1u : 0u);
                pair_commit(&bars->empty[stage]);
                if (kb == kb_count - 1) pair_commit(&bars->tfull[b]);
              }
              __syncwarp();
              issued = true;
              if (++stage == nstages) {
                stage = 0;
                phase ^= 1;
              }
            }
            if (!ok) break;
          }
          if (ok && elect_one()) pair_commit(&bars->a_empty);  // the query rows may be replaced once these MMAs complete
          __syncwarp();
        }
        if (!ok && issued) {  // wait for this thread's MMAs before TMEM is freed (bounded)
          if (elect_one()) pair_commit(&bars->drain);
          __syncwarp();
          mbar_wait(&bars->drain, 0, nullptr, nullptr, 0);
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsHigh));
    const int q = warp & 3;          // TMEM lane quarter this warp may access
    const int h = (warp - 4) >> 2;   // column half of every tile
    const int r = q * 32 + lane;
    constexpr int C = kListC;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * kSliceN);
    const float sc = out_scale ? *out_scale : 1.f;
    const uint32_t tempty0 = peer_addr(smem_u32(&bars->tempty[0]), 0);
    int64_t g = 0;
    int seg = 0;
    bool ok = true;
    for (int64_t w = w_begin; w < w_end && ok; ++seg) {
      const Seg sg = segment_at(w, w_end, n_tiles, qblocks, none);
      const int share = (int)(sg.qb % shares);
      int rot = 0;
      w += sg.t1 - sg.t0;
      const int64_t ra = sg.qb / shares * kPairRows + rank * kTM + r;
      const bool row_ok = ra < n_rows;
      const int64_t i = a_rows ? (row_ok ? (int64_t)a_rows[ra] : -1) : ra;
      RowList<C> L;
      L.clear();
      for (int t = sg.t0; t < sg.t1; ++t, ++g) {
        const int b = (int)(g & 1);
        const bool got = mbar_wait(&bars->tfull[b], (uint32_t)(g >> 1) & 1u, abort, err, 5);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // written before the segment's query rows were loaded, which its
        // first accumulator waited for
        if (t == sg.t0) rot = *reinterpret_cast<volatile int*>(&bars->rot[seg & 1]);
        const int kt = (t + rot < n_tiles ? t + rot : t + rot - n_tiles) * shares + share;
        const uint32_t jb = (uint32_t)kt * kTN + (uint32_t)(h * kSliceN);
        const uint32_t tb = lane_base + (uint32_t)(b * kTN);
        auto release = [&] {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) pair_arrive(tempty0 + (uint32_t)(b * sizeof(uint64_t)));
        };
        fold_slice<C>(tb, jb, (uint32_t)n, (uint32_t)i, L, release);
      }
      if (!ok) break;
      L.flush((uint32_t)n, (uint32_t)i);
      float* ov;
      int32_t* oi;
      if (sg.t0 == 0 && sg.t1 == n_tiles) {  // whole block: final lists
        if (!row_ok) continue;
        ov = cand_val + (i * shares + share) * kCandC;
        oi = cand_idx + (i * shares + share) * kCandC;
      } else {
        const int64_t slot = (pair * 2 + (seg == 0 ? 0 : 1)) * kPairRows + rank * kTM + r;
        ov = part_val + slot * kCandC;
        oi = part_idx + slot * kCandC;
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        ov[h * C + c] = L.lv[c] * sc;
        oi[h * C + c] = L.li[c];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // no CTA leaves while its peer may still signal it or read its keys
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// Lists of the query blocks split between runs: per row and column half, the
// 16 best of the pieces' lists (each piece holds the best of its own key
// tiles, so the result is the best of the whole half).  A thread
// per row (kRows: 128, or 256 for pairs) and half; blocks that one run covered
// return at once.  A piece's 16 entries are loaded together, and a block's
// threads are spread over CTAs of 128: with one entry at a time, both halves in
// one thread and a CTA per block, the eight pieces a block has at n = 2000 took
// 80 us of a call of 185 us.
// Block qb's work items are [x0, x1) = [qb n_tiles, (qb + 1) n_tiles), or
// [blk_ptr[qb], blk_ptr[qb + 1]) in tile-list mode (a block with no tiles
// gets empty lists).
constexpr int kMergeThreads = 128;
template <int kRows>
__global__ void __launch_bounds__(kMergeThreads)
k_merge_lists(int n_tiles, int64_t work, int64_t ctas, const int64_t* __restrict__ blk_ptr,
              const float* __restrict__ part_val, const int32_t* __restrict__ part_idx,
              const int32_t* __restrict__ a_rows, int64_t n_rows, int shares, float* __restrict__ cand_val,
              int32_t* __restrict__ cand_idx) {
  static_assert(kLists == 2 && kListC == 16, "a thread per half, four 16-byte loads per list");
  const int64_t qb = blockIdx.x;
  const int64_t x0 = blk_ptr ? blk_ptr[qb] : qb * n_tiles;
  const int64_t x1 = blk_ptr ? blk_ptr[qb + 1] : x0 + n_tiles;
  const int t = blockIdx.y * kMergeThreads + threadIdx.x;
  const int r = t % kRows, h = t / kRows;
  const int64_t ra = qb / shares * kRows + r;
  if (ra >= n_rows) return;
  const int64_t i = (a_rows ? (int64_t)a_rows[ra] : ra) * shares + qb % shares;  // the lists' row
  constexpr int C = kListC;
  float* ov = cand_val + i * kCandC + h * C;
  int32_t* oi = cand_idx + i * kCandC + h * C;
  float lv[C];
  int32_t li[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    lv[c] = -INFINITY;
    li[c] = -1;
  }
  // the list run cc left for the block
  auto load = [&](int64_t cc, float (&v)[C], int32_t (&j)[C]) {
    const int64_t b = range_begin(cc, work, ctas);
    const int64_t slot = (cc * 2 + (b >= x0 ? 0 : 1)) * kRows + r;  // run cc starts inside the block: its first segment
    const float4* pv = reinterpret_cast<const float4*>(part_val + slot * kCandC + h * C);
    const int4* pi = reinterpret_cast<const int4*>(part_idx + slot * kCandC + h * C);
#pragma unroll
    for (int q = 0; q < C / 4; ++q) {
      const float4 f = pv[q];
      const int4 g = pi[q];
      v[4 * q] = f.x, v[4 * q + 1] = f.y, v[4 * q + 2] = f.z, v[4 * q + 3] = f.w;
      j[4 * q] = g.x, j[4 * q + 1] = g.y, j[4 * q + 2] = g.z, j[4 * q + 3] = g.w;
    }
  };
  if (x0 < x1) {
    const int64_t c0 = ((x0 + 1) * ctas + work - 1) / work - 1;  // the CTA whose range holds x0
    if (range_begin(c0 + 1, work, ctas) >= x1) return;           // covered whole: its lists are final
    load(c0, lv, li);  // the first piece is the list so far
    for (int64_t cc = c0 + 1; cc < ctas && range_begin(cc, work, ctas) < x1; ++cc) {
      float v[C];
      int32_t j[C];
      load(cc, v, j);
      // the piece is sorted: nothing after its first entry that does not pass can pass
#pragma unroll
      for (int e = 0; e < C; ++e) {
        if (!(j[e] >= 0 && v[e] > lv[C - 1])) break;
        sorted_insert<C>(lv, li, v[e], j[e]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < C / 4; ++q) {
    reinterpret_cast<float4*>(ov)[q] = make_float4(lv[4 * q], lv[4 * q + 1], lv[4 * q + 2], lv[4 * q + 3]);
    reinterpret_cast<int4*>(oi)[q] = make_int4(li[4 * q], li[4 * q + 1], li[4 * q + 2], li[4 * q + 3]);
  }
}

// pipeline depth and dynamic shared memory for kb_count blocks of A
ancka_status tc_smem(int kb_count, int* nstages, size_t* smem) {
  const size_t fixed = 1024 + (size_t)kb_count * kABytes + sizeof(Bars);
  int ns = (int)((kMaxSmem - fixed) / kBBytes);
  if (ns > kMaxStages) ns = kMaxStages;
  if (ns < 2) {
    set_error("tensor-core contraction: not enough shared memory for two stages");
    return ANCKA_ERR_UNSUPPORTED;
  }
  // at least ~120 KB so that one CTA owns an SM and its 512 TMEM columns
  size_t sm = fixed + (size_t)ns * kBBytes;
  if (sm < 120 * 1024) sm = 120 * 1024;
  *nstages = ns;
  *smem = sm;
  return ANCKA_OK;
}

// ---------------------------------------------------------------------------
// Symmetric contraction (the scores are symmetric: s_ij = s_ji).
//
// Only the pairs j > i are multiplied: the tiles (query block qb, key tile t)
// with t >= qb / 2, in stream-K runs as above.  Every row-half (the keys of
// one column half of the 256-key tiles, the halves of the two lists) has a
// threshold L, the 16th-best score of that row-half over every 8th key tile
// (the list kernel with key_stride 8): at least 16 keys of the full half
// score >= L.  A tile's score s_ij is appended to row i's buffer when s_ij >=
// L_i (row path, half = the key's column half) and to row j's buffer when
// s_ij >= L_j (column path, half = (i mod 256) / 128 = qb & 1, the same for
// the whole CTA); a per-32-key minimum of the column thresholds skips most
// chunks.  k_sym_select then takes each row-half's 16 best, which are the
// lists of a full sweep: a key left out scored below L or below the 16th
// collected score.  A row whose buffer overflowed gets empty lists, which
// the certificate sends to the exact fallback.
// ---------------------------------------------------------------------------
constexpr int kSymStride = 8;  // key tiles of the sampled pass

// first work item of query block qb: sum over q < qb of (n_tiles - q / 2)
__device__ __forceinline__ int64_t sym_start(int64_t qb, int64_t n_tiles) {
  const int64_t a = qb >> 1;
  const int64_t s = (qb & 1) ? a * a : a * (a - 1);
  return qb * n_tiles - s;
}

// the query block holding work item w (binary search over qb)
__device__ __forceinline__ int64_t sym_block(int64_t w, int64_t qblocks, int64_t n_tiles) {
  int64_t lo = 0, hi = qblocks - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (sym_start(mid, n_tiles) <= w) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// The contraction stages (row-half, key, score) entries: each epilogue warp
// reserves blocks of kSymBlock entries with one atomic and fills them without
// waiting on atomics (unused tails are marked -1); k_sym_scatter then appends
// the entries to per-row-half buffers.
constexpr int kSymBlock = 256;

struct SymArgs {
  const float* L;      // 2 x lstride thresholds (half-major); lstride = 256 x key tiles
  const float* Lmin;   // 2 x (lstride / 32) minima over 32 consecutive rows
  int32_t* st_slot;    // staging: row * 2 + half, -1 unused
  int32_t* st_key;
  float* st_val;
  unsigned long long* st_count;  // entries reserved (may exceed st_cap: overflow)
  int64_t st_cap;
};

__device__ __forceinline__ void sym_stage(const SymArgs& sa, int64_t pos, int32_t slot, int32_t key, float v) {
  if (pos < sa.st_cap) {
    sa.st_slot[pos] = slot;
    sa.st_key[pos] = key;
    sa.st_val[pos] = v;
  }
}

__global__ void __launch_bounds__(kThreads, 1)
k_knn_sym(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int64_t n,
          int64_t n_pad, int64_t qblocks, int kb_count, int nstages, SymArgs sa, int* __restrict__ err) {
  constexpr int kTK = 64;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = sA + kb_count * kABytes;
  Bars* bars = reinterpret_cast<Bars*>(sB + nstages * kBBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_tiles = ceil_div(n_pad, kTN);
  const int64_t work = sym_start(qblocks, n_tiles);
  const int64_t w_begin = range_begin(blockIdx.x, work, gridDim.x);
  const int64_t w_end = range_begin((int64_t)blockIdx.x + 1, work, gridDim.x);
  volatile int* abort = &bars->abort;
  if (threadIdx.x == 0) {
    for (int s = 0; s < nstages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    mbar_init(&bars->a_full, 1);
    mbar_init(&bars->a_empty, 1);
    mbar_init(&bars->tfull[0], 1);
    mbar_init(&bars->tfull[1], 1);
    mbar_init(&bars->tempty[0], kEpiWarps);
    mbar_init(&bars->tempty[1], kEpiWarps);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&bars->tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  // segment of a run: (qb, t0, t1) with t in [qb / 2, n_tiles)
  auto segment = [&](int64_t w, int64_t& qb, int64_t& t0, int64_t& t1) {
    qb = sym_block(w, qblocks, n_tiles);
    t0 = (qb >> 1) + (w - sym_start(qb, n_tiles));
    t1 = w_end - w < n_tiles - t0 ? t0 + (w_end - w) : n_tiles;
  };

  if (warp == 0) {
    if (lane == 0) {
      bool pending[kMaxStages];
      uint32_t pend_par[kMaxStages];
      for (int s = 0; s < kMaxStages; ++s) pending[s] = false;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int seg = 0;
      for (int64_t w = w_begin; w < w_end && ok; ++seg) {
        int64_t qb, t0, t1;
        segment(w, qb, t0, t1);
        w += t1 - t0;
        if (seg > 0 && !mbar_wait(&bars->a_empty, (uint32_t)((seg - 1) & 1), abort, err, 6)) {
          ok = false;
          break;
        }
        mbar_expect_tx(&bars->a_full, (uint32_t)(kb_count * kABytes));
        for (int kb = 0; kb < kb_count; ++kb)
          tma_load_2d(smem_u32(sA + kb * kABytes), &tmA, kb * kTK, (int)(qb * kTM), &bars->a_full);
        for (int64_t t = t0; t < t1 && ok; ++t) {
          for (int kb = 0; kb < kb_count; ++kb) {
            if (!mbar_wait(&bars->empty[stage], phase ^ 1, abort, err, 1)) {
              ok = false;
              break;
            }
            pending[stage] = false;
            mbar_expect_tx(&bars->full[stage], (uint32_t)kBBytes);
            tma_load_2d(smem_u32(sB + stage * kBBytes), &tmB, kb * kTK, (int)(t * kTN), &bars->full[stage]);
            pending[stage] = true;
            pend_par[stage] = phase;
            if (++stage == nstages) {
              stage = 0;
              phase ^= 1;
            }
          }
        }
      }
      if (!ok) {
        if (seg > 0) mbar_wait(&bars->a_full, (uint32_t)((seg - 1) & 1), nullptr, nullptr, 0);
        for (int s = 0; s < nstages; ++s)
          if (pending[s]) mbar_wait(&bars->full[s], pend_par[s], nullptr, nullptr, 0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0;
      bool issued = false;
      int64_t g = 0;
      int seg = 0;
      for (int64_t w = w_begin; w < w_end && ok; ++seg) {
        int64_t qb, t0, t1;
        segment(w, qb, t0, t1);
        w += t1 - t0;
        if (!mbar_wait(&bars->a_full, (uint32_t)(seg & 1), abort, err, 2)) {
          ok = false;
          break;
        }
        for (int64_t t = t0; t < t1; ++t, ++g) {
          const int b = (int)(g & 1);
          const uint32_t use = (uint32_t)(g >> 1);
          if (!mbar_wait(&bars->tempty[b], (use & 1) ^ 1, abort, err, 3)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(b * kTN);
          for (int kb = 0; kb < kb_count; ++kb) {
            if (!mbar_wait(&bars->full[stage], phase, abort, err, 4)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA + kb * kABytes);
            const uint32_t b0 = smem_u32(sB + stage * kBBytes);
#pragma unroll
            for (int kk = 0; kk < kMmaPerStage; ++kk)
              umma_bf16(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), (kb | kk) != 0 ? 1u : 0u);
            issued = true;
            umma_commit(&bars->empty[stage]);
            if (++stage == nstages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (!ok) break;
          umma_commit(&bars->tfull[b]);
        }
        if (ok) umma_commit(&bars->a_empty);
      }
      if (!ok && issued) {
        umma_commit(&bars->drain);
        mbar_wait(&bars->drain, 0, nullptr, nullptr, 0);
      }
    }
  } else {
    const int ew = warp - 2;
    const int q = warp & 3;
    const int h = ew >> 2;  // column half of the tile = the row path's list half
    const int r = q * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
    int64_t g = 0;
    bool ok = true;
    int64_t blk_base = 0;  // the warp's staging block (uniform over the warp)
    int blk_cap = 0, blk_used = 0;
    for (int64_t w = w_begin; w < w_end && ok;) {
      int64_t qb, t0, t1;
      segment(w, qb, t0, t1);
      w += t1 - t0;
      const int64_t i = qb * kTM + r;
      const int64_t lstride = n_tiles * kTN;
      const float Lrow = i < n ? sa.L[(int64_t)h * lstride + i] : INFINITY;
      const int hc = (int)(qb & 1);  // the column path's list half
      const float* Lc = sa.L + (int64_t)hc * lstride;
      const float* Lm = sa.Lmin + (int64_t)hc * (lstride / 32);
      for (int64_t t = t0; t < t1; ++t, ++g) {
        const int b = (int)(g & 1);
        const uint32_t use = (uint32_t)(g >> 1);
        const int64_t jb = t * kTN + h * kSliceN;
        // the tile's column thresholds (lane: keys jb + 4 lane .. + 3) and
        // per-chunk minima, loaded before the wait so that their latency hides
        const float4 lcol = *reinterpret_cast<const float4*>(Lc + jb + 4 * lane);
        const float4 lmin4 = *reinterpret_cast<const float4*>(Lm + (jb >> 5));
        const bool got = mbar_wait(&bars->tfull[b], use & 1, abort, err, 5);
        if (!__all_sync(0xffffffffu, got)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t tb = lane_base + (uint32_t)(b * kTN + h * kSliceN);
#pragma unroll 1
        for (int c = 0; c < kSliceN / 32; ++c) {
          uint32_t rv[32];
          tmem_ld32_issue(tb + (uint32_t)(c * 32), rv);
          tmem_wait();
          pin(rv);
          const int64_t j0 = jb + c * 32;
          // keys j0 + e with i < j < n
          const int64_t lo = i + 1 - j0, hi = n - j0;
          const int e0 = lo < 0 ? 0 : (lo > 32 ? 32 : (int)lo);
          const int e1 = hi < 0 ? 0 : (hi > 32 ? 32 : (int)hi);
          uint32_t vm = 0;
          if (e1 > e0) vm = (e1 - e0 == 32 ? 0xffffffffu : ((1u << (e1 - e0)) - 1u)) << e0;
          float m[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) m[u] = fmaxf(__uint_as_float(rv[u]), __uint_as_float(rv[u + 16]));
#pragma unroll
          for (int u2 = 8; u2 >= 1; u2 >>= 1)
#pragma unroll
            for (int u = 0; u < u2; ++u) m[u] = fmaxf(m[u], m[u + u2]);
          const float mx = vm ? m[0] : -INFINITY;
          uint32_t pr = 0, pc = 0;
          if (__any_sync(0xffffffffu, mx >= Lrow)) {  // row path
#pragma unroll
            for (int e = 0; e < 32; ++e) pr |= (__uint_as_float(rv[e]) >= Lrow ? 1u : 0u) << e;
            pr &= vm;
          }
          const float lmin = c == 0 ? lmin4.x : c == 1 ? lmin4.y : c == 2 ? lmin4.z : lmin4.w;
          if (__any_sync(0xffffffffu, mx >= lmin)) {  // column path
#pragma unroll
            for (int e4 = 0; e4 < 8; ++e4) {  // chunk c's thresholds sit in lanes 8c .. 8c + 7
              const int src = c * 8 + e4;
              const float t0v = __shfl_sync(0xffffffffu, lcol.x, src);
              const float t1v = __shfl_sync(0xffffffffu, lcol.y, src);
              const float t2v = __shfl_sync(0xffffffffu, lcol.z, src);
              const float t3v = __shfl_sync(0xffffffffu, lcol.w, src);
              pc |= (__uint_as_float(rv[4 * e4]) >= t0v ? 1u : 0u) << (4 * e4);
              pc |= (__uint_as_float(rv[4 * e4 + 1]) >= t1v ? 1u : 0u) << (4 * e4 + 1);
              pc |= (__uint_as_float(rv[4 * e4 + 2]) >= t2v ? 1u : 0u) << (4 * e4 + 2);
              pc |= (__uint_as_float(rv[4 * e4 + 3]) >= t3v ? 1u : 0u) << (4 * e4 + 3);
            }
            pc &= vm;
          }
          // the warp's entries: one exclusive prefix, one block reservation when needed
          const int cl = __popc(pr) + __popc(pc);
          int incl = cl;
#pragma unroll
          for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
          }
          const int ctot = __shfl_sync(0xffffffffu, incl, 31);
          if (ctot > 0) {
            if (blk_used + ctot > blk_cap) {
              for (int e = blk_used + lane; e < blk_cap; e += 32) sym_stage(sa, blk_base + e, -1, -1, 0.f);
              const int nblk = (ctot + kSymBlock - 1) / kSymBlock;
              unsigned long long b = 0;
              if (lane == 0) b = atomicAdd(sa.st_count, (unsigned long long)nblk * kSymBlock);
              blk_base = (int64_t)__shfl_sync(0xffffffffu, b, 0);
              blk_cap = nblk * kSymBlock;
              blk_used = 0;
            }
            int64_t pos = blk_base + blk_used + (incl - cl);
            while (pr) {
              const int e = __ffs(pr) - 1;
              pr &= pr - 1;
              sym_stage(sa, pos++, (int32_t)(i * 2 + h), (int32_t)(j0 + e), pick32(rv, e));
            }
            while (pc) {
              const int e = __ffs(pc) - 1;
              pc &= pc - 1;
              sym_stage(sa, pos++, (int32_t)((j0 + e) * 2 + hc), (int32_t)i, pick32(rv, e));
            }
            blk_used += ctot;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->tempty[b]);
      }
    }
    for (int e = blk_used + lane; e < blk_cap; e += 32) sym_stage(sa, blk_base + e, -1, -1, 0.f);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// the staged entries into per-row-half buffers (cnt counts past cap); a
// staging overflow marks every row (overflow flag), so that all go to the
// exact fallback
__global__ void k_sym_scatter(const int32_t* __restrict__ st_slot, const int32_t* __restrict__ st_key,
                              const float* __restrict__ st_val, const unsigned long long* __restrict__ st_count,
                              int64_t st_cap, int32_t* __restrict__ cnt, float* __restrict__ bufv,
                              int32_t* __restrict__ bufi, int cap, int32_t* __restrict__ overflow) {
  const unsigned long long tot = *st_count;
  if (tot > (unsigned long long)st_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *overflow = 1;
    return;
  }
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)tot;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t slot = st_slot[q];
    if (slot < 0) continue;
    const int pos = atomicAdd(&cnt[slot], 1);
    if (pos < cap) {
      bufv[(int64_t)slot * cap + pos] = st_val[q];
      bufi[(int64_t)slot * cap + pos] = st_key[q];
    }
  }
}

// thresholds from the sampled lists: L[h][i] = the 16th score of row i's
// half-h list (sorted descending), -inf if that list is not full; rows >= n
// +inf; Lmin[h][g] = min over rows 32g .. 32g + 31 (lstride a multiple of 256)
__global__ void k_sym_thresholds(const float* __restrict__ cand_val, const int32_t* __restrict__ cand_idx,
                                 int64_t n, int64_t lstride, float* __restrict__ L, float* __restrict__ Lmin) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= lstride) return;
  const int64_t n_pad = lstride;
  for (int h = 0; h < 2; ++h) {
    float v = INFINITY;
    if (i < n) {
      const int64_t last = i * kCandC + h * kListC + (kListC - 1);
      v = cand_idx[last] >= 0 ? cand_val[last] : -INFINITY;
    }
    L[(int64_t)h * n_pad + i] = v;
    float mn = v;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
    if ((threadIdx.x & 31) == 0) Lmin[(int64_t)h * (n_pad / 32) + (i >> 5)] = mn;
  }
}

// each row's two lists: the 16 best collected entries per half, sorted
// descending; a row with an overflowing half gets two empty lists (sent to
// the exact fallback by the certificate)
__global__ void k_sym_select(const int32_t* __restrict__ cnt, const float* __restrict__ bufv,
                             const int32_t* __restrict__ bufi, int cap, int64_t n,
                             const int32_t* __restrict__ overflow, float* __restrict__ cand_val,
                             int32_t* __restrict__ cand_idx) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool over = *overflow || cnt[i * 2] > cap || cnt[i * 2 + 1] > cap;
  constexpr int C = kListC;
  for (int h = 0; h < 2; ++h) {
    float lv[C];
    int32_t li[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      lv[c] = -INFINITY;
      li[c] = -1;
    }
    if (!over) {
      const int64_t slot = i * 2 + h;
      const int c_n = cnt[slot];
      for (int e = 0; e < c_n; ++e) {
        const float v = bufv[slot * cap + e];
        if (v > lv[C - 1]) sorted_insert<C>(lv, li, v, bufi[slot * cap + e]);
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      cand_val[i * kCandC + h * C + c] = lv[c];
      cand_idx[i * kCandC + h * C + c] = li[c];
    }
  }
}

__global__ void k_gather_rows(const uint8_t* __restrict__ x, int row_bytes, const int32_t* __restrict__ rows,
                              int64_t n_a, int64_t n_a_pad, uint8_t* __restrict__ out) {
  const int64_t r = blockIdx.x;
  if (r >= n_a_pad) return;
  const uint4* src = r < n_a ? reinterpret_cast<const uint4*>(x + (int64_t)rows[r] * row_bytes) : nullptr;
  uint4* dst = reinterpret_cast<uint4*>(out + r * row_bytes);
  for (int c = threadIdx.x; c < row_bytes / 16; c += blockDim.x) dst[c] = src ? src[c] : make_uint4(0, 0, 0, 0);
}

// One persistent CTA per SM (at most one per work item); list mode adds the
// partial-list area and the merge of split query blocks.
template <bool kCollect>
ancka_status launch_tc(Workspace& ws, const CUtensorMap& ta, const CUtensorMap& tb, int64_t n, int64_t n_pad,
                       int64_t n_rows, int kb_count, int d, float* cand_val, int32_t* cand_idx,
                       const CollectArgs& ca, int32_t* err, cudaStream_t s, int key_stride = 1) {
  // MMAs over the last 128-byte feature block: K = 16 features each; the
  // padding past d is zero and needs none
  const int per_kb = 64, per_mma = 16;
  const int rem = d - per_kb * (kb_count - 1);
  const int k_last = (rem >= 1 && rem <= per_kb) ? (int)ceil_div(rem, per_mma) : kMmaPerStage;
  int nstages;
  size_t smem;
  ANCKA_TRY(tc_smem(kb_count, &nstages, &smem));
  int sms = 152, dev = 0;
  ANCKA_CUDA(cudaGetDevice(&dev));
  ANCKA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t qblocks = ceil_div(n_rows, kTM);
  const int n_tiles = (int)ceil_div(ceil_div(n_pad, kTN), key_stride);
  const int64_t work = ca.blk_ptr ? ca.blk_work : qblocks * n_tiles;
  const int64_t ctas = std::max<int64_t>(1, std::min<int64_t>(sms, work));
  float* part_val = nullptr;
  int32_t* part_idx = nullptr;
  if (!kCollect) {
    ANCKA_TRY(ws.alloc(&part_val, (size_t)ctas * 2 * kTM * kCandC));
    ANCKA_TRY(ws.alloc(&part_idx, (size_t)ctas * 2 * kTM * kCandC));
  }
  unsigned long long* tick = nullptr;  // tiles issued by all CTAs (re-aligns whole blocks' key order)
  if (kCollect) ANCKA_TRY(ws.zeros(&tick, 1));
  ANCKA_CUDA(cudaFuncSetAttribute(k_knn_tc<kCollect>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  k_knn_tc<kCollect><<<(unsigned)ctas, kTcThreads, smem, s>>>(ta, tb, n, n_pad, qblocks, kb_count, k_last,
                                                                   nstages, key_stride, cand_val, cand_idx,
                                                                   part_val, part_idx, ca, tick, err);
  ANCKA_LAUNCHED();
  if (!kCollect) {
    k_merge_lists<kTM><<<dim3((unsigned)qblocks, 2 * kTM / kMergeThreads), kMergeThreads, 0, s>>>(n_tiles, work, ctas, ca.blk_ptr, part_val, part_idx, ca.a_rows,
                                                    n_rows, 1, cand_val, cand_idx);
    ANCKA_LAUNCHED();
  }
  return ANCKA_OK;
}

// The full sweep by CTA pairs: every row's two lists over all keys (rows of
// a_rows, written at their own row index, or rows 0..n-1).
template <bool kE4M3>
ancka_status launch_pair(Workspace& ws, const CUtensorMap& ta, const CUtensorMap& tb, int64_t n, int64_t n_pad,
                         const int32_t* a_rows, int64_t n_rows, int kb_count, int d, float* cand_val,
                         int32_t* cand_idx, const float* out_scale, int32_t* err, cudaStream_t s, int shares = 1) {
  const int per_kb = kE4M3 ? 128 : 64, per_mma = kE4M3 ? 32 : 16;  // k_last as in launch_tc
  const int rem = d - per_kb * (kb_count - 1);
  const int k_last = (rem >= 1 && rem <= per_kb) ? (int)ceil_div(rem, per_mma) : kMmaPerStage;
  const size_t fixed = 1024 + (size_t)kb_count * kABytes + sizeof(PairBars);
  const int nstages = (int)std::min<size_t>(kPairMaxStages, (kMaxSmem - fixed) / kPairBBytes);
  const size_t smem = fixed + (size_t)nstages * kPairBBytes;  // > 120 KB for every kb_count: one CTA per SM
  if (nstages < 4) {
    set_error("tensor-core contraction: not enough shared memory for four stages");
    return ANCKA_ERR_UNSUPPORTED;
  }
  int sms = 152, dev = 0;
  ANCKA_CUDA(cudaGetDevice(&dev));
  ANCKA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t qblocks = ceil_div(n_rows, kPairRows) * shares;
  const int n_tiles = (int)ceil_div(ceil_div(n_pad, kTN), shares);
  const int64_t work = qblocks * n_tiles;
  const int64_t pairs = std::max<int64_t>(1, std::min<int64_t>(sms / 2, work));
  float* part_val;
  int32_t* part_idx;
  unsigned long long* tick;
  ANCKA_TRY(ws.alloc(&part_val, (size_t)pairs * 2 * kPairRows * kCandC));
  ANCKA_TRY(ws.alloc(&part_idx, (size_t)pairs * 2 * kPairRows * kCandC));
  ANCKA_TRY(ws.zeros(&tick, 1));
  auto kernel = k_knn_pair<kE4M3, false>;
  if constexpr (!kE4M3)
    if (shares > 1) kernel = k_knn_pair<kE4M3, true>;
  ANCKA_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  kernel<<<(unsigned)(2 * pairs), kTcThreads, smem, s>>>(
      ta, tb, n, n_pad, qblocks, kb_count, k_last, nstages, cand_val, cand_idx, out_scale, part_val, part_idx,
      a_rows, n_rows, shares, tick, err);
  ANCKA_LAUNCHED();
  k_merge_lists<kPairRows><<<dim3((unsigned)qblocks, 2 * kPairRows / kMergeThreads), kMergeThreads, 0, s>>>(n_tiles, work, pairs, nullptr, part_val, part_idx,
                                                                   a_rows, n_rows, shares, cand_val, cand_idx);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

int64_t sym_start_host(int64_t qb, int64_t n_tiles) {
  const int64_t a = qb >> 1;
  return qb * n_tiles - ((qb & 1) ? a * a : a * (a - 1));
}

// off by default: on the measured workloads the symmetric form is slower than
// the full sweep (its fixed thresholds admit ~8x more candidates than the
// full sweep's running ones, so its epilogue does about twice the work per
// tile over half the tiles)
std::atomic<int64_t> g_sym_min_rows{INT64_MAX};

// BF16 lists by the symmetric contraction (sampled thresholds, the j > i
// tiles with both paths, selection)
ancka_status knn_candidates_bf16_sym(Workspace& ws, const PrepOut& pr, int64_t n, const CUtensorMap& ta,
                                     const CUtensorMap& tb, int kb_count, float* cand_val, int32_t* cand_idx,
                                     int32_t* err, cudaStream_t s) {
  // 1. sampled lists: every kSymStride-th key tile
  float* sv;
  int32_t* si;
  ANCKA_TRY(ws.alloc(&sv, (size_t)n * kCandC));
  ANCKA_TRY(ws.alloc(&si, (size_t)n * kCandC));
  CollectArgs none{};
  const ancka_status st = launch_tc<false>(ws, ta, tb, n, pr.n_pad, n, kb_count, pr.d, sv, si, none,
                                                  err, s, kSymStride);
  if (st != ANCKA_OK) return st;
  // 2. thresholds
  const int64_t n_tiles = ceil_div(pr.n_pad, kTN);
  const int64_t lstride = n_tiles * kTN;
  float *L, *Lmin;
  ANCKA_TRY(ws.alloc(&L, (size_t)2 * lstride));
  ANCKA_TRY(ws.alloc(&Lmin, (size_t)2 * (lstride / 32)));
  k_sym_thresholds<<<(unsigned)(lstride / 256), 256, 0, s>>>(sv, si, n, lstride, L, Lmin);
  ANCKA_LAUNCHED();
  // 3. the j > i tiles, both paths
  constexpr int kCap = 320;  // ~16 x kSymStride entries expected per row-half
  SymArgs sa{L, Lmin, nullptr, nullptr, nullptr, nullptr, 0};
  sa.st_cap = n * 2 * 16 * kSymStride * 5 / 2 + (int64_t)8 * kThreads / 32 * kSymBlock * 152;
  ANCKA_TRY(ws.alloc(&sa.st_slot, (size_t)sa.st_cap));
  ANCKA_TRY(ws.alloc(&sa.st_key, (size_t)sa.st_cap));
  ANCKA_TRY(ws.alloc(&sa.st_val, (size_t)sa.st_cap));
  ANCKA_TRY(ws.zeros(&sa.st_count, 1));
  int32_t *cnt, *bufi, *overflow;
  float* bufv;
  ANCKA_TRY(ws.zeros(&cnt, (size_t)n * 2));
  ANCKA_TRY(ws.alloc(&bufv, (size_t)n * 2 * kCap));
  ANCKA_TRY(ws.alloc(&bufi, (size_t)n * 2 * kCap));
  ANCKA_TRY(ws.zeros(&overflow, 1));
  int nstages;
  size_t smem;
  ANCKA_TRY(tc_smem(kb_count, &nstages, &smem));
  int sms = 152, dev = 0;
  ANCKA_CUDA(cudaGetDevice(&dev));
  ANCKA_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t qblocks = ceil_div(n, kTM);
  const int64_t work = sym_start_host(qblocks, n_tiles);
  const int64_t ctas = std::min<int64_t>(sms, work);
  ANCKA_CUDA(cudaFuncSetAttribute(k_knn_sym, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  k_knn_sym<<<(unsigned)ctas, kThreads, smem, s>>>(ta, tb, n, pr.n_pad, qblocks, kb_count, nstages, sa, err);
  ANCKA_LAUNCHED();
  // 4. staged entries into the row-half buffers, then the two lists of every row
  k_sym_scatter<<<(unsigned)(4 * sms), 256, 0, s>>>(sa.st_slot, sa.st_key, sa.st_val, sa.st_count, sa.st_cap, cnt,
                                                   bufv, bufi, kCap, overflow);
  ANCKA_LAUNCHED();
  k_sym_select<<<(unsigned)ceil_div(n, 128), 128, 0, s>>>(cnt, bufv, bufi, kCap, n, overflow, cand_val, cand_idx);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

}  // namespace

bool knn_tc_available() { return true; }

int knn_tc_max_dp() { return 512; }

ancka_status knn_candidates_bf16(Workspace& ws, const PrepOut& pr, int64_t n, float* cand_val, int32_t* cand_idx,
                                 int32_t* err, cudaStream_t s) {
  const int kb_count = pr.dp / 64;
  if (pr.dp % 64 != 0 || kb_count < 1 || pr.dp > knn_tc_max_dp()) {
    set_error("BF16 contraction supports up to %d features (got %d)", knn_tc_max_dp(), pr.dp);
    return ANCKA_ERR_UNSUPPORTED;
  }
  CUtensorMap ta, tb;
  ANCKA_TRY(make_map(&ta, pr.xb, pr.dp, pr.n_pad, kTM, 2));
  if (n >= g_sym_min_rows.load(std::memory_order_relaxed)) {
    ANCKA_TRY(make_map(&tb, pr.xb, pr.dp, pr.n_pad, kTN, 2));
    return knn_candidates_bf16_sym(ws, pr, n, ta, tb, kb_count, cand_val, cand_idx, err, s);
  }
  ANCKA_TRY(make_map(&tb, pr.xb, pr.dp, pr.n_pad, kTN / 2, 2));
  return launch_pair<false>(ws, ta, tb, n, pr.n_pad, nullptr, n, kb_count, pr.d, cand_val, cand_idx, nullptr, err, s);
}

// two lists per row and share of the key tiles (see k_knn_pair)
ancka_status knn_candidates_bf16_shares(Workspace& ws, const PrepOut& pr, int64_t n, int shares, float* cand_val,
                                        int32_t* cand_idx, int32_t* err, cudaStream_t s) {
  CUtensorMap ta, tb;
  ANCKA_TRY(make_map(&ta, pr.xb, pr.dp, pr.n_pad, kTM, 2));
  ANCKA_TRY(make_map(&tb, pr.xb, pr.dp, pr.n_pad, kTN / 2, 2));
  return launch_pair<false>(ws, ta, tb, n, pr.n_pad, nullptr, n, pr.dp / 64, pr.d, cand_val, cand_idx, nullptr, err, s,
                            shares);
}

void knn_set_symmetric_min_rows(int64_t n_min) { g_sym_min_rows.store(n_min, std::memory_order_relaxed); }

ancka_status knn_candidates_fp8(Workspace& ws, const PrepOut& pr, int64_t n, float* cand_val, int32_t* cand_idx,
                                int32_t* err, cudaStream_t s) {
  const int kb_count = pr.dp8 / 128;
  if (!pr.x8 || pr.dp8 % 128 != 0 || kb_count < 1 || pr.dp8 > knn_tc_max_dp_fp8()) {
    set_error("FP8 contraction supports up to %d features (got %d)", knn_tc_max_dp_fp8(), pr.dp8);
    return ANCKA_ERR_UNSUPPORTED;
  }
  CUtensorMap ta, tb;
  ANCKA_TRY(make_map(&ta, pr.x8, pr.dp8, pr.n_pad, kTM, 1));
  ANCKA_TRY(make_map(&tb, pr.x8, pr.dp8, pr.n_pad, kTN / 2, 1));
  return launch_pair<true>(ws, ta, tb, n, pr.n_pad, nullptr, n, kb_count, pr.d, cand_val, cand_idx, pr.inv_s2, err, s);
}

int knn_tc_max_dp_fp8() { return 1024; }

// BF16 lists for the n_a rows listed in rows (written at their global rows)
ancka_status knn_list_gathered_bf16(Workspace& ws, const PrepOut& pr, int64_t n, const int32_t* rows, int64_t n_a,
                                    float* cand_val, int32_t* cand_idx, int32_t* err, cudaStream_t s) {
  const int kb_count = pr.dp / 64;
  const int64_t n_a_pad = round_up(n_a, kTM);
  __nv_bfloat16* af;
  ANCKA_TRY(ws.alloc(&af, (size_t)n_a_pad * pr.dp));
  k_gather_rows<<<(unsigned)n_a_pad, 64, 0, s>>>(reinterpret_cast<const uint8_t*>(pr.xb), pr.dp * 2, rows, n_a,
                                                 n_a_pad, reinterpret_cast<uint8_t*>(af));
  ANCKA_LAUNCHED();
  CUtensorMap ta, tb;
  ANCKA_TRY(make_map(&ta, af, pr.dp, n_a_pad, kTM, 2));
  ANCKA_TRY(make_map(&tb, pr.xb, pr.dp, pr.n_pad, kTN / 2, 2));
  return launch_pair<false>(ws, ta, tb, n, pr.n_pad, rows, n_a, kb_count, pr.d, cand_val, cand_idx, nullptr, err, s);
}

ancka_status knn_lists_bf16(Workspace& ws, const __nv_bfloat16* a, int64_t a_rows_total, const int32_t* rows,
                           int64_t n_rows, const __nv_bfloat16* keys, int64_t n_keys, int64_t keys_pad, int dp, int d,
                           const int64_t* blk_ptr, const int32_t* blk_tiles, int64_t blk_work, bool no_self,
                           float* cand_val, int32_t* cand_idx, int32_t* err, cudaStream_t s) {
  const int kb_count = dp / 64;
  if (dp % 64 != 0 || kb_count < 1 || dp > knn_tc_max_dp()) {
    set_error("BF16 contraction supports up to %d features (got %d)", knn_tc_max_dp(), dp);
    return ANCKA_ERR_UNSUPPORTED;
  }
  CUtensorMap ta, tb;
  if (rows) {
    const int64_t n_a_pad = round_up(n_rows, kTM);
    __nv_bfloat16* af;
    ANCKA_TRY(ws.alloc(&af, (size_t)n_a_pad * dp));
    k_gather_rows<<<(unsigned)n_a_pad, 64, 0, s>>>(reinterpret_cast<const uint8_t*>(a), dp * 2, rows, n_rows,
                                                   n_a_pad, reinterpret_cast<uint8_t*>(af));
    ANCKA_LAUNCHED();
    ANCKA_TRY(make_map(&ta, af, dp, n_a_pad, kTM, 2));
  } else {
    ANCKA_TRY(make_map(&ta, a, dp, round_up(a_rows_total, kTM), kTM, 2));
  }
  ANCKA_TRY(make_map(&tb, keys, dp, keys_pad, kTN, 2));
  CollectArgs ca{rows, n_rows, nullptr, nullptr, nullptr, 0};
  ca.blk_ptr = blk_ptr;
  ca.blk_tiles = blk_tiles;
  ca.blk_work = blk_work;
  ca.no_self = no_self ? 1 : 0;
  return launch_tc<false>(ws, ta, tb, n_keys, keys_pad, n_rows, kb_count, d, cand_val, cand_idx, ca, err, s);
}

ancka_status knn_collect_bf16(Workspace& ws, const PrepOut& pr, int64_t n, const int32_t* rows, int64_t n_a,
                              const float* thr, int32_t* cnt, int32_t* buf, int cap, int32_t* err, cudaStream_t s) {
  const int kb_count = pr.dp / 64;
  const int64_t n_a_pad = round_up(n_a, kTM);
  __nv_bfloat16* af;
  ANCKA_TRY(ws.alloc(&af, (size_t)n_a_pad * pr.dp));
  k_gather_rows<<<(unsigned)n_a_pad, 64, 0, s>>>(reinterpret_cast<const uint8_t*>(pr.xb), pr.dp * 2, rows, n_a,
                                                 n_a_pad, reinterpret_cast<uint8_t*>(af));
  ANCKA_LAUNCHED();
  CUtensorMap ta, tb;
  ANCKA_TRY(make_map(&ta, af, pr.dp, n_a_pad, kTM, 2));
  ANCKA_TRY(make_map(&tb, pr.xb, pr.dp, pr.n_pad, kTN, 2));
  CollectArgs ca{rows, n_a, thr, cnt, buf, cap};
  return launch_tc<true>(ws, ta, tb, n, pr.n_pad, n_a, kb_count, pr.d, nullptr, nullptr, ca, err, s);
}

}  // namespace ancka
