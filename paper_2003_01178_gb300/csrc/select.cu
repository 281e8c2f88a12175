// Selection (Section 3.2 query Q0, Section 4.2 query Q3) as one persistent kernel.
//
// Per tile: BlockLoad (bulk copy into a shared-memory stage) -> BlockPred (range
// predicate into a per-thread bitmap in registers) -> BlockScan (a warp scan of packed
// per-thread counts, then one warp scans the warps' totals) -> one output reservation
// per tile -> BlockShuffle (each warp compacts its rows into its own shared-memory
// run) -> BlockStore (coalesced stores of each warp's run).
//
// Each warp owns a contiguous run of ITEMS*32 rows of the tile (lane l reads the
// 4-value groups j*128 + 4l, j < ITEMS/4) and compacts its selected values in input
// order into its own shared-memory run.  A first block barrier publishes the warp totals
// (the stage goes back to the copy engine right after it); warp 0 turns them into
// offsets and makes the tile's single output reservation; after a second barrier every
// warp stores its run with coalesced writes.  In the unordered mode a tile without
// matches stops after the first barrier.  Full tiles read the stage without tail checks.
//
// Output reservation: mode 0 adds the tile's count to the global cursor with one
// atomic (the paper's scheme); mode 1 (select_ordered_kernel) turns the tiles' counts into
// positions in tile order (tile ids handed out in order by an atomic counter, so a tile
// only waits on tiles that running blocks already hold) and the result is in input order.
#include <cooperative_groups.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "pipeline.cuh"
#include "tiles.h"

namespace crys {
namespace {

constexpr uint64_t kFlagAggregate = 1ull << 62;
constexpr uint64_t kFlagInclusive = 2ull << 62;
constexpr uint64_t kValueMask = (1ull << 62) - 1;

struct SelectArgs {
  const int32_t* x;
  int64_t n;
  int32_t lo, hi;
  uint32_t span;  // hi - lo; only used when lo <= hi
  int32_t* out;
  unsigned long long* count;  // cursor (mode 0) / final count (mode 1)
  uint64_t* tile_state;       // mode 1: one status word per tile
  unsigned int* tile_counter; // mode 1: next tile id (scratch header, word 0)
  unsigned int* block_counter; // mode 1: blocks that have started (the first one scans)
  unsigned int* abort_word;   // mode 1: set by the first block of this call that gives up
  uint32_t tile_base;         // mode 1: first tile id handed out (0 unless a test stalls)
  uint64_t wait_ns;           // mode 1: bound of a wait for a count or a position
  int32_t* err;
  int32_t stages;
};

// BlockLoad + BlockPred of one warp: its rows warp*WROWS + j*128 + lane*4 + e of the staged
// tile, values into v and the predicate's bitmap returned.  A full tile (all but possibly
// the last) reads the stage without tail checks; rows past the copied groups of a ragged
// tile come from `gcol`.
template <int THREADS, int ITEMS>
__device__ __forceinline__ uint32_t load_pred(const int32_t* st, const int32_t* gcol, int valid, int32_t lo,
                                              uint32_t span, int32_t (&v)[ITEMS]) {
  constexpr int TILE = THREADS * ITEMS, VEC = ITEMS / 4, WROWS = ITEMS * kWarp;
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const int bulk = valid & ~3;
  uint32_t bits = 0;
  auto body = [&](auto full_tag) {
    constexpr bool FULL = decltype(full_tag)::value;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
      const int p = warp * WROWS + j * 128 + lane * 4;
      const int4 q = FULL ? *reinterpret_cast<const int4*>(st + p) : stage_read4(st, gcol, p, bulk, valid);
      v[4 * j + 0] = q.x;
      v[4 * j + 1] = q.y;
      v[4 * j + 2] = q.z;
      v[4 * j + 3] = q.w;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // lo <= v <= hi as one unsigned comparison (span = hi - lo, lo <= hi)
        const bool hit = (FULL || p + e < valid) &&
                         static_cast<uint32_t>(v[4 * j + e]) - static_cast<uint32_t>(lo) <= span;
        bits |= static_cast<uint32_t>(hit) << (4 * j + e);
      }
    }
  };
  if (valid == TILE)
    body(std::true_type{});
  else
    body(std::false_type{});
  return bits;
}

// BlockScan + BlockShuffle of one warp: its selected values, in input order, to `dst`; returns
// how many.  One warp scan covers the per-lane counts of all ITEMS/4 groups at once
// (group j's count in byte j; a group's warp total is at most 128).
template <int ITEMS>
__device__ __forceinline__ int compact_warp(const int32_t (&v)[ITEMS], uint32_t bits, int32_t* dst) {
  constexpr int VEC = ITEMS / 4;
  const int lane = threadIdx.x % kWarp;
  uint32_t packed = 0;
#pragma unroll
  for (int j = 0; j < VEC; ++j) packed |= static_cast<uint32_t>(__popc((bits >> (4 * j)) & 0xFu)) << (8 * j);
  const uint32_t incl = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(packed), lane));
  const uint32_t excl = incl - packed;
  const uint32_t totals = __shfl_sync(0xFFFFFFFFu, incl, kWarp - 1);
  int run = 0;
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    int pos = run + static_cast<int>((excl >> (8 * j)) & 0xFFu);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (bits & (1u << (4 * j + e))) dst[pos++] = v[4 * j + e];
    }
    run += static_cast<int>((totals >> (8 * j)) & 0xFFu);
  }
  return run;
}

template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS) select_kernel(SelectArgs a) {
  constexpr int TILE = THREADS * ITEMS;
  constexpr int VEC = ITEMS / 4;
  constexpr int WARPS = THREADS / kWarp;
  constexpr int WROWS = ITEMS * kWarp;  // rows of a tile owned by one warp, contiguous
  static_assert(ITEMS % 4 == 0 && VEC <= 4, "4..16 items per thread");
  static_assert(WARPS <= kWarp, "one warp scans the warp totals");

  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int S = a.stages;
  int32_t* stages = reinterpret_cast<int32_t*>(smem_raw);    // S x TILE
  int32_t* wbuf_all = stages + S * TILE;                     // per-warp compaction runs
  __shared__ StageRing ring;
  __shared__ int32_t wtot[WARPS];
  __shared__ int32_t woff[WARPS];
  __shared__ long long out_base;

  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  int32_t* wbuf = wbuf_all + warp * WROWS;
  const int64_t ntiles = (a.n + TILE - 1) / TILE;
  const uint64_t pol = policy_evict_first();
  int64_t issued = 0;  // thread 0 only

  auto issue = [&](int s) {
    const int64_t t = static_cast<int64_t>(blockIdx.x) + issued * gridDim.x;
    ++issued;
    if (t >= ntiles) {
      ring.tile[s] = -1;
      return;
    }
    ring.tile[s] = t;
    const int64_t row = t * TILE;
    const int64_t valid = (a.n - row) < TILE ? (a.n - row) : TILE;
    ring_issue(&ring.full[s], stages + s * TILE, TILE, &a.x, 1, row, valid, pol);
  };

  ring_init(ring, S);
  if (tid == 0)
    for (int s = 0; s < S; ++s) issue(s);
  __syncthreads();

  for (int64_t k = 0;; ++k) {
    const int s = static_cast<int>(k % S);
    const int64_t t = ring.tile[s];
    if (t < 0) break;
    if (!ring_wait(ring, k, S, a.err)) {
      if (tid == 0) ring_drain(ring, k, S, a.err);
      return;
    }
    const int32_t* st = stages + s * TILE;
    const int64_t row0 = t * TILE;
    const int valid = static_cast<int>((a.n - row0) < TILE ? (a.n - row0) : TILE);

    int32_t v[ITEMS];
    const uint32_t bits = load_pred<THREADS, ITEMS>(st, a.x + row0, valid, a.lo, a.span, v);
    const int run = compact_warp<ITEMS>(v, bits, wbuf);
    if (lane == 0) wtot[warp] = run;
    __syncthreads();  // every warp has read the stage and published its count
    // A tile without matches needs no reservation and no store: every thread sees the
    // same warp totals, so the whole block skips the second barrier together.  (The
    // totals are next written after the next iteration's stage barrier.)
    int tile_total = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) tile_total += wtot[w];
    if (tile_total == 0) {
      if (tid == 0) {
        fence_proxy_async_smem();
        issue(s);
      }
      continue;
    }
    if (warp == 0) {
      if (lane == 0) {  // the stage is free: refill it now, while the tile is written
        fence_proxy_async_smem();
        issue(s);
      }
      const int32_t x = lane < WARPS ? wtot[lane] : 0;
      const int32_t inc = warp_inclusive_scan(x, lane);
      if (lane < WARPS) woff[lane] = inc - x;
      const int32_t total = __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
      if (lane == 0) {
        long long base = static_cast<long long>(atomicAdd(a.count, static_cast<unsigned long long>(total)));
        if (base + total > a.n) {
          set_error(a.err, CRYS_DEV_BOUNDS);
          base = -1;
        }
        out_base = base;
      }
    }
    __syncthreads();
    const long long base = out_base;
    if (base < 0) {  // out of bounds: abandon uniformly
      if (tid == 0) ring_drain(ring, k + 1, S, a.err);
      return;
    }
    // BlockStore: each warp writes its run with coalesced stores.
    int32_t* dst = a.out + base + woff[warp];
    for (int i = lane; i < run; i += kWarp) dst[i] = wbuf[i];
  }
}

// ---------------------------------------------------------------- input order

// Selection in input order as one persistent kernel.  Every tile publishes its count in
// its status word; one block, the first to start, turns the counts into output positions
// in tile order (the scanner) and writes each position back into the tile's word, which
// only that tile's block polls.
//
// Why one scanner: a look-back per tile makes hundreds of blocks read the same few words
// that are being written, and those reads are what bounds it.  At 2^29 rows, half
// selected: 3.84 ms with one thread per block walking back word by word, 2.84 / 3.43 /
// 5.00 ms with a warp reading 64 / 128 / 256 words per round trip (each tile's work is the
// same; only the number of words read differs).  Here a word is read by one warp, until it
// is there, and by its own tile: 0.64 ms, against 0.55 ms of the unordered kernel.
//
// A worker block has three roles: WARPS consumer warps, a scan warp and a producer
// thread.  A stage of its ring goes: filled by a bulk copy -> compacted in place (each
// warp's selected values to the front of its own part) -> stored once the tile's output
// position is known -> refilled.  The consumers store kDefer tiles behind the one they
// compact, so the way to the scanner and back does not stop the block.
constexpr int kDefer = 2;
constexpr int kChunk = 128;  // status words a scanner warp takes at a time

struct OrderedShared {
  uint64_t full[kMaxStages];   // the tile's bulk copy has landed (1 arrival + tx bytes)
  uint64_t count[kMaxStages];  // every consumer warp has compacted and counted
  uint64_t ready[kMaxStages];  // the scan warp has written base and woff
  uint64_t empty[kMaxStages];  // every consumer warp has stored its part
  int64_t tile[kMaxStages];    // tile of the stage, -1: no more tiles
  long long base[kMaxStages];  // first output row of the tile, -1: given up
  uint64_t running;            // scanner: selected rows of the chunks before next_chunk
  int64_t next_chunk;          // scanner: chunk whose turn it is
  int32_t gave_up;
  uint32_t ticket;             // 0: this block is the scanner
};

// The scanner: warp w of the block takes the chunks w, w + WARPS, ... of kChunk status words,
// reads each until it is published and, once the earlier chunks are done, hands out
// positions to the published words in front of the first missing one.  (Not only to whole
// chunks: a worker holds several tiles and counts the later ones after storing the first.)
template <int WARPS>
__device__ void scan_tiles(const SelectArgs& a, OrderedShared& sh, int64_t ntiles) {
  constexpr int R = kChunk / kWarp;
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  volatile int32_t* gave_up = &sh.gave_up;
  volatile int64_t* turn = &sh.next_chunk;
  for (int64_t c = warp; c * kChunk < ntiles; c += WARPS) {
    const int64_t i0 = c * kChunk + lane;
    uint64_t w[R];
#pragma unroll
    for (int r = 0; r < R; ++r) w[r] = i0 + r * kWarp < ntiles ? 0ull : kFlagAggregate;
    ScanWait wait = {};
    uint32_t spins = 0;
    int handed = 0;  // words of the chunk whose position is out
    int there = 0;   // published words in front of the first missing one
    uint32_t before[R], total = 0;  // their exclusive prefix and sum
    while (handed < kChunk) {
      if (there < kChunk) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (w[r] == 0ull) w[r] = ld_relaxed_u64(&a.tile_state[i0 + r * kWarp]);
        there = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint32_t none = __ballot_sync(0xFFFFFFFFu, w[r] == 0ull);
          if (there == r * kWarp) there += none ? __ffs(none) - 1 : kWarp;
        }
        total = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint32_t x = r * kWarp + lane < there ? static_cast<uint32_t>(w[r] & kValueMask) : 0u;
          const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(x), lane));
          before[r] = total + inc - x;
          total += __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
        }
      }
      const bool mine = __shfl_sync(0xFFFFFFFFu, static_cast<int>(*turn == c), 0) != 0;
      if (there == handed || !mine) {
        if (++spins % 32 == 0) {
          // ids from tile_base on are handed out in order: the first missing tile is among them
          const int64_t held_at = there < kChunk ? c * kChunk + there + 1 - static_cast<int64_t>(a.tile_base) : 0;
          if (!__all_sync(0xFFFFFFFFu, scan_look(&wait, a.tile_counter, held_at, a.abort_word, a.wait_ns, a.err))) {
            if (lane == 0) *gave_up = 1;
            return;
          }
        }
        if (__any_sync(0xFFFFFFFFu, *gave_up)) return;
        continue;
      }
      // this chunk's turn: the critical section is one shared-memory read and one write
      __threadfence_block();
      __syncwarp();  // lane 0 saw the turn: its fence orders every lane's read
      const uint64_t base = sh.running;  // written before the turn was passed on
      __syncwarp();
      if (there == kChunk && lane == 0) {
        sh.running = base + total;
        __threadfence_block();
        *turn = c + 1;
        if ((c + 1) * kChunk >= ntiles) *a.count = static_cast<unsigned long long>(base + total);
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int pos = r * kWarp + lane;
        if (pos >= handed && pos < there && i0 + r * kWarp < ntiles)
          st_relaxed_u64(&a.tile_state[i0 + r * kWarp], kFlagInclusive | (base + before[r]));
      }
      handed = there;
    }
  }
}

template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS + 2 * kWarp) select_ordered_kernel(SelectArgs a) {
  constexpr int TILE = THREADS * ITEMS;
  constexpr int WARPS = THREADS / kWarp;
  constexpr int WROWS = ITEMS * kWarp;  // rows of a tile owned by one warp, contiguous
  static_assert(ITEMS % 4 == 0 && ITEMS <= 16 && WARPS <= kWarp, "4..16 items per thread, one warp scans the warps");

  extern __shared__ __align__(128) unsigned char smem_raw[];
  int32_t* stages = reinterpret_cast<int32_t*>(smem_raw);  // S x TILE
  const int S = a.stages;
  __shared__ OrderedShared sh;
  __shared__ int32_t wtot[kMaxStages][WARPS];
  __shared__ int32_t woff[kMaxStages][WARPS];
  __shared__ int32_t ttot[kMaxStages];

  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const int64_t ntiles = (a.n + TILE - 1) / TILE;
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.count[s], WARPS);
      mbar_init(&sh.ready[s], 1);
      mbar_init(&sh.empty[s], WARPS);
    }
    sh.running = 0;
    sh.next_chunk = 0;
    sh.gave_up = 0;
    fence_barrier_init();
    sh.ticket = atomicAdd(a.block_counter, 1u);
  }
  __syncthreads();
  volatile int32_t* gave_up = &sh.gave_up;

  if (sh.ticket == 0) {  // the first block to start: it runs, whatever happens to the others
    scan_tiles<WARPS + 2>(a, sh, ntiles);
    return;
  }

  if (warp == WARPS + 1) {  // producer: tile ids in order, a bulk copy per free stage
    if (lane != 0) return;
    const uint64_t pol = policy_evict_first();
    int64_t k = 0, first = 0;  // copies first..k-1 may be in flight at the end
    for (;; ++k) {
      const int s = static_cast<int>(k % S);
      first = k > S ? k - S : 0;
      if (k >= S) {
        const uint32_t addr = smem_u32(&sh.empty[s]), parity = static_cast<uint32_t>((k / S - 1) & 1);
        const uint64_t t0 = global_timer_ns();
        while (!mbar_try_wait(addr, parity) && !*gave_up)
          if (global_timer_ns() - t0 > kWaitBoundNs) {
            set_error(a.err, CRYS_DEV_TIMEOUT);
            *gave_up = 1;
          }
        if (*gave_up) break;
      }
      const int64_t t = static_cast<int64_t>(a.tile_base) + static_cast<int64_t>(atomicAdd(a.tile_counter, 1u));
      if (t >= ntiles) {
        sh.tile[s] = -1;
        mbar_arrive(&sh.full[s]);  // this stage's previous copy was consumed: not waited for again
        first = k >= S ? k - S + 1 : 0;
        break;
      }
      sh.tile[s] = t;
      const int64_t row = t * TILE;
      ring_issue(&sh.full[s], stages + s * TILE, TILE, &a.x, 1, row, (a.n - row) < TILE ? (a.n - row) : TILE, pol);
    }
    // every copy lands before the block ends, also when the other warps gave up early
    for (int64_t j = first; j < k; ++j)
      mbar_wait_bounded(&sh.full[j % S], static_cast<uint32_t>((j / S) & 1), a.err);
    return;
  }

  if (warp == WARPS) {  // scan warp: a tile's count out, the position of an earlier one back
    // Waits for the position of iteration j's tile and passes it to the consumers.
    auto position = [&](int64_t j) -> bool {
      const int s = static_cast<int>(j % S);
      long long base = -1;
      if (lane == 0) {
        const uint64_t* word = &a.tile_state[sh.tile[s]];
        SpinGuard guard;
        uint64_t w = ld_relaxed_u64(word);
        while ((w >> 62) != 2u && guard.go_on(a.abort_word, a.wait_ns, a.err)) w = ld_relaxed_u64(word);
        if ((w >> 62) == 2u) base = static_cast<long long>(w & kValueMask);
        if (base >= 0 && base + ttot[s] > a.n) {
          set_error(a.err, CRYS_DEV_BOUNDS);
          base = -1;
        }
        sh.base[s] = base;
        if (base < 0) *gave_up = 1;
        mbar_arrive(&sh.ready[s]);
      }
      return __shfl_sync(0xFFFFFFFFu, static_cast<int>(base >= 0), 0) != 0;
    };
    for (int64_t k = 0;; ++k) {
      const int s = static_cast<int>(k % S);
      const uint32_t parity = static_cast<uint32_t>((k / S) & 1);
      bool ok = mbar_wait_bounded(&sh.full[s], parity, a.err);
      const int64_t t = sh.tile[s];
      if (ok && t < 0) {
        for (int64_t j = k > kDefer ? k - kDefer : 0; j < k; ++j)
          if (!position(j)) return;
        return;
      }
      ok = ok && mbar_wait_bounded(&sh.count[s], parity, a.err);
      if (!__all_sync(0xFFFFFFFFu, ok)) {
        if (lane == 0) *gave_up = 1;
        return;
      }
      const int32_t x = lane < WARPS ? wtot[s][lane] : 0;
      const int32_t inc = warp_inclusive_scan(x, lane);
      if (lane < WARPS) woff[s][lane] = inc - x;
      if (lane == kWarp - 1) {
        ttot[s] = inc;
        st_relaxed_u64(&a.tile_state[t], kFlagAggregate | static_cast<uint64_t>(inc));
      }
      __syncwarp();
      if (k >= kDefer && !position(k - kDefer)) return;
    }
  }

  // consumer warps
  // BlockStore of iteration j's tile: this warp's run with coalesced stores, then its part of
  // the stage is free.  False when the tile's position never came.
  auto store = [&](int64_t j) -> bool {
    const int s = static_cast<int>(j % S);
    if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(&sh.ready[s], static_cast<uint32_t>((j / S) & 1), a.err)))
      return false;
    const long long base = sh.base[s];
    if (base < 0) return false;
    const int run = wtot[s][warp];
    const int32_t* src = stages + s * TILE + warp * WROWS;
    int32_t* dst = a.out + base + woff[s][warp];
    for (int i = lane; i < run; i += kWarp) dst[i] = src[i];
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.empty[s]);
    return true;
  };
  for (int64_t k = 0;; ++k) {
    const int s = static_cast<int>(k % S);
    if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(&sh.full[s], static_cast<uint32_t>((k / S) & 1), a.err))) {
      if (lane == 0) *gave_up = 1;
      return;
    }
    const int64_t t = sh.tile[s];
    if (t < 0) {
      for (int64_t j = k > kDefer ? k - kDefer : 0; j < k; ++j)
        if (!store(j)) return;
      return;
    }
    int32_t* st = stages + s * TILE;
    const int64_t row0 = t * TILE;
    const int valid = static_cast<int>((a.n - row0) < TILE ? (a.n - row0) : TILE);
    int32_t v[ITEMS];
    const uint32_t bits = load_pred<THREADS, ITEMS>(st, a.x + row0, valid, a.lo, a.span, v);
    __syncwarp();  // the warp's part has been read: compact in place
    const int run = compact_warp<ITEMS>(v, bits, st + warp * WROWS);
    __syncwarp();
    if (lane == 0) {
      wtot[s][warp] = run;
      mbar_arrive(&sh.count[s]);
    }
    if (k >= kDefer && !store(k - kDefer)) return;
  }
}

// ---------------------------------------------------------------- small columns
//
// Up to kSmallRows rows are selected by one cluster of 8 blocks, in input order: a block counts
// its share of the rows, writes the count to every block's shared memory, and stores.  The
// wait that shows that the other blocks run lies behind the loads and the block's own count.
// No scratch and no cleared counter, so the call is one launch; it is launches that bound
// small calls (100,003 rows: 11.8 us per call with two clearings and the tiled kernel, 6.2 us
// with this one).  The line is what 8 blocks hold in registers, 16 rows per thread; without an
// order half of that, for the tiled kernel needs one clearing less there (three quarters and
// all of 65536 rows 6.2 against 6.5 us, of 131072 rows 8.2 against 6.3).  The values go through
// shared memory so that a warp's stores are consecutive: stored from the registers, all of
// 65536 rows took 7.7 us.
constexpr int kSmallBlocks = 8;
constexpr int kSmallThreads = 1024;
constexpr int kSmallVec = 4;  // groups of 4 rows per thread
constexpr int64_t kSmallRows = int64_t{kSmallBlocks} * kSmallThreads * kSmallVec * 4;
constexpr int64_t kSmallRowsAnyOrder = kSmallRows / 2;

__global__ void __cluster_dims__(kSmallBlocks, 1, 1) __launch_bounds__(kSmallThreads)
    select_small_kernel(const int32_t* __restrict__ x, int n, int32_t lo, uint32_t span, int32_t* __restrict__ out,
                        long long* count, int32_t* err) {
  namespace cg = cooperative_groups;
  cluster_arrive_relaxed();  // this block runs; waited for before the first store to another block
  constexpr int WARPS = kSmallThreads / kWarp;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto kept = reinterpret_cast<int32_t(*)[128 * kSmallVec]>(smem_raw);  // per warp
  __shared__ int32_t wtot[WARPS];
  __shared__ int32_t totals_of[kSmallBlocks];  // every block's count, written by that block
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  // this block's rows [first, last), 128 * vec consecutive ones per warp
  const int share = ((n + kSmallBlocks - 1) / kSmallBlocks + 3) & ~3;
  const int first = min(rank * share, n), last = min(first + share, n);
  const int vec = (last - first + kSmallThreads * 4 - 1) / (kSmallThreads * 4);
  const int row0 = first + warp * 128 * vec + lane * 4;
  int32_t v[4 * kSmallVec];
  uint32_t bits = 0;
#pragma unroll
  for (int j = 0; j < kSmallVec; ++j) {
    const int r = row0 + j * 128;
    if (j < vec && r + 4 <= last) {
      const int4 q = *reinterpret_cast<const int4*>(x + r);  // first and r are multiples of 4
      v[4 * j + 0] = q.x;
      v[4 * j + 1] = q.y;
      v[4 * j + 2] = q.z;
      v[4 * j + 3] = q.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[4 * j + e] = j < vec && r + e < last ? x[r + e] : 0;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool hit = j < vec && r + e < last && static_cast<uint32_t>(v[4 * j + e]) - static_cast<uint32_t>(lo) <= span;
      bits |= static_cast<uint32_t>(hit) << (4 * j + e);
    }
  }
  // the warp's selected values to its own part of shared memory, then one scan of the warps
  const int run = compact_warp<4 * kSmallVec>(v, bits, kept[warp]);
  if (lane == 0) wtot[warp] = run;
  __syncthreads();
  cluster_wait();  // every block runs: their shared memory may be written
  if (warp == 0) {
    const int32_t t = wtot[lane];
    const int32_t inc = warp_inclusive_scan(t, lane);
    wtot[lane] = inc - t;
    const int32_t total = __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
    if (lane < kSmallBlocks) *cluster.map_shared_rank(&totals_of[rank], lane) = total;
  }
  cluster.sync();  // the counts are there: a block reads its own copy of them
  int base = 0;
#pragma unroll
  for (int b = 0; b < kSmallBlocks; ++b) base += b < rank ? totals_of[b] : 0;
  if (base < 0 || base + totals_of[rank] > n) {  // the same in every thread of the block
    if (tid == 0) set_error(err, CRYS_DEV_BOUNDS);
    return;
  }
  if (rank == kSmallBlocks - 1 && tid == 0) *count = static_cast<long long>(base) + totals_of[rank];
  int32_t* dst = out + base + wtot[warp];
  for (int i = lane; i < run; i += kWarp) dst[i] = kept[warp][i];
}

template <int THREADS, int ITEMS>
int launch(SelectArgs a, bool ordered, cudaStream_t s) {
  constexpr int TILE = THREADS * ITEMS;
  const size_t tile_bytes = static_cast<size_t>(TILE) * sizeof(int32_t);
  const int64_t ntiles = (a.n + TILE - 1) / TILE;
  if (ordered) {
    // About 24 consumer warps per SM, the stages sharing what shared memory is left: a tile
    // being filled, one being compacted and kDefer waiting for their position need 4 stages.
    // 2^29 rows, half selected, 256 x 16: 0.64 ms at 3 blocks per SM (4 stages), 0.92 at 4
    // (3 stages), 0.83 at 2 (6 stages); storing one tile behind instead of two, 0.77.
    a.stages = stages_for(tile_bytes, 2048, THREADS >= 512 ? 2 : 24 * kWarp / THREADS);
    const size_t smem = static_cast<size_t>(a.stages) * tile_bytes;
    auto k = select_ordered_kernel<THREADS, ITEMS>;
    if (!allow_smem(k, smem)) return CRYS_ECUDA;
    k<<<persistent_grid(k, THREADS + 2 * kWarp, smem, ntiles + 1), THREADS + 2 * kWarp, smem, s>>>(a);
  } else {
    // The select body is issue-bound: keep about 32 warps per SM resident and give each
    // block the stages that still fit.
    a.stages = stages_for(tile_bytes, tile_bytes + 1024, (32 * kWarp) / THREADS);
    const size_t smem = static_cast<size_t>(a.stages + 1) * tile_bytes;
    auto k = select_kernel<THREADS, ITEMS>;
    if (!allow_smem(k, smem)) return CRYS_ECUDA;
    k<<<persistent_grid(k, THREADS, smem, ntiles), THREADS, smem, s>>>(a);
  }
  note_launch();
  return check_launch();
}

constexpr int kOp = CRYS_OP_SELECT;

int64_t min_tile() {
  int64_t m = INT64_MAX;
  for (int i = 0; i < kNumVariants[kOp]; ++i) {
    const int64_t t = static_cast<int64_t>(kTiles[kOp][i].threads) * kTiles[kOp][i].items;
    if (t < m) m = t;
  }
  return m;
}

}  // namespace
}  // namespace crys

extern "C" int crys_select(const int32_t* x, int64_t n, int32_t lo, int32_t hi, int32_t* out,
                           int64_t* d_count, int order_preserving, void* d_temp,
                           size_t* temp_bytes, crys_stream stream) {
  using namespace crys;
  if (n < 0 || (order_preserving != 0 && order_preserving != 1)) return CRYS_EINVAL;
  const int64_t max_tiles = (n + min_tile() - 1) / min_tile();
  const size_t need = order_preserving ? (static_cast<size_t>(max_tiles) * 8 + 256) : 0;
  if (!d_temp && temp_bytes) {
    *temp_bytes = need;
    return CRYS_OK;
  }
  if (need && (!d_temp || !temp_bytes)) return CRYS_EINVAL;
  if (need && *temp_bytes < need) return CRYS_ENOMEM;
  if (!d_count || (n > 0 && (!x || !out))) return CRYS_EINVAL;
  if (n > 0 && !aligned16(x)) return CRYS_EINVAL;
  if (need && (reinterpret_cast<uintptr_t>(d_temp) & 255u)) return CRYS_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  uint32_t stall_base = 0;
  uint64_t stall_ns = kWaitBoundNs;
  const bool stalled = n > 0 && lo <= hi && order_preserving && take_stall(CRYS_OP_SELECT, &stall_base, &stall_ns);
  const bool any_tile = set_tile_variant(kOp) < 0;
  if (n > 0 && n <= (order_preserving ? kSmallRows : kSmallRowsAnyOrder) && lo <= hi && !stalled && any_tile) {
    int32_t* err = device_error_word();
    if (!err) return CRYS_ECUDA;
    constexpr size_t smem = sizeof(int32_t) * 4 * kSmallVec * kSmallThreads;
    if (!allow_smem(select_small_kernel, smem)) return CRYS_ECUDA;
    select_small_kernel<<<kSmallBlocks, kSmallThreads, smem, s>>>(x, static_cast<int>(n), lo,
                                                              static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo), out,
                                                              reinterpret_cast<long long*>(d_count), err);
    if (check_launch() == CRYS_OK) {
      note_launch();
      return CRYS_OK;
    }  // a cluster this large was refused (a stream that owns few SMs): by tiles
  }
  if (cudaMemsetAsync(d_count, 0, sizeof(int64_t), s) != cudaSuccess) return CRYS_ECUDA;
  if (n == 0) return CRYS_OK;
  if (lo > hi) {  // empty range: nothing selected (d_count already zeroed)
    if (order_preserving && cudaMemsetAsync(d_temp, 0, need, s) != cudaSuccess) return CRYS_ECUDA;
    return CRYS_OK;
  }
  SelectArgs a;
  a.x = x;
  a.n = n;
  a.lo = lo;
  a.hi = hi;
  a.span = static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo);
  a.out = out;
  a.count = reinterpret_cast<unsigned long long*>(d_count);
  a.tile_counter = nullptr;
  a.block_counter = nullptr;
  a.abort_word = nullptr;
  a.tile_state = nullptr;
  a.tile_base = 0;
  a.wait_ns = kWaitBoundNs;
  a.err = device_error_word();
  if (!a.err) return CRYS_ECUDA;
  const int variant = tile_variant(CRYS_OP_SELECT);
  if (order_preserving) {
    a.tile_counter = static_cast<unsigned int*>(d_temp);
    a.block_counter = static_cast<unsigned int*>(d_temp) + 1;
    a.abort_word = static_cast<unsigned int*>(d_temp) + 32;  // polled: not in the counters' line
    a.tile_state = reinterpret_cast<uint64_t*>(static_cast<char*>(d_temp) + 256);
    a.tile_base = stall_base;
    a.wait_ns = stall_ns;
    // only the words of the chosen shape's tiles are read
    const int64_t tile = static_cast<int64_t>(kTiles[kOp][variant].threads) * kTiles[kOp][variant].items;
    if (cudaMemsetAsync(d_temp, 0, 256 + static_cast<size_t>((n + tile - 1) / tile) * 8, s) != cudaSuccess)
      return CRYS_ECUDA;
  }
  const bool ord = order_preserving != 0;
  switch (variant) {
    case 1: return launch<kTiles[kOp][1].threads, kTiles[kOp][1].items>(a, ord, s);
    case 2: return launch<kTiles[kOp][2].threads, kTiles[kOp][2].items>(a, ord, s);
    case 3: return launch<kTiles[kOp][3].threads, kTiles[kOp][3].items>(a, ord, s);
    default: return launch<kTiles[kOp][0].threads, kTiles[kOp][0].items>(a, ord, s);
  }
}

// ---------------------------------------------------------------------------
// Allocation-free order-preserving selection: the tiles' status words are a static device
// array of this file instead of caller-supplied memory.

namespace crys {
namespace {

static_assert(CRYS_SELECT_STATIC_SCRATCH_BYTES >= 256 + (CRYS_SELECT_STATIC_MAX_ROWS / 512) * 8,
              "static scratch covers the smallest tile shape");

static __device__ __align__(256) unsigned char g_select_scratch[CRYS_SELECT_STATIC_SCRATCH_BYTES];

constexpr int kMaxStaticDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxStaticDevices] = {};

// Device address of g_select_scratch on the current device (looked up once per device
// with that device current; the host-side name is only a stand-in for the symbol).
void* static_scratch() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxStaticDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_select_scratch) != cudaSuccess) return nullptr;
    g_static_ptr[dev] = ptr;
  }
  return g_static_ptr[dev];
}

}  // namespace
}  // namespace crys

extern "C" int crys_select_static(const int32_t* x, int64_t n, int32_t lo, int32_t hi,
                                  int32_t* out, int64_t* d_count, crys_stream stream) {
  using namespace crys;
  if (n < 0 || n > CRYS_SELECT_STATIC_MAX_ROWS) return CRYS_EINVAL;
  size_t need = 0;
  if (crys_select(nullptr, n, lo, hi, nullptr, nullptr, 1, nullptr, &need, stream) != CRYS_OK)
    return CRYS_EINVAL;
  if (need > CRYS_SELECT_STATIC_SCRATCH_BYTES) return CRYS_EINVAL;
  void* scratch = static_scratch();
  if (!scratch) return CRYS_ECUDA;
  size_t have = CRYS_SELECT_STATIC_SCRATCH_BYTES;
  // crys_select clears the words it uses (none for a column of one cluster) on `stream` first.
  return crys_select(x, n, lo, hi, out, d_count, 1, scratch, &have, stream);
}
