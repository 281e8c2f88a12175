// Radix partitioning without stability, and the two operators built on it:
//
//  * crys_sort_msb - the most-significant-digit radix sort the paper's GPU sort number
//    comes from (Section 4.4): one or two partition passes on the leading bits, then every
//    bucket is sorted inside one thread block (localsort.cuh).  Unstable, as in the paper.
//  * crys_join_partitioned - the radix-partitioned hash join Section 4.3 sets beside the
//    no-partitioning join for build sides far beyond the caches: both sides are split by
//    hash bits in two passes so that each build partition's table fits in shared memory,
//    then each partition is built and probed there.
//
// A partition pass moves (key, value) pairs by a digit of at most 8 bits inside each of up
// to 256 segments (the buckets of the previous pass): a histogram kernel counts the digits
// of every segment, a scan kernel turns the counts into the start of every (segment, digit)
// bucket, and a scatter kernel ranks a tile's pairs by digit with shared-memory atomics
// (hence unstable), reserves each digit's run of the tile with one global atomic per digit,
// sorts the tile in shared memory and stores each run with consecutive addresses.  No pass
// waits on another block, so nothing here spins.
#include "common.cuh"
#include "keyrange.cuh"
#include "localsort.cuh"

namespace crys {
namespace {

constexpr int kBuckets = 256;
constexpr int kHistThreads = 256;
constexpr int kHistItems = 8;
constexpr int kPartThreads = 512;
constexpr int kPartItems = 12;
constexpr int kPartTile = kPartThreads * kPartItems;  // rows per tile of a partition pass

// Join digits: bits of the multiplicative hash key * 2654435769 from the top down.
struct HashDigit {
  uint32_t shift, mask;
  __device__ __forceinline__ HashDigit load() const { return *this; }
  __device__ __forceinline__ uint32_t operator()(int32_t k) const {
    return ((static_cast<uint32_t>(k) * 2654435769u) >> shift) & mask;
  }
};

// Sort digits: bits of the key's place in the key range (keyrange.cuh).
struct RangeDigit {
  const KeyRange* range;
  uint32_t shift, mask;
  struct Fn {
    KeyRange r;
    uint32_t shift, mask;
    __device__ __forceinline__ uint32_t operator()(int32_t k) const { return (r.place(k) >> shift) & mask; }
  };
  __device__ __forceinline__ Fn load() const { return Fn{*range, shift, mask}; }
};

// Segments of a pass: segment s covers rows [begin[s], begin[s] + size[s]) and owns the
// tiles [tile_start[s], tile_start[s + 1]) of the pass (tile_start has count + 1 entries).
struct Segs {
  const uint32_t* begin;
  const uint32_t* size;
  const uint32_t* tile_start;
  int32_t count;
};

// Rows of tile `b`, which belongs to segment `seg`.
struct TileAt {
  int valid;
  uint32_t row0;
};

__device__ __forceinline__ TileAt tile_rows(const Segs& S, int seg, uint32_t b, int rows) {
  const uint32_t off = (b - S.tile_start[seg]) * static_cast<uint32_t>(rows);
  const uint32_t rem = S.size[seg] - off;
  return TileAt{static_cast<int>(rem < static_cast<uint32_t>(rows) ? rem : static_cast<uint32_t>(rows)),
                S.begin[seg] + off};
}

// Segment of tile `b` (a tile that exists): the last one that starts at or before it and is
// not empty, by binary search.
__device__ __forceinline__ int find_segment(const Segs& S, uint32_t b) {
  int lo = 0, hi = S.count;  // tile_start[lo] <= b < tile_start[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    if (S.tile_start[mid] <= b)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// Block-wide exclusive scan of one value per thread (THREADS <= 1024); also returns the
// total.  `tmp` holds one word per warp and one more.
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* tmp, uint32_t* total) {
  constexpr int WARPS = THREADS / kWarp;
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(x), lane));
  if (lane == kWarp - 1) tmp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < WARPS ? tmp[lane] : 0u;
    const uint32_t wi = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(w), lane));
    if (lane < WARPS) tmp[lane] = wi - w;
    if (lane == WARPS - 1) tmp[WARPS] = wi;  // the total, beside the warps' offsets
  }
  __syncthreads();
  const uint32_t r = tmp[warp] + inc - x;
  *total = tmp[WARPS];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------- segment set-up

// One segment covering rows [0, n).
__global__ void seg_init_kernel(uint32_t n, int rows, uint32_t* begin, uint32_t* size, uint32_t* tile_start) {
  begin[0] = 0;
  size[0] = n;
  tile_start[0] = 0;
  tile_start[1] = (n + static_cast<uint32_t>(rows) - 1) / static_cast<uint32_t>(rows);
}

// Tile prefix of `n` segments from their sizes: one block of 32 warps, any n.  A warp sums a
// contiguous share of the sizes, 32 at a time, one block scan joins the shares, and the warp
// goes over its share again.  (65536 segments with a contiguous share per thread: 0.12 ms.)
__global__ void __launch_bounds__(1024) tile_prefix_kernel(const uint32_t* __restrict__ size, int n, int rows,
                                                           uint32_t* __restrict__ tile_start) {
  __shared__ uint32_t share_start[kWarp];
  constexpr int kAhead = 8;  // loads in flight
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const int share = ((n + 1023) / 1024) * kWarp;  // segments per warp, whole groups of 32
  const int first = warp * share, last = min(first + share, n);
  auto tiles = [&](int i) {
    return i < last ? (size[i] + static_cast<uint32_t>(rows) - 1) / static_cast<uint32_t>(rows) : 0u;
  };
  uint32_t sum = 0;
  for (int i = first; i < last; i += kAhead * kWarp) {
    uint32_t t[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) t[j] = tiles(i + j * kWarp + lane);
#pragma unroll
    for (int j = 0; j < kAhead; ++j) sum += t[j];
  }
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) share_start[warp] = sum;
  __syncthreads();
  if (warp == 0) {
    const uint32_t x = share_start[lane];
    const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(x), lane));
    share_start[lane] = inc - x;
    if (lane == kWarp - 1) tile_start[n] = inc;
  }
  __syncthreads();
  uint32_t run = share_start[warp];
  for (int i = first; i < last; i += kAhead * kWarp) {
    uint32_t t[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) t[j] = tiles(i + j * kWarp + lane);
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(t[j]), lane));
      const int at = i + j * kWarp + lane;
      if (at < last) tile_start[at] = run + inc - t[j];
      run += __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
    }
  }
}

// ---------------------------------------------------------------- one partition pass

// Digit counts of every segment.  A persistent block takes a contiguous range of the
// pass's tiles (so it stays in one segment for many tiles), counts in shared memory and
// adds its counts to the segment's when the segment changes and at the end.
template <typename Digit>
__global__ void __launch_bounds__(kHistThreads) part_hist_kernel(const int32_t* __restrict__ keys, Segs S,
                                                                 const __grid_constant__ Digit digit, int digits,
                                                                 uint32_t* hist) {
  constexpr int kCopies = 4;
  constexpr int kStep = kHistThreads * kHistItems;
  __shared__ uint32_t h[kCopies][kBuckets];
  const int tid = threadIdx.x;
  const auto f = digit.load();
  for (int i = tid; i < kCopies * kBuckets; i += kHistThreads) (&h[0][0])[i] = 0;
  const uint32_t total = S.tile_start[S.count];
  const uint32_t t0 = static_cast<uint32_t>((static_cast<uint64_t>(total) * blockIdx.x) / gridDim.x);
  const uint32_t t1 = static_cast<uint32_t>((static_cast<uint64_t>(total) * (blockIdx.x + 1)) / gridDim.x);
  if (t0 >= t1) return;
  uint32_t* mine = h[(tid / kWarp) % kCopies];
  const uint64_t pol = policy_evict_first();
  int seg = find_segment(S, t0);
  auto flush = [&]() {
    __syncthreads();
    for (int d = tid; d < digits; d += kHistThreads) {
      uint32_t c = 0;
#pragma unroll
      for (int r = 0; r < kCopies; ++r) {
        c += h[r][d];
        h[r][d] = 0;
      }
      if (c) atomicAdd(&hist[seg * digits + d], c);
    }
    __syncthreads();
  };
  __syncthreads();
  for (uint32_t b = t0; b < t1; ++b) {
    if (b >= S.tile_start[seg + 1]) {
      flush();
      while (b >= S.tile_start[seg + 1]) ++seg;
    }
    const TileAt at = tile_rows(S, seg, b, kPartTile);
    for (int base = 0; base < at.valid; base += kStep) {
      int32_t k[kHistItems];
#pragma unroll
      for (int i = 0; i < kHistItems; ++i) {
        const int idx = base + i * kHistThreads + tid;
        k[i] = idx < at.valid ? ld_stream(keys + at.row0 + idx, pol) : 0;
      }
#pragma unroll
      for (int i = 0; i < kHistItems; ++i)
        if (base + i * kHistThreads + tid < at.valid) atomicAdd(&mine[f(k[i])], 1u);
    }
  }
  flush();
}

// A cursor per bucket.  Every tile adds to every cursor of its segment, and adds to one 32-byte
// sector wait for each other, so the cursors of a first pass, where all tiles share one
// segment, have a sector each; those of a second pass are four to a sector.
constexpr int kCursorStrideA = 8, kCursorStrideB = 2;

// Bucket starts of every segment: begin of the segment plus the exclusive prefix of its
// digit counts.  One block of 256 threads per segment.
__global__ void __launch_bounds__(kBuckets) part_scan_kernel(const uint32_t* hist, const uint32_t* seg_begin, int digits,
                                                             uint32_t* cursor, int stride, uint32_t* bucket_begin) {
  __shared__ uint32_t tmp[kWarp + 1];
  const int d = threadIdx.x;
  const int i = static_cast<int>(blockIdx.x) * digits + d;
  uint32_t total;
  const uint32_t ex = block_exclusive_scan<kBuckets>(d < digits ? hist[i] : 0u, tmp, &total);
  if (d < digits) {
    const uint32_t b = seg_begin[blockIdx.x] + ex;
    cursor[i * stride] = b;
    bucket_begin[i] = b;
  }
}

template <typename Digit>
struct ScatterArgs {
  const int32_t* kin;
  const int32_t* vin;
  int32_t* kout;
  int32_t* vout;
  Segs S;
  Digit digit;
  int32_t digits;
  uint32_t* cursor;  // [segments][digits], `stride` words apart: next free row of each bucket
  int32_t stride;
  int32_t* err;
};

// One tile of 6144 pairs per block, three blocks per SM.  The tile is what a digit's run is
// cut from (24 rows on average at 256 digits; 2048-row tiles wrote 8-row runs), and the keys
// and values go through the same registers one after the other, so that three blocks fit
// and one's loads and barriers hide behind the others' work: at 2^28 pairs 1.01 ms per pass
// against 1.09 with 8192-row tiles, two blocks per SM and both columns in registers, and
// 1.50 with 2048-row tiles and counters per warp.  Latency bounds it: issue is active half
// of the cycles, the L1 pipe 65%, DRAM 40%.
template <typename Digit>
__global__ void __launch_bounds__(kPartThreads, 3) part_scatter_kernel(const __grid_constant__ ScatterArgs<Digit> a) {
  extern __shared__ __align__(16) int32_t part_smem[];
  int32_t* sk = part_smem;               // the tile's keys in bucket order
  int32_t* sv = part_smem + kPartTile;   // and values
  __shared__ uint32_t count[kBuckets];   // rows of each digit
  __shared__ uint32_t lstart[kBuckets];  // tile-local start of each digit's run
  __shared__ uint32_t gshift[kBuckets];  // global row minus tile-local position (mod 2^32)
  __shared__ uint32_t tmp[kWarp + 1];
  __shared__ int seg_sh;
  const int tid = threadIdx.x;
  const uint32_t b = blockIdx.x;
  if (b >= a.S.tile_start[a.S.count]) return;
  if (tid < kBuckets) count[tid] = 0;
  if (tid < a.S.count && a.S.tile_start[tid] <= b && b < a.S.tile_start[tid + 1]) seg_sh = tid;  // one of at most 256
  const auto f = a.digit.load();
  __syncthreads();
  const int seg = seg_sh;
  const TileAt at = tile_rows(a.S, seg, b, kPartTile);
  const uint64_t pol = policy_evict_first();
  int32_t k[kPartItems];   // keys, then values
  uint32_t r[kPartItems];  // digit << 16 | rank inside the tile's rows of that digit, then place in the tile
#pragma unroll
  for (int i = 0; i < kPartItems; ++i) {
    const int idx = i * kPartThreads + tid;
    k[i] = idx < at.valid ? ld_stream(a.kin + at.row0 + idx, pol) : 0;
  }
  if (tid == 0) {  // the values are read after the keys are placed: on their way to L2 meanwhile
    const uint32_t mis = static_cast<uint32_t>((reinterpret_cast<uintptr_t>(a.vin + at.row0) & 15u) / 4);
    const uint32_t lead = mis ? 4 - mis : 0;
    const uint32_t words = static_cast<uint32_t>(at.valid) > lead ? (at.valid - lead) & ~3u : 0u;
    if (words) bulk_prefetch_l2(a.vin + at.row0 + lead, words * 4);
  }
#pragma unroll
  for (int i = 0; i < kPartItems; ++i)
    if (i * kPartThreads + tid < at.valid) {
      const uint32_t d = f(k[i]);
      r[i] = (d << 16) | atomicAdd(&count[d], 1u);
    }
  __syncthreads();
  bool bad = false;
  {
    const uint32_t run = tid < a.digits ? count[tid] : 0u;
    uint32_t total;
    const uint32_t ls = block_exclusive_scan<kPartThreads>(run, tmp, &total);
    if (run) {
      const uint32_t g = atomicAdd(&a.cursor[(seg * a.digits + tid) * a.stride], run);
      // the run must stay inside its segment (it does whenever the counts came from these
      // keys); otherwise the tile is reported and dropped rather than written out of place
      bad = g < a.S.begin[seg] || g + run > a.S.begin[seg] + a.S.size[seg];
      if (bad) set_error(a.err, CRYS_DEV_BOUNDS);
      lstart[tid] = ls;
      gshift[tid] = g - ls;
    }
  }
  if (__syncthreads_or(bad)) return;
#pragma unroll
  for (int i = 0; i < kPartItems; ++i)
    if (i * kPartThreads + tid < at.valid) {
      const uint32_t p = lstart[r[i] >> 16] + (r[i] & 0xFFFFu);
      sk[p] = k[i];
      r[i] = p;
    }
#pragma unroll
  for (int i = 0; i < kPartItems; ++i) {
    const int idx = i * kPartThreads + tid;
    k[i] = idx < at.valid ? ld_stream(a.vin + at.row0 + idx, pol) : 0;
  }
#pragma unroll
  for (int i = 0; i < kPartItems; ++i)
    if (i * kPartThreads + tid < at.valid) sv[r[i]] = k[i];
  __syncthreads();
#pragma unroll 4
  for (int j = tid; j < at.valid; j += kPartThreads) {
    const int32_t key = sk[j];
    const uint32_t g = gshift[f(key)] + static_cast<uint32_t>(j);
    a.kout[g] = key;
    a.vout[g] = sv[j];
  }
}

// ---------------------------------------------------------------- partitioned join
//
// After both sides are partitioned by the same hash bits, build partition p's table in
// shared memory (linear probing, 4096 slots at most 9/16 full or kJoinSlots at most 3/4) and
// probe the tiles of probe partition p against it.  Persistent blocks take contiguous ranges
// of probe tiles, so a block works through whole partitions in order, builds each table
// once, and has the copy engine bring the next tile's rows into L2 while it probes.  A
// build partition too large for shared memory gets a table in global scratch at 4 x its
// first row (its capacity is at most 4 x its rows, so the regions of different partitions
// do not overlap), built beforehand.  Each block adds its sum and matches with one atomic
// each.
//
// The multiplicative hash key * 2654435769 is one-to-one on 32 bits and its top bits are the
// partition, so inside a partition the remaining bits ("rest") stand for the key: they are
// what the shared-memory table holds, as 32-bit words beside 32-bit values, and their own
// top bits are the home slot.  An insert is one 32-bit compare-and-swap, a probe one 4-byte
// read and, on a hit, another.  With 8-byte (key, value) slots, a second hash and half the
// threads without rows, the kernel took 2.43 ms at 2^27 x 2^28 rows; now 1.04 ms.

constexpr int kJoinThreads = 512;
constexpr int kJoinItems = 10;
constexpr int kJoinTile = kJoinThreads * kJoinItems;  // probe rows per tile
constexpr int kJoinSlots = 8192;                      // largest table in shared memory: 64 KB
constexpr uint32_t kNoRest = 0xFFFFFFFFu;             // an empty slot

struct JoinArgs {
  const int32_t* bkey;  // build side, partitioned
  const int32_t* bval;
  const uint32_t* b_begin;  // [partitions]
  const uint32_t* b_count;  // [partitions]
  const int32_t* pkey;      // probe side, partitioned
  const int32_t* ppay;
  Segs probe;               // probe partitions with their tile prefix
  int32_t bits;             // hash bits that chose the partition
  uint64_t* arena;          // global tables of oversized build partitions (4 x build rows)
  unsigned long long* sum;
  unsigned long long* matches;
  int32_t* err;
};

// Slot of a key in an oversized partition's table: the MurmurHash3 32-bit finaliser
// (Appleby), independent of the multiplicative hash whose top bits chose the partition.
__device__ __forceinline__ uint32_t slot_hash(int32_t k) {
  uint32_t h = static_cast<uint32_t>(k);
  h ^= h >> 16;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return h;
}

// The single partition of a join whose build side needs no partitioning.
__global__ void one_partition_kernel(uint32_t nb, uint32_t np, int rows, uint32_t* b_begin, uint32_t* b_count,
                                     uint32_t* p_begin, uint32_t* p_size, uint32_t* p_tiles) {
  b_begin[0] = 0;
  b_count[0] = nb;
  p_begin[0] = 0;
  p_size[0] = np;
  p_tiles[0] = 0;
  p_tiles[1] = (np + static_cast<uint32_t>(rows) - 1) / static_cast<uint32_t>(rows);
}

// log2 slots of a build partition's table in shared memory: 4096 or kJoinSlots; 0 when the rows
// would fill more than three quarters of those.  The line between the two lies above
// partitions of 2048 rows on average: fuller tables cost more probing steps than the larger ones
// cost clearing.  2^27 probes, random keys, a tenth of them matching: 161M build rows (2458 per
// partition) 4.16 ms with the line at 2304 rows, 5.24 with 3072; 199M rows 4.82 and 7.07
// (6.54 with tables at most half full).
__device__ __forceinline__ int join_log2_slots(uint32_t rows) {
  return rows <= 2304u ? 12 : rows <= 3u * kJoinSlots / 4u ? 13 : 0;
}

// Capacity of an oversized partition's table: a power of two of at least twice its rows.
__device__ __forceinline__ uint32_t join_capacity(uint32_t rows) {
  uint32_t cap = 2;
  while (cap < 2u * rows) cap <<= 1;
  return cap;
}

// Inserts the rows of build partition p into `table` (cap slots, already empty).
__device__ __forceinline__ void join_insert(const JoinArgs& a, int64_t bb, uint32_t bn, uint64_t* table, uint32_t cap,
                                            int nthreads) {
  const uint32_t mask = cap - 1;
  for (uint32_t i = threadIdx.x; i < bn; i += nthreads) {
    const int32_t key = a.bkey[bb + i];
    const uint64_t packed = static_cast<uint64_t>(static_cast<uint32_t>(key)) |
                            (static_cast<uint64_t>(static_cast<uint32_t>(a.bval[bb + i])) << 32);
    uint32_t h = slot_hash(key) & mask;
    for (uint32_t step = 0; step < cap; ++step) {
      const uint64_t prev = atomicCAS(reinterpret_cast<unsigned long long*>(table + h), kEmptySlot, packed);
      if (prev == kEmptySlot) break;
      if (static_cast<uint32_t>(prev) == static_cast<uint32_t>(key)) {
        set_error(a.err, CRYS_DEV_DUP_KEY);
        break;
      }
      h = (h + 1) & mask;
    }
  }
}

// Build partitions too large for shared memory get their table in the global arena, built
// once here before any probe reads it.  A block looks at `per_block` partitions, one per
// thread, and builds the tables of those that are too large, one after the other: 32 when
// few can be, one when the partitions average more than 4096 rows and most are.
constexpr int kLargeParts = 32;

__global__ void __launch_bounds__(kJoinThreads) join_build_large_kernel(const __grid_constant__ JoinArgs a, int parts, int per_block) {
  __shared__ int list[kLargeParts];
  __shared__ int found;
  if (threadIdx.x == 0) found = 0;
  __syncthreads();
  const int mine = static_cast<int>(blockIdx.x) * per_block + static_cast<int>(threadIdx.x);
  if (static_cast<int>(threadIdx.x) < per_block && mine < parts && join_log2_slots(a.b_count[mine]) == 0) list[atomicAdd(&found, 1)] = mine;
  __syncthreads();
  for (int j = 0; j < found; ++j) {
    const int p = list[j];
    const uint32_t bn = a.b_count[p];
    const uint32_t cap = join_capacity(bn);
    const int64_t bb = a.b_begin[p];
    uint64_t* table = a.arena + 4 * bb;
    for (uint32_t i = threadIdx.x; i < cap; i += kJoinThreads) table[i] = kEmptySlot;
    __syncthreads();
    join_insert(a, bb, bn, table, cap, kJoinThreads);
  }
}

// Bulk L2 prefetch of rows [row, row + rows) of a column (whole 16-byte groups inside the
// range; a partial group at either end is left to the demand loads).
__device__ __forceinline__ void prefetch_rows(const int32_t* col, int64_t row, int64_t rows) {
  const uintptr_t first = (reinterpret_cast<uintptr_t>(col + row) + 15u) & ~uintptr_t{15};
  const uintptr_t last = reinterpret_cast<uintptr_t>(col + row + rows) & ~uintptr_t{15};
  if (last > first) bulk_prefetch_l2(reinterpret_cast<const void*>(first), static_cast<uint32_t>(last - first));
}

// The table of one build partition in shared memory.
struct JoinTable {
  alignas(16) uint32_t rest[kJoinSlots];
  int32_t value[kJoinSlots];
  int32_t odd_value;  // value of the one key whose rest equals kNoRest (no partitioning only)
  int32_t odd;        // whether it is there
};

__global__ void __launch_bounds__(kJoinThreads, 3) join_partition_kernel(const __grid_constant__ JoinArgs a) {
  extern __shared__ __align__(16) unsigned char join_smem[];
  JoinTable& tab = *reinterpret_cast<JoinTable*>(join_smem);
  __shared__ uint64_t red[kJoinThreads / kWarp];
  const int tid = threadIdx.x;
  // a persistent block takes a contiguous range of the probe tiles: tiles of one partition
  // are adjacent, so a block mostly works through whole partitions in order
  const uint32_t total = a.probe.tile_start[a.probe.count];
  const uint32_t t0 = static_cast<uint32_t>((static_cast<uint64_t>(total) * blockIdx.x) / gridDim.x);
  const uint32_t t1 = static_cast<uint32_t>((static_cast<uint64_t>(total) * (blockIdx.x + 1)) / gridDim.x);
  const uint32_t rest_mask = a.bits ? (1u << (32 - a.bits)) - 1u : 0xFFFFFFFFu;
  const uint64_t pol = policy_evict_first();
  uint64_t sum = 0;
  uint32_t matches = 0;
  int built = -1;  // partition whose table is in shared memory
  int p = t0 < t1 ? find_segment(a.probe, t0) : 0;
  for (uint32_t b = t0; b < t1; ++b) {
    while (b >= a.probe.tile_start[p + 1]) ++p;
    const TileAt at = tile_rows(a.probe, p, b, kJoinTile);
    const int64_t bb = a.b_begin[p];
    const uint32_t bn = a.b_count[p];
    const int log2_slots = join_log2_slots(bn);
    if (tid == 0 && b + 1 < t1) {  // the next tile's rows travel to L2 meanwhile
      int q = p;
      while (b + 1 >= a.probe.tile_start[q + 1]) ++q;
      const TileAt nx = tile_rows(a.probe, q, b + 1, kJoinTile);
      prefetch_rows(a.pkey, nx.row0, nx.valid);
      prefetch_rows(a.ppay, nx.row0, nx.valid);
      if (q != p) {
        prefetch_rows(a.bkey, a.b_begin[q], a.b_count[q]);
        prefetch_rows(a.bval, a.b_begin[q], a.b_count[q]);
      }
    }
    int32_t k[kJoinItems];
#pragma unroll
    for (int i = 0; i < kJoinItems; ++i) {
      const int idx = i * kJoinThreads + tid;
      k[i] = idx < at.valid ? ld_stream(a.pkey + at.row0 + idx, pol) : 0;
    }
    if (log2_slots == 0) {  // the arena's table is built already
      const uint64_t* table = a.arena + 4 * bb;
      const uint32_t cap = join_capacity(bn), mask = cap - 1;
      constexpr int G = kJoinItems / 2;  // first slots in flight together
#pragma unroll
      for (int i0 = 0; i0 < kJoinItems; i0 += G) {
        uint64_t s[G];
        int32_t pay[G];
#pragma unroll
        for (int j = 0; j < G; ++j)
          pay[j] = (i0 + j) * kJoinThreads + tid < at.valid ? ld_stream(a.ppay + at.row0 + (i0 + j) * kJoinThreads + tid, pol) : 0;
#pragma unroll
        for (int j = 0; j < G; ++j)
          s[j] = (i0 + j) * kJoinThreads + tid < at.valid ? table[slot_hash(k[i0 + j]) & mask] : kEmptySlot;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int idx = (i0 + j) * kJoinThreads + tid;
          const int32_t key = k[i0 + j];
          uint32_t h = slot_hash(key) & mask;
          for (uint32_t step = 0; idx < at.valid && step < cap; ++step) {
            const uint64_t cur = step == 0 ? s[j] : table[h];
            if (cur == kEmptySlot) break;
            if (static_cast<uint32_t>(cur) == static_cast<uint32_t>(key)) {
              sum += static_cast<uint64_t>(static_cast<int64_t>(pay[j]) * static_cast<int32_t>(cur >> 32));
              matches += 1;
              break;
            }
            h = (h + 1) & mask;
          }
        }
      }
      continue;
    }
    const uint32_t mask = (1u << log2_slots) - 1u;
    const int home = max(32 - a.bits - log2_slots, 0);  // (fewer rest bits than slots: the low slots)
    if (built != p) {
      __syncthreads();  // the previous partition's probes are done with the table
      for (uint32_t i = tid; i < (mask + 1) / 4; i += kJoinThreads)
        reinterpret_cast<uint4*>(tab.rest)[i] = make_uint4(kNoRest, kNoRest, kNoRest, kNoRest);
      if (tid == 0) tab.odd = 0;
      __syncthreads();
      for (uint32_t i = tid; i < bn; i += kJoinThreads) {
        const uint32_t rest = (static_cast<uint32_t>(a.bkey[bb + i]) * 2654435769u) & rest_mask;
        const int32_t value = a.bval[bb + i];
        if (rest == kNoRest) {
          if (atomicExch(&tab.odd, 1)) set_error(a.err, CRYS_DEV_DUP_KEY);
          tab.odd_value = value;
          continue;
        }
        uint32_t h = rest >> home;
        while (true) {  // at most three quarters full: a free slot is met
          const uint32_t prev = atomicCAS(&tab.rest[h], kNoRest, rest);
          if (prev == kNoRest) {
            tab.value[h] = value;
            break;
          }
          if (prev == rest) {
            set_error(a.err, CRYS_DEV_DUP_KEY);
            break;
          }
          h = (h + 1) & mask;
        }
      }
      __syncthreads();
      built = p;
    }
    // probe: the first slot of every row is read before any is examined, then the rows that
    // are neither found nor missed walk on together; k becomes the slot of a found row
    uint32_t found = 0;
    uint32_t s[kJoinItems];
#pragma unroll
    for (int i = 0; i < kJoinItems; ++i) {
      k[i] = static_cast<int32_t>((static_cast<uint32_t>(k[i]) * 2654435769u) & rest_mask);
      s[i] = tab.rest[static_cast<uint32_t>(k[i]) >> home];
    }
#pragma unroll
    for (int i = 0; i < kJoinItems; ++i) {
      const uint32_t rest = static_cast<uint32_t>(k[i]);
      const bool real = i * kJoinThreads + tid < at.valid;
      uint32_t h = rest >> home;
      if (real && rest == kNoRest) {
        if (tab.odd) {
          sum += static_cast<uint64_t>(static_cast<int64_t>(a.ppay[at.row0 + i * kJoinThreads + tid]) * tab.odd_value);
          matches += 1;
        }
      } else if (real) {
        uint32_t cur = s[i];
        while (cur != rest && cur != kNoRest) {
          h = (h + 1) & mask;
          cur = tab.rest[h];
        }
        found |= static_cast<uint32_t>(cur == rest) << i;
      }
      k[i] = static_cast<int32_t>(h);
    }
    int32_t pay[kJoinItems];
#pragma unroll
    for (int i = 0; i < kJoinItems; ++i)
      pay[i] = (found >> i) & 1u ? ld_stream(a.ppay + at.row0 + i * kJoinThreads + tid, pol) : 0;
#pragma unroll
    for (int i = 0; i < kJoinItems; ++i)
      if ((found >> i) & 1u) sum += static_cast<uint64_t>(static_cast<int64_t>(pay[i]) * tab.value[k[i]]);
    matches += __popc(found);
  }
  const uint64_t bs = block_sum_u64<kJoinThreads>(sum, red);
  const uint64_t bm = block_sum_u64<kJoinThreads>(matches, red);
  if (tid == 0) {
    if (bs) atomicAdd(a.sum, static_cast<unsigned long long>(bs));
    if (a.matches && bm) atomicAdd(a.matches, static_cast<unsigned long long>(bm));
  }
}

// ---------------------------------------------------------------- host side

size_t up256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

// A bump allocator over caller scratch (every region 256-byte aligned).
struct Carve {
  char* base;
  size_t off = 0;
  explicit Carve(void* p) : base(static_cast<char*>(p)) {}
  template <typename T>
  T* take(size_t count) {
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += up256(count * sizeof(T));
    return p;
  }
};

// Device arrays of one partition level of one side.
struct Level {
  uint32_t* seg_begin;     // [segments] (level B: the bucket starts and counts of level A)
  uint32_t* seg_size;      // [segments]
  uint32_t* tile_start;    // [segments + 1]
  uint32_t* hist;          // [segments][digits]
  uint32_t* cursor;        // [segments][digits], stride words apart
  int stride;
  uint32_t* bucket_begin;  // [segments][digits]
};

int64_t tiles_bound(int64_t n, int segments, int rows) { return (n + rows - 1) / rows + segments; }

Level carve_level(Carve& c, int segments, int digits) {
  const size_t buckets = static_cast<size_t>(segments) * digits;
  Level L;
  L.seg_begin = c.take<uint32_t>(segments);
  L.seg_size = c.take<uint32_t>(segments);
  L.tile_start = c.take<uint32_t>(segments + 1);
  L.hist = c.take<uint32_t>(buckets);
  L.stride = segments == 1 ? kCursorStrideA : kCursorStrideB;
  L.cursor = c.take<uint32_t>(buckets * L.stride);
  L.bucket_begin = c.take<uint32_t>(buckets);
  return L;
}

// One partition pass over the segments of L (already set up): histogram, scan, scatter.
template <typename Digit>
int run_pass(const Level& L, int segments, int digits, int64_t n, const int32_t* kin, const int32_t* vin, int32_t* kout,
             int32_t* vout, Digit f, int32_t* err, cudaStream_t s) {
  if (cudaMemsetAsync(L.hist, 0, static_cast<size_t>(segments) * digits * 4, s) != cudaSuccess) return CRYS_ECUDA;
  Segs S{L.seg_begin, L.seg_size, L.tile_start, segments};
  const int64_t grid = tiles_bound(n, segments, kPartTile);
  const int64_t hist_grid = grid < static_cast<int64_t>(sm_count()) * 8 ? grid : static_cast<int64_t>(sm_count()) * 8;
  part_hist_kernel<<<static_cast<unsigned>(hist_grid), kHistThreads, 0, s>>>(kin, S, f, digits, L.hist);
  note_launch();
  part_scan_kernel<<<static_cast<unsigned>(segments), kBuckets, 0, s>>>(L.hist, L.seg_begin, digits, L.cursor,
                                                                        L.stride, L.bucket_begin);
  note_launch();
  ScatterArgs<Digit> a{kin, vin, kout, vout, S, f, digits, L.cursor, L.stride, err};
  const size_t smem = static_cast<size_t>(kPartTile) * 8;
  if (!allow_smem(part_scatter_kernel<Digit>, smem)) return CRYS_ECUDA;
  part_scatter_kernel<Digit><<<static_cast<unsigned>(grid), kPartThreads, smem, s>>>(a);
  note_launch();
  return check_launch();
}

// The buckets of level A as the segments of level B.
int next_level(const Level& A, Level& B, int segments, cudaStream_t s) {
  B.seg_begin = A.bucket_begin;
  B.seg_size = A.hist;
  tile_prefix_kernel<<<1, 1024, 0, s>>>(A.hist, segments, kPartTile, B.tile_start);
  note_launch();
  return check_launch();
}

bool no_overlap(const void* a, size_t na, const void* b, size_t nb) {
  const char* x = static_cast<const char*>(a);
  const char* y = static_cast<const char*>(b);
  return x + na <= y || y + nb <= x;
}

// Hash bits of the join's partitioning for a build side of nb rows: partitions of about
// 2048 rows (a 4096-slot table, a quarter of the shared-memory table), at most 16 bits in
// two passes of at most 8.
int join_bits(int64_t nb) {
  int bits = 0;
  while (bits < 16 && (nb >> bits) > 2048) ++bits;
  return bits;
}

}  // namespace
}  // namespace crys

extern "C" int crys_sort_msb(const int32_t* keys_in, const int32_t* vals_in, int32_t* keys_out, int32_t* vals_out,
                             int64_t n, void* d_temp, size_t* temp_bytes, crys_stream stream) {
  using namespace crys;
  if (n < 0 || n > (1ll << 31) - 1) return CRYS_EINVAL;
  const int bits = range_bits(n, kLocalCap);
  const int b2 = bits > 8 ? bits - 8 : 0, digits2 = 1 << b2;
  // scratch: a (key, value) buffer of n rows, the key range and the two levels' arrays
  auto layout = [&](void* base, int32_t** tk, int32_t** tv, KeyRange** range, Level* A, Level* B) {
    Carve c(base);
    *tk = c.take<int32_t>(static_cast<size_t>(n));
    *tv = c.take<int32_t>(static_cast<size_t>(n));
    *range = c.take<KeyRange>(1);
    *A = carve_level(c, 1, kBuckets);
    *B = carve_level(c, kBuckets, digits2);
    return c.off;
  };
  int32_t *tk, *tv;
  KeyRange* range;
  Level A, B;
  const size_t need = layout(nullptr, &tk, &tv, &range, &A, &B);
  if (!d_temp && temp_bytes) {
    *temp_bytes = need;
    return CRYS_OK;
  }
  if (n == 0) return CRYS_OK;
  if (!d_temp || !temp_bytes) return CRYS_EINVAL;
  if (*temp_bytes < need) return CRYS_ENOMEM;
  if (!keys_in || !vals_in || !keys_out || !vals_out || (reinterpret_cast<uintptr_t>(d_temp) & 255u)) return CRYS_EINVAL;
  const size_t nb = static_cast<size_t>(n) * 4;
  if (!no_overlap(keys_out, nb, keys_in, nb) || !no_overlap(keys_out, nb, vals_in, nb) ||
      !no_overlap(vals_out, nb, keys_in, nb) || !no_overlap(vals_out, nb, vals_in, nb) ||
      !no_overlap(keys_out, nb, vals_out, nb))
    return CRYS_EINVAL;
  layout(d_temp, &tk, &tv, &range, &A, &B);
  int32_t* err = device_error_word();
  if (!err) return CRYS_ECUDA;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const uint32_t rows = static_cast<uint32_t>(n);
  if (bits == 0)  // one block sorts everything
    return launch_local_sort<false>(LocalArgs{keys_in, vals_in, keys_out, vals_out, nullptr, nullptr, rows, err}, 1, s);
  // (its counts lie in the output's keys, read in 16-byte groups)
  if (aligned16(keys_out) && small_sort_fits(n) &&
      launch_small_sort(keys_in, vals_in, tk, tv, keys_out, vals_out, n, range, s) == CRYS_OK)
    return CRYS_OK;  // (refused on a stream that owns few SMs: by a pass)
  if (launch_key_range(keys_in, n, bits, range, nullptr, s) != CRYS_OK) return CRYS_ECUDA;
  // level A: the whole array by the leading 8 bits
  seg_init_kernel<<<1, 1, 0, s>>>(rows, kPartTile, A.seg_begin, A.seg_size, A.tile_start);
  note_launch();
  int32_t* ak = b2 ? keys_out : tk;
  int32_t* av = b2 ? vals_out : tv;
  int rc = run_pass(A, 1, kBuckets, n, keys_in, vals_in, ak, av, RangeDigit{range, static_cast<uint32_t>(b2), 0xFFu}, err, s);
  if (rc != CRYS_OK) return rc;
  const Level* last = &A;
  if (b2) {
    // level B: each of the 256 buckets by the next bits, output -> scratch buffers
    rc = next_level(A, B, kBuckets, s);
    if (rc != CRYS_OK) return rc;
    rc = run_pass(B, kBuckets, digits2, n, ak, av, tk, tv, RangeDigit{range, 0u, static_cast<uint32_t>(digits2 - 1)}, err, s);
    if (rc != CRYS_OK) return rc;
    last = &B;
  }
  // every bucket sorted by its remaining bits, scratch -> output
  return launch_local_sort<true>(LocalArgs{tk, tv, keys_out, vals_out, last->bucket_begin, last->hist, rows, err},
                                 static_cast<unsigned>(1u << bits), s);
}

extern "C" int crys_join_partitioned(const int32_t* bkeys, const int32_t* bvals, int64_t nb, const int32_t* fk,
                                     const int32_t* payload, int64_t np, int64_t* d_sum, int64_t* d_matches,
                                     void* d_temp, size_t* temp_bytes, crys_stream stream) {
  using namespace crys;
  if (nb < 0 || np < 0 || nb > (1ll << 30) || np > (1ll << 31) - 1) return CRYS_EINVAL;
  const int bits = join_bits(nb);
  const int b1 = (bits + 1) / 2, b2 = bits / 2;
  const int parts1 = 1 << b1;
  // bucket d of pass-2 segment g is partition (g << b2) + d
  const int parts = 1 << bits;
  struct Side {
    int32_t *k1, *v1, *k2, *v2;  // rows after pass 1 and after pass 2
    Level A, B;
  };
  struct Parts {  // the partitions the join kernel reads
    uint32_t* b_begin;
    uint32_t* b_count;
    uint32_t* p_begin;
    uint32_t* p_size;
    uint32_t* p_tiles;
    uint64_t* arena;
  };
  auto layout = [&](void* base, Side* R, Side* P, Parts* J) {
    Carve c(base);
    for (Side* sd : {R, P}) {
      const size_t rows = static_cast<size_t>(sd == R ? nb : np);
      sd->k1 = c.take<int32_t>(rows);
      sd->v1 = c.take<int32_t>(rows);
      sd->k2 = c.take<int32_t>(rows);
      sd->v2 = c.take<int32_t>(rows);
      sd->A = carve_level(c, 1, parts1);
      sd->B = carve_level(c, parts1, 1 << b2);
    }
    J->b_begin = c.take<uint32_t>(1);
    J->b_count = c.take<uint32_t>(1);
    J->p_begin = c.take<uint32_t>(1);
    J->p_size = c.take<uint32_t>(1);
    J->p_tiles = c.take<uint32_t>(static_cast<size_t>(parts) + 1);
    J->arena = c.take<uint64_t>(static_cast<size_t>(4) * static_cast<size_t>(nb > 0 ? nb : 1));
    return c.off;
  };
  Side R, P;
  Parts J;
  const size_t need = layout(nullptr, &R, &P, &J);
  if (!d_temp && temp_bytes) {
    *temp_bytes = need;
    return CRYS_OK;
  }
  if (!d_sum) return CRYS_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (!clear_results(d_sum, d_matches, s)) return CRYS_ECUDA;
  if (nb == 0 || np == 0) return CRYS_OK;
  if (!d_temp || !temp_bytes) return CRYS_EINVAL;
  if (*temp_bytes < need) return CRYS_ENOMEM;
  if (!bkeys || !bvals || !fk || !payload || (reinterpret_cast<uintptr_t>(d_temp) & 255u)) return CRYS_EINVAL;
  layout(d_temp, &R, &P, &J);
  int32_t* err = device_error_word();
  if (!err) return CRYS_ECUDA;
  // both sides partitioned by the same hash bits: pass 1 by the top b1 bits, pass 2 by
  // the next b2 bits inside each pass-1 partition
  const HashDigit f1{static_cast<uint32_t>(32 - b1), static_cast<uint32_t>(parts1 - 1)};
  const HashDigit f2{static_cast<uint32_t>(32 - bits), static_cast<uint32_t>((1 << b2) - 1)};
  Side* sides[2] = {&R, &P};
  const int32_t* in_k[2] = {bkeys, fk};
  const int32_t* in_v[2] = {bvals, payload};
  const int64_t rows[2] = {nb, np};
  const int32_t* fin_k[2] = {bkeys, fk};
  const int32_t* fin_v[2] = {bvals, payload};
  const uint32_t* fin_begin[2] = {nullptr, nullptr};
  const uint32_t* fin_count[2] = {nullptr, nullptr};
  for (int w = 0; w < 2 && bits > 0; ++w) {
    Side& sd = *sides[w];
    seg_init_kernel<<<1, 1, 0, s>>>(static_cast<uint32_t>(rows[w]), kPartTile, sd.A.seg_begin, sd.A.seg_size, sd.A.tile_start);
    note_launch();
    int rc = run_pass(sd.A, 1, parts1, rows[w], in_k[w], in_v[w], sd.k1, sd.v1, f1, err, s);
    if (rc != CRYS_OK) return rc;
    fin_k[w] = sd.k1;
    fin_v[w] = sd.v1;
    fin_begin[w] = sd.A.bucket_begin;
    fin_count[w] = sd.A.hist;
    if (b2 == 0) continue;
    rc = next_level(sd.A, sd.B, parts1, s);
    if (rc != CRYS_OK) return rc;
    rc = run_pass(sd.B, parts1, 1 << b2, rows[w], sd.k1, sd.v1, sd.k2, sd.v2, f2, err, s);
    if (rc != CRYS_OK) return rc;
    fin_k[w] = sd.k2;
    fin_v[w] = sd.v2;
    fin_begin[w] = sd.B.bucket_begin;
    fin_count[w] = sd.B.hist;
  }
  const uint32_t* b_begin = fin_begin[0];
  const uint32_t* b_count = fin_count[0];
  const uint32_t* p_begin = fin_begin[1];
  const uint32_t* p_size = fin_count[1];
  if (bits == 0) {  // one partition: the inputs as they are
    one_partition_kernel<<<1, 1, 0, s>>>(static_cast<uint32_t>(nb), static_cast<uint32_t>(np), kJoinTile, J.b_begin, J.b_count, J.p_begin, J.p_size, J.p_tiles);
    note_launch();
    b_begin = J.b_begin;
    b_count = J.b_count;
    p_begin = J.p_begin;
    p_size = J.p_size;
  } else {
    tile_prefix_kernel<<<1, 1024, 0, s>>>(fin_count[1], parts, kJoinTile, J.p_tiles);
    note_launch();
  }
  JoinArgs a;
  a.bkey = fin_k[0];
  a.bval = fin_v[0];
  a.b_begin = b_begin;
  a.b_count = b_count;
  a.pkey = fin_k[1];
  a.ppay = fin_v[1];
  a.probe = Segs{p_begin, p_size, J.p_tiles, parts};
  a.bits = bits;
  a.arena = J.arena;
  a.sum = reinterpret_cast<unsigned long long*>(d_sum);
  a.matches = reinterpret_cast<unsigned long long*>(d_matches);
  a.err = err;
  const int per_block = (nb >> bits) > 4096 ? 1 : kLargeParts;
  join_build_large_kernel<<<static_cast<unsigned>((parts + per_block - 1) / per_block), kJoinThreads, 0, s>>>(a, parts, per_block);
  note_launch();
  const size_t smem = sizeof(JoinTable);
  if (!allow_smem(join_partition_kernel, smem)) return CRYS_ECUDA;
  const int per_sm = blocks_per_sm(reinterpret_cast<const void*>(join_partition_kernel), kJoinThreads, smem);
  int64_t grid = tiles_bound(np, parts, kJoinTile);
  if (grid > static_cast<int64_t>(per_sm) * sm_count()) grid = static_cast<int64_t>(per_sm) * sm_count();
  join_partition_kernel<<<static_cast<unsigned>(grid), kJoinThreads, smem, s>>>(a);
  note_launch();
  return check_launch();
}
