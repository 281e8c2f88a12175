// Stable radix sort of (key, value) pairs (Section 4.4), by signed key.
//
// Two plans, chosen on the device from the keys:
//  * buckets: the keys are spread over up to 2^16 buckets of about 4096 rows by their leading
//    bits - one stable radix pass of 8 bits, or two, low bits first - and every bucket is
//    then sorted inside one thread block (localsort.cuh).  The leading bits are those of a
//    key's place between the smallest and largest key of a sample (keyrange.cuh), so narrow
//    ranges fill the buckets too.  One kernel reads the keys and counts all buckets, which
//    gives the passes' bucket starts and shows whether any bucket is too large for a block.
//  * digits: when one is (heavily repeated or clustered keys), when a sample of the keys differs
//    in at most three bytes or shows more than eight rows per key value (keyrange.cuh), or
//    when there are too many rows, the least-significant-digit sort: 8-bit digits, a stable
//    pass per digit from the low one to the high one.  Digits that have one value in all
//    keys are skipped.
//
// A pass is ONE kernel: a thread block takes the next tile id from an atomic counter, ranks
// its keys stably inside the block (per-warp multisplit: keys are processed warp-striped,
// round by round, so rank order equals input order), publishes its per-digit counts, places
// keys and values in shared memory in sorted order while scanner blocks turn all tiles'
// counts into positions, and stores each digit's run with consecutive addresses.  So a
// pass reads 8N and writes 8N.
//
// The paper notes that its V100 kernels could partition only 7 bits per stable pass
// because each thread kept a 2^r histogram in registers; the per-warp shared-memory
// multisplit used here keeps 8-bit stable passes.
//
// 2^28 random pairs: 4.37 ms by buckets (0.23 ms counting, two passes of 1.23 ms, 1.59 ms in
// the blocks).  Four passes by digits, each with a decoupled look-back, took 6.10 ms.
#include "common.cuh"
#include "keyrange.cuh"
#include "localsort.cuh"
#include "multisplit.cuh"
#include "pipeline.cuh"
#include "tiles.h"

namespace crys {
namespace {

constexpr int kPasses = 4;
constexpr uint32_t kFlagAggregate = 1u << 30;
constexpr uint32_t kFlagInclusive = 2u << 30;
constexpr uint32_t kValueMask = (1u << 30) - 1;
// Largest sort by buckets: 2^16 buckets of 4096 rows on average.
constexpr int64_t kMaxBucketRows = int64_t{4096} << 16;

__device__ __forceinline__ uint32_t digit_of(int32_t key, int pass) {
  const uint32_t d = (static_cast<uint32_t>(key) >> (8 * pass)) & 0xFFu;
  return pass == kPasses - 1 ? d ^ 0x80u : d;
}

// What the passes do, written on the device; one per sort, in its scratch.
struct SortHead {
  unsigned int tile_counter[kPasses];
  unsigned int abort_word;   // set by the first block of this sort that gives up
  unsigned int counted;      // blocks of the counting kernels that have finished
  unsigned int digits_counted;
  unsigned int crowded;      // a bucket is too large for a block, or the keys are few (keyrange.cuh)
  uint32_t buckets;          // 1: sorted by buckets, 0: by digits
  uint32_t passes;           // passes that do work; pass j writes to the output when an even number follows
  KeyRange range;
  uint32_t shift[kPasses], mask[kPasses];  // a pass's digit
};
static_assert(sizeof(SortHead) <= 256, "the head has 256 bytes of the scratch");

// A pass's digit of a key: bits of its place in the key range, or of the key itself with the
// sign bit flipped.
template <bool PLACE>
struct PassDigit {
  KeyRange range;
  uint32_t shift, mask;
  __device__ __forceinline__ uint32_t operator()(int32_t k) const {
    const uint32_t x = PLACE ? range.place(k) : static_cast<uint32_t>(k) ^ 0x80000000u;
    return (x >> shift) & mask;
  }
};

// ---------------------------------------------------------------- counting the buckets

constexpr int kCountThreads = 1024;

// Exclusive prefix of 256 values held in shared memory, by the first 8 warps of the block.
__device__ __forceinline__ void scan256(const uint32_t* in, uint32_t* out, uint32_t* tmp) {
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  uint32_t inc = 0;
  if (tid < kRadix) {
    inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(in[tid]), lane));
    if (lane == kWarp - 1) tmp[warp] = inc;
  }
  __syncthreads();
  if (tid < kRadix) {
    uint32_t base = 0;
    for (int w = 0; w < warp; ++w) base += tmp[w];
    out[tid] = base + inc - in[tid];
  }
  __syncthreads();
}

// Rows per bucket.  Every block counts its share of the keys in shared memory, two 16-bit
// counters per word, and stops as soon as one of its buckets is too large for a block (which
// also keeps the counters from running over: at most 16 more rows per thread follow).  The
// block that finishes last turns the counts into the passes' bucket starts and the buckets'
// first rows.
__global__ void __launch_bounds__(kCountThreads, 1) count_buckets_kernel(const int32_t* __restrict__ keys, int64_t n, int bits,
                                                                         SortHead* head, uint32_t* counts,
                                                                         uint32_t* bucket_begin, uint32_t* base) {
  extern __shared__ __align__(16) uint32_t bins[];  // 2^bits 16-bit counters
  __shared__ uint32_t col[kRadix], row[kRadix], scanned[kRadix], tmp[kRadix / kWarp];
  __shared__ unsigned int ticket;
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const int words = 1 << (bits - 1);
  if (__syncthreads_or(head->crowded != 0u)) return;  // decided already (head->buckets stays 0)
  for (int i = tid; i < words; i += kCountThreads) bins[i] = 0;
  const KeyRange range = head->range;
  const uint64_t pol = policy_evict_first();
  __syncthreads();
  bool over = false;
  auto add = [&](int32_t k) {
    const uint32_t b = range.place(k), half = 16u * (b & 1u);
    over |= ((atomicAdd(&bins[b >> 1], 1u << half) >> half) & 0xFFFFu) >= static_cast<uint32_t>(kLocalCap);
  };
  const int64_t nvec = n / 4;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kCountThreads;
  int64_t v = static_cast<int64_t>(blockIdx.x) * kCountThreads + tid;
  volatile unsigned int* crowded = &head->crowded;
  constexpr int kVecs = 4;  // in flight per thread
  for (int step = 0; v < nvec && !over; ++step, v += kVecs * stride) {
    if (step % 8 == 7 && *crowded) break;
    int4 q[kVecs];
#pragma unroll
    for (int j = 0; j < kVecs; ++j)
      if (v + j * stride < nvec) q[j] = ld_stream_v4(keys + 4 * (v + j * stride), pol);
#pragma unroll
    for (int j = 0; j < kVecs; ++j)
      if (v + j * stride < nvec) {
        add(q[j].x);
        add(q[j].y);
        add(q[j].z);
        add(q[j].w);
      }
  }
  if (blockIdx.x == 0 && 4 * nvec + tid < n) add(keys[4 * nvec + tid]);  // the last 0..3 keys
  if (over) *crowded = 1;
  __syncthreads();
  if (!*crowded) {
    for (int i = tid; i < words; i += kCountThreads) {
      const uint32_t w = bins[i];
      if (w & 0xFFFFu) atomicAdd(&counts[2 * i], w & 0xFFFFu);
      if (w >> 16) atomicAdd(&counts[2 * i + 1], w >> 16);
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) ticket = atomicAdd(&head->counted, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  // the last block: 256 buckets per row (the second pass's digit), one warp per row
  const int rows = bits > 8 ? 1 << (bits - 8) : 1;
  if (tid < kRadix) col[tid] = row[tid] = 0;
  __syncthreads();
  uint32_t most = 0;
  for (int r = warp; r < rows; r += kCountThreads / kWarp) {
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < kRadix / kWarp; ++j) {
      const uint32_t c = __ldcg(&counts[r * kRadix + j * kWarp + lane]);
      most = max(most, c);
      sum += c;
      if (c) atomicAdd(&col[j * kWarp + lane], c);
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) row[r] = sum;
  }
  if (__syncthreads_or(most > static_cast<uint32_t>(kLocalCap) || *crowded != 0)) return;  // head->buckets stays 0
  scan256(col, scanned, tmp);
  if (tid < kRadix) base[tid] = scanned[tid];
  __syncthreads();
  scan256(row, scanned, tmp);
  if (tid < kRadix && rows > 1) base[kRadix + tid] = scanned[tid];
  for (int r = warp; r < rows; r += kCountThreads / kWarp) {
    uint32_t run = scanned[r];
#pragma unroll
    for (int j = 0; j < kRadix / kWarp; ++j) {
      const uint32_t c = __ldcg(&counts[r * kRadix + j * kWarp + lane]);
      const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(c), lane));
      bucket_begin[r * kRadix + j * kWarp + lane] = run + inc - c;
      run += __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
    }
  }
  if (tid == 0) {
    head->buckets = 1;
    head->passes = rows > 1 ? 2 : 1;
    head->shift[0] = 0;
    head->mask[0] = kRadix - 1;
    head->shift[1] = 8;
    head->mask[1] = static_cast<uint32_t>(rows - 1);
  }
}

// ---------------------------------------------------------------- counting the digits

constexpr int kHistThreads = 512;
constexpr int kHistCopies = 4;  // shared-memory copies of the 4x256 histogram

// Rows per value of every digit; the block that finishes last turns them into the passes'
// bucket starts.  Nothing to do when the sort goes by buckets.
__global__ void __launch_bounds__(kHistThreads) sort_hist_kernel(const int32_t* __restrict__ keys,
                                                                  int64_t n, unsigned int* hist, SortHead* head,
                                                                  uint32_t* base) {
  __shared__ unsigned int h[kHistCopies][kPasses * kRadix];
  __shared__ unsigned int ticket;
  __shared__ int varies[kPasses];
  if (head->buckets) return;
  for (int i = threadIdx.x; i < kHistCopies * kPasses * kRadix; i += kHistThreads)
    (&h[0][0])[i] = 0;
  __syncthreads();
  unsigned int* mine = h[(threadIdx.x / kWarp) % kHistCopies];
  const uint64_t pol = policy_evict_first();
  const int64_t nvec = n / 4;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kHistThreads;
  for (int64_t v = static_cast<int64_t>(blockIdx.x) * kHistThreads + threadIdx.x; v < nvec; v += stride) {
    const int4 q = ld_stream_v4(keys + 4 * v, pol);
    const int32_t k4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int p = 0; p < kPasses; ++p) atomicAdd(&mine[p * kRadix + digit_of(k4[e], p)], 1u);
  }
  if (blockIdx.x == 0) {
    for (int64_t i = 4 * nvec + threadIdx.x; i < n; i += kHistThreads) {
      const int32_t k = keys[i];
#pragma unroll
      for (int p = 0; p < kPasses; ++p) atomicAdd(&mine[p * kRadix + digit_of(k, p)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kPasses * kRadix; i += kHistThreads) {
    unsigned int c = 0;
#pragma unroll
    for (int r = 0; r < kHistCopies; ++r) c += h[r][i];
    if (c) atomicAdd(hist + i, c);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) ticket = atomicAdd(&head->digits_counted, 1u);
  __syncthreads();
  if (ticket != gridDim.x - 1) return;
  __threadfence();
  // warp p: does digit p vary, and the starts of its values
  const int lane = threadIdx.x % kWarp, p = threadIdx.x / kWarp;
  if (p < kPasses) {
    bool all = false;
    for (int c0 = 0; c0 < kRadix; c0 += kWarp) all |= __ldcg(&hist[p * kRadix + c0 + lane]) == static_cast<uint32_t>(n);
    const bool constant = __any_sync(0xFFFFFFFFu, all) != 0;
    if (lane == 0) varies[p] = !constant;
  }
  __syncthreads();
  int passes = 0;
  for (int q = 0; q < kPasses; ++q) passes += varies[q];
  if (p < kPasses && (varies[p] || (passes == 0 && p == 0))) {  // (one key value: one pass copies the rows)
    int slot = 0;
    for (int q = 0; q < p; ++q) slot += varies[q];
    unsigned int carry = 0;
    for (int c0 = 0; c0 < kRadix; c0 += kWarp) {
      const unsigned int x = __ldcg(&hist[p * kRadix + c0 + lane]);
      const unsigned int inc = static_cast<unsigned int>(warp_inclusive_scan(static_cast<int32_t>(x), lane));
      base[slot * kRadix + c0 + lane] = carry + inc - x;
      carry += __shfl_sync(0xFFFFFFFFu, inc, kWarp - 1);
    }
    if (lane == 0) {
      head->shift[slot] = static_cast<uint32_t>(8 * p);
      head->mask[slot] = kRadix - 1;
    }
  }
  if (threadIdx.x == 0) head->passes = passes ? passes : 1;
}

// ---------------------------------------------------------------- one pass

struct PassArgs {
  const int32_t *keys_in, *vals_in;  // the sort's input, scratch and output columns
  int32_t *keys_tmp, *vals_tmp;
  int32_t *keys_out, *vals_out;
  int64_t n;
  int pass;
  SortHead* head;
  const unsigned int* digit_base;  // 256 bucket starts of this pass
  uint32_t* status;                // per tile x digit: the tile's count, then its position
  uint32_t tile_base;              // first tile id handed out (0 unless a test stalls)
  uint64_t wait_ns;                // bound of a wait for a count or a position
  int32_t* err;
};

// Columns of one pass.
struct PassCols {
  const int32_t *kin, *vin;
  int32_t *kout, *vout;
};

template <int THREADS>
struct PassShared {
  alignas(4) uint16_t whist[THREADS / kWarp][kRadix];  // per-warp digit counts, then offsets
  uint32_t tile_start[kRadix];              // tile-local start of each digit run
  uint32_t out_shift[kRadix];               // global position minus local position (mod 2^32)
  uint32_t scan_tmp[kRadix / kWarp];
  uint32_t tile;
};

// The scanners: kScanners blocks, the first of a pass to start, turn the tiles' digit counts
// into exclusive prefixes over the tiles, 32 digits each (one per lane).  Warp w takes the
// chunks w, w + WARPS, ... of kScanTiles tiles, reads each count until it is published and,
// once the earlier chunks are done, hands out the prefixes of the published tiles in front
// of the first missing one.
//
// A decoupled look-back, where every tile's block reads earlier tiles' words itself, finished
// 22 to 26 tiles per microsecond whatever the tile's size (hundreds of blocks read the words
// that are being written), so a pass over 2^28 rows took 1.5 ms with 8192-row tiles and 3.0
// with 4096-row tiles.
constexpr int kScanners = kRadix / kWarp;
constexpr int kScanTiles = 16;

struct ScanShared {
  uint32_t running[kWarp];  // rows of the digit in the chunks before `turn`
  int64_t turn;             // chunk whose turn it is
  int32_t gave_up;
};

template <int WARPS>
__device__ void scan_tiles(const PassArgs& a, int scanner, int64_t tiles, ScanShared& sh) {
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  if (threadIdx.x < kWarp) sh.running[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    sh.turn = 0;
    sh.gave_up = 0;
  }
  __syncthreads();
  volatile int64_t* turn = &sh.turn;
  volatile int32_t* gave_up = &sh.gave_up;
  volatile uint32_t* running = sh.running;
  for (int64_t c = warp; c * kScanTiles < tiles; c += WARPS) {
    const int64_t first = c * kScanTiles;
    const int chunk = static_cast<int>(tiles - first < kScanTiles ? tiles - first : kScanTiles);
    uint32_t* word = a.status + first * kRadix + scanner * kWarp + lane;  // the chunk's first tile
    uint32_t w[kScanTiles];
#pragma unroll
    for (int r = 0; r < kScanTiles; ++r) w[r] = 0;
    ScanWait wait = {};
    uint32_t spins = 0;
    int handed = 0, there = 0;  // tiles whose prefixes are out; published tiles in front
    while (handed < chunk) {
      if (there < chunk) {
#pragma unroll
        for (int r = 0; r < kScanTiles; ++r)
          if (r >= there && r < chunk && w[r] == 0u) w[r] = ld_relaxed_u32(word + r * kRadix);
        there = 0;
#pragma unroll
        for (int r = 0; r < kScanTiles; ++r)
          if (there == r && __all_sync(0xFFFFFFFFu, w[r] != 0u)) there = r + 1;
      }
      const bool mine = __shfl_sync(0xFFFFFFFFu, static_cast<int>(*turn == c), 0) != 0;
      if (there == handed || !mine) {
        if (++spins % 32 == 0) {
          // the first kScanners tickets are no tiles, then ids from tile_base on are handed out in order
          const int64_t held_at = there < chunk ? first + there + 1 + kScanners - static_cast<int64_t>(a.tile_base) : 0;
          if (!__all_sync(0xFFFFFFFFu, scan_look(&wait, &a.head->tile_counter[a.pass], held_at, &a.head->abort_word,
                                                 a.wait_ns, a.err))) {
            if (lane == 0) *gave_up = 1;
            return;
          }
        }
        if (__any_sync(0xFFFFFFFFu, *gave_up)) return;
        continue;
      }
      __threadfence_block();
      __syncwarp();  // lane 0 saw the turn: its fence orders every lane's read
      uint32_t run = running[lane];
      if (there == chunk) {  // the turn goes on before the stores
        uint32_t total = 0;
#pragma unroll
        for (int r = 0; r < kScanTiles; ++r) total += w[r] & kValueMask;
        running[lane] = run + total;
        __syncwarp();
        if (lane == 0) {
          __threadfence_block();  // after every lane's sum
          *turn = c + 1;
        }
      }
#pragma unroll
      for (int r = 0; r < kScanTiles; ++r) {
        if (r >= handed && r < there) st_relaxed_u32(word + r * kRadix, kFlagInclusive | run);
        run += w[r] & kValueMask;
      }
      handed = there;
    }
  }
}

// This tile's rows of one digit: counted in the tiles before it.  False when that never came.
// The word is cleared for the next pass: its scanner is done with it once the prefix is
// there, and nobody else reads it.
__device__ __forceinline__ bool prefix_of(const PassArgs& a, uint32_t* word, uint32_t* excl) {
  SpinGuard guard;
  uint32_t w = ld_relaxed_u32(word);
  while ((w >> 30) != 2u) {
    if (!guard.go_on(&a.head->abort_word, a.wait_ns, a.err)) return false;
    w = ld_relaxed_u32(word);
  }
  st_relaxed_u32(word, 0u);
  *excl = w & kValueMask;
  return true;
}

// One tile.
template <int THREADS, int ITEMS, typename Digit>
__device__ __forceinline__ void pass_tile(const PassArgs& a, const PassCols& cols, const Digit digit, int64_t tile,
                                          int32_t* sk, int32_t* sv, PassShared<THREADS>& sh) {
  constexpr int WARPS = THREADS / kWarp;
  constexpr int TILE = THREADS * ITEMS;
  static_assert(THREADS >= kRadix && TILE < 65536, "one thread per digit, 16-bit counters");
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const int64_t row0 = tile * TILE;
  const int valid = static_cast<int>((a.n - row0) < TILE ? (a.n - row0) : TILE);
  const int lim = valid - warp * (kWarp * ITEMS) - lane;  // item i of this thread exists while 32 i < lim
  const int32_t* kin = cols.kin + row0 + warp * (kWarp * ITEMS) + lane;
  const int32_t* vin = cols.vin + row0 + warp * (kWarp * ITEMS) + lane;
  const uint64_t pol = policy_evict_first();
  int32_t k[ITEMS];  // keys, then values
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) k[i] = i * kWarp < lim ? ld_stream(kin + i * kWarp, pol) : 0;
  if (tid == 0 && valid >= 4)  // the values are read after the keys are placed: on their way to L2
    bulk_prefetch_l2(cols.vin + row0, static_cast<uint32_t>(valid & ~3) * 4u);

  // Stable per-warp ranking, warp-striped: item i of lane l in warp w is tile position
  // w*32*ITEMS + i*32 + l, so the rows of round i come before those of round i + 1.
  uint32_t r[ITEMS];  // digit << 16 | rank in the warp, then place in the tile
  static_assert(WARPS * kRadix <= TILE, "the warps' tables fit the place of the sorted tile");
  uint2* table = reinterpret_cast<uint2*>(sk) + warp * kRadix;
  for (int i = lane; i < kRadix / 2; i += kWarp) reinterpret_cast<uint4*>(table)[i] = make_uint4(0, 0, 0, 0);
  __syncwarp();
  if (valid == TILE)
    rank_rows<ITEMS, true>(k, lim, digit, table, r);
  else
    rank_rows<ITEMS, false>(k, lim, digit, table, r);
  for (int i = lane; i < kRadix; i += kWarp) sh.whist[warp][i] = static_cast<uint16_t>(table[i].y);
  __syncthreads();

  // Per digit: exclusive offsets of the warps, the tile's count (published for the later
  // tiles) and its start in the tile.
  uint32_t count = 0;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      const uint32_t c = sh.whist[w][tid];
      sh.whist[w][tid] = static_cast<uint16_t>(count);
      count += c;
    }
    st_relaxed_u32(a.status + tile * kRadix + tid, kFlagAggregate | count);
    const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(count), lane));
    if (lane == kWarp - 1) sh.scan_tmp[warp] = inc;
    sh.tile_start[tid] = inc - count;
  }
  __syncthreads();
  if (tid < kRadix) {
    uint32_t wbase = 0;
    for (int w = 0; w < warp; ++w) wbase += sh.scan_tmp[w];
    sh.tile_start[tid] += wbase;
  }
  __syncthreads();

  // BlockShuffle: keys and values to their sorted positions of the tile
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    if (i * kWarp < lim) {
      const uint32_t d = r[i] >> 16;
      r[i] = sh.tile_start[d] + sh.whist[warp][d] + (r[i] & 0xFFFFu);
      sk[r[i]] = k[i];
    }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) k[i] = i * kWarp < lim ? ld_stream(vin + i * kWarp, pol) : 0;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    if (i * kWarp < lim) sv[r[i]] = k[i];

  // Global positions; the scanner has mostly answered by now.
  bool failed = false;
  if (tid < kRadix) {
    uint32_t excl = 0;
    failed = !prefix_of(a, a.status + tile * kRadix + tid, &excl);
    const uint32_t start = a.digit_base[tid] + excl;
    // the digit's run [start, start + count) of this tile must land inside the output
    if (!failed && count && static_cast<int64_t>(start) + count > a.n) {
      set_error(a.err, CRYS_DEV_BOUNDS);
      failed = true;
    }
    sh.out_shift[tid] = start - sh.tile_start[tid];
  }
  if (__syncthreads_or(failed)) return;
  // BlockStore in sorted order: each digit run is written with consecutive addresses.
#pragma unroll 4
  for (int i = tid; i < valid; i += THREADS) {
    const int32_t key = sk[i];
    const uint32_t g = sh.out_shift[digit(key)] + static_cast<uint32_t>(i);  // checked per digit above
    cols.kout[g] = key;
    cols.vout[g] = sv[i];
  }
}

// Resident blocks per SM a tile shape's shared memory and 65536 registers allow.
constexpr int pass_blocks(int threads, int items) {
  const int smem = 227 * 1024 / (threads * items * 8 + threads * 16 + 4 * 1024);
  const int regs = 65536 / (threads * (2 * items + 18));
  return smem < regs ? smem : regs;
}

template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, pass_blocks(THREADS, ITEMS)) sort_pass_kernel(const __grid_constant__ PassArgs a) {
  constexpr int TILE = THREADS * ITEMS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  int32_t* sk = reinterpret_cast<int32_t*>(smem_raw);  // the tile's keys in sorted order
  int32_t* sv = sk + TILE;                             // and values
  __shared__ PassShared<THREADS> sh;
  const int tid = threadIdx.x;
  const int passes = static_cast<int>(a.head->passes);
  if (a.pass >= passes) return;
  // the last pass writes to the output, the one before to the scratch, and so on
  const bool to_out = (passes - 1 - a.pass) % 2 == 0;
  PassCols cols;
  cols.kin = a.pass == 0 ? a.keys_in : to_out ? a.keys_tmp : a.keys_out;
  cols.vin = a.pass == 0 ? a.vals_in : to_out ? a.vals_tmp : a.vals_out;
  cols.kout = to_out ? a.keys_out : a.keys_tmp;
  cols.vout = to_out ? a.vals_out : a.vals_tmp;
  const uint32_t shift = a.head->shift[a.pass], mask = a.head->mask[a.pass];
  const bool buckets = a.head->buckets != 0;
  const KeyRange range = a.head->range;
  if (tid == 0)  // a sort whose earlier pass gave up does no further work (tile id past the end)
    sh.tile = ld_relaxed_u32(&a.head->abort_word) ? 0xFFFFFFFFu : atomicAdd(&a.head->tile_counter[a.pass], 1u);
  __syncthreads();
  const uint32_t ticket = sh.tile;
  if (ticket < static_cast<uint32_t>(kScanners)) {
    __shared__ ScanShared scan;
    scan_tiles<THREADS / kWarp>(a, static_cast<int>(ticket), (a.n + TILE - 1) / TILE, scan);
    return;
  }
  const int64_t tile = static_cast<int64_t>(ticket) - kScanners + a.tile_base;
  if (ticket == 0xFFFFFFFFu || tile * TILE >= a.n) return;
  if (buckets)
    pass_tile<THREADS, ITEMS>(a, cols, PassDigit<true>{range, shift, mask}, tile, sk, sv, sh);
  else
    pass_tile<THREADS, ITEMS>(a, cols, PassDigit<false>{KeyRange{}, shift, mask}, tile, sk, sv, sh);
}

struct Layout {
  size_t tmp_keys, tmp_vals, hist, base, counters, status, total;
  int64_t tiles;
};

size_t up256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

int64_t min_tile() {
  int64_t m = INT64_MAX;
  for (int i = 0; i < kNumVariants[CRYS_OP_SORT]; ++i) {
    const int64_t t = static_cast<int64_t>(kTiles[CRYS_OP_SORT][i].threads) * kTiles[CRYS_OP_SORT][i].items;
    if (t < m) m = t;
  }
  return m;
}

Layout layout(int64_t n) {
  Layout L;
  L.tiles = (n + min_tile() - 1) / min_tile();
  size_t off = 0;
  L.tmp_keys = off;
  off += up256(static_cast<size_t>(n) * 4);
  L.tmp_vals = off;
  off += up256(static_cast<size_t>(n) * 4);
  L.hist = off;
  off += up256(kPasses * kRadix * 4);
  L.base = off;
  off += up256(kPasses * kRadix * 4);
  L.counters = off;
  off += 256;
  L.status = off;
  off += up256(static_cast<size_t>(L.tiles) * kRadix * 4);
  L.total = off;
  return L;
}

// Where the bucket plan keeps its counts and first rows (2^bits words each), or NULL when
// the scratch has no room for them: with up to 256 buckets in the starts of passes that the
// plan does not run, otherwise behind the status words of the tile shape in use.
uint32_t* bucket_words(char* temp, const Layout& L, int bits, int64_t tiles) {
  if (bits <= 8) return reinterpret_cast<uint32_t*>(temp + L.base) + kRadix;
  const size_t at = L.status + up256(static_cast<size_t>(tiles) * kRadix * 4);
  const size_t need = (size_t{2} << bits) * 4;
  return at + need <= L.total ? reinterpret_cast<uint32_t*>(temp + at) : nullptr;
}

template <int THREADS, int ITEMS>
int run_sort(const int32_t* keys_in, const int32_t* vals_in, int32_t* keys_out, int32_t* vals_out, int64_t n, char* temp,
             const Layout& L, uint32_t stall_base, uint64_t stall_ns, cudaStream_t s) {
  constexpr int TILE = THREADS * ITEMS;
  const int64_t tiles = (n + TILE - 1) / TILE;
  const size_t smem = static_cast<size_t>(TILE) * 8;
  auto kernel = sort_pass_kernel<THREADS, ITEMS>;
  if (!allow_smem(kernel, smem)) return CRYS_ECUDA;
  SortHead* head = reinterpret_cast<SortHead*>(temp + L.counters);
  uint32_t* base = reinterpret_cast<uint32_t*>(temp + L.base);
  int32_t* err = device_error_word();
  if (!err) return CRYS_ECUDA;
  const int bits = n <= kMaxBucketRows ? range_bits(n, kLocalCap) : 0;
  uint32_t* counts = bits ? bucket_words(temp, L, bits, tiles) : nullptr;
  const int64_t buckets = int64_t{1} << bits;
  // One clearing: the histogram, the head, the status words (every tile of a pass clears its
  // own again) and, right behind them, the counts of more than 256 buckets.
  size_t cleared = L.status + up256(static_cast<size_t>(tiles) * kRadix * 4) - L.hist;
  if (counts && bits > 8) cleared += static_cast<size_t>(buckets) * 4;
  if (cudaMemsetAsync(temp + L.hist, 0, cleared, s) != cudaSuccess) return CRYS_ECUDA;
  if (counts) {
    if (launch_key_range(keys_in, n, bits, &head->range, &head->crowded, s) != CRYS_OK) return CRYS_ECUDA;
    const size_t bins = static_cast<size_t>(buckets) * 2;
    if (!allow_smem(count_buckets_kernel, size_t{2} << 16)) return CRYS_ECUDA;
    // a block for every 16 rows per thread, at most one per SM
    int64_t grid = (n + 16 * kCountThreads - 1) / (16 * kCountThreads);
    if (grid > sm_count()) grid = sm_count();
    count_buckets_kernel<<<static_cast<unsigned>(grid), kCountThreads, bins, s>>>(keys_in, n, bits, head, counts,
                                                                                 counts + buckets, base);
    note_launch();
  }
  int64_t hist_grid = (n + 16 * kHistThreads - 1) / (16 * kHistThreads);
  if (hist_grid > sm_count() * 4) hist_grid = sm_count() * 4;
  sort_hist_kernel<<<static_cast<unsigned>(hist_grid), kHistThreads, 0, s>>>(keys_in, n, reinterpret_cast<unsigned int*>(temp + L.hist),
                                                                           head, base);
  note_launch();
  if (check_launch() != CRYS_OK) return CRYS_ECUDA;
  PassArgs a;
  a.keys_in = keys_in;
  a.vals_in = vals_in;
  a.keys_tmp = reinterpret_cast<int32_t*>(temp + L.tmp_keys);
  a.vals_tmp = reinterpret_cast<int32_t*>(temp + L.tmp_vals);
  a.keys_out = keys_out;
  a.vals_out = vals_out;
  a.n = n;
  a.head = head;
  a.status = reinterpret_cast<uint32_t*>(temp + L.status);
  a.err = err;
  for (int p = 0; p < kPasses; ++p) {
    a.tile_base = p == 0 ? stall_base : 0u;
    a.wait_ns = p == 0 ? stall_ns : kWaitBoundNs;
    a.pass = p;
    a.digit_base = base + p * kRadix;
    kernel<<<static_cast<unsigned int>(tiles + kScanners), THREADS, smem, s>>>(a);
    note_launch();
    if (check_launch() != CRYS_OK) return CRYS_ECUDA;
  }
  if (!counts) return CRYS_OK;
  LocalArgs l{keys_out, vals_out, keys_out, vals_out, counts + buckets, counts, static_cast<uint32_t>(n), err,
              &head->buckets, &head->abort_word};
  return launch_local_sort<false>(l, static_cast<unsigned>(buckets), s);
}

constexpr int kOp = CRYS_OP_SORT;

}  // namespace
}  // namespace crys

extern "C" int crys_sort(const int32_t* keys_in, const int32_t* vals_in, int32_t* keys_out,
                         int32_t* vals_out, int64_t n, void* d_temp, size_t* temp_bytes,
                         crys_stream stream) {
  using namespace crys;
  if (n < 0 || n > static_cast<int64_t>(kValueMask)) return CRYS_EINVAL;
  const Layout L = layout(n);
  if (!d_temp && temp_bytes) {
    *temp_bytes = L.total;
    return CRYS_OK;
  }
  if (n == 0) return CRYS_OK;
  if (!d_temp || !temp_bytes) return CRYS_EINVAL;
  if (*temp_bytes < L.total) return CRYS_ENOMEM;
  if (!keys_in || !vals_in || !keys_out || !vals_out || !aligned16(keys_in) || !aligned16(vals_in) ||
      !aligned16(keys_out) || !aligned16(vals_out))
    return CRYS_EINVAL;
  if (reinterpret_cast<uintptr_t>(d_temp) & 255u) return CRYS_EINVAL;
  auto overlaps = [n](const void* a, const void* b) {
    const char* x = static_cast<const char*>(a);
    const char* y = static_cast<const char*>(b);
    return x < y + n * 4 && y < x + n * 4;
  };
  if (overlaps(keys_out, keys_in) || overlaps(keys_out, vals_in) || overlaps(vals_out, keys_in) ||
      overlaps(vals_out, vals_in) || overlaps(keys_out, vals_out))
    return CRYS_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* temp = static_cast<char*>(d_temp);
  uint32_t stall_base = 0;
  uint64_t stall_ns = kWaitBoundNs;
  // a test's stall applies to the first pass: a stalled sort goes by passes, whatever its size
  const bool stalled = take_stall(CRYS_OP_SORT, &stall_base, &stall_ns);
  const bool any_tile = set_tile_variant(kOp) < 0;
  if (n <= kLocalCap && any_tile && !stalled) {  // one block sorts everything
    int32_t* err = device_error_word();
    if (!err) return CRYS_ECUDA;
    return launch_local_sort<false>(
        LocalArgs{keys_in, vals_in, keys_out, vals_out, nullptr, nullptr, static_cast<uint32_t>(n), err}, 1, s);
  }
  if (!stalled && any_tile && small_sort_fits(n) &&
      launch_small_sort(keys_in, vals_in, reinterpret_cast<int32_t*>(temp + L.tmp_keys),
                        reinterpret_cast<int32_t*>(temp + L.tmp_vals), keys_out, vals_out, n, temp + L.counters, s) == CRYS_OK)
    return CRYS_OK;  // (refused on a stream that owns few SMs: by passes)
  // up to 2^20 rows (one pass by buckets) the smallest tile, so that more SMs have one
  switch (any_tile && n <= (1 << 20) ? kNumVariants[kOp] - 1 : tile_variant(kOp)) {
    case 1: return run_sort<kTiles[kOp][1].threads, kTiles[kOp][1].items>(keys_in, vals_in, keys_out, vals_out, n, temp, L, stall_base, stall_ns, s);
    case 2: return run_sort<kTiles[kOp][2].threads, kTiles[kOp][2].items>(keys_in, vals_in, keys_out, vals_out, n, temp, L, stall_base, stall_ns, s);
    case 3: return run_sort<kTiles[kOp][3].threads, kTiles[kOp][3].items>(keys_in, vals_in, keys_out, vals_out, n, temp, L, stall_base, stall_ns, s);
    default: return run_sort<kTiles[kOp][0].threads, kTiles[kOp][0].items>(keys_in, vals_in, keys_out, vals_out, n, temp, L, stall_base, stall_ns, s);
  }
}
