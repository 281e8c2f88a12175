// Sorts of up to 2^20 pairs in ONE launch, for crys_sort and crys_sort_msb (the result is
// stable).  The steps of the larger sort would be a dozen launches and clearings here, and the
// host needs 3 to 4 us for each; the work itself takes less.
//
// A cooperative launch of a block per SM (fewer for few rows, up to 211 where the blocks would
// hold too many), each holding up to 4992 rows, with a grid barrier between the steps:
//  1. smallest and largest key;
//  2. every block ranks its rows stably by the bucket of their key (up to 256 buckets over the
//     key range) and publishes its bucket counts;
//  3. every block sums the counts of the blocks before it and stores its rows, bucket by
//     bucket, to the scratch columns;
//  4. the blocks sort the buckets (localsort.cuh) into the output.  A key range of at most
//     256 values leaves nothing to sort: step 3 writes the output.
// When a bucket is too large for a block, steps 2 and 3 are repeated for the 8-bit digits of
// key - smallest instead, from the low one to the high one (each block takes its rows of the
// previous digit's result again).
//
// 100,003 random pairs: 60 us per call with the larger sort's steps, 22 us here; 2^20 pairs: 84
// and 46 us.  What bounds it is latency: three grid barriers of about 2 us each and a few
// dependent trips to L2 between them, at one block per SM.
#include "common.cuh"
#include "localsort.cuh"
#include "multisplit.cuh"

namespace crys {
namespace {

constexpr int kThreads = kLocalThreads;
constexpr int kItems = kLocalItems;
constexpr int kWarps = kThreads / kWarp;
constexpr int kRows = kThreads * kItems;  // rows a block holds
static_assert(kRows < 65536, "16-bit counts");

// One per call, cleared before it.
struct SmallHead {
  unsigned int arrived;     // blocks at the grid barriers so far
  unsigned int abort_word;  // set by the first block that gives up
  unsigned int high;        // largest key, sign bit flipped
  unsigned int low;         // complement of the smallest key, sign bit flipped
};

struct SmallArgs {
  const int32_t *keys_in, *vals_in;
  int32_t *keys_tmp, *vals_tmp;
  int32_t *keys_out, *vals_out;
  uint32_t n;
  uint32_t share;    // rows per block
  uint32_t buckets;  // at most kRadix
  SmallHead* head;
  int32_t* err;
};

struct SplitShared {
  int32_t keys[kRows];  // first the warps' ranking tables, then the rows in bucket order
  int32_t vals[kRows];
  alignas(4) uint16_t whist[kWarps][kRadix];  // per-warp counts, then offsets
  uint32_t start[kRadix];                     // the digit's first row in the block
  uint32_t dest[kRadix];                      // its first row in the result minus `start`
  uint32_t total[kRadix], before[kRadix];     // rows of all blocks, of the blocks before this one
  uint32_t tmp[kWarps + 1];
};
static_assert(sizeof(uint2) * kRadix * kWarps <= sizeof(int32_t) * 2 * kRows, "the tables fit the place of the rows");

union SmallShared {
  LocalShared local;
  SplitShared split;
};
static_assert(sizeof(SplitShared) <= offsetof(LocalShared, loaded), "the copy barrier stays valid");

// Grid barrier number `k` (1, 2, ...).  False when the wait ran out.
__device__ __forceinline__ bool grid_barrier(const SmallArgs& a, unsigned int k) {
  __threadfence();
  asm volatile("fence.proxy.async;" ::: "memory");  // rows stored here may be read by a bulk copy
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    atomicAdd(&a.head->arrived, 1u);
    SpinGuard guard;
    while (ok && ld_relaxed_u32(&a.head->arrived) < k * gridDim.x)
      ok = guard.go_on(&a.head->abort_word, kWaitBoundNs, a.err);
    __threadfence();
  }
  const bool all = !__syncthreads_or(!ok);
  asm volatile("fence.proxy.async;" ::: "memory");
  return all;
}

// Bucket of a key: evenly over [lo, lo + span]; the key's offset itself for at most 256 values.
struct BucketDigit {
  uint32_t lo, scale;
  __device__ __forceinline__ uint32_t operator()(int32_t k) const {
    const uint32_t off = static_cast<uint32_t>(k) - lo;
    return scale ? __umulhi(off, scale) : off;
  }
};
struct ByteDigit {
  uint32_t lo, shift;
  __device__ __forceinline__ uint32_t operator()(int32_t k) const {
    return ((static_cast<uint32_t>(k) - lo) >> shift) & 255u;
  }
};

// Ranks the block's rows k (row first + warp * 32 * per + 32 i + lane for item i < per, present
// while 32 i < lim) by digit and publishes the block's counts in its row of `matrix`.
template <typename Digit>
__device__ __forceinline__ void split_count(SplitShared& sh, const int32_t (&k)[kItems], int lim, const Digit& digit,
                                            uint32_t (&r)[kItems], uint16_t* matrix) {
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  uint2* table = reinterpret_cast<uint2*>(sh.keys) + warp * kRadix;
  for (int i = lane; i < kRadix / 2; i += kWarp) reinterpret_cast<uint4*>(table)[i] = make_uint4(0, 0, 0, 0);
  __syncwarp();
  rank_rows<kItems, false>(k, lim, digit, table, r);
  for (int i = lane; i < kRadix; i += kWarp) sh.whist[warp][i] = static_cast<uint16_t>(table[i].y);
  __syncthreads();
  uint32_t count = 0;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = sh.whist[w][tid];
      sh.whist[w][tid] = static_cast<uint16_t>(count);
      count += c;
    }
    __stcg(&matrix[blockIdx.x * kRadix + tid], static_cast<uint16_t>(count));
    sh.total[tid] = sh.before[tid] = 0;
  }
  uint32_t all;
  const uint32_t ex = local_scan(count, sh.tmp, &all);
  if (tid < kRadix) sh.start[tid] = ex;
  __syncthreads();
}

// Sums every block's counts (a warp per row of the matrix, 8 digits per lane): sh.total,
// and sh.dest from the sums of the blocks before this one.  Returns the largest total.
__device__ __forceinline__ uint32_t split_offsets(SplitShared& sh, const uint16_t* matrix) {
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  uint32_t all[8] = {}, before[8] = {};
#pragma unroll 4
  for (uint32_t b = warp; b < gridDim.x; b += kWarps) {
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(matrix + b * kRadix) + lane);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t c = j % 2 ? w[j / 2] >> 16 : w[j / 2] & 0xFFFFu;
      all[j] += c;
      before[j] += b < blockIdx.x ? c : 0u;
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    atomicAdd(&sh.total[lane * 8 + j], all[j]);
    atomicAdd(&sh.before[lane * 8 + j], before[j]);
  }
  __syncthreads();
  const uint32_t t = tid < kRadix ? sh.total[tid] : 0u;
  uint32_t sum;
  const uint32_t base = local_scan(t, sh.tmp, &sum);
  if (tid < kRadix) sh.dest[tid] = base + sh.before[tid] - sh.start[tid];
  uint32_t most = __reduce_max_sync(0xFFFFFFFFu, t);
  __syncthreads();
  if (lane == 0) sh.tmp[warp] = most;
  __syncthreads();
  most = __reduce_max_sync(0xFFFFFFFFu, sh.tmp[min(lane, kWarps - 1)]);
  __syncthreads();
  return most;
}

// Stores the block's rows, in digit order, to kout / vout.
template <typename Digit>
__device__ __forceinline__ void split_store(const SmallArgs& a, SplitShared& sh, const int32_t (&k)[kItems], int lim,
                                            const int32_t* vals, int count, const Digit& digit, uint32_t (&r)[kItems],
                                            int32_t* kout, int32_t* vout) {
  const int warp = threadIdx.x / kWarp;
#pragma unroll
  for (int i = 0; i < kItems; ++i)
    if (i * kWarp < lim) {
      const uint32_t d = r[i] >> 16;
      r[i] = sh.start[d] + sh.whist[warp][d] + (r[i] & 0xFFFFu);
      sh.keys[r[i]] = k[i];
    }
  int32_t v[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) v[i] = i * kWarp < lim ? __ldcg(vals + i * kWarp) : 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i)
    if (i * kWarp < lim) sh.vals[r[i]] = v[i];
  __syncthreads();
  for (int j = threadIdx.x; j < count; j += kThreads) {
    const int32_t key = sh.keys[j];
    const uint32_t g = sh.dest[digit(key)] + static_cast<uint32_t>(j);
    if (g < a.n) {
      kout[g] = key;
      vout[g] = sh.vals[j];
    } else {
      set_error(a.err, CRYS_DEV_BOUNDS);
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kThreads, 2) small_sort_kernel(const __grid_constant__ SmallArgs a) {
  extern __shared__ __align__(128) unsigned char small_smem[];
  SmallShared& sh = *reinterpret_cast<SmallShared*>(small_smem);
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const uint32_t first = min(blockIdx.x * a.share, a.n);
  const int count = static_cast<int>(min(a.share, a.n - first));
  const int per = (count + kThreads - 1) / kThreads;  // rows per thread, warp-striped
  const int p0 = warp * (kWarp * per) + lane;
  const int lim = min(count - p0, kWarp * per);
  const uint32_t mine = first + static_cast<uint32_t>(p0);  // this thread's first row
  unsigned int barriers = 0;
  if (tid == 0) {
    mbar_init(&sh.local.loaded, 1);
    fence_barrier_init();
  }
  // 1. the key range, exact
  int32_t k[kItems];
  uint32_t high = 0, low = 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) k[i] = i * kWarp < lim ? a.keys_in[mine + i * kWarp] : 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i)
    if (i * kWarp < lim) {
      const uint32_t u = static_cast<uint32_t>(k[i]) ^ 0x80000000u;
      high = max(high, u);
      low = max(low, ~u);
    }
  high = __reduce_max_sync(0xFFFFFFFFu, high);
  low = __reduce_max_sync(0xFFFFFFFFu, low);
  if (lane == 0 && p0 - lane < count) {
    atomicMax(&a.head->high, high);
    atomicMax(&a.head->low, low);
  }
  if (!grid_barrier(a, ++barriers)) return;
  const uint32_t hi = ld_relaxed_u32(&a.head->high), lo = ~ld_relaxed_u32(&a.head->low);
  const uint32_t span = hi - lo;
  const bool direct = span < kRadix;  // a bucket per value: nothing left to sort afterwards
  const BucketDigit bucket{lo ^ 0x80000000u,
                           direct ? 0u : static_cast<uint32_t>((static_cast<uint64_t>(a.buckets) << 32) / (static_cast<uint64_t>(span) + 1))};
  // 2. counts; 3. stores.  The matrix lies in whichever of the two key columns is not written.
  uint32_t r[kItems];
  uint16_t* matrix = reinterpret_cast<uint16_t*>(direct ? a.keys_tmp : a.keys_out);
  split_count(sh.split, k, lim, bucket, r, matrix);
  if (!grid_barrier(a, ++barriers)) return;
  const uint32_t most = split_offsets(sh.split, matrix);
  if (direct || most <= static_cast<uint32_t>(kLocalCap)) {
    split_store(a, sh.split, k, lim, a.vals_in + mine, count, bucket, r, direct ? a.keys_out : a.keys_tmp,
                direct ? a.vals_out : a.vals_tmp);
    if (direct) return;
    // 4. the buckets: their rows are where every block's total says
    uint32_t begin_of = 0, size_of = 0;
    {
      uint32_t sum;
      size_of = tid < kRadix ? sh.split.total[tid] : 0u;
      begin_of = local_scan(size_of, sh.split.tmp, &sum);
    }
    if (!grid_barrier(a, ++barriers)) return;
    const LocalArgs l{a.keys_tmp, a.vals_tmp, a.keys_out, a.vals_out, nullptr, nullptr, a.n, a.err};
    __shared__ uint32_t at[2];
    uint32_t parity = 0;
    for (int b = blockIdx.x; b < kRadix; b += gridDim.x) {
      if (tid == b) {
        at[0] = begin_of;
        at[1] = size_of;
      }
      __syncthreads();
      const uint32_t begin = at[0], size = at[1];
      if (size) {
        local_sort_bucket(l, sh.local, begin, size, parity);
        parity ^= 1u;
      }
      fence_proxy_async_smem();  // the next bucket's values come by a bulk copy into the same place
      __syncthreads();  // the bucket is stored: its shared memory is free
    }
    return;
  }
  // a bucket too large for a block: by digits of key - lo
  const int passes = (32 - __clz(span) + 7) / 8;
  for (int p = 0; p < passes; ++p) {
    const bool to_out = (passes - 1 - p) % 2 == 0;
    const int32_t* kin = p == 0 ? a.keys_in : to_out ? a.keys_tmp : a.keys_out;
    const int32_t* vin = p == 0 ? a.vals_in : to_out ? a.vals_tmp : a.vals_out;
    int32_t* kout = to_out ? a.keys_out : a.keys_tmp;
    const ByteDigit digit{lo ^ 0x80000000u, static_cast<uint32_t>(8 * p)};
    if (!grid_barrier(a, ++barriers)) return;  // the previous result is complete, its counts are read
#pragma unroll
    for (int i = 0; i < kItems; ++i) k[i] = i * kWarp < lim ? __ldcg(kin + mine + i * kWarp) : 0;
    matrix = reinterpret_cast<uint16_t*>(kout);
    split_count(sh.split, k, lim, digit, r, matrix);
    if (!grid_barrier(a, ++barriers)) return;
    split_offsets(sh.split, matrix);
    if (!grid_barrier(a, ++barriers)) return;  // every block has read the counts: the column is free
    split_store(a, sh.split, k, lim, vin + mine, count, digit, r, kout, to_out ? a.vals_out : a.vals_tmp);
  }
}

}  // namespace

bool small_sort_fits(int64_t n) {
  if (n <= kLocalCap || n > (int64_t{1} << 20)) return false;
  static_assert(sizeof(SmallHead) <= 256, "the head has 256 bytes of the scratch");
  if (!allow_smem(small_sort_kernel, sizeof(SmallShared))) return false;
  const int64_t blocks =
      static_cast<int64_t>(sm_count()) *
      blocks_per_sm(reinterpret_cast<const void*>(small_sort_kernel), kThreads, sizeof(SmallShared));
  return n <= blocks * kRows;
}

int launch_small_sort(const int32_t* keys_in, const int32_t* vals_in, int32_t* keys_tmp, int32_t* vals_tmp,
                      int32_t* keys_out, int32_t* vals_out, int64_t n, void* head, cudaStream_t s) {
  int32_t* err = device_error_word();
  if (!err) return CRYS_ECUDA;
  if (cudaMemsetAsync(head, 0, sizeof(SmallHead), s) != cudaSuccess) return CRYS_ECUDA;
  // A block per SM, fewer while their rows of counts would not fit the key column (2 bytes per
  // count, 4 per row), more once they would hold too many rows.  As many buckets as blocks
  // up to 2^18 rows, so that each block sorts one; then 256, so that a bucket fits a block.
  // (With a block per 1024 rows and always 256 buckets, 5000 rows took 170 us, the blocks
  // sorting 51 buckets each; 72 us by a dozen launches.)
  int64_t grid = n / (kRadix / 2);
  if (grid > sm_count()) grid = sm_count();
  if (grid < (n + kRows - 1) / kRows) grid = (n + kRows - 1) / kRows;
  uint32_t buckets = kRadix;
  while (buckets > grid && n <= (1 << 18)) buckets /= 2;
  SmallArgs a{keys_in, vals_in, keys_tmp, vals_tmp, keys_out, vals_out, static_cast<uint32_t>(n),
              static_cast<uint32_t>((n + grid - 1) / grid), buckets, static_cast<SmallHead*>(head), err};
  void* args[] = {&a};
  if (cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(small_sort_kernel), dim3(static_cast<unsigned>(grid)),
                                  dim3(kThreads), args, sizeof(SmallShared), s) != cudaSuccess) {
    cudaGetLastError();  // the blocks do not fit the SMs of this stream together: not an error of the call
    return CRYS_ECUDA;
  }
  note_launch();
  return check_launch();
}

}  // namespace crys
