// The key range a sort partitions by: an order-preserving map of the keys onto 2^bits
// buckets.
//
// The smallest and largest of a sample of the keys, widened a little, are spread evenly over
// the buckets; keys outside them go to the first and last bucket, so the map is monotone
// for every input and the buckets are sorted afterwards whatever they hold.  Keys of a
// narrow range (dense ids, codes) thus fill all buckets like keys over all 32 bits do.
#pragma once

#include "common.cuh"

namespace crys {

struct KeyRange {
  int32_t lo;      // keys at or below it go to bucket 0
  uint32_t scale;  // buckets per key, times 2^32
  uint32_t last;   // last bucket
  __device__ __forceinline__ uint32_t place(int32_t k) const {
    const uint32_t off = static_cast<uint32_t>(max(k, lo)) - static_cast<uint32_t>(lo);
    return min(__umulhi(off, scale), last);
  }
};

constexpr int kRangeThreads = 1024;
constexpr int kRangeSamples = 8;  // per thread
// Keys that differ in at most this many bytes are sorted stably by digits, one pass per byte
// (and a count of 0.2 ms for 2^28 rows): two passes for 2^28 keys of two bytes take 3.09 ms, the
// buckets 4.8 ms when their leading bits are spread evenly; three passes for keys of three
// bytes 4.26 to 4.46 ms, the buckets 4.48 to 6.46 ms, because few key values crowd the bins of
// a bucket.  A fourth pass would add 1.2 to 1.4 ms, to more than the 4.36 ms of the buckets.
constexpr int kFewBytes = 3;

// One block: 256 runs of 32 consecutive keys, spread evenly over the column and taken by a
// warp each, always with the first and the last key.  `few`, when given, is set if the sampled
// keys differ in at most kFewBytes of their bytes.
static __global__ void __launch_bounds__(kRangeThreads) key_range_kernel(const int32_t* __restrict__ keys, int64_t n,
                                                                         int bits, KeyRange* out, uint32_t* few) {
  __shared__ int32_t slo[kRangeThreads / kWarp], shi[kRangeThreads / kWarp];
  __shared__ uint32_t sdiff[kRangeThreads / kWarp];
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  constexpr int kRuns = kRangeThreads / kWarp * kRangeSamples;
  int32_t k[kRangeSamples];
#pragma unroll
  for (int j = 0; j < kRangeSamples; ++j) {
    const int64_t run = static_cast<int64_t>(j) * (kRangeThreads / kWarp) + warp;
    const int64_t i = run * (n > kWarp ? n - kWarp : 0) / (kRuns - 1) + lane;
    k[j] = keys[i < n ? i : n - 1];
  }
  const int32_t ref = keys[0];
  int32_t lo = k[0], hi = k[0];
  uint32_t diff = static_cast<uint32_t>(k[0] ^ ref);
#pragma unroll
  for (int j = 1; j < kRangeSamples; ++j) {
    lo = min(lo, k[j]);
    hi = max(hi, k[j]);
    diff |= static_cast<uint32_t>(k[j] ^ ref);
  }
  lo = __reduce_min_sync(0xFFFFFFFFu, lo);
  hi = __reduce_max_sync(0xFFFFFFFFu, hi);
  diff = __reduce_or_sync(0xFFFFFFFFu, diff);
  if (lane == 0) {
    slo[warp] = lo;
    shi[warp] = hi;
    sdiff[warp] = diff;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 0; w < kRangeThreads / kWarp; ++w) {
    lo = min(lo, slo[w]);
    hi = max(hi, shi[w]);
    diff |= sdiff[w];
  }
  // the extremes of 8192 sampled keys of an even distribution miss about 2^-13 of it at
  // either end, eight buckets of 65536: widened by 2^-8 of the range they miss nothing
  const int64_t widen = (static_cast<int64_t>(hi) - lo) / 256;
  const int64_t l = max(static_cast<int64_t>(lo) - widen, static_cast<int64_t>(INT32_MIN));
  const int64_t h = min(static_cast<int64_t>(hi) + widen, static_cast<int64_t>(INT32_MAX));
  const uint64_t span = static_cast<uint64_t>(h - l) + 1;  // 1 .. 2^32
  const uint64_t buckets = 1ull << bits;
  out->lo = static_cast<int32_t>(l);
  out->scale = span <= buckets ? 0xFFFFFFFFu : static_cast<uint32_t>((buckets << 32) / span);
  out->last = static_cast<uint32_t>(buckets - 1);
  int bytes = 0;
  for (int b = 0; b < 32; b += 8) bytes += ((diff >> b) & 255u) != 0u;
  if (few && bytes <= kFewBytes) *few = 1;
}

inline int launch_key_range(const int32_t* keys, int64_t n, int bits, KeyRange* out, uint32_t* few, cudaStream_t s) {
  key_range_kernel<<<1, kRangeThreads, 0, s>>>(keys, n, bits, out, few);
  note_launch();
  return check_launch();
}

// Bits of a key's place that are partitioned before the buckets are sorted, one block each:
// none while the rows fit one block (`cap` rows), 8 bits (one pass) up to 2^20 rows, then for
// buckets of 2048 to 4096 rows on average, at most 16 bits (two passes).
inline int range_bits(int64_t n, int cap) {
  if (n <= cap) return 0;
  int bits = 8;
  while (bits < 16 && (int64_t{4096} << bits) < n) ++bits;
  return bits;
}

}  // namespace crys
