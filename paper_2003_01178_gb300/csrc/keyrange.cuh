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
constexpr int kRangeBatch = 8;  // samples of a thread in flight together
// Keys that differ in at most this many bytes are sorted stably by digits, one pass per byte
// (and a count of 0.2 ms for 2^28 rows): two passes for 2^28 keys of two bytes take 3.09 ms, the
// buckets 4.8 ms when their leading bits are spread evenly; three passes for keys of three
// bytes 4.26 to 4.46 ms, the buckets 4.48 to 6.46 ms, because few key values crowd the bins of
// a bucket.  A fourth pass would add 1.2 to 1.4 ms, to more than the 4.36 ms of the buckets.
constexpr int kFewBytes = 3;
// Rows per key value, as estimated from the equal pairs of a sample, above which the keys are
// sorted stably by digits too: more rows share a bin of a bucket than its bins are made for.
// 36M keys of random 32-bit values, by buckets and by digits: 8 rows per value 0.94 and 0.94
// ms, 10 1.09 and 0.93, 12 1.22, 16 to 128 1.39 (four digits with a look-back 0.95); 150M keys: 8
// rows 3.45 and 3.39 ms, 12 4.10 and 3.35, 16 4.40.
constexpr int kCrowdedRows = 8;

// Rows sampled: the power of two of at least 2 sqrt(n), at most `most`.
inline int range_samples(int64_t n, int most) {
  int samples = kRangeThreads;
  while (samples < most && static_cast<int64_t>(samples) * samples < 4 * n) samples *= 2;
  return samples;
}

// Row of sample i: the first, the last, then rows drawn independently (the 32-bit finaliser of
// MurmurHash3, Appleby).  Not evenly spaced runs of rows: where a column is made of pieces with
// ranges of their own, those runs miss whole pieces, and all keys of a missed one beyond the
// sampled range go to one bucket (MSB sort of 2^28 keys in 1000 such pieces: 17.9 ms).
__device__ __forceinline__ int64_t sample_row(uint32_t i, int64_t n) {
  if (i < 2) return i == 0 ? 0 : n - 1;
  uint32_t h = i * 0x9E3779B9u;
  h ^= h >> 16;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return static_cast<int64_t>((static_cast<uint64_t>(h) * static_cast<uint64_t>(n)) >> 32);
}

// What a stable sort asks of the sample: the sort goes by digits when the sampled keys
// differ in at most kFewBytes of their bytes or more than `pairs` sampled keys are repeats.
struct FewKeys {
  uint32_t* digits;  // set to 1 then
  uint32_t pairs;
};

// One block.  FEW: with the two questions of FewKeys.  The repeats are counted with a table of
// one word per sample in shared memory: a sample puts its key into the slot that it hashes
// to and finds there the last one that did.
template <bool FEW>
static __global__ void __launch_bounds__(kRangeThreads) key_range_kernel(const int32_t* __restrict__ keys, int64_t n,
                                                                         int bits, int samples, KeyRange* out,
                                                                         const __grid_constant__ FewKeys few) {
  extern __shared__ __align__(16) uint32_t last_key[];  // FEW: `samples` words
  __shared__ int32_t slo[kRangeThreads / kWarp], shi[kRangeThreads / kWarp];
  __shared__ uint32_t sdiff[kRangeThreads / kWarp];
  __shared__ uint32_t repeats;
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const int32_t ref = keys[0];
  const int slot_shift = __clz(samples) + 1;  // samples is a power of two
  if (FEW) {
    // no slot holds a key of its own at first: 0 hashes to slot 0, 1 to another one
    for (int i = threadIdx.x; i < samples; i += kRangeThreads) last_key[i] = i == 0;
    if (threadIdx.x == 0) repeats = 0;
    __syncthreads();
  }
  int32_t lo = ref, hi = ref;
  uint32_t diff = 0, mine = 0;
  for (int i0 = threadIdx.x; i0 < samples; i0 += kRangeBatch * kRangeThreads) {
    int32_t k[kRangeBatch];
#pragma unroll
    for (int j = 0; j < kRangeBatch; ++j) {
      const int i = i0 + j * kRangeThreads;
      k[j] = i < samples ? keys[sample_row(static_cast<uint32_t>(i), n)] : ref;
    }
#pragma unroll
    for (int j = 0; j < kRangeBatch; ++j) {
      lo = min(lo, k[j]);
      hi = max(hi, k[j]);
      diff |= static_cast<uint32_t>(k[j] ^ ref);
      const uint32_t key = static_cast<uint32_t>(k[j]);
      // (a thread that has met enough of them puts no more: hot keys would queue for one slot)
      if (FEW && mine <= few.pairs && i0 + j * kRangeThreads < samples)
        mine += atomicExch(&last_key[(key * 2654435769u) >> slot_shift], key) == key;
    }
  }
  if (FEW) {
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) atomicAdd(&repeats, mine);
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
  // the extremes of 1024 to 8192 sampled keys of an even distribution miss 2^-10 to 2^-13 of it
  // at either end: widened by 2^-8 of the range they miss nothing
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
  if (FEW && (bytes <= kFewBytes || repeats > few.pairs)) *few.digits = 1;
}

// `digits`, when given, is set if a stable sort of the keys should go by digits.
inline int launch_key_range(const int32_t* keys, int64_t n, int bits, KeyRange* out, uint32_t* digits, cudaStream_t s) {
  if (!digits) {
    key_range_kernel<false><<<1, kRangeThreads, 0, s>>>(keys, n, bits, range_samples(n, 8192), out, FewKeys{});
  } else {
    const int samples = range_samples(n, 32768);
    // Of S samples with q rows per value, S^2 q / 2n pairs are equal; the table sees 2/e of
    // them (the others have a key of the same slot between the two): 12 to 47 at the line, so
    // the count's own spread moves it by less than a third.  (More samples cost more than a
    // sharper line gives: twice as many take 8 to 17 us longer at 9M to 36M rows.)
    const double pairs = kCrowdedRows * 0.7358 * samples * samples / (2.0 * static_cast<double>(n));
    const size_t smem = static_cast<size_t>(samples) * 4;
    if (!allow_smem(key_range_kernel<true>, size_t{32768} * 4)) return CRYS_ECUDA;
    key_range_kernel<true><<<1, kRangeThreads, smem, s>>>(keys, n, bits, samples, out, FewKeys{digits, static_cast<uint32_t>(pairs)});
  }
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
