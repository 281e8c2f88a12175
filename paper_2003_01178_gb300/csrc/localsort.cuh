// Sort of one bucket inside a thread block: the last step of the sorts that first partition
// their rows into buckets by the keys' leading bits (crys_sort_msb, crys_sort).
//
// A bucket of at most kLocalCap rows is sorted in shared memory by ONE counting step and a
// short fix-up.  The block finds the bucket's smallest and largest key, so any bucket works
// whatever bits it was partitioned by, and spreads the keys over up to 8192 bins by the
// leading bits of key - smallest; one shared-memory atomic per row gives its place in its
// bin.  With more bins than rows a bin holds one or two rows, and a row's rank inside its
// bin is found by comparing it with the others there, by (remaining key bits, row), which
// makes the result stable.  When bins are crowded (repeated keys) the block instead runs
// stable 8-bit digit passes, as many as the bucket's key range has bytes.
//
// What bounds it: issue slots (about 60% busy) and about 39 shared-memory wavefronts per 32 rows
// (atomics, the random bin and place accesses), against 24 at HBM speed.  65536 buckets of
// 4096 rows: 1.59 ms (159 instructions per row; 1.79 with branches around every compare); four
// stable 4-bit passes over (low bits, row) words took 3.94 ms.
#pragma once

#include "common.cuh"

namespace crys {

// 3 blocks per SM either way; a sort of 2^28 pairs in 65536 buckets takes 4.21 ms with 384 x 13,
// 4.29 with 512 x 10 or 384 x 14, 4.40 with 256 x 18 (4 blocks), 4.69 with 256 x 20.
constexpr int kLocalThreads = 384;
constexpr int kLocalItems = 13;
constexpr int kLocalCap = kLocalThreads * kLocalItems;  // 4992 rows
constexpr int kLocalBinBits = 13;
constexpr int kLocalBins = 1 << kLocalBinBits;  // two 16-bit counters per word
constexpr int kLocalWarps = kLocalThreads / kWarp;
constexpr int kLocalScan = (kLocalBins / 8 + kLocalThreads - 1) / kLocalThreads;  // 8-bin groups a thread scans
constexpr uint32_t kLocalCrowded = 24;  // rows in one bin above which digit passes are cheaper
static_assert(kLocalCap <= kLocalBins, "a row index takes kLocalBinBits bits");

struct LocalArgs {
  const int32_t* kin;  // rows of the buckets; kin may be kout and vin may be vout
  const int32_t* vin;
  int32_t* kout;
  int32_t* vout;
  const uint32_t* begin;  // first row of each bucket (NULL: one bucket, rows [0, n))
  const uint32_t* count;  // rows of each bucket
  uint32_t n;
  int32_t* err;
  const uint32_t* go = nullptr;    // no work unless *go is set (NULL: always)
  const uint32_t* stop = nullptr;  // no work once *stop is set (NULL: never)
};

struct LocalShared {
  alignas(16) int32_t vals[kLocalCap + 8];  // the bucket's values in row order, shifted by at most 3 words
  alignas(16) uint32_t words[kLocalCap];    // (low key bits, row) by bin; then the sorted keys
  union {
    alignas(16) uint32_t bins[kLocalScan * kLocalThreads * 4 + 4];  // counts, then starts, two per word
    struct {
      uint16_t order[kLocalCap];                  // row of each sorted position
      uint16_t whist[kLocalWarps][256];           // digit passes: per-warp counts, then offsets
    } out;
  };
  uint32_t digit_start[256];
  uint32_t tmp[kLocalWarps + 1];
  int32_t lo[kLocalWarps], hi[kLocalWarps];
  uint64_t loaded;
};

// Block-wide exclusive scan of one value per thread; also returns the total.
__device__ __forceinline__ uint32_t local_scan(uint32_t x, uint32_t* tmp, uint32_t* total) {
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const uint32_t inc = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(x), lane));
  if (lane == kWarp - 1) tmp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < kLocalWarps ? tmp[lane] : 0u;
    const uint32_t wi = static_cast<uint32_t>(warp_inclusive_scan(static_cast<int32_t>(w), lane));
    if (lane < kLocalWarps) tmp[lane] = wi - w;
    if (lane == kLocalWarps - 1) tmp[kLocalWarps] = wi;
  }
  __syncthreads();
  *total = tmp[kLocalWarps];
  return tmp[warp] + inc - x;
}

// Stable position of this thread's rows by the 8-bit digit (v >> shift) & 255.  The rows are
// warp-striped: item i of the thread is row warp * 32 * per + i * 32 + lane, `real` marks
// those that exist.  pos receives each row's position in digit order; on return
// digit_start holds the digits' starts (every thread may read it).
__device__ __forceinline__ void local_rank(LocalShared& sh, const uint32_t (&v)[kLocalItems], uint32_t real, int per,
                                           int shift, uint32_t (&pos)[kLocalItems]) {
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  for (int i = tid; i < kLocalWarps * 256; i += kLocalThreads) (&sh.out.whist[0][0])[i] = 0;
  __syncthreads();
  const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i) {
    if (i >= per) continue;  // the same in every thread
    const bool have = (real >> i) & 1u;
    const uint32_t d = (v[i] >> shift) & 255u;
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, have);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const uint32_t bit = (d >> b) & 1u;
      const uint32_t vote = __ballot_sync(0xFFFFFFFFu, bit);
      peers &= bit ? vote : ~vote;
    }
    const uint32_t before = have ? sh.out.whist[warp][d] : 0u;
    __syncwarp();
    pos[i] = before + __popc(peers & lt_mask);
    if (have && (peers & lt_mask) == 0) sh.out.whist[warp][d] = static_cast<uint16_t>(before + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  uint32_t run = 0;
  if (tid < 256) {
#pragma unroll
    for (int w = 0; w < kLocalWarps; ++w) {
      const uint32_t c = sh.out.whist[w][tid];
      sh.out.whist[w][tid] = static_cast<uint16_t>(run);
      run += c;
    }
  }
  uint32_t total;
  const uint32_t start = local_scan(run, sh.tmp, &total);
  if (tid < 256) sh.digit_start[tid] = start;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i)
    if ((real >> i) & 1u) {
      const uint32_t d = (v[i] >> shift) & 255u;
      pos[i] += sh.digit_start[d] + sh.out.whist[warp][d];
    }
}

// Smallest and largest of one value pair per thread, in every thread.
__device__ __forceinline__ void local_range(LocalShared& sh, int32_t& lo, int32_t& hi) {
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  lo = __reduce_min_sync(0xFFFFFFFFu, lo);
  hi = __reduce_max_sync(0xFFFFFFFFu, hi);
  if (lane == 0) {
    sh.lo[warp] = lo;
    sh.hi[warp] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xFFFFFFFFu, sh.lo[min(lane, kLocalWarps - 1)]);
  hi = __reduce_max_sync(0xFFFFFFFFu, sh.hi[min(lane, kLocalWarps - 1)]);
}

// A bucket of more than kLocalCap rows, through global memory: stable 8-bit digit passes of
// the bytes its key range has, kin -> kout -> kin ..., chunk by chunk with the digit
// positions carried along, and a last copy when the result ends in kin.  Correct for
// every bucket; slow, and only for heavily repeated leading bits.  kin and kout differ.
static __device__ __noinline__ void local_sort_large(const LocalArgs& a, LocalShared& sh, int64_t begin, int64_t size) {
  __shared__ uint32_t digit_base[256];
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  int32_t* bufk[2] = {const_cast<int32_t*>(a.kin) + begin, a.kout + begin};
  int32_t* bufv[2] = {const_cast<int32_t*>(a.vin) + begin, a.vout + begin};
  int32_t lo = INT32_MAX, hi = INT32_MIN;
  for (int64_t i = tid; i < size; i += kLocalThreads) {
    lo = min(lo, bufk[0][i]);
    hi = max(hi, bufk[0][i]);
  }
  local_range(sh, lo, hi);
  const uint32_t span = static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo);
  const int passes = (32 - __clz(span) + 7) / 8;
  for (int pass = 0; pass < passes; ++pass) {
    const int shift = 8 * pass;
    const int32_t *sk = bufk[pass & 1], *sv = bufv[pass & 1];
    int32_t *dk = bufk[(pass + 1) & 1], *dv = bufv[(pass + 1) & 1];
    __syncthreads();
    if (tid < 256) digit_base[tid] = 0;
    __syncthreads();
    for (int64_t i = tid; i < size; i += kLocalThreads)
      atomicAdd(&digit_base[((static_cast<uint32_t>(sk[i]) - static_cast<uint32_t>(lo)) >> shift) & 255u], 1u);
    __syncthreads();
    uint32_t total;
    const uint32_t start = local_scan(tid < 256 ? digit_base[tid] : 0u, sh.tmp, &total);
    if (tid < 256) digit_base[tid] = start;
    for (int64_t c0 = 0; c0 < size; c0 += kLocalCap) {
      const int cnt = static_cast<int>((size - c0) < kLocalCap ? (size - c0) : kLocalCap);
      uint32_t v[kLocalItems], pos[kLocalItems], real = 0;
      int32_t val[kLocalItems];
#pragma unroll
      for (int i = 0; i < kLocalItems; ++i) {
        const int p = warp * (kWarp * kLocalItems) + i * kWarp + lane;
        v[i] = p < cnt ? static_cast<uint32_t>(sk[c0 + p]) - static_cast<uint32_t>(lo) : 0u;
        val[i] = p < cnt ? sv[c0 + p] : 0;
        real |= static_cast<uint32_t>(p < cnt) << i;
      }
      local_rank(sh, v, real, kLocalItems, shift, pos);
      uint32_t counted = 0;  // rows of digit tid in this chunk
      if (tid < 256) counted = (tid < 255 ? sh.digit_start[tid + 1] : static_cast<uint32_t>(cnt)) - sh.digit_start[tid];
#pragma unroll
      for (int i = 0; i < kLocalItems; ++i)
        if ((real >> i) & 1u) {
          const uint32_t d = (v[i] >> shift) & 255u;
          const int64_t g = static_cast<int64_t>(digit_base[d]) + (pos[i] - sh.digit_start[d]);
          dk[g] = static_cast<int32_t>(v[i] + static_cast<uint32_t>(lo));
          dv[g] = val[i];
        }
      __syncthreads();
      if (tid < 256) digit_base[tid] += counted;
      __syncthreads();
    }
    __threadfence_block();
    __syncthreads();
  }
  if (passes % 2 == 0)
    for (int64_t i = tid; i < size; i += kLocalThreads) {
      bufk[1][i] = bufk[0][i];
      bufv[1][i] = bufv[0][i];
    }
}

// A bucket with crowded bins: stable 8-bit digit passes over the `bits` bits of key - lo,
// through words and order.  (A function of its own that reads the keys again, so that the
// usual path keeps its registers.)
static __device__ __noinline__ void local_sort_digits(const LocalArgs& a, LocalShared& sh, uint32_t begin, int cnt, int per,
                                               int32_t lo, int bits) {
  const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
  const int p0 = warp * (kWarp * per) + lane;
  uint32_t v[kLocalItems], row[kLocalItems], at[kLocalItems], real = 0;
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i) {
    const int p = p0 + i * kWarp;
    const bool have = i < per && p < cnt;
    real |= static_cast<uint32_t>(have) << i;
    row[i] = static_cast<uint32_t>(p);
    at[i] = static_cast<uint32_t>(p);  // one key value only: no pass, the rows stay as they are
    v[i] = have ? static_cast<uint32_t>(a.kin[begin + p]) - static_cast<uint32_t>(lo) : 0u;
  }
  for (int shift = 0; shift < max(bits, 1); shift += 8) {
    if (bits > 0) local_rank(sh, v, real, per, shift, at);
    const bool last = shift + 8 >= bits;
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i)
      if ((real >> i) & 1u) {
        sh.words[at[i]] = v[i] + (last ? static_cast<uint32_t>(lo) : 0u);
        sh.out.order[at[i]] = static_cast<uint16_t>(row[i]);
      }
    __syncthreads();
    if (last) break;
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i)
      if ((real >> i) & 1u) {
        v[i] = sh.words[p0 + i * kWarp];
        row[i] = sh.out.order[p0 + i * kWarp];
      }
  }
}

// Sorts rows [begin, begin + size) of one bucket, 1 <= size <= kLocalCap, by the whole block.
// sh.loaded is an initialised barrier whose phases before `parity` are complete.
__device__ __forceinline__ void local_sort_bucket(const LocalArgs& a, LocalShared& sh, uint32_t begin, uint32_t size,
                                                  uint32_t parity) {
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const int cnt = static_cast<int>(size);
  const int per = (cnt + kLocalThreads - 1) / kLocalThreads;  // rows per thread, warp-striped
  // the values travel to shared memory meanwhile: whole 16-byte groups by a bulk copy
  const int32_t* vsrc = a.vin + begin;
  const int skew = static_cast<int>((reinterpret_cast<uintptr_t>(vsrc) & 15u) / 4);
  const int bulk = (cnt + skew) & ~3;  // words copied, from the group that holds the first value
  if (tid == 0) {
    mbar_arrive_expect_tx(&sh.loaded, static_cast<uint32_t>(bulk) * 4u);
    if (bulk) bulk_load(sh.vals, vsrc - skew, static_cast<uint32_t>(bulk) * 4u, &sh.loaded, policy_evict_first());
  }
  const int p0 = warp * (kWarp * per) + lane;
  // item i of this thread is row p0 + 32 i; it exists while 32 i < lim
  const int lim = min(cnt - p0, kWarp * per);
  uint32_t v[kLocalItems], at[kLocalItems];
  const uint32_t some = static_cast<uint32_t>(a.kin[begin]);  // stands in for rows that do not exist
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i) {
    v[i] = some;
    if (i < per && i * kWarp < lim) v[i] = static_cast<uint32_t>(a.kin[begin + p0 + i * kWarp]);
  }
  for (int i = tid; i < kLocalScan * kLocalThreads; i += kLocalThreads)
    reinterpret_cast<uint4*>(sh.bins)[i] = make_uint4(0, 0, 0, 0);
  int32_t lo = static_cast<int32_t>(some), hi = lo;
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i)
    if (i < per) {
      lo = min(lo, static_cast<int32_t>(v[i]));
      hi = max(hi, static_cast<int32_t>(v[i]));
    }
  local_range(sh, lo, hi);  // its barrier also orders the cleared bins and the copy's barrier
  const uint32_t span = static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo);
  const int bits = 32 - __clz(span);
  const int shift = bits > kLocalBinBits ? bits - kLocalBinBits : 0;
#pragma unroll
  for (int i = 0; i < kLocalItems; ++i) {
    if (i >= per) break;
    v[i] -= static_cast<uint32_t>(lo);
    const uint32_t bin = v[i] >> shift, half = 16u * (bin & 1u);
    at[i] = 0;
    if (i * kWarp < lim) at[i] = (atomicAdd(&sh.bins[bin >> 1], 1u << half) >> half) & 0xFFFFu;  // rows of the bin before this one
  }
  __syncthreads();
  // starts of the bins, 13 bits, with the bin's rows above them (7: seven or more): each
  // thread takes consecutive bins
  uint32_t c[4 * kLocalScan], sum = 0, most = 0;
#pragma unroll
  for (int g = 0; g < kLocalScan; ++g) {
    const uint4 q = reinterpret_cast<const uint4*>(sh.bins)[kLocalScan * tid + g];
    c[4 * g] = q.x; c[4 * g + 1] = q.y; c[4 * g + 2] = q.z; c[4 * g + 3] = q.w;
  }
#pragma unroll
  for (int j = 0; j < 4 * kLocalScan; ++j) {
    const uint32_t x = c[j] & 0xFFFFu, y = c[j] >> 16;
    most = max(most, max(x, y));
    c[j] = (sum | (min(x, 7u) << kLocalBinBits)) | (((sum + x) | (min(y, 7u) << kLocalBinBits)) << 16);
    sum += x + y;
  }
  uint32_t total;
  const uint32_t base = local_scan(sum, sh.tmp, &total);
  const uint32_t base2 = base | (base << 16);
#pragma unroll
  for (int g = 0; g < kLocalScan; ++g)
    reinterpret_cast<uint4*>(sh.bins)[kLocalScan * tid + g] =
        make_uint4(c[4 * g] + base2, c[4 * g + 1] + base2, c[4 * g + 2] + base2, c[4 * g + 3] + base2);
  if (kLocalScan * kLocalThreads * 8 == kLocalBins && tid == 0) sh.bins[kLocalBins / 2] = total;  // the last bin's end
  const bool crowded = __syncthreads_or(most > kLocalCrowded) != 0;
  if (!crowded) {
    constexpr uint32_t kStart = kLocalBins - 1u;
    const uint16_t* bins = reinterpret_cast<const uint16_t*>(sh.bins);
    const uint32_t low = (1u << shift) - 1u;
    auto word = [&](int i) { return ((v[i] & low) << kLocalBinBits) | static_cast<uint32_t>(p0 + i * kWarp); };
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i) {
      if (i >= per) break;
      const uint32_t entry = bins[v[i] >> shift];
      if (i * kWarp < lim) sh.words[(entry & kStart) + at[i]] = word(i);
      at[i] |= entry << 8;  // place in the bin (at most kLocalCrowded), start and rows of the bin
    }
    __syncthreads();
    // Rank inside the bin: no other row in 61% of the cases, one in 30%, two in 8% (half a row
    // per bin on average).  The next two rows of the bin, cyclically, are compared without a
    // branch (in a smaller bin they are the row itself), more in a loop.
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i) {
      if (i >= per) break;
      const uint32_t r = at[i] & 255u, s = (at[i] >> 8) & kStart, rows = at[i] >> (8 + kLocalBinBits);
      const uint32_t mine = word(i);
      const uint32_t o1 = r + 1u == rows ? 0u : r + 1u, o2 = o1 + 1u == rows ? 0u : o1 + 1u;
      uint32_t less = static_cast<uint32_t>(sh.words[s + o1] < mine) + static_cast<uint32_t>(sh.words[s + o2] < mine);
      if (rows > 3u) {
        const uint32_t e = (rows < 7u ? s + rows : bins[(v[i] >> shift) + 1] & kStart);
        less = 0;
        for (uint32_t j = s; j < e; ++j) less += sh.words[j] < mine;
      }
      at[i] = s + less;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i) {
      if (i >= per) break;
      if (i * kWarp < lim) {
        sh.words[at[i]] = v[i] + static_cast<uint32_t>(lo);
        sh.out.order[at[i]] = static_cast<uint16_t>(p0 + i * kWarp);
      }
    }
  } else {
    local_sort_digits(a, sh, begin, cnt, per, lo, bits);
  }
  // the last 16-byte group of the values, when the copy did not cover it
  if (tid >= bulk - skew && tid < cnt && bulk <= skew) sh.vals[skew + tid] = vsrc[tid];
  if (bulk > skew && tid < cnt - (bulk - skew)) sh.vals[bulk + tid] = vsrc[bulk - skew + tid];
  const bool ok = mbar_wait_bounded(&sh.loaded, parity, a.err);
  if (__syncthreads_or(!ok)) return;
#pragma unroll 4
  for (int q = tid; q < cnt; q += kLocalThreads) {
    a.kout[begin + q] = static_cast<int32_t>(sh.words[q]);
    a.vout[begin + q] = sh.vals[skew + sh.out.order[q]];
  }
}

// A bucket of more than kLocalCap rows that one cut of its key range divides into two parts that
// fit the block: the rows move from kin to kout, the lower part first, and the parts are sorted
// there.  Any other bucket goes through global memory.  (Not stable; a function of its own,
// so that the usual path keeps its registers.)  The buckets of 327M evenly spread rows hold
// kLocalCap rows on average: 328M rows take 6.96 ms, with all larger buckets through global memory
// 10.95; 400M rows 9.98 and 18.6.
static __device__ __noinline__ void local_sort_split(const LocalArgs& a, LocalShared& sh, uint32_t begin, uint32_t size) {
  __shared__ uint32_t cut, next[2];  // last bin of the lower part; next row of each part
  const int tid = threadIdx.x, lane = tid % kWarp;
  const int32_t *kin = a.kin + begin, *vin = a.vin + begin;
  int32_t lo = INT32_MAX, hi = INT32_MIN;
  for (uint32_t i = tid; i < size; i += kLocalThreads) {
    lo = min(lo, kin[i]);
    hi = max(hi, kin[i]);
  }
  if (tid < 256) sh.digit_start[tid] = 0;
  if (tid == 0) cut = 256;
  local_range(sh, lo, hi);
  const int bits = 32 - __clz(static_cast<uint32_t>(hi) - static_cast<uint32_t>(lo));
  const int shift = bits > 8 ? bits - 8 : 0;
  auto bin = [&](int32_t k) { return (static_cast<uint32_t>(k) - static_cast<uint32_t>(lo)) >> shift; };
  if (size <= 2u * kLocalCap)
    for (uint32_t i = tid; i < size; i += kLocalThreads) atomicAdd(&sh.digit_start[bin(kin[i])], 1u);
  __syncthreads();
  const uint32_t rows = tid < 256 ? sh.digit_start[tid] : 0u;
  uint32_t total;
  const uint32_t upto = local_scan(rows, sh.tmp, &total) + rows;
  if (tid < 256 && upto <= static_cast<uint32_t>(kLocalCap) && upto + kLocalCap >= size) atomicMin(&cut, static_cast<uint32_t>(tid));
  __syncthreads();
  const uint32_t last = cut;
  if (size > 2u * kLocalCap || last == 256u) {
    local_sort_large(a, sh, begin, size);
    return;
  }
  if (static_cast<uint32_t>(tid) == last) {
    next[0] = 0;
    next[1] = upto;
  }
  if (tid == 0) {
    mbar_init(&sh.loaded, 1);
    fence_barrier_init();
  }
  __syncthreads();
  const uint32_t lower = next[1];
  __syncthreads();
  for (uint32_t i0 = 0; i0 < size; i0 += kLocalThreads) {
    const uint32_t i = i0 + tid;
    const int32_t k = i < size ? kin[i] : 0, v = i < size ? vin[i] : 0;
    const uint32_t up = bin(k) > last ? 1u : 0u;
#pragma unroll
    for (uint32_t part = 0; part < 2; ++part) {
      const uint32_t mine = __ballot_sync(0xFFFFFFFFu, i < size && up == part);
      uint32_t at = 0;
      if (lane == 0 && mine) at = atomicAdd(&next[part], static_cast<uint32_t>(__popc(mine)));
      at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(mine & ((1u << lane) - 1u));
      if (i < size && up == part) {
        a.kout[begin + at] = k;
        a.vout[begin + at] = v;
      }
    }
  }
  asm volatile("fence.proxy.async;" ::: "memory");  // the values stored here are read by a bulk copy
  __syncthreads();
  const LocalArgs l{a.kout, a.vout, a.kout, a.vout, nullptr, nullptr, a.n, a.err};
  for (uint32_t part = 0; part < 2; ++part) {
    const uint32_t rows_of = part ? size - lower : lower;
    local_sort_bucket(l, sh, begin + (part ? lower : 0u), rows_of, part);
    fence_proxy_async_smem();  // the other part's values come by a bulk copy into the same place
    __syncthreads();
  }
}

// One block per bucket.  kLarge: buckets above kLocalCap are divided or sorted through global
// memory (needs kin != kout); without it they are reported (CRYS_DEV_BOUNDS) and left alone.
template <bool kLarge>
__global__ void __launch_bounds__(kLocalThreads, 3) local_sort_kernel(const __grid_constant__ LocalArgs a) {
  extern __shared__ __align__(128) unsigned char local_smem[];
  LocalShared& sh = *reinterpret_cast<LocalShared*>(local_smem);
  if ((a.go && *a.go == 0u) || (a.stop && *a.stop != 0u)) return;
  const uint32_t begin = a.begin ? a.begin[blockIdx.x] : 0u;
  const uint32_t size = a.begin ? a.count[blockIdx.x] : a.n;
  if (size == 0) return;
  if (size > static_cast<uint32_t>(kLocalCap)) {
    if (kLarge)
      local_sort_split(a, sh, begin, size);
    else if (threadIdx.x == 0)
      set_error(a.err, CRYS_DEV_BOUNDS);
    return;
  }
  if (threadIdx.x == 0) {
    mbar_init(&sh.loaded, 1);
    fence_barrier_init();
  }
  local_sort_bucket(a, sh, begin, size, 0);
}

// Sorts `buckets` buckets (one block each).
template <bool kLarge>
inline int launch_local_sort(const LocalArgs& a, unsigned buckets, cudaStream_t s) {
  auto k = local_sort_kernel<kLarge>;
  if (!allow_smem(k, sizeof(LocalShared))) return CRYS_ECUDA;
  k<<<buckets, kLocalThreads, sizeof(LocalShared), s>>>(a);
  note_launch();
  return check_launch();
}

}  // namespace crys
