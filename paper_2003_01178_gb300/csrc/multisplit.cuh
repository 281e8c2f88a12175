// Stable ranking of a warp's rows by an 8-bit digit, shared by the radix sorts.
#pragma once

#include "common.cuh"

namespace crys {

constexpr int kRadix = 256;

// Ranks of a warp's rows among its rows of the same digit, in row order.  Round i holds item i
// of every lane; a lane's rank is (rows of its digit in earlier rounds) + (lanes below it
// with the same digit), rows past the end taking part in no group (FULL: there are none).
// `table` has a (lanes of this round, rows so far) pair per digit, all zero at the start; the
// second words are the warp's digit counts at the end.
//
// The lanes with the same digit are found in turn by eight ballots and by OR-ing the lane's bit
// into the table: the ballots keep the ALU busy (68% of its peak when all rounds use them,
// 123 instructions per row), the table the shared-memory pipe (83%, 78 instructions), and
// alternating them uses both.  2^28 random pairs, whole sort: all ballots 4.91 ms, all table
// 4.94, one round in two 4.74, one in four by either 4.79 and 4.89.  A shared-memory atomic
// per row with a repair of the lanes that share a digit took 5.14 (its repair loop is serial).
template <int ITEMS, bool FULL, typename Digit>
__device__ __forceinline__ void rank_rows(const int32_t (&k)[ITEMS], int lim, const Digit& digit, uint2* table,
                                          uint32_t (&r)[ITEMS]) {
  const uint32_t lane_bit = 1u << (threadIdx.x % kWarp), below = lane_bit - 1u;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const bool real = FULL || i * kWarp < lim;
    if (!FULL && !__any_sync(0xFFFFFFFFu, real)) break;  // no row of the warp in this round or later
    const uint32_t d = real ? digit(k[i]) : 0u;
    const uint32_t entry = smem_u32(table + d);
    uint32_t peers, before = 0;
    if (i % 2 == 0) {
      if (real) atomicOr(&table[d].x, lane_bit);
      __syncwarp();
      asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(peers), "=r"(before) : "r"(entry) : "memory");
      __syncwarp();
      if (real && (peers & below) == 0)
        asm volatile("st.volatile.shared.v2.u32 [%0], {%1, %2};" ::"r"(entry), "r"(0u), "r"(before + __popc(peers))
                     : "memory");
    } else {
      peers = FULL ? 0xFFFFFFFFu : __ballot_sync(0xFFFFFFFFu, real);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const uint32_t bit = (d >> b) & 1u;
        const uint32_t vote = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? vote : ~vote;
      }
      if (real) before = *reinterpret_cast<volatile uint32_t*>(&table[d].y);
      __syncwarp();
      if (real && (peers & below) == 0) *reinterpret_cast<volatile uint32_t*>(&table[d].y) = before + __popc(peers);
    }
    r[i] = (d << 16) | (before + __popc(peers & below));
    __syncwarp();
  }
}

}  // namespace crys
