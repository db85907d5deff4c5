// Warp-level ranking shared by the onesweep passes (tj_radix.cu, tj_word.cu) and
// the partition-resident join (tj_fused.cu): stable ranks of a warp's rows by a
// small digit, found with one ballot per digit bit (rank_items), with a
// per-warp table of lane masks for the low 7 bits and one ballot per higher
// bit (rank_items_or), or some rows each way (wrank).
#pragma once

#include <stdint.h>

#include "tj_internal.cuh"

namespace tj {

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Stable ranks of a warp's rows by digit.  Row i*32 + lane of the warp holds
// digit dr[i] (low 16 bits); rows at or beyond nv are padding.  Lanes with the
// same digit are found by one ballot per digit bit; the group's highest lane
// adds the group size to the warp's 16-bit counter of that digit (two per
// word; items in order, so ranks follow row order), and the rank (returned
// base + lanes of the group below this one) goes to the high 16 bits of dr[i].
template <int NB, int ITEMS>
__device__ __forceinline__ void rank_items(uint32_t (&dr)[ITEMS], int nv, uint32_t* wh) {
  const int lane = threadIdx.x & 31;
  const uint32_t ltm = lanemask_lt();
  constexpr int kHalf = ITEMS % 4 == 0 ? 4 : (ITEMS % 3 == 0 ? 3 : (ITEMS % 2 == 0 ? 2 : 1));
#pragma unroll
  for (int i0 = 0; i0 < ITEMS; i0 += kHalf) {
    uint32_t peers[kHalf];
#pragma unroll
    for (int h = 0; h < kHalf; ++h) {
      const bool ok = (i0 + h) * 32 + lane < nv;
      const uint32_t v = __ballot_sync(0xFFFFFFFFu, ok);
      peers[h] = ok ? v : ~v;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
#pragma unroll
      for (int h = 0; h < kHalf; ++h) {
        const int32_t m = (int32_t)(dr[i0 + h] << (31 - b)) >> 31;  // bit b: -1, else 0
        const uint32_t x = __ballot_sync(0xFFFFFFFFu, m != 0);
        peers[h] &= ~(x ^ (uint32_t)m);  // lanes whose bit b equals this lane's
      }
    }
#pragma unroll
    for (int h = 0; h < kHalf; ++h) {
      const int i = i0 + h;
      const bool ok = i * 32 + lane < nv;
      const int leader = 31 - __clz(peers[h]);
      const uint32_t d = dr[i] & 0xFFFFu;
      const uint32_t sh = (d & 1u) * 16u;
      uint32_t base = 0u;
      if (ok && leader == lane)
        base = (atomicAdd(&wh[d >> 1], (uint32_t)__popc(peers[h]) << sh) >> sh) & 0xFFFFu;
      base = __shfl_sync(0xFFFFFFFFu, base, leader);
      dr[i] |= (base + __popc(peers[h] & ltm)) << 16;
    }
  }
}

// Stable ranks as rank_items, with the lanes of each digit found through a
// per-warp table of lane masks in shared memory (wm[min(bins, 128)], zero on
// entry and on exit): every lane ORs its bit into the word of its digit's low
// 7 bits, the warp reads the words back, one ballot per higher digit bit (NH
// of them) drops the lanes that differ above, and each group's highest lane
// clears the word.  One shared atomic and NH ballots per row instead of one
// ballot per digit bit; the tables of all warps must fit the slot-index array.
template <int NH, int ITEMS>
__device__ __forceinline__ void rank_items_or(uint32_t (&dr)[ITEMS], int nv, uint32_t* wh,
                                              uint32_t* wm) {
  const int lane = threadIdx.x & 31;
  const uint32_t ltm = lanemask_lt();
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    if (i * 32 >= nv) break;  // the warp's remaining items are padding
    const bool ok = i * 32 + lane < nv;
    const uint32_t d = dr[i] & 0xFFFFu;
    const uint32_t w = d & 127u;
    if (ok) atomicOr(&wm[w], 1u << lane);
    __syncwarp();
    uint32_t peers = ok ? wm[w] : (1u << lane);
#pragma unroll
    for (int b = 7; b < 7 + NH; ++b) {
      const int32_t m = (int32_t)(d << (31 - b)) >> 31;  // bit b: -1, else 0
      const uint32_t x = __ballot_sync(0xFFFFFFFFu, m != 0);
      peers &= ~(x ^ (uint32_t)m);
    }
    __syncwarp();
    const int leader = 31 - __clz(peers);
    const uint32_t sh = (d & 1u) * 16u;
    uint32_t base = 0u;
    if (ok && leader == lane) {
      wm[w] = 0u;
      base = (atomicAdd(&wh[d >> 1], (uint32_t)__popc(peers) << sh) >> sh) & 0xFFFFu;
    }
    __syncwarp();
    base = __shfl_sync(0xFFFFFFFFu, base, leader);
    dr[i] |= (base + __popc(peers & ltm)) << 16;
  }
}

__device__ __forceinline__ uint32_t lanemask_gt() {
  uint32_t m;
  asm volatile("mov.u32 %0, %%lanemask_gt;" : "=r"(m));
  return m;
}

// 16-bit values, two a register.
template <int N>
struct Half {
  uint32_t v[(N + 1) / 2];
  __device__ __forceinline__ uint32_t get(int i) const {
    return (i & 1) ? v[i >> 1] >> 16 : v[i >> 1] & 0xFFFFu;
  }
  // i in ascending order: the even one sets the register, the odd one adds
  __device__ __forceinline__ void set(int i, uint32_t x) {
    if (i & 1)
      v[i >> 1] |= x << 16;
    else
      v[i >> 1] = x;
  }
  __device__ __forceinline__ void put(int i, uint32_t x) {
    v[i >> 1] = __byte_perm(v[i >> 1], x, (i & 1) ? 0x5410 : 0x3254);
  }
};

// items ranked together by wrank
template <int ITEMS>
__host__ __device__ constexpr int wrank_group() {
  return ITEMS % 4 == 0 ? 4 : (ITEMS % 3 == 0 ? 3 : (ITEMS % 2 == 0 ? 2 : 1));
}

// Stable ranks of a warp's words, item i of the warp being 32 consecutive
// rows with digit(i) (NB bits): rows of the digit earlier in the warp (`cnt`,
// of 16 or 32 bits, and `masks` zero on entry; groups of items at or beyond row
// nv are skipped, rows beyond it in the last group counted).  All
// lanes read the warp's count of their digit and the digit's highest lane
// stores the new one.  The lanes of equal digit are found for MAXM of
// every G items through a table of lane masks by the digit's low 7 bits (each
// lane ORs its bit in, reads the word back, and the group's highest lane
// clears it) with a ballot per higher bit, for the others by a ballot per
// digit bit.  Ballots cost issue slots, the table conflicting shared-memory
// accesses, and each alone bounds the pass: 10^8 words by a 7-bit digit take
// 526 us with ballots only, 527 with the table only, 500 with two of four
// items each way (GB300, 512 threads x 16 words). With 8 and 9 bits three of four
// through the table are 1-2% better than two (sort of 10^8 int64 2.79 -> 2.76 ms,
// 3x10^7 hashed keys 1.36 -> 1.34, join of 10^8 x 4x10^8 under 256 MiB 13.97 -> 13.86).
template <int NB, int ITEMS, int MAXM, typename C, typename D>
__device__ __forceinline__ void wrank(const D& digit, Half<ITEMS>& rank, C* cnt, uint32_t* masks,
                                      int nv = 32 * ITEMS) {
  const uint32_t bit = 1u << (threadIdx.x & 31), ltm = lanemask_lt(), gtm = lanemask_gt();
  constexpr int G = wrank_group<ITEMS>();
  constexpr int MX = MAXM < G ? MAXM : G;
#pragma unroll
  for (int i0 = 0; i0 < ITEMS; i0 += G) {
    if (nv < 32 * ITEMS && i0 * 32 >= nv) break;
    uint32_t d[G], peers[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
      d[h] = digit(i0 + h);
      peers[h] = 0xFFFFFFFFu;
    }
#pragma unroll
    for (int h = 0; h < MX; ++h) atomicOr(&masks[h * 128 + (d[h] & 127u)], bit);
    __syncwarp();
#pragma unroll
    for (int h = 0; h < MX; ++h) peers[h] = masks[h * 128 + (d[h] & 127u)];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
#pragma unroll
      for (int h = 0; h < G; ++h) {
        if (h < MX && b < 7) continue;
        const bool p = (d[h] & (1u << b)) != 0u;
        const uint32_t x = __ballot_sync(0xFFFFFFFFu, p);
        peers[h] &= p ? x : ~x;  // lanes whose bit b equals this lane's
      }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < MX; ++h)
      if ((peers[h] & gtm) == 0u) masks[h * 128 + (d[h] & 127u)] = 0u;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < G; ++h) {
      C* c = cnt + d[h];
      const uint32_t base = *c;
      __syncwarp();
      if ((peers[h] & gtm) == 0u) *c = (C)(base + __popc(peers[h]));
      rank.set(i0 + h, base + __popc(peers[h] & ltm));
      __syncwarp();
    }
  }
}

// Decoupled look-back over one 64-bit word a tile (STRIDE words apart), by one
// warp: the sum of the words before tile t back to the first inclusive one. Each
// round trip reads the 32 WORDS newest predecessors not yet summed and sums the run of
// ready words; the sum of 62-bit words is three sums of 21 bits (redux), shorter
// than ten shuffles in a wait that every later tile inherits. Bounded wait:
// *err = TJ_ERR_TIMEOUT.
template <int STRIDE, int WORDS>
__device__ __forceinline__ uint64_t chain_prefix(const uint64_t* words, int64_t t, int* err) {
  const int lane = threadIdx.x & 31;
  uint64_t prefix = 0;
  int64_t k = t - 1;  // newest predecessor not yet summed
  int spins = 0;
  bool done = t == 0;
  while (!done) {
    uint64_t v[WORDS];
#pragma unroll
    for (int q = 0; q < WORDS; ++q) {
      const int64_t i = k - 32 * q - lane;
      v[q] = kFlagInc64;
      if (i >= 0)
        asm volatile("ld.volatile.global.u64 %0, [%1];"
                     : "=l"(v[q])
                     : "l"(words + i * STRIDE)
                     : "memory");
    }
    uint64_t x = 0;
    int take = 0;  // words summed
#pragma unroll
    for (int q = 0; q < WORDS; ++q) {
      if (done || take != 32 * q) break;
      const uint64_t f = v[q] & ~kValMask64;
      const uint32_t notready = __ballot_sync(0xFFFFFFFFu, f == 0ull);
      const uint32_t inc = __ballot_sync(0xFFFFFFFFu, f == kFlagInc64);
      const int first_nr = notready ? __ffs(notready) - 1 : 32;
      const int first_inc = inc ? __ffs(inc) - 1 : 32;
      done = first_inc < first_nr;
      const int n = done ? first_inc + 1 : first_nr;  // lanes summed
      if (lane < n) x += v[q] & kValMask64;
      take += n;
    }
    const uint32_t s0 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)x & 0x1FFFFFu);
    const uint32_t s1 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(x >> 21) & 0x1FFFFFu);
    const uint32_t s2 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(x >> 42));
    prefix += (uint64_t)s0 + ((uint64_t)s1 << 21) + ((uint64_t)s2 << 42);
    k -= take;
    if (take != 0) {
      spins = 0;
    } else {
      if (++spins > kSpinLimit) {
        if (lane == 0) atomicExch(err, (int)TJ_ERR_TIMEOUT);
        break;
      }
      __nanosleep(32);
    }
  }
  return prefix;
}

}  // namespace tj
