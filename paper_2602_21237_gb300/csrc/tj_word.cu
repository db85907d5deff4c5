// Radix passes over folded rows: the tensor-path sort (paper Sec. 4.2) and the
// route / MSD passes of the join, on rows of one 64-bit word.
//
// A row (key, id) whose key offset and id fit 64 bits together is one word,
//   w = (key - wlo) << ib | (id - ilo),
// made by the first pass as it reads the caller's columns and taken apart
// again only where ids (or keys) are written.  Against separate key and id
// arrays every pass in between moves 8 bytes a row instead of 16 (64-bit
// rows), and a row is one load, one shared-memory slot and one store instead
// of two of each plus an index.
//
// Rows too wide for one word (64-bit keys whose range and ids need more than 64
// bits) travel as "wide" rows, the key as it is beside a 32-bit id, when their
// ids' range fits 32 bits.
//
// The ids' range is a sample's.  The few ids outside it (a sentinel in some rows, say)
// fold as codes, which have the id's top bit, their values go to a table beside the
// words, and one pass over the result puts them back (k_far_ids).
//
// k_wsweep is one onesweep pass (decoupled look-back, as k_onesweep in
// tj_radix.cu) over a tile of kWThreads * ITEMS rows: take the digits, rank
// them inside the warp, move the words to their tile-sorted slots in shared
// memory, write the slots out in order.
#include <algorithm>
#include <type_traits>

#include "tj_internal.cuh"
#include "tj_warp.cuh"

namespace tj {

namespace {

__device__ __forceinline__ uint32_t wld_volatile(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void wst_volatile(uint32_t* p, uint32_t v) {
  asm volatile("st.volatile.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
template <typename Job>
__device__ __forceinline__ int find_job_w(const Job* jobs, int num_jobs, int64_t t) {
  int lo = 0, hi = num_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].tile0 <= t)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Digit of a word: bits [shift, shift + n) of w - lo.  HI: shift >= 32 and lo
// is a multiple of 2^32 (keys of at most 32 bits sit in the word's upper
// half), so one 32-bit subtract and shift give it.
template <bool HI>
__device__ __forceinline__ uint32_t wdigit(uint64_t w, uint64_t lo, int shift, uint32_t mask) {
  if (HI) return (((uint32_t)(w >> 32) - (uint32_t)(lo >> 32)) >> (shift & 31)) & mask;
  return (uint32_t)((w - lo) >> shift) & mask;
}

// Batch of a word under equal-width ranges: (clamp(key) - lo) >> shift, all
// as offsets from the words' first key (rlo: the range's first key, span: its
// width).  HI as above: the key offset lies in the upper 32 bits.
template <bool HI>
__device__ __forceinline__ uint32_t wroute_radix(uint64_t w, int ib, uint64_t rlo, uint64_t span,
                                                 int shift) {
  if (HI) {
    const uint32_t x = (uint32_t)(w >> 32) >> (ib & 31), l = (uint32_t)rlo;
    const uint32_t y = x < l ? 0u : min(x - l, (uint32_t)span);
    return y >> shift;
  }
  const uint64_t x = w >> ib;
  uint64_t y = x < rlo ? 0ull : x - rlo;
  y = y < span ? y : span;
  return (uint32_t)(y >> shift);
}

// Batch of a word under the cut table: the number of cuts <= key (offsets from
// the words' first key), through the radix index over the cuts (the same
// number of halvings on every lane; see RadixJob::route_tab).
__device__ __forceinline__ uint32_t wroute_cuts(uint64_t w, int ib, uint64_t rlo,
                                                const uint64_t* s_cuts, const uint16_t* s_tab,
                                                int steps, int ushift) {
  const uint64_t key = w >> ib;
  const uint64_t x = key < rlo ? 0ull : key - rlo;
  uint32_t b;
  if (ushift >= 0) {
    const uint64_t u = x >> ushift;
    b = u < (uint64_t)(kRouteBuckets - 1) ? (uint32_t)u : (uint32_t)(kRouteBuckets - 1);
  } else {
    const int nb = 64 - __clzll((long long)x);
    b = nb < 6 ? (uint32_t)x : (uint32_t)((nb << 5) | ((x >> (nb - 6)) & 31ull));
  }
  int a = s_tab[b];
  int n = (int)s_tab[b + 1] - a;
  for (int i = 0; i < steps; ++i) {
    const int half = n >> 1;
    const bool go = n > 0 && s_cuts[a + half] <= key;
    a = go ? a + half + 1 : a;
    n = go ? n - half - 1 : half;
  }
  return (uint32_t)a;
}

// Per-warp ranking tables of a pass: digit counts, lane masks.
__host__ __device__ constexpr size_t wtable_bytes(int nbits) {
  return (size_t)kWWarps * 4u * (((size_t)1 << (nbits < 2 ? 2 : nbits)) + 128u * kWMaskItems);
}

// Shared memory: the tile's words in tile-sorted order, overlaid with the
// ranking tables (dead before the words move; wide rows: keys, then ids) |
// global base and tile
// count per digit | end of each batch's region (guarded route passes) | cut
// keys, radix index and slot digits (route passes by the cut table).
template <int ITEMS>
__host__ __device__ constexpr size_t wsweep_smem_bytes(int nbits, int mode, bool guard, bool wide) {
  const size_t stage = (wide ? 12u : 8u) * (size_t)kWThreads * ITEMS;
  const size_t bins = (size_t)1 << nbits;
  return (stage > wtable_bytes(nbits) ? stage : wtable_bytes(nbits)) + 8u * bins +
         (mode != kModeSort && guard ? 4u * bins : 0u) +
         (mode == kModeCuts ? 8u * bins + 2u * (kRouteBuckets + 8) +
                                  (size_t)(nbits <= 8 ? 1 : 2) * kWThreads * ITEMS
                            : 0u);
}

template <int ITEMS, typename D>
__device__ __forceinline__ void wrank_bits(const D& digit, int nbits, Half<ITEMS>& rank,
                                           uint32_t* cnt, uint32_t* masks) {
  switch (nbits) {
    case 0:  // one digit value
    case 1: wrank<1, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 2: wrank<2, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 3: wrank<3, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 4: wrank<4, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 5: wrank<5, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 6: wrank<6, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 7: wrank<7, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 8: wrank<8, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    case 9: wrank<9, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
    default: wrank<10, ITEMS, kWMaskItems>(digit, rank, cnt, masks); break;
  }
}

// Sum look-back words (newest predecessor first) into `prefix` up to the first
// inclusive one, stopping at one not published yet; returns the words used.
template <int W>
__device__ __forceinline__ int wlookback(const uint32_t (&v)[W], uint32_t& prefix, bool& done) {
  int used = 0;
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    if (used != k) break;
    const uint32_t f = v[k] & ~kValMask;
    if (f == 0u) break;
    acc += v[k] & kValMask;
    ++used;
    if (f == kFlagInc) {
      done = true;
      break;
    }
  }
  prefix += acc;
  return used;
}

}  // namespace

// One pass over a tile of kWThreads * ITEMS rows:
//   1. digits, 16 bits a row in registers (from the key column, or the words'
//      upper halves when the key is there), and stable ranks inside each warp;
//   2. per digit: sum over the warps, publish to the look-back chain, scan;
//   3. the rows are read again, from L2 (RAW_IN: keys and ids, folded; far ids get
//      a code; a row whose key offset does not fit, or one far id too many, sets
//      *err = kErrFold), and move to
//      their tile-sorted slots in shared memory, after the digits' threads have
//      finished the look-back (bounded wait);
//   4. slots in order -> global: each digit's run lands contiguously (RAW_OUT:
//      as key and id columns).
// Reading a row twice, L2's bandwidth being idle, keeps only its digit and rank
// in registers while the tile is ranked. Holding the words there spilled at
// 512 threads x 16 rows, two CTAs a multiprocessor (64 registers), above all
// where columns are folded: 5x10^8 rows by an 8-bit batch digit took 4.44 ms,
// now 3.08 ms (12 GB); 10^8 words take 491 / 535 / 594 us by 7 / 8 / 9 bits
// against 500 / 538 / 618. What bounds the pass is the ranking (see wrank):
// without it and the look-back the same tiles move at the copy rate.
// Rows beyond the tile's end carry the largest digit, so they rank last and
// need no test before step 4.
// MODE: kModeSort (a digit of w - lo), kModeRadix or kModeCuts (route passes:
// the batch under equal-width ranges or the cut table).  HI: see wdigit.
// After a row failed to fold, the folding pass's other tiles and the later passes
// return at once: a RAW_OUT pass never overwrites the caller's columns with such rows,
// and a join whose one far key the sample of its key range missed loses half of the
// route pass on average, not all of it (far key in the middle of S, 10^8 x 4x10^8 rows
// under 256 MiB: 22.6 ms, now 21.5; columns from the start 18.8).
// WIDE: rows are a key and a 32-bit id (src / dst columns of 8 and 4 bytes; a
// pass after the first reads the ids where the one before wrote them).
template <typename K, bool RAW_IN, bool RAW_OUT, int MODE, bool HI, bool WIDE, int ITEMS>
__global__ void __launch_bounds__(kWThreads, kWMinB)
    k_wsweep(const RadixJob<K>* __restrict__ jobs, int num_jobs, int64_t total_tiles, int pass,
             uint32_t* __restrict__ tile_counter, int* __restrict__ err,
             const int32_t* __restrict__ tile_job) {
  using U = typename UnsignedOf<K>::type;
  constexpr int TILE = kWThreads * ITEMS;
  static_assert(TILE <= 65536, "16-bit positions within a tile");
  static_assert(!WIDE || (sizeof(K) == 8 && !HI && MODE == kModeSort), "wide rows: 64-bit sorts");
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_warp[kWWarps];
  __shared__ uint32_t s_t;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    // (only passes that fold set kErrFold, so all tiles of another pass agree; a tile
    // of a folding pass that waits for one which stopped here goes on without it)
    const bool stop =
        wld_volatile(reinterpret_cast<const uint32_t*>(err)) == (uint32_t)kErrFold;
    const uint32_t ticket = atomicAdd(tile_counter, 1u);
    s_t = stop ? 0xFFFFFFFFu : ticket;
  }
  __syncthreads();
  const int64_t t = s_t;
  if (t >= total_tiles) return;
  const int j = tile_job ? tile_job[t] : find_job_w(jobs, num_jobs, t);
  const RadixJob<K>* J = jobs + j;
  if (pass >= J->passes) return;
  // tiles of a job are numbered in 32 bits (n < 2^30 rows)
  const int lt = (int)(t - J->tile0);
  const int64_t row0 = (int64_t)lt * TILE;
  const int nvalid = (int)min((int64_t)TILE, J->n - row0);
  const int shift = J->shift[pass], nbits = J->bits[pass];
  const int bins = 1 << nbits;
  const uint32_t mask = (uint32_t)bins - 1u;
  const uint64_t lo = J->lo;
  const int ib = J->ib;
  const uint64_t idm = (1ull << ib) - 1ull;

  uint64_t* const stage = reinterpret_cast<uint64_t*>(smem);
  const size_t tab_bytes = wtable_bytes(nbits);
  constexpr size_t kStage = (WIDE ? 12u : 8u) * (size_t)TILE;
  const size_t area = kStage > tab_bytes ? kStage : tab_bytes;
  uint32_t* const stage_v = reinterpret_cast<uint32_t*>(smem + 8u * (size_t)TILE);  // WIDE
  uint32_t* const s_gbase = reinterpret_cast<uint32_t*>(smem + area);
  uint32_t* const s_cnt = s_gbase + bins;
  uint32_t* const s_rend = s_cnt + bins;
  const bool guard = MODE != kModeSort && J->route_end != nullptr;
  uint64_t* const s_cuts =
      reinterpret_cast<uint64_t*>(smem + area + 8u * bins + (guard ? 4u * bins : 0u));
  uint16_t* const s_tab = reinterpret_cast<uint16_t*>(s_cuts + bins);
  uint16_t* const s_dig = s_tab + (kRouteBuckets + 8);
  uint8_t* const s_dig8 = reinterpret_cast<uint8_t*>(s_dig);
  const bool dig8 = nbits <= 8;
  const uint64_t span = J->route_hi;  // route passes: the range's width
  const int rsteps = J->route_steps, rshift = J->route_shift;

  auto digit = [&](uint64_t w) -> uint32_t {
    if (MODE == kModeRadix) return wroute_radix<HI>(w, ib, lo, span, shift);
    if (MODE == kModeCuts) return wroute_cuts(w, ib, lo, s_cuts, s_tab, rsteps, rshift);
    return wdigit<HI>(w, lo, shift, mask);
  };

  // 1. digits.  A row past the end takes the largest digit any row can have.
  const int wbase = warp * 32 * ITEMS + lane;
  const uint64_t pad = MODE == kModeCuts ? ~0ull
                       : MODE == kModeRadix ? (lo + span) << ib
                                            : lo + ((uint64_t)mask << shift);
  const uint64_t* __restrict__ wp = reinterpret_cast<const uint64_t*>(J->src_k[pass]) + row0;
  const K* __restrict__ kp = J->src_k[pass] + row0;
  using Part = typename std::conditional<RAW_IN, K,
                                         typename std::conditional<HI, uint32_t, uint64_t>::type>::type;
  Part part[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int r = wbase + i * 32;
    if constexpr (RAW_IN)
      part[i] = r < nvalid ? kp[r] : K(0);
    else if constexpr (HI)
      part[i] = r < nvalid ? reinterpret_cast<const uint32_t*>(wp)[2 * r + 1] : (uint32_t)(pad >> 32);
    else
      part[i] = r < nvalid ? wp[r] : pad;
  }
  {
    uint4* z = reinterpret_cast<uint4*>(smem);
    for (int i = tid; i < (int)(tab_bytes / 16); i += kWThreads) z[i] = make_uint4(0, 0, 0, 0);
  }
  if (MODE == kModeCuts) {
    const uint64_t* __restrict__ cuts = reinterpret_cast<const uint64_t*>(J->cuts);
    for (int i = tid; i < bins; i += kWThreads) s_cuts[i] = cuts[i];
    for (int i = tid; i <= kRouteBuckets; i += kWThreads) s_tab[i] = J->route_tab[i];
  }
  if (guard)
    for (int i = tid; i < bins; i += kWThreads) s_rend[i] = J->route_end[i];
  __syncthreads();
  Half<ITEMS> dig, rank;
  {
    const U wlo = (U)J->wlo;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      uint64_t x;
      if constexpr (RAW_IN && WIDE)
        x = wbase + i * 32 < nvalid ? (uint64_t)part[i] : pad;
      else if constexpr (RAW_IN)
        x = wbase + i * 32 < nvalid ? (uint64_t)(U)((U)part[i] - wlo) << ib : pad;
      else if constexpr (HI)
        x = (uint64_t)part[i] << 32;
      else
        x = part[i];
      dig.set(i, digit(x));
    }
  }
  auto item_digit = [&](int i) -> uint32_t { return dig.get(i); };
  uint32_t* const t_cnt = reinterpret_cast<uint32_t*>(smem);  // [warp][digit]
  uint32_t* const t_mask = t_cnt + kWWarps * bins;
  wrank_bits<ITEMS>(item_digit, nbits, rank, t_cnt + warp * bins,
                    t_mask + warp * 128 * kWMaskItems);
  __syncthreads();

  // 2. per digit (`per` consecutive ones a thread): the tile's count,
  //    published, and its exclusive prefix over (digit, warp), left in the
  //    tables
  const int per = (bins + kWThreads - 1) / kWThreads;
  const int d0 = tid * per, d1 = min(bins, d0 + per);
  uint32_t sum = 0;
  {
    const uint32_t npad = (uint32_t)(TILE - nvalid);
    uint32_t* const lb_mine = J->lookback + pass * J->lb_stride + (int64_t)lt * bins;
    // (by the cut table not always the last batch: a cut after the largest key of a
    // range of 2^k keys lies past every key that folds)
    const uint32_t dpad = npad ? digit(pad) : ~0u;
#pragma unroll 1
    for (int d = d0; d < d1; ++d) {
      uint32_t c = 0;
#pragma unroll
      for (int q = 0; q < kWWarps; ++q) c += t_cnt[q * bins + d];
      sum += c;
      s_gbase[d] = c;
      if ((uint32_t)d == dpad) c -= npad;
      s_cnt[d] = c;
      wst_volatile(lb_mine + d, (lt == 0 ? kFlagInc : kFlagAgg) | c);
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t run = x - sum;
#pragma unroll
    for (int q = 0; q < kWWarps; ++q)
      if (q < warp) run += s_warp[q];
#pragma unroll 1
    for (int d = d0; d < d1; ++d) {
      const uint32_t c = s_gbase[d];
      s_gbase[d] = run;
      uint32_t p = run;
#pragma unroll
      for (int q = 0; q < kWWarps; ++q) {
        const uint32_t v = t_cnt[q * bins + d];
        t_cnt[q * bins + d] = p;
        p += v;
      }
      run += c;
    }
  }
  __syncthreads();

  // 3. positions (the tables die here), the look-back, the move
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    rank.put(i, rank.get(i) + t_cnt[warp * bins + item_digit(i)]);
  __syncthreads();
  const uint32_t* __restrict__ hist = J->hist + pass * J->hist_stride;
  uint32_t* const lb_base = J->lookback + pass * J->lb_stride;
#pragma unroll 1
  for (int d = d0; d < d1; ++d) {
    uint32_t prefix = 0;
    if (lt > 0) {
      int k = lt - 1;  // newest predecessor not yet summed
      bool done = false;
      int spins = 0;
      while (!done) {
        uint32_t v[kLookWide];
#pragma unroll
        for (int q = 0; q < kLookWide; ++q)
          v[q] = (k - q >= 0) ? wld_volatile(lb_base + (int64_t)(k - q) * bins + d) : kFlagInc;
        const int used = wlookback<kLookWide>(v, prefix, done);
        k -= used;
        if (used == 0) {
          // (the sum so far is too small, if anything: rows stay in their digit's place)
          if (RAW_IN && sizeof(K) == 8 &&
              wld_volatile(reinterpret_cast<const uint32_t*>(err)) == (uint32_t)kErrFold)
            break;
          if (++spins > kSpinLimit) {
            atomicExch(err, (int)TJ_ERR_TIMEOUT);
            break;
          }
          __nanosleep(32);
        }
      }
      wst_volatile(lb_base + (int64_t)lt * bins + d, kFlagInc | ((prefix + s_cnt[d]) & kValMask));
    }
    s_gbase[d] = hist[d] + prefix - s_gbase[d];  // minus the digit's first slot
  }
  {
    const K* __restrict__ vp = RAW_IN ? J->fold_v + row0 : nullptr;
    const U wlo = (U)J->wlo, ilo = (U)J->ilo;
    // bits that no row of a group should have: far ids, keys that do not fit (a later
    // pass that folds meets far ids' codes, which are ids of the window to it)
    uint64_t out = 0;
    constexpr bool kCheck = RAW_IN && sizeof(K) == 8;
    const int cb = kCheck && pass == 0 ? J->cb : ib;
    const uint32_t code_bit = WIDE && cb < 32 ? 1u << cb : 0u;  // (cb is 31 or 32)
    uint32_t wide_out = 0;
    bool misfit = false;  // a key that does not fit, or a far id too many
    // (pairs of 64-bit columns: half of the rows at a time, wide ones a quarter, to
    // spare registers)
    constexpr int G = RAW_IN && WIDE                        ? ITEMS / 4
                      : (RAW_IN && sizeof(K) == 8) || WIDE ? ITEMS / 2
                                                            : ITEMS;
    static_assert(ITEMS % G == 0, "whole groups");
    const uint32_t* __restrict__ ip =
        WIDE && !RAW_IN ? reinterpret_cast<const uint32_t*>(J->dst_v[pass - 1]) + row0 : nullptr;
#pragma unroll
    for (int i0 = 0; i0 < ITEMS; i0 += G) {
      uint64_t w[G];
      uint32_t id[WIDE ? G : 1];
      if constexpr (RAW_IN && WIDE) {
        K v[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int r = wbase + (i0 + i) * 32;
          w[i] = r < nvalid ? (uint64_t)kp[r] : 0ull;
          v[i] = r < nvalid ? vp[r] : (K)ilo;
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const uint64_t io = (uint64_t)(U)((U)v[i] - ilo);
          id[i] = (uint32_t)io;
          wide_out |= (uint32_t)(io >> 32) | (id[i] & code_bit);
        }
      } else if constexpr (RAW_IN) {
        K v[G], k[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int r = wbase + (i0 + i) * 32;
          k[i] = r < nvalid ? kp[r] : K(0);
          v[i] = r < nvalid ? vp[r] : K(0);
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const uint64_t ko = (uint64_t)(U)((U)k[i] - wlo), io = (uint64_t)(U)((U)v[i] - ilo);
          if (kCheck && wbase + (i0 + i) * 32 < nvalid) out |= (io >> cb) | (ko >> (64 - ib));
          w[i] = (ko << ib) | (io & idm);
        }
      } else {
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int r = wbase + (i0 + i) * 32;
          w[i] = r < nvalid ? wp[r] : 0ull;
          if constexpr (WIDE) id[i] = r < nvalid ? ip[r] : 0u;
        }
      }
      if (kCheck && (WIDE ? wide_out != 0u : out != 0ull)) {
        // which rows: far ids get a code (here, before the rows move, it needs no
        // register beyond the group's; after all groups it held their ranks, and wide
        // folding passes took 2% more)
#pragma unroll 1
        for (int i = 0; i < G && !misfit; ++i) {
          const int r = wbase + (i0 + i) * 32;
          if (r >= nvalid) break;
          const K v = vp[r];
          if (!WIDE) misfit = ((uint64_t)(U)((U)kp[r] - wlo) >> (64 - ib)) != 0ull;
          if (((uint64_t)(U)((U)v - ilo) >> cb) == 0ull) continue;
          const uint32_t k = cb < ib ? atomicAdd(J->far_n, 1u) : (uint32_t)kFarIds;
          misfit |= k >= (uint32_t)kFarIds;
          if (misfit) break;
          J->far_ids[k] = (uint64_t)v;
#pragma unroll
          for (int q = 0; q < G; ++q)
            if (q == i) {
              if constexpr (WIDE) id[q] = (1u << cb) + k;
              else w[q] = (w[q] & ~idm) | ((1ull << cb) + k);
            }
        }
        out = 0;
        wide_out = 0;
      }
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const uint32_t pos = rank.get(i0 + i);
        stage[pos] = w[i];
        if constexpr (WIDE) stage_v[pos] = id[i];
        if (MODE == kModeCuts) {
          if (dig8)
            s_dig8[pos] = (uint8_t)dig.get(i0 + i);
          else
            s_dig[pos] = (uint16_t)dig.get(i0 + i);
        }
      }
    }
    if (misfit && wld_volatile(reinterpret_cast<const uint32_t*>(err)) == 0u)
      atomicCAS(err, 0, kErrFold);
  }
  __syncthreads();

  // 4. slots in order -> global
  uint64_t* __restrict__ dst_w = reinterpret_cast<uint64_t*>(J->dst_k[pass]);
  K* __restrict__ dst_k = J->dst_k[pass];
  K* __restrict__ dst_v = J->dst_v[pass];
  const U wlo = (U)J->wlo, ilo = (U)J->ilo;
  const uint32_t room = RAW_IN ? (uint32_t)J->dst_rows : 0u;
  bool over = false;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int q = tid + it * kWThreads;
    if (q < nvalid) {
      const uint64_t x = stage[q];
      const uint32_t d = MODE == kModeCuts ? (dig8 ? (uint32_t)s_dig8[q] : (uint32_t)s_dig[q])
                                           : digit(x);
      const uint32_t g = s_gbase[d] + (uint32_t)q;
      if constexpr (RAW_OUT && WIDE) {
        dst_k[g] = (K)x;
        dst_v[g] = (K)((U)stage_v[q] + ilo);
      } else if constexpr (RAW_OUT) {
        dst_k[g] = (K)((U)(x >> ib) + wlo);
        dst_v[g] = (K)((U)(x & idm) + ilo);
      } else {
        // batch regions sized in advance: a row past its region's end is
        // dropped and reported (the caller then routes again); rows that did
        // not fold may miscount, so a folding pass keeps to its destination
        const bool in = MODE != kModeSort && guard ? g < s_rend[d] : !RAW_IN || g < room;
        over |= !in;
        if (in) {
          dst_w[g] = x;
          if constexpr (WIDE) reinterpret_cast<uint32_t*>(dst_v)[g] = stage_v[q];
        }
      }
    }
  }
  if (MODE != kModeSort && over) atomicCAS(err, 0, (int)TJ_ERR_CAPACITY);
}

// ---------------------------------------------------------------------------
// Nearly unique keys: a sort by the leading bits, then the runs put right
// ---------------------------------------------------------------------------
// Wide keys of few duplicates are told apart by far fewer bits than they have:
// n keys spread over their range share a 27-bit prefix with n / 2^27 others on
// average. Sorting by three digits of the prefix leaves short runs of rows with
// equal prefixes, in input order; k_runs ranks each run by the whole key and
// writes the columns. 3x10^7 hashed 64-bit keys:
// eight passes of 240 us were 2.38 ms in all, three of 262 us and k_runs (183 us,
// 0.84 GB) are 1.35 ms.
//
// k_prefix_sample decides from the statistics and a sample whether that will
// do: *pairs = the number of pairs of equal prefixes among SAMPLE rows.
// Prefixes that n rows share evenly among D values give SAMPLE^2 / 2 D.
template <int SAMPLE>
__host__ __device__ constexpr size_t sample_smem_bytes() {
  return 2 * SAMPLE * (sizeof(unsigned long long) + sizeof(uint32_t));
}
template <int SAMPLE>
__global__ void __launch_bounds__(1024)
    k_prefix_sample(const int64_t* __restrict__ keys, int64_t n,
                    const KeyStats* __restrict__ stats, int prefix_bits, int min_bits,
                    uint32_t* __restrict__ pairs) {
  constexpr int kSlots = 2 * SAMPLE;
  constexpr unsigned long long kNone = ~0ull;  // (prefixes have at most 32 bits)
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long* const s_key = reinterpret_cast<unsigned long long*>(smem);
  uint32_t* const s_cnt = reinterpret_cast<uint32_t*>(s_key + kSlots);
  const unsigned long long lo = stats->min_u, range = ~stats->max_u - lo;
  const int kb = 64 - __clzll((long long)range);
  if (kb < min_bits) return;
  for (int i = threadIdx.x; i < kSlots; i += blockDim.x) {
    s_key[i] = kNone;
    s_cnt[i] = 0u;
  }
  __syncthreads();
  const int64_t step = n / SAMPLE;
#pragma unroll
  for (int u = 0; u < SAMPLE / 1024; ++u) {
    const uint32_t i = threadIdx.x + u * 1024;
    // one row of every stretch of `step`, not always the same one
    const int64_t r = i * step + (int64_t)((i * 0x9E3779B97F4A7C15ull >> 33) % (uint64_t)step);
    const unsigned long long k = (unsigned long long)keys[r] ^ 0x8000000000000000ull;
    const unsigned long long p = (k - lo) >> (kb - prefix_bits);
    uint32_t h = (uint32_t)((p * 0x9E3779B97F4A7C15ull) >> 40) & (kSlots - 1);
    while (true) {
      const unsigned long long old = atomicCAS(&s_key[h], kNone, p);
      if (old == kNone || old == p) break;
      h = (h + 1) & (kSlots - 1);
    }
    const uint32_t before = atomicAdd(&s_cnt[h], 1u);
    if (before) atomicAdd(pairs, before);
  }
}

// Rows sorted stably by key >> s -> key and id columns sorted by key. A tile's
// keys and kRunMax rows on either side come to shared memory; a row finds the
// ends of its run (rows of the same prefix) and counts the run's rows that come
// before it. A run of more than kRunMax rows is left as it is, which is right
// when its keys are in order already (one repeated key, say), and its ends are listed;
// where one is not, *err = kErrRuns and the caller sorts the listed runs by themselves.
// fix = false only writes the rows out as columns, in the order they have.
// WIDE: keys as they are and ids as 32-bit offsets; otherwise folded rows.
template <bool WIDE>
__global__ void __launch_bounds__(kRunThreads)
    k_runs(const uint64_t* __restrict__ rows, const uint32_t* __restrict__ ids, int64_t n, Fold f,
           int s, bool fix, int64_t* __restrict__ out_k, int64_t* __restrict__ out_v,
           uint32_t* __restrict__ runs, uint32_t* __restrict__ runs_n, int* __restrict__ err) {
  constexpr int kSpan = kRunTile + 2 * kRunMax;
  __shared__ uint64_t s_row[kSpan];
  const int tid = threadIdx.x;
  if (*reinterpret_cast<volatile int*>(err) == kErrFold) return;  // (nothing was sorted)
  const int64_t t0 = (int64_t)blockIdx.x * kRunTile;
  const int64_t b0 = max((int64_t)0, t0 - kRunMax);
  const int m = (int)(min(n, t0 + kRunTile + kRunMax) - b0);  // rows on chip
  const int i0 = (int)(t0 - b0);                              // the tile's first
  const int i1 = (int)min((int64_t)m, i0 + (int64_t)kRunTile);
  const uint64_t* __restrict__ src = rows + b0;
#pragma unroll
  for (int u = 0; u < kSpan / kRunThreads; ++u) {
    const int i = tid + u * kRunThreads;
    if (i < m) s_row[i] = src[i];
  }
  __syncthreads();
  // what rows are ordered by: the key's offset from the smallest
  auto key = [&](uint64_t w) -> uint64_t { return WIDE ? w - f.wlo : w >> f.ib; };
  const uint64_t idm = (1ull << f.ib) - 1ull;
  bool bad = false;
#pragma unroll 1
  for (int i = i0 + tid; i < i1; i += kRunThreads) {
    const uint64_t w = s_row[i], k = key(w), pre = k >> s;
    int pos = i;
    if (fix) {
      int a = i, before = 0;
      while (a > 0 && i - a < kRunMax) {
        const uint64_t x = key(s_row[a - 1]);
        if ((x >> s) != pre) break;
        before += x <= k;  // (rows before it of the same key stay before it)
        --a;
      }
      int e = i + 1;
      while (e < m && e - i <= kRunMax) {  // (one more, to tell runs of kRunMax + 1)
        const uint64_t x = key(s_row[e]);
        if ((x >> s) != pre) break;
        before += x < k;
        ++e;
      }
      if (e - a <= kRunMax)
        pos = a + before;
      else {  // a long run: rows in order stay where they are
        if (i > a) bad |= k < key(s_row[i - 1]);
        if (i == a || e == i + 1) {  // its first row, its last one
          const uint32_t q = atomicAdd(&runs_n[i != a], 1u);
          if (q < (uint32_t)kLongRuns) runs[(i == a ? 0 : kLongRuns) + q] = (uint32_t)(b0 + i);
        }
      }
    }
    const int64_t g = b0 + pos;
    if constexpr (WIDE) {
      out_k[g] = (int64_t)w;
      out_v[g] = (int64_t)((uint64_t)ids[b0 + i] + f.ilo);
    } else {
      out_k[g] = (int64_t)(k + f.wlo);
      out_v[g] = (int64_t)((w & idm) + f.ilo);
    }
  }
  if (bad) atomicCAS(err, 0, kErrRuns);
}

// Far ids back into a result: an id whose offset is a code takes the code's value. (No
// other row has such an id: one that had was far itself.) A read of the ids and a write
// of few: a sort of 10^8 rows with one far id takes 2.44 ms, 0.15 more than without
// (4.34 when it went back to columns, 3.43 on columns from the start).
__global__ void __launch_bounds__(256)
    k_far_ids(int64_t* __restrict__ ids, int64_t n, uint64_t ilo, uint64_t esc,
              const uint64_t* __restrict__ far_ids, uint32_t far_n) {  // esc: code 0
  constexpr int kRows = 8;
  const int64_t step = (int64_t)gridDim.x * blockDim.x * kRows;
  for (int64_t r0 = (int64_t)blockIdx.x * blockDim.x * kRows + threadIdx.x; r0 < n; r0 += step) {
    uint64_t x[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int64_t r = r0 + u * 256;
      x[u] = r < n ? (uint64_t)ids[r] - ilo - esc : ~0ull;
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u)
      if (x[u] < (uint64_t)far_n) ids[r0 + u * 256] = (int64_t)far_ids[x[u]];
  }
}

// Long runs packed one after another, to be sorted, and back: run r's rows start at row
// first[r] of the columns and at off[r] of the packed ones.
__global__ void __launch_bounds__(256)
    k_long_rows(const uint32_t* __restrict__ first, const uint32_t* __restrict__ off, int runs,
                int64_t n, int64_t* __restrict__ keys, int64_t* __restrict__ ids,
                int64_t* __restrict__ packed_k, int64_t* __restrict__ packed_v, bool back) {
  for (int64_t x = (int64_t)blockIdx.x * 256 + threadIdx.x; x < n; x += (int64_t)gridDim.x * 256) {
    int lo = 0, hi = runs - 1;  // last run with off <= x
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((int64_t)off[mid] <= x) lo = mid;
      else hi = mid - 1;
    }
    const int64_t r = (int64_t)first[lo] + (x - (int64_t)off[lo]);
    if (back) {
      keys[r] = packed_k[x];
      ids[r] = packed_v[x];
    } else {
      packed_k[x] = keys[r];
      packed_v[x] = ids[r];
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Shared memory of a launch over jobs of several digit widths: the largest of their
// layouts, from 0 bits on (a batched pair whose rows all have one key folds them in a
// pass of no digit, which stages its tile like any other).
template <int ITEMS>
size_t wsweep_launch_smem(int max_bits, int mode, bool guard, bool wide) {
  size_t m = wsweep_smem_bytes<ITEMS>(0, mode, guard, wide);
  for (int b = 1; b <= max_bits; ++b)
    m = std::max(m, wsweep_smem_bytes<ITEMS>(b, mode, guard, wide));
  return m;
}

template <typename K, bool RI, bool RO, int MODE, bool HI, bool WIDE, int ITEMS>
cudaError_t wsweep_attr() {
  const size_t m = wsweep_launch_smem<ITEMS>(kMaxDigitBits, MODE, MODE != kModeSort, WIDE);
  return cudaFuncSetAttribute(k_wsweep<K, RI, RO, MODE, HI, WIDE, ITEMS>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m);
}

template <typename K, bool RI, bool RO, int MODE, bool HI, bool WIDE, int ITEMS>
cudaError_t wsweep_go(const RadixJob<K>* d_jobs, int num_jobs, int64_t tiles, int pass,
                      int max_bits, bool guard, uint32_t* d_counter, int* d_err, cudaStream_t st,
                      const int32_t* d_tile_job) {
  if (tiles <= 0) return cudaSuccess;
  if (max_bits < 0 || max_bits > kMaxDigitBits) return cudaErrorInvalidValue;
  const size_t smem = wsweep_launch_smem<ITEMS>(max_bits, MODE, guard, WIDE);
  k_wsweep<K, RI, RO, MODE, HI, WIDE, ITEMS><<<(unsigned)tiles, kWThreads, smem, st>>>(
      d_jobs, num_jobs, tiles, pass, d_counter, d_err, d_tile_job);
  return cudaGetLastError();
}

// Calls f<RAW_IN, RAW_OUT, HI, WIDE>() for the layout asked for, if this key
// type and mode have it.  32-bit keys always sit in the upper half, and words
// to words go through the 64-bit instantiation.
template <typename K, int MODE, typename F>
cudaError_t wsweep_layout(bool raw_in, bool raw_out, bool hi, bool wide, const F& f) {
  constexpr bool k64 = sizeof(K) == 8;
  if constexpr (k64 && MODE == kModeSort) {
    if (wide) {
      if (raw_in) return f.template operator()<true, false, false, true>();
      if (raw_out) return f.template operator()<false, true, false, true>();
      return f.template operator()<false, false, false, true>();
    }
  }
  if (wide) return cudaErrorInvalidValue;
  if (raw_in) {
    if constexpr (k64 && MODE != kModeCuts)
      if (!hi) return f.template operator()<true, false, false, false>();
    return f.template operator()<true, false, true, false>();
  }
  if constexpr (MODE == kModeSort) {
    if (raw_out) {
      if constexpr (k64)
        if (!hi) return f.template operator()<false, true, false, false>();
      return f.template operator()<false, true, true, false>();
    }
    if constexpr (k64) {
      if (!hi) return f.template operator()<false, false, false, false>();
      return f.template operator()<false, false, true, false>();
    }
  }
  return cudaErrorInvalidValue;
}

template <typename K>
struct WordLaunch {
  const RadixJob<K>* jobs;
  int num_jobs;
  int64_t tiles;
  int pass, max_bits;
  bool guard;
  uint32_t* counter;
  int* err;
  cudaStream_t st;
  const int32_t* tile_job;
};
template <typename K, int MODE, int ITEMS>
struct WordGo {
  const WordLaunch<K>& a;
  template <bool RI, bool RO, bool HI, bool WIDE>
  cudaError_t operator()() const {
    return wsweep_go<K, RI, RO, MODE, HI, WIDE, ITEMS>(a.jobs, a.num_jobs, a.tiles, a.pass,
                                                       a.max_bits, a.guard, a.counter, a.err,
                                                       a.st, a.tile_job);
  }
};
template <typename K, int MODE, int ITEMS>
struct WordAttr {
  template <bool RI, bool RO, bool HI, bool WIDE>
  cudaError_t operator()() const {
    return wsweep_attr<K, RI, RO, MODE, HI, WIDE, ITEMS>();
  }
};

template <typename K>
cudaError_t launch_wsweep(const RadixJob<K>* d_jobs, int num_jobs, int64_t total_tiles, int pass,
                          int max_bits, int mode, bool raw_in, bool raw_out, bool hi, bool wide,
                          int items, bool guard, uint32_t* d_tile_counter, int* d_err,
                          cudaStream_t st, const int32_t* d_tile_job) {
  const WordLaunch<K> a = {d_jobs, num_jobs, total_tiles, pass, max_bits, guard, d_tile_counter,
                           d_err, st, d_tile_job};
  if (items == kWItems && mode == kModeSort)
    return wsweep_layout<K, kModeSort>(raw_in, raw_out, hi, wide, WordGo<K, kModeSort, kWItems>{a});
  if (items == kWItems && mode == kModeRadix)
    return wsweep_layout<K, kModeRadix>(raw_in, raw_out, hi, wide,
                                        WordGo<K, kModeRadix, kWItems>{a});
  if (items == kWItems && mode == kModeCuts)
    return wsweep_layout<K, kModeCuts>(raw_in, raw_out, hi, wide, WordGo<K, kModeCuts, kWItems>{a});
  if (items == kWItemsSmall && mode == kModeSort)
    return wsweep_layout<K, kModeSort>(raw_in, raw_out, hi, wide,
                                       WordGo<K, kModeSort, kWItemsSmall>{a});
  return cudaErrorInvalidValue;
}

// every layout of a mode (raw_in, raw_out, hi, wide in turn)
template <typename K, int MODE, int ITEMS>
cudaError_t wsweep_attrs_mode() {
  const WordAttr<K, MODE, ITEMS> f;
  for (int m = 0; m < 12; ++m) {
    const bool ri = m % 3 == 1, ro = m % 3 == 2, hi = (m / 3) & 1, wide = m / 6;
    const cudaError_t e = wsweep_layout<K, MODE>(ri, ro, hi, wide, f);
    if (e != cudaSuccess && e != cudaErrorInvalidValue) return e;  // (a layout the mode has not)
  }
  return cudaSuccess;
}

template <typename K>
cudaError_t wsweep_attrs() {
  cudaError_t e = wsweep_attrs_mode<K, kModeSort, kWItems>();
  if (e == cudaSuccess) e = wsweep_attrs_mode<K, kModeSort, kWItemsSmall>();
  if (e == cudaSuccess) e = wsweep_attrs_mode<K, kModeRadix, kWItems>();
  if (e == cudaSuccess) e = wsweep_attrs_mode<K, kModeCuts, kWItems>();
  return e;
}

cudaError_t launch_prefix_sample(const int64_t* keys, int64_t n, const KeyStats* d_stats,
                                 int prefix_bits, int min_bits, uint32_t* d_pairs,
                                 cudaStream_t st) {
  if (n < prefix_sample(n) || prefix_bits > 32 || min_bits < prefix_bits)
    return cudaErrorInvalidValue;
  if (prefix_sample(n) == 2048)
    k_prefix_sample<2048><<<1, 1024, sample_smem_bytes<2048>(), st>>>(keys, n, d_stats, prefix_bits,
                                                                      min_bits, d_pairs);
  else
    k_prefix_sample<8192><<<1, 1024, sample_smem_bytes<8192>(), st>>>(keys, n, d_stats, prefix_bits,
                                                                      min_bits, d_pairs);
  return cudaGetLastError();
}

cudaError_t launch_long_rows(const uint32_t* d_first, const uint32_t* d_off, int runs, int64_t n,
                             int64_t* keys, int64_t* ids, int64_t* packed_k, int64_t* packed_v,
                             bool back, cudaStream_t st) {
  if (n <= 0 || runs <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8);
  k_long_rows<<<grid, 256, 0, st>>>(d_first, d_off, runs, n, keys, ids, packed_k, packed_v, back);
  return cudaGetLastError();
}

cudaError_t launch_far_ids(int64_t* ids, int64_t n, const Fold& f, const uint64_t* far_ids,
                           uint32_t far_n, cudaStream_t st) {
  if (n <= 0 || far_n == 0) return cudaSuccess;
  const unsigned grid = (unsigned)std::min<int64_t>((n + 2047) / 2048, 152 * 16);
  k_far_ids<<<grid, 256, 0, st>>>(ids, n, f.ilo, 1ull << f.cb, far_ids,
                                  std::min<uint32_t>(far_n, kFarIds));
  return cudaGetLastError();
}

cudaError_t launch_runs(const uint64_t* rows, const uint32_t* ids, int64_t n, const Fold& f, int s,
                        bool fix, int64_t* out_k, int64_t* out_v, uint32_t* d_runs,
                        uint32_t* d_runs_n, int* d_err, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)((n + kRunTile - 1) / kRunTile);
  if (f.wide)
    k_runs<true><<<grid, kRunThreads, 0, st>>>(rows, ids, n, f, s, fix, out_k, out_v, d_runs,
                                                 d_runs_n, d_err);
  else
    k_runs<false><<<grid, kRunThreads, 0, st>>>(rows, ids, n, f, s, fix, out_k, out_v, d_runs,
                                                 d_runs_n, d_err);
  return cudaGetLastError();
}

cudaError_t word_init_attributes() {
  cudaError_t e = wsweep_attrs<int32_t>();
  if (e == cudaSuccess) e = wsweep_attrs<int64_t>();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_prefix_sample<2048>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sample_smem_bytes<2048>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_prefix_sample<8192>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sample_smem_bytes<8192>());
  return e;
}

#define TJ_INSTANTIATE_WORD(K)                                                                  \
  template cudaError_t launch_wsweep<K>(const RadixJob<K>*, int, int64_t, int, int, int, bool, \
                                        bool, bool, bool, int, bool, uint32_t*, int*,          \
                                        cudaStream_t, const int32_t*);
TJ_INSTANTIATE_WORD(int32_t)
TJ_INSTANTIATE_WORD(int64_t)

}  // namespace tj
