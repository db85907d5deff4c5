// Partition-resident phase of the partitioned join (paper Sec. 4.1: align
// both relations on the common key axis; Sec. 3.1: materialise once; Sec. 6:
// every pass within the working memory).
//
// After the route pass has cut R and S into key-range batches and one MSD
// onesweep pass has cut each batch into sub-batches of kFKeys consecutive key
// values (S and R rows of a sub-batch contiguous, in input order), one CTA
// per tile of a sub-batch (at most kFCapS S rows, all of the sub-batch's R
// rows) finishes the join on chip:
//   1. count the R rows per 10-bit key offset (key - the sub-batch's first
//      key) and keep each key's R id in a table (keys with several R rows:
//      the R rows sorted stably by key offset in shared memory, two LSD
//      passes of 5-bit digits);
//   2. hold the S rows in registers, count them per key offset and rank each
//      stably among the warp's rows of its key (tj_warp.cuh);
//   3. per key offset: the S rows of earlier warps and the offset of the
//      key's first pair, Sum_{k' < k} |S_k'| |R_k'| (an exclusive scan);
//   4. a decoupled look-back over the items of the group (in key order) gives
//      the tile's first output index;
//   5. write every pair (r_id, s_id) once, straight to its place: key order,
//      then S position, then R position.
// A sub-batch with more than kFCapS S rows (skewed keys) is split into tiles
// processed by separate CTAs: k_fused_hist adds each tile's counts into the
// sub-batch's totals first, and inside k_fused_join a second decoupled
// look-back over per-key count vectors gives every tile the counts of the
// tiles before it, so a hot key's rows spread over many CTAs.
//
//   k_fused_info  : per batch, the number of items (tiles), of tiles and
//                   sub-batches that need the multi-tile counts, and the
//                   largest R sub-batch (the host checks it fits on chip);
//   k_fused_items : the item list of a group in key order;
//   k_fused_hist  : per-key totals of the multi-tile sub-batches;
//   k_fused_join  : the join of one item.
#include <type_traits>

#include "tj_internal.cuh"
#include "tj_warp.cuh"

namespace tj {

namespace {

constexpr int kFWarps = kFThreads / 32;
constexpr int kFItemsS = kFCapS / kFThreads;  // S rows per thread (18)
static_assert(kFItemsS * kFThreads == kFCapS, "S tile = threads x rows per thread");
constexpr int kFItemsR = kFCapR / kFThreads;  // R rows per thread (8)
constexpr int kFKeysT = kFKeys / kFThreads;   // key offsets per thread in the scans (4)
constexpr int kFDigit = kFKeyBits / 2;        // bits per in-smem sort pass (5)
constexpr int kFBins = 1 << kFDigit;          // 32
static_assert(kFDigit * 2 == kFKeyBits, "two in-smem passes cover the key offset");
static_assert(kFKeysT == 4, "four key offsets per thread in the scans: 16-byte words");
static_assert(kFCapS <= 65536 && kFCapR <= 65536, "16-bit row indices");

__device__ __forceinline__ uint4 ld_vol_v4(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_vol_v4(uint32_t* p, uint4 v) {
  asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_vol_u64(uint64_t* p, uint64_t v) {
  asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Rows of sub-batch d of a job: its R and S row ranges (exclusive bases of
// the MSD histogram; a job without an MSD pass is one sub-batch).
template <typename K>
struct Sub {
  int64_t r0, nr, s0, ns;
};
template <typename K>
__device__ __forceinline__ Sub<K> sub_of(const FusedJob<K>& J, int d) {
  Sub<K> x;
  if (J.m == 0) {
    x.r0 = 0;
    x.nr = J.nr;
    x.s0 = 0;
    x.ns = J.ns;
  } else {
    const int nd = 1 << J.m;
    x.r0 = J.hr[d];
    x.nr = (d + 1 < nd ? (int64_t)J.hr[d + 1] : J.nr) - x.r0;
    x.s0 = J.hs[d];
    x.ns = (d + 1 < nd ? (int64_t)J.hs[d + 1] : J.ns) - x.s0;
  }
  return x;
}

// tiles of a sub-batch (0 if it cannot produce pairs)
__device__ __forceinline__ int64_t tiles_of(int64_t nr, int64_t ns) {
  return (nr > 0 && ns > 0) ? (ns + kFCapS - 1) / kFCapS : 0;
}

// Exclusive scan of v (one value per thread of a CTA of NT threads); the
// CTA's total goes to *total.  Ends with a barrier.
template <int NT, typename T>
__device__ __forceinline__ T block_excl(T v, T* s_warp, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  T pre = 0, all = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    const T z = s_warp[w];
    if (w < warp) pre += z;
    all += z;
  }
  *total = all;
  __syncthreads();
  return pre + x - v;
}

}  // namespace

// ---------------------------------------------------------------------------
// k_fused_info: one CTA per job
// ---------------------------------------------------------------------------
template <typename K>
__global__ void __launch_bounds__(kFThreads) k_fused_info(const FusedJob<K>* __restrict__ jobs,
                                                          int64_t* __restrict__ info) {
  __shared__ int64_t s_w[kFWarps];
  __shared__ int64_t s_max[kFWarps];
  const FusedJob<K>& J = jobs[blockIdx.x];
  const int nd = J.m == 0 ? 1 : 1 << J.m;
  int64_t items = 0, kbt = 0, kbs = 0, maxr = 0;
  for (int d = threadIdx.x; d < nd; d += kFThreads) {
    const Sub<K> x = sub_of(J, d);
    const int64_t t = tiles_of(x.nr, x.ns);
    items += t;
    if (t > 1) {
      kbt += t;
      kbs += 1;
    }
    if (t > 0) maxr = max(maxr, x.nr);
  }
  int64_t tot;
  int64_t* outs[3] = {&items, &kbt, &kbs};
  for (int i = 0; i < 3; ++i) {
    block_excl<kFThreads, int64_t>(*outs[i], s_w, &tot);
    if (threadIdx.x == 0) info[4 * blockIdx.x + i] = tot;
  }
  // largest R sub-batch that produces pairs
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) maxr = max(maxr, __shfl_xor_sync(0xFFFFFFFFu, maxr, o));
  if (lane == 0) s_max[warp] = maxr;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kFWarps; ++w) maxr = max(maxr, s_max[w]);
    info[4 * blockIdx.x + 3] = maxr;
  }
}

// ---------------------------------------------------------------------------
// k_fused_items: one CTA per job writes its items (sub-batches in key order,
// tiles in row order) from its first item index on
// ---------------------------------------------------------------------------
template <typename K>
__global__ void __launch_bounds__(kFThreads) k_fused_items(const FusedJob<K>* __restrict__ jobs,
                                                           FItem* __restrict__ items) {
  __shared__ int64_t s_w[kFWarps];
  const int j = blockIdx.x;
  const FusedJob<K>& J = jobs[j];
  const int nd = J.m == 0 ? 1 : 1 << J.m;
  int64_t base_i = J.item0, base_t = J.kbt0, base_s = J.kbs0;
  for (int c = 0; c < nd; c += kFThreads) {
    const int d = c + (int)threadIdx.x;
    int64_t t = 0;
    if (d < nd) {
      const Sub<K> x = sub_of(J, d);
      t = tiles_of(x.nr, x.ns);
    }
    const bool multi = t > 1;
    int64_t ti, tt, ts;
    const int64_t ei = block_excl<kFThreads, int64_t>(t, s_w, &ti);
    const int64_t et = block_excl<kFThreads, int64_t>(multi ? t : 0, s_w, &tt);
    const int64_t es = block_excl<kFThreads, int64_t>(multi ? 1 : 0, s_w, &ts);
    Sub<K> x = {0, 0, 0, 0};
    if (d < nd) x = sub_of(J, d);
    using U = typename UnsignedOf<K>::type;
    for (int64_t k = 0; k < t; ++k) {
      FItem it;
      it.rk = (uint64_t)(uintptr_t)(J.rk + x.r0);
      it.rv = (uint64_t)(uintptr_t)(J.rv + x.r0);
      it.sk = (uint64_t)(uintptr_t)(J.sk + x.s0 + k * kFCapS);
      it.sv = (uint64_t)(uintptr_t)(J.sv + x.s0 + k * kFCapS);
      it.sublo = (uint64_t)((U)J.lo + ((U)d << kFKeyBits));
      it.nr = (int32_t)x.nr;
      it.ns = (int32_t)min((int64_t)kFCapS, x.ns - k * kFCapS);
      it.job = j;
      it.dt = (uint32_t)d | ((uint32_t)k << 11);
      it.kbt = multi ? (int32_t)(base_t + et + k) : -1;
      it.kbs = multi ? (int32_t)(base_s + es) : -1;
      items[base_i + ei + k] = it;
    }
    base_i += ti;
    base_t += tt;
    base_s += ts;
  }
}

// ---------------------------------------------------------------------------
// k_fused_hist: per-key totals of the multi-tile sub-batches (one CTA per
// item; items of single-tile sub-batches return at once)
// ---------------------------------------------------------------------------
template <typename K>
__global__ void __launch_bounds__(256) k_fused_hist(const FusedJob<K>* __restrict__ jobs,
                                                    const FItem* __restrict__ items,
                                                    uint32_t* __restrict__ tot, int ib) {
  __shared__ uint32_t h[kFKeys];
  const FItem it = items[blockIdx.x];
  if (it.kbt < 0) return;
  using U = typename UnsignedOf<K>::type;
  const U sublo = (U)it.sublo;
  for (int i = threadIdx.x; i < kFKeys; i += 256) h[i] = 0u;
  __syncthreads();
  const int n = it.ns;
  const K* __restrict__ sk = reinterpret_cast<const K*>(it.sk);
  for (int i = threadIdx.x; i < n; i += 256)
    atomicAdd(&h[(uint32_t)(((U)sk[i] >> ib) - sublo) & (kFKeys - 1)], 1u);
  __syncthreads();
  uint32_t* T = tot + (size_t)it.kbs * kFKeys;
  for (int i = threadIdx.x; i < kFKeys; i += 256)
    if (h[i]) atomicAdd(&T[i], h[i]);
}

// ---------------------------------------------------------------------------
// in-smem stable sort of n <= ITEMS * kFThreads rows by their 10-bit key
// offset: two LSD passes of 5-bit digits; the sorted row order lands in pb
// (pa holds the order after the first pass)
// ---------------------------------------------------------------------------
template <int ITEMS>
__device__ __forceinline__ void sort_offsets(const uint16_t* __restrict__ koff, int n,
                                             uint16_t* __restrict__ pa, uint16_t* __restrict__ pb,
                                             uint32_t* wcnt, uint16_t* wexcl, uint32_t* dbase) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wbase = warp * 32 * ITEMS;
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    const int sh = pass * kFDigit;
    uint16_t* __restrict__ outp = pass ? pb : pa;
    for (int i = tid; i < kFWarps * (kFBins / 2); i += kFThreads) wcnt[i] = 0u;
    __syncthreads();
    uint32_t dr[ITEMS];
    uint16_t idx[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const int q = wbase + i * 32 + lane;
      idx[i] = (uint16_t)(q < n ? (pass ? pa[q] : q) : 0);
      dr[i] = q < n ? ((uint32_t)koff[idx[i]] >> sh) & (kFBins - 1) : 0u;
    }
    rank_items<kFDigit, ITEMS>(dr, n - wbase, wcnt + warp * (kFBins / 2));
    __syncthreads();
    // per digit: exclusive prefix over the warps, then the digits' bases
    if (tid < kFBins) {
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kFWarps; ++w) {
        const uint32_t c = (wcnt[w * (kFBins / 2) + (tid >> 1)] >> ((tid & 1) * 16)) & 0xFFFFu;
        wexcl[w * kFBins + tid] = (uint16_t)run;
        run += c;
      }
      // warp 0 holds the 32 digits' totals: exclusive scan
      uint32_t x = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
      }
      dbase[tid] = x - run;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const int q = wbase + i * 32 + lane;
      if (q < n) {
        const uint32_t d = dr[i] & 0xFFFFu;
        outp[dbase[d] + wexcl[warp * kFBins + d] + (dr[i] >> 16)] = idx[i];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// k_fused_join: one CTA per item
// ---------------------------------------------------------------------------
// Shared memory: per-warp counters of the key offsets (two 16-bit counters a
// word) and lane-mask tables of the ranking | per key offset: the
// sub-batch's R rows (two 16-bit counters a word) and the entry a row reads
// to write its pairs | the R rows' key offsets, sorted by key offset
// (stably) when a key has several R rows.  About 48 KB: four CTAs a
// multiprocessor, which their 64 registers a thread allow too.
// What a row of key offset k needs to write its pairs, in one 16-byte load:
// the position of the key's first pair for this tile's rows within the
// sub-batch's output (~0: no R row has the key), and the key's R id (one R
// row per key) or the start of its sorted R run (several).
template <typename K>
struct alignas(16) KeyEnt {
  uint64_t a;
  K r;
};

template <typename K>
struct FusedSmem {
  uint16_t wh[kFWarps][kFKeys];
  union {
    uint32_t wm[kFWarps][128 * kFMaskItems];  // dead before the R rows are sorted
    struct {
      uint16_t r_pa[kFCapR];
      uint16_t r_pb[kFCapR];
    };
  };
  uint32_t cR[kFKeys / 2];
  KeyEnt<K> ent[kFKeys];
  uint16_t r_koff[kFCapR];
  uint32_t wcnt[kFWarps * (kFBins / 2)];
  uint16_t wexcl[kFWarps * kFBins];
  uint32_t dbase[kFBins];
  uint64_t s_w64[kFWarps];
  uint64_t s_wc[kFWarps];
  uint32_t s_w32[kFWarps];
  uint64_t s_base;
  uint32_t s_item;
  uint32_t s_pairs;    // the tile's pairs, summed warp by warp
  uint32_t s_arrived;  // warps that have added theirs
};

template <typename K>
size_t fused_smem_bytes() {
  return sizeof(FusedSmem<K>);
}

// One item: a tile of <= kFCapS S rows of a sub-batch and all its R rows.
//   1. R rows: count per key offset; a key's first R id goes to a table (a
//      key with several R rows sets a flag: then the R rows are sorted by key
//      offset, stably, and each key's run is used);
//   2. S rows (warp w owns 32 kFItemsS consecutive ones, item u of a lane is
//      the warp's row 32 u + lane) counted per key offset and ranked stably
//      within the warp by key offset (wrank); the rows are read again (from
//      L2) when their pairs are written, so only ranks stay in registers;
//   3. per key offset: the S rows of earlier warps (prefix over the warps'
//      counters), of earlier tiles of the sub-batch (look-back over count
//      vectors), and the key's first pair, Sum_{k' < k} |S_k'| |R_k'|;
//   4. the chained scan over the group's items gives the tile's first pair;
//   5. each S row's pairs go to their final position straight from registers.
// Eight warps a CTA, four CTAs a multiprocessor: the per-warp counter tables
// are cleared and summed for every item, so few warps with many rows each pay
// less for them, and four items in different phases hide each other's waits.
// Separate columns hold key offsets beside the ids and keep half of a thread's 64-bit
// S ids in registers at a time, three CTAs a multiprocessor: at 64 registers they
// spilled 304 bytes a thread, now 44 at 80 (join of 10^8 x 4x10^8 rows whose ids do not
// fold, under 256 MiB: 20.02 ms, now 18.70; 2x10^7 x 8x10^7 without a budget 3.62 and
// 3.40; only the halves 19.78, only three CTAs 18.84).
#ifndef TJ_FUSED_MINB
#define TJ_FUSED_MINB 4
#endif
#ifndef TJ_FUSED_MINB_COLUMNS
#define TJ_FUSED_MINB_COLUMNS 3
#endif
// An item's pair count needs only the R counts (each row has its key's), so it is
// published before the ranking, half of an item's time, and the chained scan reads
// 128 words a round trip, most of them ready: join of 10^8 x 4x10^8 rows under
// 256 MiB 14.50 -> 13.95 ms (publishing after the ranking; 32 words 14.05).
constexpr int kFChainWords = 4;
// WORDS: the rows are folded (tj_word.cu), R and S words at it.rk and it.sk.
template <typename K, bool WORDS>
__global__ void __launch_bounds__(kFThreads, WORDS ? TJ_FUSED_MINB : TJ_FUSED_MINB_COLUMNS)
    k_fused_join(const FItem* __restrict__ items, WordFmt f,
                 int64_t n_items, uint32_t* __restrict__ item_counter,
                 uint64_t* __restrict__ item_lb, uint32_t* __restrict__ kb_lb,
                 const uint32_t* __restrict__ kb_tot, K* __restrict__ out, int64_t capacity,
                 const int64_t* __restrict__ out_base, int64_t* __restrict__ total,
                 int* __restrict__ err) {
  using Elem = typename std::conditional<WORDS, uint64_t, K>::type;
  const uint64_t idm = (1ull << f.ib) - 1ull;
  // key offset within the sub-batch, id of a word
  auto koff = [&](Elem e, uint32_t sublo) -> uint32_t {
    return ((WORDS ? (uint32_t)((uint64_t)e >> f.ib) : (uint32_t)e) - sublo) & (kFKeys - 1);
  };
  auto word_id = [&](uint64_t e) -> K { return (K)((e & idm) + f.ilo); };
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FusedSmem<K>& S = *reinterpret_cast<FusedSmem<K>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    S.s_item = atomicAdd(item_counter, 1u);
    S.s_pairs = S.s_arrived = 0u;
  }
  // counters and tables start at zero
  {
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < (int)(sizeof(S.wh) / 16); i += kFThreads)
      reinterpret_cast<uint4*>(S.wh)[i] = z;
    for (int i = tid; i < (int)(sizeof(S.wm) / 16); i += kFThreads)
      reinterpret_cast<uint4*>(S.wm)[i] = z;
    for (int i = tid; i < (int)(sizeof(S.cR) / 16); i += kFThreads)
      reinterpret_cast<uint4*>(S.cR)[i] = z;
  }
  __syncthreads();
  const int64_t ii = S.s_item;
  if (ii >= n_items) return;
  const FItem it = items[ii];
  const int t = (int)(it.dt >> 11);
  const bool multi_tile = it.kbt >= 0;
  const uint32_t sublo = (uint32_t)it.sublo;  // offsets below 2^10: 32 bits suffice
  const int nr = it.nr;  // <= kFCapR (the host checked)
  const int ns = it.ns;
  const K* __restrict__ g_rv = reinterpret_cast<const K*>(it.rv);
  const K* __restrict__ g_sv = reinterpret_cast<const K*>(it.sv);

  // 1. the tile's global loads in flight at once: S keys (the S ids are loaded
  //    when the pairs are written), half of the R rows there is room for
  const int wrow = warp * 32 * kFItemsS;
  const Elem* __restrict__ g_rk = reinterpret_cast<const Elem*>(it.rk);
  const Elem* __restrict__ g_sk = reinterpret_cast<const Elem*>(it.sk);
  // a row past the end takes the last key offset: it ranks after all rows
  const Elem pad = WORDS ? (Elem)((it.sublo + (kFKeys - 1)) << f.ib)
                         : (Elem)(it.sublo + (kFKeys - 1));
  Elem skey[kFItemsS];
#pragma unroll
  for (int u = 0; u < kFItemsS; ++u) {
    const int row = wrow + u * 32 + lane;
    skey[u] = row < ns ? g_sk[row] : pad;
  }
  // (columns keep the key offsets, 16 bits a row, from here on: their ids are read
  // when the pairs are written, and folded rows give the offset again with the id)
  Half<kFItemsS> rank, dig;
  if constexpr (!WORDS) {
#pragma unroll
    for (int u = 0; u < kFItemsS; ++u) dig.set(u, koff(skey[u], sublo));
  }
  auto row_digit = [&](int u) -> uint32_t {
    if constexpr (WORDS) return koff(skey[u], sublo);
    else return dig.get(u);
  };
  // R rows: counts per key offset, a key's first R id in the table
  bool dup = false;
#pragma unroll 1
  for (int u0 = 0; u0 * kFThreads < nr; u0 += kFItemsR / 2) {
    Elem rkey[kFItemsR / 2];
    K rid_v[WORDS ? 1 : kFItemsR / 2];
#pragma unroll
    for (int u = 0; u < kFItemsR / 2; ++u) {
      const int i = tid + (u0 + u) * kFThreads;
      rkey[u] = i < nr ? g_rk[i] : Elem(0);
      if constexpr (!WORDS) rid_v[u] = i < nr ? g_rv[i] : K(0);
    }
#pragma unroll
    for (int u = 0; u < kFItemsR / 2; ++u) {
      const int i = tid + (u0 + u) * kFThreads;
      if (i < nr) {
        const uint32_t o = koff(rkey[u], sublo);
        K rid;
        if constexpr (WORDS) rid = word_id(rkey[u]);
        else rid = rid_v[u];
        S.r_koff[i] = (uint16_t)o;
        const uint32_t sh = (o & 1u) * 16u;  // counts <= kFCapR: the halves never carry
        if (((atomicAdd(&S.cR[o >> 1], 1u << sh) >> sh) & 0xFFFFu) == 0u)
          S.ent[o].r = rid;  // the key's R id, kept unless the key has several
        else
          dup = true;
      }
    }
  }
  dup = __syncthreads_or(dup) != 0;  // R counts complete
  // 2. the tile's pairs: every S row has as many as its key has R rows. Summed
  //    and published before the rows are ranked, so that the items after this
  //    one find the word when they come to the chained scan
  {
    uint32_t c = 0;  // (at most kFCapS kFCapR in a tile)
#pragma unroll
    for (int u = 0; u < kFItemsS; ++u)
      if (wrow + u * 32 + lane < ns)
        c += reinterpret_cast<const uint16_t*>(S.cR)[row_digit(u)];
    c = __reduce_add_sync(0xFFFFFFFFu, c);
    if (lane == 0) {
      atomicAdd(&S.s_pairs, c);
      __threadfence_block();
      if (atomicAdd(&S.s_arrived, 1u) == kFWarps - 1)  // the last warp: the sum is whole
        st_vol_u64(item_lb + ii, (ii == 0 ? kFlagInc64 : kFlagAgg64) | atomicAdd(&S.s_pairs, 0u));
    }
  }
  //    S rows counted and ranked
  wrank<kFKeyBits, kFItemsS, kFMaskItems>(row_digit, rank, S.wh[warp], S.wm[warp], ns - wrow);
  __syncthreads();  // counts complete, ranks done

  // 3. per key offset (four per thread, two 16-bit counters a word): the S rows
  //    of earlier warps, and the tile's count
  const int k0 = kFKeysT * tid;
  uint32_t cs[kFKeysT];
  {
    uint2 run = make_uint2(0u, 0u);  // the 16-bit halves never carry (counts <= kFCapS)
#pragma unroll
    for (int w = 0; w < kFWarps; ++w) {
      uint2* c = reinterpret_cast<uint2*>(&S.wh[w][k0]);
      const uint2 v = *c;
      *c = run;
      run.x += v.x;
      run.y += v.y;
    }
    cs[0] = run.x & 0xFFFFu;
    cs[1] = run.x >> 16;
    cs[2] = run.y & 0xFFFFu;
    cs[3] = run.y >> 16;
    if (tid == kFThreads - 1) {
      // the last warp with rows ranked its last group whole: those past the
      // end were counted as the last key offset
      constexpr int kGroup = 32 * wrank_group<kFItemsS>();
      const int local = (ns - 1) % (32 * kFItemsS) + 1;
      cs[3] -= (uint32_t)((local + kGroup - 1) / kGroup * kGroup - local);
    }
  }
  // multi-tile sub-batches: publish this tile's counts (look-back over the
  // sub-batch's tiles, one word per key offset)
  uint32_t* lb_mine = multi_tile ? kb_lb + (size_t)it.kbt * kFKeys : nullptr;
  if (multi_tile) {
    const uint32_t fl = t == 0 ? kFlagInc : kFlagAgg;
    st_vol_v4(lb_mine + k0, make_uint4(fl | cs[0], fl | cs[1], fl | cs[2], fl | cs[3]));
  }
  // keys with several R rows: their R rows sorted by key offset
  if (dup) sort_offsets<kFItemsR>(S.r_koff, nr, S.r_pa, S.r_pb, S.wcnt, S.wexcl, S.dbase);
  uint32_t pr[kFKeysT] = {0u, 0u, 0u, 0u};
  if (multi_tile && t > 0) {
    // decoupled look-back over the earlier tiles of the sub-batch (a window
    // of kLB predecessors per round trip, the four key offsets in lockstep;
    // tile 0 publishes inclusive counts, so the walk ends there at the
    // latest; bounded wait)
    constexpr int kLB = 4;
    const int64_t first = it.kbt - t;  // a sub-batch's tiles have consecutive slots
    int64_t p = it.kbt - 1;
    uint32_t open = 0xFu;  // key offsets without an inclusive word yet
    int spins = 0;
    while (open != 0u) {
      uint4 v[kLB];
#pragma unroll
      for (int q = 0; q < kLB; ++q)
        v[q] = p - q >= first ? ld_vol_v4(kb_lb + (size_t)(p - q) * kFKeys + k0)
                              : make_uint4(kFlagInc, kFlagInc, kFlagInc, kFlagInc);
      int used = 0;
#pragma unroll
      for (int q = 0; q < kLB; ++q) {
        const uint32_t x[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
        bool ready = true;
#pragma unroll
        for (int e = 0; e < kFKeysT; ++e) ready &= (x[e] & ~kValMask) != 0u;
        if (used != q || !ready) continue;  // an earlier one is not published yet
        ++used;
#pragma unroll
        for (int e = 0; e < kFKeysT; ++e)
          if ((open >> e) & 1u) {
            pr[e] += x[e] & kValMask;
            if ((x[e] & ~kValMask) == kFlagInc) open &= ~(1u << e);
          }
      }
      p -= used;
      if (used == 0) {
        if (++spins > kSpinLimit) {
          atomicExch(err, (int)TJ_ERR_TIMEOUT);
          break;
        }
        __nanosleep(32);
      }
    }
    st_vol_v4(lb_mine + k0, make_uint4(kFlagInc | ((pr[0] + cs[0]) & kValMask),
                                       kFlagInc | ((pr[1] + cs[1]) & kValMask),
                                       kFlagInc | ((pr[2] + cs[2]) & kValMask),
                                       kFlagInc | ((pr[3] + cs[3]) & kValMask)));
  }
  uint32_t cr[kFKeysT], tot[kFKeysT];
  {
    const uint2 c4 = *reinterpret_cast<const uint2*>(&S.cR[2 * tid]);
    cr[0] = c4.x & 0xFFFFu;
    cr[1] = c4.x >> 16;
    cr[2] = c4.y & 0xFFFFu;
    cr[3] = c4.y >> 16;
    uint4 t4 = make_uint4(cs[0], cs[1], cs[2], cs[3]);
    if (multi_tile)
      t4 = *reinterpret_cast<const uint4*>(kb_tot + (size_t)it.kbs * kFKeys + k0);
    tot[0] = t4.x;
    tot[1] = t4.y;
    tot[2] = t4.z;
    tot[3] = t4.w;
  }
  // one pass over the key offsets: the exclusive scan of the keys' pairs in
  // the sub-batch (the first pair of each key) and of their R rows (run
  // starts), with the sum of earlier tiles' pairs
  const uint64_t cnt_tile = S.s_pairs;
  uint64_t total_sub, before;
  {
    uint64_t a = 0, c = 0;  // scanned, summed
    uint32_t r = 0;                // scanned
#pragma unroll
    for (int e = 0; e < kFKeysT; ++e) {
      a += (uint64_t)tot[e] * cr[e];
      c += (uint64_t)pr[e] * cr[e];
      r += cr[e];
    }
    uint64_t xa = a;
    uint32_t xr = r;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t ya = __shfl_up_sync(0xFFFFFFFFu, xa, o);
      const uint32_t yr = __shfl_up_sync(0xFFFFFFFFu, xr, o);
      if (lane >= o) {
        xa += ya;
        xr += yr;
      }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    }
    if (lane == 31) {
      S.s_w64[warp] = xa;
      S.s_w32[warp] = xr;
    }
    if (lane == 0) {
      S.s_wc[warp] = c;
    }
    __syncthreads();
    uint64_t pa = 0, ta = 0, tc = 0;
    uint32_t pr32 = 0;
#pragma unroll
    for (int w = 0; w < kFWarps; ++w) {
      const uint64_t va = S.s_w64[w];
      if (w < warp) {
        pa += va;
        pr32 += S.s_w32[w];
      }
      ta += va;
      tc += S.s_wc[w];
    }
    uint64_t eo = pa + xa - a;     // first pair of key k0 in the sub-batch
    uint32_t er = pr32 + xr - r;  // first sorted R row of key k0
#pragma unroll
    for (int e = 0; e < kFKeysT; ++e) {
      // the key's first pair for this tile's rows: after the earlier tiles';
      // with several R rows a key's run start replaces its R id
      S.ent[k0 + e].a = cr[e] ? eo + (uint64_t)pr[e] * cr[e] : ~0ull;
      if (dup) S.ent[k0 + e].r = (K)er;
      eo += (uint64_t)tot[e] * cr[e];
      er += cr[e];
    }
    total_sub = ta;
    before = tc;
  }

  // the S ids (folded rows: the words again, from L2), needed when the pairs
  // are written: their loads in flight while warp 0 runs the chained scan
  using SRow = typename std::conditional<WORDS, uint64_t, K>::type;
  // (64-bit columns, whose digits take registers too: half of them, and the other half
  // after those are written, prefetched to L2)
  constexpr int kHold = !WORDS && sizeof(K) == 8 ? kFItemsS / 2 : kFItemsS;
  static_assert(kFItemsS % kHold == 0, "whole groups");
  const SRow* __restrict__ g_srow =
      WORDS ? reinterpret_cast<const SRow*>(it.sk) : reinterpret_cast<const SRow*>(g_sv);
  SRow srow[kHold];
  auto load_rows = [&](int u0) {
#pragma unroll
    for (int h = 0; h < kHold; ++h) {
      const int row = wrow + (u0 + h) * 32 + lane;
      srow[h] = row < ns ? g_srow[row] : SRow(0);
    }
  };
  load_rows(0);
#pragma unroll
  for (int u = kHold; u < kFItemsS; ++u)
    if (wrow + u * 32 + lane < ns)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(g_srow + (wrow + u * 32 + lane)));
  // 4. chained scan over the group's items (warp 0): the tile's first pair
  if (warp == 0) {
    const uint64_t prefix = chain_prefix<1, kFChainWords>(item_lb, ii, err);
    if (lane == 0 && ii != 0)
      st_vol_u64(item_lb + ii, kFlagInc64 | ((prefix + cnt_tile) & kValMask64));
    if (lane == 0) {
      const int64_t gb = out_base ? *out_base : 0;
      S.s_base = (uint64_t)gb + prefix;
      if (ii == n_items - 1) *total = gb + (int64_t)(prefix + cnt_tile);
    }
  }
  __syncthreads();
  const uint64_t E = S.s_base;      // absolute index of this tile's first pair
  const uint64_t base = E - before;  // the sub-batch's first pair
  // the tile's pairs lie anywhere in its sub-batch's: write nothing unless
  // all of them fit (the host reports TJ_ERR_CAPACITY)
  if (base + total_sub > (uint64_t)capacity) return;

  // 5. every S row's pairs, in key order, then S position, then R position
  using P = typename PairOf<K>::type;
  const bool vec = (((uintptr_t)out) & (2 * sizeof(K) - 1)) == 0;
  const uint16_t* wx = S.wh[warp];
#pragma unroll
  for (int u = 0; u < kFItemsS; ++u) {
    if (u > 0 && u % kHold == 0) load_rows(u);
    if (wrow + u * 32 + lane >= ns) continue;
    uint32_t k;
    K s_id;
    if constexpr (WORDS) {
      k = koff(srow[u % kHold], sublo);
      s_id = word_id(srow[u % kHold]);
    } else {
      k = dig.get(u);
      s_id = srow[u % kHold];
    }
    const KeyEnt<K> en = S.ent[k];
    if (en.a == ~0ull) continue;  // no R row has the key
    // S rows of the key before this one in the tile: earlier warps, earlier
    // lanes and items of this warp
    const uint32_t within = wx[k] + rank.get(u);
    if (!dup) {
      const uint64_t pos = base + en.a + within;
      if (vec) {
        P pr2;
        pr2.x = en.r;
        pr2.y = s_id;
        *reinterpret_cast<P*>(out + 2 * pos) = pr2;
      } else {
        out[2 * pos] = en.r;
        out[2 * pos + 1] = s_id;
      }
    } else {
      const uint32_t c = (S.cR[k >> 1] >> ((k & 1u) * 16u)) & 0xFFFFu;
      const uint64_t pos = base + en.a + (uint64_t)within * c;
      const uint32_t r0 = (uint32_t)en.r;
      const K* __restrict__ rv = g_rv;  // R ids in the order of the key's run
      for (uint32_t j = 0; j < c; ++j) {
        const uint32_t row = S.r_pb[r0 + j];
        if constexpr (WORDS) out[2 * (pos + j)] = word_id(g_rk[row]);
        else out[2 * (pos + j)] = rv[row];
        out[2 * (pos + j) + 1] = s_id;
      }
    }
  }
}

// ---------------------------------------------------------------------------
template <typename K>
cudaError_t launch_fused_info(const FusedJob<K>* d_jobs, int nj, int64_t* d_info,
                              cudaStream_t st) {
  if (nj <= 0) return cudaSuccess;
  k_fused_info<K><<<nj, kFThreads, 0, st>>>(d_jobs, d_info);
  return cudaGetLastError();
}

template <typename K>
cudaError_t launch_fused_prep(const FusedJob<K>* d_jobs, int nj, FItem* d_items, int64_t n_items,
                              bool any_multi, uint32_t* d_kb_tot, cudaStream_t st, WordFmt f) {
  if (nj <= 0 || n_items <= 0) return cudaSuccess;
  // folded rows: the pointers step 8 bytes a row whatever K
  const auto* w_jobs = reinterpret_cast<const FusedJob<int64_t>*>(d_jobs);
  if (f.ib)
    k_fused_items<int64_t><<<nj, kFThreads, 0, st>>>(w_jobs, d_items);
  else
    k_fused_items<K><<<nj, kFThreads, 0, st>>>(d_jobs, d_items);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !any_multi) return e;
  if (f.ib)
    k_fused_hist<int64_t><<<(unsigned)n_items, 256, 0, st>>>(w_jobs, d_items, d_kb_tot, f.ib);
  else
    k_fused_hist<K><<<(unsigned)n_items, 256, 0, st>>>(d_jobs, d_items, d_kb_tot, 0);
  return cudaGetLastError();
}

template <typename K>
cudaError_t launch_fused_join(const FusedJob<K>* d_jobs, const FItem* d_items, int64_t n_items,
                              uint32_t* d_item_counter, uint64_t* d_item_lb, uint32_t* d_kb_lb,
                              const uint32_t* d_kb_tot, K* out, int64_t capacity,
                              const int64_t* d_out_base, int64_t* d_total, int* d_err,
                              cudaStream_t st, WordFmt f) {
  (void)d_jobs;  // the items carry what the join needs
  if (n_items <= 0) return cudaSuccess;
  if (f.ib)
    k_fused_join<K, true><<<(unsigned)n_items, kFThreads, fused_smem_bytes<K>(), st>>>(
        d_items, f, n_items, d_item_counter, d_item_lb, d_kb_lb, d_kb_tot, out, capacity,
        d_out_base, d_total, d_err);
  else
    k_fused_join<K, false><<<(unsigned)n_items, kFThreads, fused_smem_bytes<K>(), st>>>(
        d_items, f, n_items, d_item_counter, d_item_lb, d_kb_lb, d_kb_tot, out, capacity,
        d_out_base, d_total, d_err);
  return cudaGetLastError();
}

template <typename K, bool WORDS>
cudaError_t fused_attr() {
  return cudaFuncSetAttribute(k_fused_join<K, WORDS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)fused_smem_bytes<K>());
}

cudaError_t fused_init_attributes() {
  cudaError_t e = fused_attr<int32_t, false>();
  if (e == cudaSuccess) e = fused_attr<int32_t, true>();
  if (e == cudaSuccess) e = fused_attr<int64_t, false>();
  if (e == cudaSuccess) e = fused_attr<int64_t, true>();
  return e;
}

#define TJ_INSTANTIATE_FUSED(K)                                                                 \
  template cudaError_t launch_fused_info<K>(const FusedJob<K>*, int, int64_t*, cudaStream_t);   \
  template cudaError_t launch_fused_prep<K>(const FusedJob<K>*, int, FItem*, int64_t, bool,     \
                                            uint32_t*, cudaStream_t, WordFmt);                  \
  template cudaError_t launch_fused_join<K>(const FusedJob<K>*, const FItem*, int64_t,          \
                                            uint32_t*, uint64_t*, uint32_t*, const uint32_t*,   \
                                            K*, int64_t, const int64_t*, int64_t*, int*,        \
                                            cudaStream_t, WordFmt);
TJ_INSTANTIATE_FUSED(int32_t)
TJ_INSTANTIATE_FUSED(int64_t)

}  // namespace tj
