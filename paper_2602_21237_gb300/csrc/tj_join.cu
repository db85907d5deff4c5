// Join of two key-sorted relations on their common key axis (paper Sec. 4.1)
// with a single final materialisation of (r_id, s_id) pairs (Sec. 3.1).
//
//   k_tile_ranges : for every tile of up to kJTile sorted S rows, the range [a, b)
//                   of sorted R rows whose keys lie between the tile's first
//                   and last key (two searches per tile), written with the
//                   tile's rows and job as one 64-byte descriptor;
//   k_join        : per S tile, fused count -> scan -> write:
//                     1. read the tile's descriptor, stage its S rows and its
//                        R range (in chunks of kRCap rows, up to 8) in shared
//                        memory with cp.async;
//                     2. look every S row's key up in each chunk: in a table key
//                        -> (first, end) of its run of R rows where the chunk's
//                        keys are dense, else by a search of its sorted rows;
//                     3. which gives its match count and run start;
//                     4. a decoupled look-back over all tiles of all jobs
//                        (the words in the tiles' descriptors) gives
//                        the tile's first output index;
//                     5. write the pairs, ordered by key, S position, R
//                        position, if they fit the caller's capacity.
//                   Tiles whose R range exceeds the on-chip chunks (S sparse
//                   against R) search a strided sample of the range on chip,
//                   then one stride of R in global memory.
#include "tj_internal.cuh"
#include "tj_warp.cuh"

namespace tj {

template <typename Job>
__device__ __forceinline__ int find_job_j(const Job* jobs, int num_jobs, int64_t t) {
  int lo = 0, hi = num_jobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].tile0 <= t)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// How a join kernel reads rows: W = 0, separate columns (an element is a key);
// W = 1, folded rows (tj_word.cu), keys of up to 63 bits; W = 2, folded rows
// whose key offset lies in the word's upper half (compared in 32 bits); W = 3,
// separate columns with 32-bit ids.  V: an element of the id column.
template <typename K, int W>
struct RowOf {
  using E = uint64_t;
  using V = uint64_t;  // (no id column)
  using Key = uint64_t;
  static __device__ __forceinline__ Key key(E e, int ib) { return e >> ib; }
};
template <typename K>
struct RowOf<K, 0> {
  using E = K;
  using V = K;
  using Key = K;
  static __device__ __forceinline__ Key key(E e, int) { return e; }
};
template <typename K>
struct RowOf<K, 3> {
  using E = K;
  using V = uint32_t;
  using Key = K;
  static __device__ __forceinline__ Key key(E e, int) { return e; }
};
template <typename K>
struct RowOf<K, 2> {
  using E = uint64_t;
  using V = uint64_t;
  using Key = uint32_t;
  static __device__ __forceinline__ Key key(E e, int ib) {
    return (uint32_t)(e >> 32) >> (ib & 31);
  }
};
template <typename K>
__device__ __forceinline__ K word_id(uint64_t w, const WordFmt& f) {
  return (K)((w & ((1ull << f.ib) - 1ull)) + f.ilo);
}
static_assert(kRCap < 0xFFFF, "run bounds are packed in 16 bits");

// Entries of the on-chip table: a chunk of R whose keys span at most that many
// values has one entry per value. (Separate columns, W = 0, leave shared memory for
// half as many.) In other chunks each S row searches the sorted R rows: filling a
// hash table of them took longer (5x10^6 x 5x10^6 int32 rows over 31 bits 589 us,
// now 537; 2^23 x 2^23 clustered rows 997, now 914; 2x10^6 x 8x10^6 516, now 525).
template <int W>
__host__ __device__ constexpr int tab_slots() {
  return W == 0 ? kJTile : 2 * kJTile;
}

__device__ __forceinline__ void st_volatile_u64(uint64_t* p, uint64_t v) {
  asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// ---------------------------------------------------------------------------
// k_tile_ranges: one warp per S tile.  Lanes 0-15 find the first R row with
// key >= the tile's first key, lanes 16-31 the first R row with key > the
// tile's last key, each by a 16-ary search (16 probes per round trip); lane 0
// writes the tile's descriptor, so a join tile needs one load to start.
template <typename K, int W>
__global__ void k_tile_ranges(const JoinJob<K>* __restrict__ jobs, int num_jobs,
                              int64_t total_tiles, JTile<K>* __restrict__ tiles,
                              const int32_t* __restrict__ tile_job, int ib,
                              const int* __restrict__ err) {
  using Row = RowOf<K, W>;
  using E = typename Row::E;
  using V = typename Row::V;
  const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (t >= total_tiles) return;  // whole warps leave together
  const int lane = threadIdx.x & 31, sub = lane & 15;
  const bool upper = lane >= 16;
  const uint32_t half = upper ? 0xFFFF0000u : 0x0000FFFFu;
  const int j = tile_job ? tile_job[t] : find_job_j(jobs, num_jobs, t);
  const JoinJob<K>* J = jobs + j;
  if (err && *err != 0) {  // the rows did not fold: empty tiles, nothing is joined
    if (lane == 0) {
      JTile<K> d = {};
      d.sk = J->sk;
      d.rk = J->rk;
      d.lt = t - J->tile0;
      d.j = j;
      tiles[t] = d;
    }
    return;
  }
  const int64_t row0 = (t - J->tile0) * J->trows;
  const int64_t row1 = min(J->ns, row0 + J->trows);
  const E* __restrict__ s = reinterpret_cast<const E*>(J->sk);
  const E* __restrict__ r = reinterpret_cast<const E*>(J->rk);
  const auto key = Row::key(upper ? s[row1 - 1] : s[row0], ib);
  auto below = [&](int64_t i) {
    const auto x = Row::key(r[i], ib);
    return upper ? !(key < x) : (x < key);
  };
  // invariant: every row before lo satisfies the predicate, none from hi on
  // (predicate: r[i] < key for the lower bound, r[i] <= key for the upper)
  int64_t lo = 0, hi = J->nr;
  while (true) {
    const int64_t len = hi - lo;
    if (__all_sync(0xFFFFFFFFu, len <= 16)) break;
    const int64_t step = (len + 15) / 16;
    const int64_t p = lo + sub * step;
    bool pred = false;
    if (len > 16 && p < hi) pred = below(p);
    const int c = __popc(__ballot_sync(0xFFFFFFFFu, pred) & half);
    if (len > 16) {
      // probes 0..c-1 satisfy the predicate, probe c (if any) does not
      const int64_t lo0 = lo;
      if (c > 0) lo = lo0 + (int64_t)(c - 1) * step + 1;
      if (c < 16) hi = min(hi, lo0 + (int64_t)c * step);
    }
  }
  const int64_t p = lo + sub;
  const bool pred = p < hi && below(p);
  const int64_t res = lo + __popc(__ballot_sync(0xFFFFFFFFu, pred) & half);
  const int64_t b = __shfl_sync(0xFFFFFFFFu, res, 16);
  if (lane == 0) {
    JTile<K> d;
    d.sk = J->sk + row0;
    d.sv = reinterpret_cast<const K*>(reinterpret_cast<const V*>(J->sv) + row0);
    d.rk = J->rk + res;
    d.rv = reinterpret_cast<const K*>(reinterpret_cast<const V*>(J->rv) + res);
    d.lt = t - J->tile0;
    d.nrr = b - res;
    d.nv = (int32_t)(row1 - row0);
    d.j = j;
    d.chain = 0;
    tiles[t] = d;
  }
}

// ---------------------------------------------------------------------------
#ifndef TJ_JTHREADS
#define TJ_JTHREADS 512
#endif
#ifndef TJ_JMINB
#define TJ_JMINB 2
#endif
constexpr int kJThreads = TJ_JTHREADS;          // threads per join CTA
constexpr int kJWarps = kJThreads / 32;
constexpr int kJItems = kJTile / kJThreads;     // S rows per thread
static_assert(kJItems * kJThreads == kJTile, "join tile = threads x items");
// Most matches a row may have for its thread to write them one after another
// (the matches of neighbouring rows share sectors); beyond, every output index
// of the tile finds its row by a binary search.
constexpr uint32_t kJDirect = 16;
static_assert(kJSparse % kJThreads == 0, "whole rounds of a sparse tile's rows");
// R rows a sparse tile takes on chip at once: the room of the table and of the S
// rows it has not.
template <int W>
__host__ __device__ constexpr int sparse_rcap() {
  return W == 0 || W == 3 ? 3 * kRCap : 4 * kRCap;
}
// Wide rows (W = 3) use no table in any tile: their keys are seldom dense, and
// searching takes the whole R range of a tile of as many R rows at once.
// Against 2048-row chunks hashed one after another: join of 2 x 2^26 rows of clustered
// 40-bit keys 7.23 -> 6.22 ms (join kernel 1.8 -> 0.8). Dense keys stay with the table:
// join of 10^7 x 4x10^7 rows 1.48 ms by table, 1.63 by search.
template <int W>
__host__ __device__ constexpr int search_rcap() {
  return W == 3 ? 9 * kRCap / 4 : kRCap;
}
constexpr int kSparseChunks = 2;  // and how often (beyond: searched in global memory)

// Shared memory: S keys | R keys | S ids | R ids (kJTile or kRCap elements and
// kPad more each) | table[tab_slots] u32; folded rows: S words | R words |
// table.  Each staged array starts up to kPad
// elements into its area (its first element keeps the source's address modulo
// 16, so that all but a head and a tail move in 16-byte copies).  After the
// probe the many-matches write path (which reads ids from global memory)
// keeps per-row offsets (u64) and run starts (u32) from the start of it.
template <typename K>
__host__ __device__ constexpr int join_pad() {
  return 16 / (int)sizeof(K);
}
template <typename K, int W>
constexpr size_t join_smem_bytes() {
  using E = typename RowOf<K, W>::E;
  using V = typename RowOf<K, W>::V;
  constexpr bool ids = W == 0 || W == 3;
  return sizeof(E) * (size_t)(kJTile + join_pad<E>() + kRCap + join_pad<E>()) +
         (ids ? sizeof(V) * (size_t)(kJTile + join_pad<V>() + kRCap + join_pad<V>()) : 0) +
         sizeof(uint32_t) * tab_slots<W>();
}
template <typename K, int W>
constexpr size_t sparse_smem_bytes() {
  using E = typename RowOf<K, W>::E;
  using V = typename RowOf<K, W>::V;
  constexpr bool ids = W == 0 || W == 3;
  return sizeof(E) * (size_t)(kJSparse + join_pad<E>() + sparse_rcap<W>() + join_pad<E>()) +
         (ids ? sizeof(V) * (size_t)(kJSparse + join_pad<V>() + sparse_rcap<W>() + join_pad<V>())
              : 0);
}
static_assert(sizeof(int64_t) * (kJTile + 2 + search_rcap<3>() + 2) +
                      sizeof(uint32_t) * (kJTile + 4 + search_rcap<3>() + 4) <=
                  join_smem_bytes<int64_t, 3>(),
              "searched tiles of wide rows fit the join's shared memory");
static_assert(sparse_smem_bytes<int32_t, 0>() <= join_smem_bytes<int32_t, 0>() &&
                  sparse_smem_bytes<int64_t, 0>() <= join_smem_bytes<int64_t, 0>() &&
                  sparse_smem_bytes<int64_t, 2>() <= join_smem_bytes<int64_t, 2>() &&
                  sparse_smem_bytes<int64_t, 3>() <= join_smem_bytes<int64_t, 3>(),
              "sparse tiles fit the join's shared memory");
static_assert(sizeof(uint64_t) * (kJTile + kRCap) >= (sizeof(uint64_t) + sizeof(uint32_t)) * kJTile,
              "offsets and run starts fit in the folded rows' shared memory");
static_assert(sizeof(int32_t) * (2 * kJTile + 2 * kRCap) >=
                  (sizeof(uint64_t) + sizeof(uint32_t)) * kJTile,
              "offsets and run starts fit in the join's shared memory");

// Asynchronous global -> shared copy of n elements into dst (16-byte aligned,
// kPad elements of slack): returns where the copy starts, dst plus the
// source's misalignment, so both sides agree modulo 16; the head and tail
// elements around the 16-byte chunks are copied one by one.  Every thread of
// the CTA calls it.
template <typename K>
__device__ __forceinline__ K* join_copy_async(K* dst, const K* __restrict__ src, int n) {
  const uint32_t mis = (uint32_t)((uintptr_t)src & 15u);  // a multiple of sizeof(K)
  K* d = dst + mis / sizeof(K);
  const uint32_t sd = (uint32_t)__cvta_generic_to_shared(d);
  constexpr int kPer = 16 / (int)sizeof(K);
  const int head = min(n, mis ? (int)((16u - mis) / sizeof(K)) : 0);
  const int chunks = (n - head) / kPer;
  for (int i = threadIdx.x; i < head; i += kJThreads)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sd + (uint32_t)(i * sizeof(K))),
                 "l"(src + i), "n"(sizeof(K))
                 : "memory");
  for (int c = threadIdx.x; c < chunks; c += kJThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sd + (uint32_t)(head * sizeof(K)) +
                                                                   16u * c),
                 "l"(src + head + c * kPer)
                 : "memory");
  for (int i = head + chunks * kPer + threadIdx.x; i < n; i += kJThreads)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sd + (uint32_t)(i * sizeof(K))),
                 "l"(src + i), "n"(sizeof(K))
                 : "memory");
  return d;
}

// One join tile: up to kJTile consecutive rows of sorted S against the range [a, b)
// of sorted R whose keys lie between the tile's first and last key.
//   1. S keys and ids and the first chunk of the R range go to shared memory
//      (cp.async); warp w owns S rows [w*32*kJItems, ...), item u = 32 rows;
//   2. per chunk of the R range (kRCap rows, at most kMaxChunks): every S
//      row's match count and run start, from a table of the chunk's keys by value
//      (entry: first and end of the key's run) where they are dense, else by a
//      search; wider R ranges are searched through a strided sample
//      staged on chip, then within one stride in global memory;
//   3. the tile's total goes to the decoupled look-back chain over all tiles
//      (warp 0, 32 predecessors per round trip), which yields the tile's
//      first output index;
//   4. at most kJDirect matches a row: each row's first output index comes
//      from ballots (one match at most, a foreign-key join) or shuffles over
//      the warp and from the warps' totals; otherwise the tile's counts are
//      scanned and each output index finds its S row.
// Output order: key, then S position, then R position.
template <typename K, int W>
__global__ void __launch_bounds__(kJThreads, TJ_JMINB)
    k_join(int64_t total_tiles, JTile<K>* tiles, WordFmt f, uint32_t* __restrict__ tile_counter,
           K* __restrict__ out, int64_t capacity, const int64_t* __restrict__ out_base,
           int64_t* __restrict__ job_out, int64_t* __restrict__ total, int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Row = RowOf<K, W>;
  using E = typename Row::E;
  using Key = typename Row::Key;
  const int ib = f.ib;
  using V = typename Row::V;
  constexpr bool kIds = W == 0 || W == 3;  // an id column beside the keys
  constexpr int kTabSlots = tab_slots<W>();
  constexpr int kPad = join_pad<E>(), kPadV = join_pad<V>();
  // an id column's element as the caller's id
  auto id_of = [&](V v) -> K { return W == 3 ? (K)((uint64_t)v + f.ilo) : (K)v; };
  __shared__ uint64_t s_wsum[kJWarps];
  __shared__ uint32_t s_wmax[kJWarps];
  __shared__ uint64_t s_base;
  __shared__ uint32_t s_t;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_t = atomicAdd(tile_counter, 1u);
  __syncthreads();
  const int64_t t = s_t;
  if (t >= total_tiles) return;
  const JTile<K> T = tiles[t];
  const int j = T.j;
  const int64_t nrr = T.nrr;
  const int64_t lt = T.lt;
  const int nv = T.nv;
  const E* __restrict__ rk_g = reinterpret_cast<const E*>(T.rk);
  const V* __restrict__ rv_g = reinterpret_cast<const V*>(T.rv);
  // id of R row i of the tile's range, read from global memory
  auto rid_g = [&](int64_t i) -> K {
    if constexpr (!kIds) return word_id<K>(rk_g[i], f);
    else return id_of(rv_g[i]);
  };
  // staging areas (16-byte aligned); a sparse tile has no table and more of R
  const bool sparse = nv <= kJSparse;
  const bool search = W == 3 || sparse;
  const int srows = sparse ? kJSparse : kJTile;
  const int rcap = sparse ? sparse_rcap<W>() : search_rcap<W>();
  E* const b_sk = reinterpret_cast<E*>(smem);
  E* const b_rk = b_sk + srows + kPad;
  V* const b_sv = reinterpret_cast<V*>(b_rk + rcap + kPad);  // (kIds only)
  V* const b_rv = b_sv + srows + kPadV;
  uint32_t* s_ht = kIds ? reinterpret_cast<uint32_t*>(b_rv + kRCap + kPadV)
                        : reinterpret_cast<uint32_t*>(b_sv);
  const int64_t nchunks = (nrr + rcap - 1) / rcap;
  const bool onchip = nchunks <= (sparse ? kSparseChunks : kMaxChunks);

  // 1. stage S and the first R chunk
  const E* s_sk = join_copy_async<E>(b_sk, reinterpret_cast<const E*>(T.sk), nv);
  const V* s_sv = b_sv;
  E* s_rk = b_rk;  // the staged R chunk (where its copy starts)
  V* s_rv = b_rv;
  if constexpr (kIds) s_sv = join_copy_async<V>(b_sv, reinterpret_cast<const V*>(T.sv), nv);
  if (onchip && nchunks > 0) {
    const int nc0 = (int)min((int64_t)rcap, nrr);
    s_rk = join_copy_async<E>(b_rk, rk_g, nc0);
    if constexpr (kIds) s_rv = join_copy_async<V>(b_rv, rv_g, nc0);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");

  // 2. probe (a short tile's rows are spread over all warps, 32 at a time)
  const int wits = (nv + kJThreads - 1) / kJThreads;  // items of a warp
  const int wbase = warp * 32 * wits;
  uint32_t cnt[kJItems], start[kJItems];
#pragma unroll
  for (int u = 0; u < kJItems; ++u) cnt[u] = start[u] = 0u;
  if (onchip) {
    for (int64_t c = 0; c < nchunks; ++c) {
      const int c0 = (int)(c * rcap);
      const int nc = (int)min((int64_t)rcap, nrr - c0);
      if (c > 0) {
        __syncthreads();  // the previous chunk's probes are done
        s_rk = join_copy_async<E>(b_rk, rk_g + c0, nc);
        if constexpr (kIds) s_rv = join_copy_async<V>(b_rv, rv_g + c0, nc);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      for (int i = tid; !search && i < kTabSlots / 4; i += kJThreads)
        reinterpret_cast<uint4*>(s_ht)[i] = make_uint4(0u, 0u, 0u, 0u);
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      const Key cf = Row::key(s_rk[0], ib), cl = Row::key(s_rk[nc - 1], ib);
      if (!search && (uint64_t)cl - (uint64_t)cf < (uint64_t)kTabSlots) {
        // dense keys: entry key - cf holds the key's run (first | end << 16),
        // each half written by the run's first or last row
        uint16_t* const s_run = reinterpret_cast<uint16_t*>(s_ht);
        for (int i = tid; i < nc; i += kJThreads) {
          const Key key = Row::key(s_rk[i], ib);
          const uint32_t d = (uint32_t)((uint64_t)key - (uint64_t)cf);
          if (i == 0 || key != Row::key(s_rk[i - 1], ib)) s_run[2 * d] = (uint16_t)i;
          if (i == nc - 1 || key != Row::key(s_rk[i + 1], ib))
            s_run[2 * d + 1] = (uint16_t)(i + 1);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kJItems; ++u) {
          const int q = wbase + u * 32 + lane;
          if (u >= wits || q >= nv) continue;
          const Key key = Row::key(s_sk[q], ib);
          if (key < cf || cl < key) continue;
          const uint32_t w = s_ht[(uint32_t)((uint64_t)key - (uint64_t)cf)];
          if (w == 0u) continue;
          if (cnt[u] == 0u) start[u] = (uint32_t)c0 + (w & 0xFFFFu);
          cnt[u] += (w >> 16) - (w & 0xFFFFu);
        }
        continue;
      }
      // each S row searches the chunk
#pragma unroll
      for (int u = 0; u < kJItems; ++u) {
        const int q = wbase + u * 32 + lane;
        if (u >= wits || q >= nv) continue;
        const Key key = Row::key(s_sk[q], ib);
        if (key < cf || cl < key) continue;
        int a = 0, n = nc;
        while (n > 0) {
          const int half = n >> 1;
          const bool go = Row::key(s_rk[a + half], ib) < key;
          a = go ? a + half + 1 : a;
          n = go ? n - half - 1 : half;
        }
        // (a < nc: the chunk's last key is not below this one)
        if (Row::key(s_rk[a], ib) != key) continue;
        // the run's end, by steps that double while it goes on, then by halving: a walk
        // of it by one lane held up every later tile's chained scan (10^7 R rows of
        // 5000 keys, 10^6 S rows of which 1000 match: 1049 us, now 505)
        int in = 0, past = 1;  // rows of the run after row a, rows to probe next
        while (a + past < nc && Row::key(s_rk[a + past], ib) == key) {
          in = past;
          past *= 2;
        }
        past = min(past, nc - a);
        while (past - in > 1) {
          const int mid = (in + past) >> 1;
          if (Row::key(s_rk[a + mid], ib) == key) in = mid;
          else past = mid;
        }
        if (cnt[u] == 0u) start[u] = (uint32_t)(c0 + a);
        cnt[u] += (uint32_t)past;
      }
    }
    if (nchunks == 0) asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // Wide R range (S sparse against R): every stride-th R key goes to shared
    // memory; a row's bound is found among those samples on chip, then inside
    // one stride of R in global memory, all rows of a thread in lockstep
    // (independent loads in flight together).
    const int64_t stride = (nrr + kRCap - 1) / kRCap;
    const int m = (int)((nrr + stride - 1) / stride);
    for (int i = tid; i < m; i += kJThreads) s_rk[i] = rk_g[(int64_t)i * stride];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    int steps = 0;  // halvings that empty a range of `stride` rows
    while (((int64_t)1 << steps) <= stride) ++steps;
    Key key[kJItems];
#pragma unroll
    for (int u = 0; u < kJItems; ++u) {
      const int q = wbase + u * 32 + lane;
      key[u] = u < wits && q < nv ? Row::key(s_sk[q], ib) : Key(0);
    }
    // bound 0: first R row with key >= the row's key; 1: first with key >
    // (offsets into the range: nrr < 2^30)
    const int nr32 = (int)nrr;
    auto search = [&](int bound, int (&lo)[kJItems]) {
      int n[kJItems];
#pragma unroll
      for (int u = 0; u < kJItems; ++u) {
        // samples before a satisfy the predicate (sample < key, or <= key)
        int a = 0, c = m;
        while (a < c) {
          const int mid = (a + c) >> 1;
          const Key x = Row::key(s_rk[mid], ib);
          const bool pr = bound ? !(key[u] < x) : (x < key[u]);
          a = pr ? mid + 1 : a;
          c = pr ? c : mid;
        }
        // rows up to sample a - 1 satisfy it, sample a (if any) does not
        lo[u] = a == 0 ? 0 : (int)((a - 1) * stride + 1);
        const int hi = a == m ? nr32 : (int)(a * stride);
        n[u] = hi - lo[u];
      }
      for (int it = 0; it < steps; ++it) {
#pragma unroll
        for (int u = 0; u < kJItems; ++u) {
          const int half = n[u] >> 1;
          const Key r = Row::key(rk_g[min(lo[u] + half, nr32 - 1)], ib);  // in range even when n == 0
          const bool go = n[u] > 0 && (bound ? !(key[u] < r) : (r < key[u]));
          lo[u] = go ? lo[u] + half + 1 : lo[u];
          n[u] = go ? n[u] - half - 1 : half;
        }
      }
    };
    int lo[kJItems];
    search(0, lo);
    // a match and no equal key right after it: one match (the common case of
    // unique R keys); otherwise the upper bound is searched too
    uint32_t more = 0u;
#pragma unroll
    for (int u = 0; u < kJItems; ++u) {
      const bool valid = u < wits && wbase + u * 32 + lane < nv;
      const Key r0 = Row::key(rk_g[min(lo[u], nr32 - 1)], ib);
      const Key r1 = Row::key(rk_g[min(lo[u] + 1, nr32 - 1)], ib);
      const bool e0 = valid && lo[u] < nr32 && r0 == key[u];
      const bool e1 = e0 && lo[u] + 1 < nr32 && r1 == key[u];
      start[u] = (uint32_t)lo[u];
      cnt[u] = e0 ? 1u : 0u;
      more |= (e1 ? 1u : 0u) << u;
    }
    if (__any_sync(0xFFFFFFFFu, more != 0u)) {
      int hi[kJItems];
      search(1, hi);
#pragma unroll
      for (int u = 0; u < kJItems; ++u)
        if ((more >> u) & 1u) cnt[u] = (uint32_t)(hi[u] - lo[u]);
    }
  }

  // 3. the tile's total, its warps' prefixes and the chained scan over tiles
  uint64_t mysum = 0;
  uint32_t mymax = 0;
#pragma unroll
  for (int u = 0; u < kJItems; ++u) {
    mysum += cnt[u];
    mymax = max(mymax, cnt[u]);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) mysum += __shfl_xor_sync(0xFFFFFFFFu, mysum, o);
  mymax = __reduce_max_sync(0xFFFFFFFFu, mymax);
  if (lane == 0) {
    s_wsum[warp] = mysum;
    s_wmax[warp] = mymax;
  }
  __syncthreads();
  uint64_t C = 0, wpre = 0;
#pragma unroll
  for (int w = 0; w < kJWarps; ++w) {
    const uint64_t x = s_wsum[w];
    if (w < warp) wpre += x;
    C += x;
    mymax = max(mymax, s_wmax[w]);  // the tile's largest match count
  }
  // chained scan over all tiles by warp 0 (the first tile is inclusive at once)
  if (warp == 0) {
    uint64_t* const mine = &tiles[t].chain;
    if (lane == 0) st_volatile_u64(mine, (t == 0 ? kFlagInc64 : kFlagAgg64) | (C & kValMask64));
    const uint64_t prefix = chain_prefix<(int)(sizeof(JTile<K>) / 8), 1>(&tiles[0].chain, t, err);
    if (lane == 0 && t != 0) st_volatile_u64(mine, kFlagInc64 | ((prefix + C) & kValMask64));
    if (lane == 0) {
      s_base = prefix;
      if (lt == 0 && job_out) job_out[j] = (int64_t)prefix;
      // the end of this launch's output (absolute when the launch has a base)
      if (t == total_tiles - 1) *total = (int64_t)(prefix + C) + (out_base ? *out_base : 0);
    }
  }
  __syncthreads();
  // output index of this tile's first pair: the group's base (the partitioned
  // join writes several groups one after another) plus the chained prefix
  const uint64_t first = s_base + (out_base ? (uint64_t)*out_base : 0ull);
  if (first + C > (uint64_t)capacity) return;  // the host reports TJ_ERR_CAPACITY

  // 4. write
  if (mymax <= kJDirect) {
    using P = typename PairOf<K>::type;
    const bool vec = (((uintptr_t)out) & (2 * sizeof(K) - 1)) == 0;
    const uint32_t ltm = lanemask_lt();
    // R rows of the chunk still in shared memory (the last one) are read
    // there, earlier ones from global memory
    const uint32_t cres = onchip && nchunks > 0 ? (uint32_t)((nchunks - 1) * rcap) : ~0u;
    const bool single = mymax <= 1u;
    K* __restrict__ const o_w = out + 2 * (first + wpre);  // the warp's first pair
    uint32_t off = 0;  // (a warp has at most 32 kJItems kJDirect pairs)
#pragma unroll
    for (int u = 0; u < kJItems; ++u) {
      const uint32_t c = cnt[u];
      uint32_t before, all;  // pairs of lower lanes, of the warp's 32 rows
      if (single) {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, c != 0u);
        before = __popc(m & ltm);
        all = __popc(m);
      } else {
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
          if (lane >= o) x += y;
        }
        before = x - c;
        all = __shfl_sync(0xFFFFFFFFu, x, 31);
      }
      if (c != 0u) {
        K* __restrict__ o = o_w + 2 * (off + before);
        const uint32_t st0 = start[u];
        K sid;
        if constexpr (!kIds) sid = word_id<K>(s_sk[wbase + u * 32 + lane], f);
        else sid = id_of(s_sv[wbase + u * 32 + lane]);
        for (uint32_t r = st0; r < st0 + c; ++r, o += 2) {
          K rid;
          if constexpr (!kIds) rid = r >= cres ? word_id<K>(s_rk[r - cres], f) : rid_g(r);
          else rid = r >= cres ? id_of(s_rv[r - cres]) : rid_g(r);
          if (vec) {
            P pr;
            pr.x = rid;
            pr.y = sid;
            *reinterpret_cast<P*>(o) = pr;
          } else {
            o[0] = rid;
            o[1] = sid;
          }
        }
      }
      off += all;
    }
  } else {
    // many matches: per-row counts -> exclusive offsets, then each output
    // index finds its S row by binary search
    uint64_t* s_off = reinterpret_cast<uint64_t*>(smem);
    uint32_t* s_rs = reinterpret_cast<uint32_t*>(s_off + kJTile);
#pragma unroll
    for (int u = 0; u < kJItems; ++u) {
      const int q = wbase + u * 32 + lane;
      if (u < wits && q < nv) {
        s_off[q] = cnt[u];
        s_rs[q] = start[u];
      }
    }
    __syncthreads();
    {
      constexpr int kPer = kJTile / kJThreads;
      uint64_t v[kPer];
      uint64_t sum = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int q = tid * kPer + i;
        v[i] = q < nv ? s_off[q] : 0ull;
        sum += v[i];
      }
      uint64_t x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
      }
      __syncthreads();  // every thread has read its counts
      if (lane == 31) s_wsum[warp] = x;
      __syncthreads();
      uint64_t pre = 0;
#pragma unroll
      for (int w = 0; w < kJWarps; ++w)
        if (w < warp) pre += s_wsum[w];
      uint64_t run = pre + x - sum;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int q = tid * kPer + i;
        if (q < nv) s_off[q] = run;
        run += v[i];
      }
    }
    __syncthreads();
    const V* __restrict__ sv_g = reinterpret_cast<const V*>(T.sv);
    const E* __restrict__ sk_g = reinterpret_cast<const E*>(T.sk);
    K* __restrict__ o = out + 2 * first;
    for (uint64_t x = tid; x < C; x += kJThreads) {
      int lo = 0, hi = nv - 1;  // last q with s_off[q] <= x
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_off[mid] <= x)
          lo = mid;
        else
          hi = mid - 1;
      }
      const uint64_t r = s_rs[lo] + (x - s_off[lo]);
      o[2 * x] = rid_g((int64_t)r);
      if constexpr (!kIds) o[2 * x + 1] = word_id<K>(sk_g[lo], f);
      else o[2 * x + 1] = id_of(sv_g[lo]);
    }
  }
}

// ---------------------------------------------------------------------------
template <typename K>
cudaError_t launch_tile_ranges(const JoinJob<K>* d_jobs, int num_jobs, int64_t total_tiles,
                               JTile<K>* d_tiles, cudaStream_t st, const int32_t* d_tile_job,
                               WordFmt f, const int* d_err) {
  if (total_tiles <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)((total_tiles * 32 + kThreads - 1) / kThreads);
  if (f.ib)  // words: the pointers step 8 bytes a row whatever K
    k_tile_ranges<int64_t, 1><<<grid, kThreads, 0, st>>>(
        reinterpret_cast<const JoinJob<int64_t>*>(d_jobs), num_jobs, total_tiles,
        reinterpret_cast<JTile<int64_t>*>(d_tiles), d_tile_job, f.ib, d_err);
  else if (f.wide)
    k_tile_ranges<K, 3><<<grid, kThreads, 0, st>>>(d_jobs, num_jobs, total_tiles, d_tiles,
                                                   d_tile_job, 0, d_err);
  else
    k_tile_ranges<K, 0><<<grid, kThreads, 0, st>>>(d_jobs, num_jobs, total_tiles, d_tiles,
                                                   d_tile_job, 0, d_err);
  return cudaGetLastError();
}

// Tile -> job maps of one group of a partitioned join: blocks [0, nr) fill
// the radix map from the radix jobs, the rest the join map from the join jobs.
template <typename K>
__global__ void k_group_maps(const RadixJob<K>* __restrict__ rjobs, int nr,
                             int32_t* __restrict__ rmap, const JoinJob<K>* __restrict__ jjobs,
                             int32_t* __restrict__ jmap, int tile) {
  const int b = blockIdx.x;
  if (b < nr) {
    const int64_t t0 = rjobs[b].tile0;
    const int64_t nt = (rjobs[b].n + tile - 1) / tile;
    for (int64_t t = threadIdx.x; t < nt; t += blockDim.x) rmap[t0 + t] = b;
  } else {
    const int j = b - nr;
    const int64_t t0 = jjobs[j].tile0;
    const int64_t nt = (jjobs[j].ns + jjobs[j].trows - 1) / jjobs[j].trows;
    for (int64_t t = threadIdx.x; t < nt; t += blockDim.x) jmap[t0 + t] = j;
  }
}

template <typename K>
cudaError_t launch_group_maps(const RadixJob<K>* d_rjobs, int nr, int32_t* d_rmap,
                              const JoinJob<K>* d_jjobs, int nj, int32_t* d_jmap,
                              cudaStream_t st, int tile) {
  if (nr + nj <= 0) return cudaSuccess;
  k_group_maps<K><<<nr + nj, 256, 0, st>>>(d_rjobs, nr, d_rmap, d_jjobs, d_jmap, tile);
  return cudaGetLastError();
}

template <typename K>
__global__ void k_fill_join_tile_job(const JoinJob<K>* __restrict__ jobs,
                                     int32_t* __restrict__ map) {
  const int j = blockIdx.x;
  const int64_t t0 = jobs[j].tile0;
  const int64_t nt = (jobs[j].ns + jobs[j].trows - 1) / jobs[j].trows;
  for (int64_t t = threadIdx.x; t < nt; t += blockDim.x) map[t0 + t] = j;
}

template <typename K>
cudaError_t launch_fill_join_tile_job(const JoinJob<K>* d_jobs, int num_jobs, int32_t* d_map,
                                      cudaStream_t st) {
  if (num_jobs <= 0) return cudaSuccess;
  k_fill_join_tile_job<K><<<num_jobs, 128, 0, st>>>(d_jobs, d_map);
  return cudaGetLastError();
}

template <typename K>
cudaError_t launch_join(int64_t total_tiles, JTile<K>* d_tiles, uint32_t* d_tile_counter, K* out, int64_t capacity,
                        const int64_t* d_out_base, int64_t* d_job_out, int64_t* d_total,
                        int* d_err, cudaStream_t st, WordFmt f) {
  if (total_tiles <= 0) return cudaSuccess;
#define TJ_JOIN(W)                                                                            \
  k_join<K, W><<<(unsigned)total_tiles, kJThreads, join_smem_bytes<K, W>(), st>>>(            \
      total_tiles, d_tiles, f, d_tile_counter, out, capacity, d_out_base,         \
      d_job_out, d_total, d_err)
  if (f.wide) {
    if constexpr (sizeof(K) == 8) TJ_JOIN(3);
  } else if (f.ib >= 32) {
    TJ_JOIN(2);
  } else if (f.ib > 0) {
    if constexpr (sizeof(K) == 8) TJ_JOIN(1);  // 32-bit rows always have ib = 32
  } else {
    TJ_JOIN(0);
  }
#undef TJ_JOIN
  return cudaGetLastError();
}

// Jobs without join tiles (empty S, or skipped) take the first output index of
// the next job that has tiles, or the total; entry num_jobs is the total.
template <typename K>
__global__ void k_fix_job_out(const JoinJob<K>* __restrict__ jobs, int num_jobs,
                              int64_t total_tiles, int64_t* __restrict__ job_out,
                              const int64_t* __restrict__ total) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > num_jobs) return;
  if (j == num_jobs) {
    job_out[j] = total_tiles > 0 ? *total : 0;
    return;
  }
  const int64_t t0 = jobs[j].tile0;
  const bool has_tiles = jobs[j].ns > 0;
  if (has_tiles) return;
  if (t0 >= total_tiles) {
    job_out[j] = total_tiles > 0 ? *total : 0;
  } else {
    const int k = find_job_j(jobs, num_jobs, t0);
    job_out[j] = job_out[k];
  }
}

template <typename K>
cudaError_t launch_fix_job_out(const JoinJob<K>* d_jobs, int num_jobs, int64_t total_tiles,
                               int64_t* d_job_out, const int64_t* d_total, cudaStream_t st) {
  const int grid = (num_jobs + 1 + kThreads - 1) / kThreads;
  k_fix_job_out<K><<<grid, kThreads, 0, st>>>(d_jobs, num_jobs, total_tiles, d_job_out, d_total);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// k_cross: the pairs of single-key batches, streamed (one CTA per kXPairs
// consecutive pairs of a batch): pair p = i * nr + j of a batch is (R id j,
// S id i), so for nr = 1 (a foreign key's heavy value) a CTA reads 4096
// consecutive S ids and writes 4096 consecutive pairs.
template <typename K, bool WORDS>
__global__ void __launch_bounds__(kXThreads)
    k_cross(const CrossJob<K>* __restrict__ jobs, int num_jobs, WordFmt f, K* __restrict__ out,
            int64_t capacity, const int64_t* __restrict__ base_in, int64_t* __restrict__ base_out,
            int64_t run_pairs) {
  const int64_t b = blockIdx.x;
  int lo = 0, hi = num_jobs - 1;  // last job whose first CTA is <= b
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].blk0 <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  const CrossJob<K> J = jobs[lo];
  auto id = [&](const K* p, int64_t i) -> K {
    if constexpr (WORDS) return word_id<K>(reinterpret_cast<const uint64_t*>(p)[i], f);
    else return p[i];
  };
  const int64_t base = *base_in;
  if (b == 0 && threadIdx.x == 0) *base_out = base + run_pairs;
  const int64_t np = J.nr * J.ns;
  const int64_t o = base + J.off;
  if (o + np > capacity) return;  // the host reports TJ_ERR_CAPACITY
  const int64_t p0 = (b - J.blk0) * kXPairs;
  const int64_t p1 = min(np, p0 + kXPairs);
  using P = typename PairOf<K>::type;
  const bool vec = (((uintptr_t)out) & (2 * sizeof(K) - 1)) == 0;
  if (J.nr == 1) {
    const K r = id(J.rv, 0);
    for (int64_t p = p0 + threadIdx.x; p < p1; p += kXThreads) {
      const K sid = id(J.sv, p);
      if (vec) {
        P v;
        v.x = r;
        v.y = sid;
        *reinterpret_cast<P*>(out + 2 * (o + p)) = v;
      } else {
        out[2 * (o + p)] = r;
        out[2 * (o + p) + 1] = sid;
      }
    }
  } else {
    for (int64_t p = p0 + threadIdx.x; p < p1; p += kXThreads) {
      const int64_t i = p / J.nr, j = p - i * J.nr;
      out[2 * (o + p)] = id(J.rv, j);
      out[2 * (o + p) + 1] = id(J.sv, i);
    }
  }
}

template <typename K>
cudaError_t launch_cross(const CrossJob<K>* d_jobs, int num_jobs, int64_t blocks, K* out,
                         int64_t capacity, const int64_t* d_base, int64_t* d_next,
                         int64_t run_pairs, cudaStream_t st, WordFmt f) {
  if (num_jobs <= 0 || blocks <= 0) return cudaErrorInvalidValue;
  if (f.ib)
    k_cross<K, true><<<(unsigned)blocks, kXThreads, 0, st>>>(d_jobs, num_jobs, f, out, capacity,
                                                             d_base, d_next, run_pairs);
  else
    k_cross<K, false><<<(unsigned)blocks, kXThreads, 0, st>>>(d_jobs, num_jobs, f, out, capacity,
                                                              d_base, d_next, run_pairs);
  return cudaGetLastError();
}

template <typename K, int W>
cudaError_t join_attr() {
  return cudaFuncSetAttribute(k_join<K, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)join_smem_bytes<K, W>());
}

cudaError_t join_init_attributes() {
  cudaError_t e = join_attr<int32_t, 0>();
  if (e == cudaSuccess) e = join_attr<int32_t, 2>();
  if (e == cudaSuccess) e = join_attr<int64_t, 0>();
  if (e == cudaSuccess) e = join_attr<int64_t, 1>();
  if (e == cudaSuccess) e = join_attr<int64_t, 2>();
  if (e == cudaSuccess) e = join_attr<int64_t, 3>();
  return e;
}

#define TJ_INSTANTIATE_JOIN(K)                                                                  \
  template cudaError_t launch_tile_ranges<K>(const JoinJob<K>*, int, int64_t, JTile<K>*,        \
                                             cudaStream_t, const int32_t*, WordFmt, const int*); \
  template cudaError_t launch_fill_join_tile_job<K>(const JoinJob<K>*, int, int32_t*,            \
                                                    cudaStream_t);                              \
  template cudaError_t launch_join<K>(int64_t, JTile<K>*, uint32_t*, K*,        \
                                      int64_t, const int64_t*, int64_t*, int64_t*, int*,          \
                                      cudaStream_t, WordFmt);                                     \
  template cudaError_t launch_cross<K>(const CrossJob<K>*, int, int64_t, K*, int64_t,            \
                                       const int64_t*, int64_t*, int64_t, cudaStream_t,         \
                                       WordFmt);                                                  \
  template cudaError_t launch_fix_job_out<K>(const JoinJob<K>*, int, int64_t, int64_t*,          \
                                             const int64_t*, cudaStream_t);                     \
  template cudaError_t launch_group_maps<K>(const RadixJob<K>*, int, int32_t*, const JoinJob<K>*, \
                                            int, int32_t*, cudaStream_t, int);
TJ_INSTANTIATE_JOIN(int32_t)
TJ_INSTANTIATE_JOIN(int64_t)

}  // namespace tj
