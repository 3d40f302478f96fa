// Ranking of the selected candidates by partition (Algorithm 1, step 15: |x| descending, ties by ascending index).
//
// The selection has left every client's candidates in coarse buckets, ranges of the sort key inv = keytop - key whose
// starts are known, in no particular order inside a bucket.  k_rank_split moves the candidates of a client with large
// buckets on into sub-buckets (the next bits of inv); k_rank then ranks whole buckets in shared memory by (inv, index) and
// writes them out in order.  The order is total, so the result does not depend on how the candidates arrived.  Against a
// stable radix sort of the same keys (three passes of 9 bits) a candidate is moved once or twice instead of three times
// and costs one counting and one placing shared-memory atomic per move instead of a stable rank among the lanes of a warp.
#include "cvlc_common.cuh"

namespace cvlc {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kRankThreads = 512;
constexpr uint32_t kCellBits = 12, kCells = 1u << kCellBits;  // value ranges a tile is spread over before its items are compared
constexpr uint32_t kCompareAll = 48;    // a cell of up to this many items is ranked by comparing each with all,
constexpr uint32_t kWarpCell = 1024;    // one of up to this many is sorted by one warp, a larger one by the block

typedef unsigned long long u64;

// status and mode of the call, the same for all threads of a block
__device__ __forceinline__ bool rank_skips(const EncHeader* hdr) {
  __shared__ int s_skip;
  if (threadIdx.x == 0) s_skip = *reinterpret_cast<const volatile int32_t*>(&hdr->status) != 0 || hdr->lsd != kRankPartition;
  __syncthreads();
  return s_skip != 0;
}

// (no candidate lies above keytop: the selection has checked that the update is the plan's)
__device__ __forceinline__ uint32_t inv_of(u64 item, uint32_t keytop) { return keytop - (uint32_t)(item >> 32); }

// ===================================================================================
// partition of the coarse buckets into sub-buckets
// ===================================================================================
// Tiles of kSplitTile consecutive candidates, held in registers.  A tile spans few coarse buckets, so its sub-buckets are a
// short range of counters: count, reserve each sub-bucket's room with one global atomic, place.  The next tile's candidates are
// requested before the current one is placed.  16 bytes per candidate; the stores are scattered 8 bytes at a time and merge in
// the L2.

constexpr int kSplitItems = 8;  // per thread
constexpr uint32_t kSplitTile = kRankThreads * kSplitItems;
static_assert(kSplitTile == kRankSplitTile, "tiles of the partition");

__global__ void __launch_bounds__(kRankThreads, 2)
k_rank_split(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L) {
  extern __shared__ uint32_t s_at[];  // [kRankSubs] counts, then next places
  __shared__ uint32_t s_next;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (rank_skips(hdr)) return;
  const uint32_t n = batch.n, tickets = hdr->split_tiles * n;
  if (tickets == 0) return;
  const int tid = threadIdx.x;
  const ClientRank* rank = reinterpret_cast<const ClientRank*>(ws + L.off_rank);
  const u64* buf_a = reinterpret_cast<const u64*>(ws + L.off_buf_a);
  u64 it[kSplitItems];
  auto request = [&](uint32_t t) {
    if (t >= tickets) return;
    const uint32_t tile = t / n, c = t - tile * n, first = tile * kSplitTile, have = rank[c].n;
    const u64* __restrict__ src = buf_a + (size_t)c * L.capacity + first;
    const uint32_t m = first < have ? have - first : 0u;
#pragma unroll
    for (int u = 0; u < kSplitItems; ++u)
      if ((uint32_t)tid + u * kRankThreads < m) it[u] = src[tid + u * kRankThreads];
  };
  if (tid == 0) s_next = atomicAdd(&hdr->split_ticket, 1u);
  __syncthreads();
  uint32_t t = s_next;
  request(t);
  while (t < tickets) {
    __syncthreads();  // everyone has read the ticket
    if (tid == 0) s_next = atomicAdd(&hdr->split_ticket, 1u);
    const uint32_t tile = t / n, c = t - tile * n;
    const ClientRank r = rank[c];
    const uint32_t first = tile * kSplitTile;
    const bool on = r.split && first < r.n;
    const uint32_t m = on ? ((r.n - first < kSplitTile) ? r.n - first : kSplitTile) : 0u;
    const uint32_t sh_coarse = 19 + r.group, sh = sh_coarse - r.sub_bits;
    uint32_t s0 = 0, ns = 0;
    if (on) {
      // the candidates are in bucket order: the sub-buckets of the tile lie between those of its ends
      const u64* __restrict__ src = buf_a + (size_t)c * L.capacity + first;
      s0 = (inv_of(src[0], r.keytop) >> sh_coarse) << r.sub_bits;
      const uint32_t s1 = ((inv_of(src[m - 1], r.keytop) >> sh_coarse) + 1) << r.sub_bits;
      ns = (s1 > s0 && s1 - s0 <= kRankSubs) ? s1 - s0 : 0u;
    }
    for (uint32_t i = tid; i < ns; i += kRankThreads) s_at[i] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSplitItems; ++u) {
      const uint32_t s = (inv_of(it[u], r.keytop) >> sh) - s0;
      if ((uint32_t)tid + u * kRankThreads < m && s < ns) atomicAdd(s_at + s, 1u);
    }
    __syncthreads();
    const uint32_t next = s_next;
    uint32_t* room = reinterpret_cast<uint32_t*>(ws + L.off_sub_pos) + (size_t)c * kRankSubs + s0;
    for (uint32_t i = tid; i < ns; i += kRankThreads) {
      const uint32_t v = s_at[i];
      if (v) s_at[i] = atomicAdd(room + i, v);
    }
    __syncthreads();
    u64 cur[kSplitItems];
#pragma unroll
    for (int u = 0; u < kSplitItems; ++u) cur[u] = it[u];
    request(next);
    u64* __restrict__ dst = reinterpret_cast<u64*>(ws + L.off_buf_b) + (size_t)c * L.capacity;
#pragma unroll
    for (int u = 0; u < kSplitItems; ++u) {
      const uint32_t s = (inv_of(cur[u], r.keytop) >> sh) - s0;
      if ((uint32_t)tid + u * kRankThreads < m && s < ns) {
        const uint32_t p = atomicAdd(s_at + s, 1u);
        if (p < r.n) dst[p] = cur[u];
      }
    }
    t = next;
  }
}

// ===================================================================================
// final ranking
// ===================================================================================

struct RankShared {
  u64 items[kRankItems + 2];  // values (see to_value): all distinct, ordered like the ranks
  uint32_t zero[4];           // cell[-1] = 0: where the first cell starts
  uint32_t cell[kCells];      // counts, then starts, then (after placing) ends of the cells
};

// A candidate as a value to rank: the key's complement in the high word, index << 1 | sign in the low word.
__device__ __forceinline__ u64 to_value(u64 item) {
  const uint32_t lo = (uint32_t)item;
  return ((u64)~(uint32_t)(item >> 32) << 32) | (u64)__funnelshift_l(lo, lo, 1);
}
__device__ __forceinline__ u64 to_item(u64 value) {
  const uint32_t lo = (uint32_t)value;
  return ((u64)~(uint32_t)(value >> 32) << 32) | (u64)__funnelshift_r(lo, lo, 1);
}

// exclusive scan of the cells in place by the whole block; returns the total
__device__ __forceinline__ uint32_t scan_cells(uint32_t* cell) {
  __shared__ uint32_t s_warp[kRankThreads / 32];
  constexpr int kVec = kCells / kRankThreads / 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4* mine = reinterpret_cast<uint4*>(cell) + kVec * tid;
  uint4 a[kVec];
  uint32_t sum = 0;
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    a[i] = mine[i];
    sum += a[i].x + a[i].y + a[i].z + a[i].w;
  }
  uint32_t incl = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  // the warps' totals: lane w holds warp w's
  const uint32_t wt = lane < kRankThreads / 32 ? s_warp[lane] : 0u;
  const uint32_t total = __reduce_add_sync(kFull, wt);
  uint32_t run = __reduce_add_sync(kFull, lane < warp ? wt : 0u) + incl - sum;
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    uint4 e;
    e.x = run;
    e.y = e.x + a[i].x;
    e.z = e.y + a[i].y;
    e.w = e.z + a[i].z;
    run = e.w + a[i].w;
    mine[i] = e;
  }
  __syncthreads();
  return total;
}

// Sorts items[0 .. n) in place by `threads` threads (t0 = the caller's number among them; `sync` waits for all of them): a bitonic
// network whose comparators all point the same way, so that the places behind the last item (larger than all) need no comparing.
template <class Sync>
__device__ __forceinline__ void bitonic_sort(u64* items, uint32_t n, uint32_t t0, uint32_t threads, Sync&& sync) {
  uint32_t size = 1;
  while (size < n) size <<= 1;
  for (uint32_t k = 2; k <= size; k <<= 1) {
    for (uint32_t j = k / 2; j > 0; j >>= 1) {
      // first step of a merge (j = k / 2): i against its mirror image in the run of k; then against i + j.  Four pairs at a time:
      // their loads, then their stores.
      const uint32_t flip = (j == k / 2) ? k - 1 : j;
      for (uint32_t ta = t0; ta < size / 2; ta += 4 * threads) {
        u64 a[4], b[4];
        uint32_t i[4], p[4];
        bool on[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t t = ta + threads * u;
          i[u] = ((t & ~(j - 1)) << 1) | (t & (j - 1));
          p[u] = i[u] ^ flip;
          on[u] = t < size / 2 && p[u] < n;
          a[u] = on[u] ? items[i[u]] : 0ull;
          b[u] = on[u] ? items[p[u]] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (on[u] && a[u] > b[u]) {
            items[i[u]] = b[u];
            items[p[u]] = a[u];
          }
        }
      }
      sync();
    }
  }
}

// by the whole block: sorts items[0 .. n) and writes them out
__device__ __noinline__ void rank_by_block(u64* items, uint32_t n, u64* __restrict__ out) {
  bitonic_sort(items, n, threadIdx.x, kRankThreads, [] { __syncthreads(); });
  for (uint32_t i = threadIdx.x; i < n; i += kRankThreads) out[i] = to_item(items[i]);
  __syncthreads();
}

// A boundary near rank x of the m values of src, all in [lo, hi): a value and how many of src lie below it.  The range around the
// rank is narrowed until at most kCutRest values are left in it; the boundary is where that range starts.  A function of the set
// of values and x alone, so that neighbouring tiles agree on it.
constexpr uint32_t kCutRest = kRankItems - kRankWindow;
struct Cut {
  u64 value;
  uint32_t below;
};
__device__ __noinline__ Cut cut_near(RankShared& s, const u64* __restrict__ src, uint32_t m, u64 lo, u64 hi, uint32_t x) {
  __shared__ uint32_t s_cell, s_below, s_count;
  const int tid = threadIdx.x;
  Cut cut{lo, 0};
  for (int level = 0; level < 8 && lo < hi; ++level) {  // 63 bits, 12 a level
    const u64 span = hi - lo - 1;
    const int sh = span < kCells ? 0 : 64 - __clzll((long long)span) - (int)kCellBits;  // span >> sh below kCells
    for (uint32_t i = tid; i < kCells; i += kRankThreads) s.cell[i] = 0;
    if (tid == 0) s_cell = s_below = s_count = 0;
    __syncthreads();
    for (uint32_t i = tid; i < m; i += kRankThreads) {
      const u64 v = to_value(src[i]);
      if (v >= lo && v < hi) atomicAdd(&s.cell[(uint32_t)((v - lo) >> sh)], 1u);
    }
    __syncthreads();
    const uint32_t total = scan_cells(s.cell);
    // the last cell that starts at or below the rank
    const uint32_t at = x - cut.below;
    for (uint32_t i = tid; i < kCells; i += kRankThreads) {
      const uint32_t b = s.cell[i], e = (i + 1 < kCells) ? s.cell[i + 1] : total;
      if (b <= at && at < e) {
        s_cell = i;
        s_below = b;
        s_count = e - b;
      }
    }
    __syncthreads();
    const uint32_t cell = s_cell, below = s_below, count = s_count;
    __syncthreads();
    lo += (u64)cell << sh;
    hi = lo + (1ull << sh) < hi ? lo + (1ull << sh) : hi;
    cut.value = lo;
    cut.below += below;
    if (count <= kCutRest || sh == 0) break;
  }
  return cut;
}

// Ranks a .. b (about) of a bucket that a block cannot hold, m values in [lo, hi): equal or nearly equal keys.  src and out differ.
__device__ __noinline__ void rank_part(RankShared& s, const u64* __restrict__ src, uint32_t m, u64 lo, u64 hi, uint32_t a, uint32_t b,
                                       u64* __restrict__ out) {
  __shared__ uint32_t s_n;
  const int tid = threadIdx.x;
  const Cut from = a == 0 ? Cut{lo, 0} : cut_near(s, src, m, lo, hi, a);
  const Cut to = b >= m ? Cut{hi, m} : cut_near(s, src, m, lo, hi, b);
  if (tid == 0) s_n = 0;
  __syncthreads();
  for (uint32_t i = tid; i < m; i += kRankThreads) {
    const u64 v = to_value(src[i]);
    if (v >= from.value && v < to.value) {
      const uint32_t p = atomicAdd(&s_n, 1u);
      if (p < kRankItems) s.items[p] = v;
    }
  }
  __syncthreads();
  const uint32_t got = s_n < kRankItems ? s_n : kRankItems;  // at most a window and kCutRest
  __syncthreads();
  rank_by_block(s.items, got, out + from.below);
}

// Cells of equal or nearly equal keys (a layer's clipped outliers, values on a grid), first item | items << 16: every warp sorts
// some of them, the block the largest.
__device__ __noinline__ void rank_big_cells(RankShared& s, const uint32_t* big, uint32_t n_big, u64* __restrict__ out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool any_huge = false;
  for (uint32_t g = 0; g < n_big; ++g) any_huge |= (big[g] >> 16) > kWarpCell;
  for (uint32_t g = warp; g < n_big; g += kRankThreads / 32) {
    const uint32_t b0 = big[g] & 0xFFFFu, n = big[g] >> 16;
    if (n > kWarpCell) continue;
    bitonic_sort(s.items + b0, n, lane, 32, [] { __syncwarp(); });
    for (uint32_t i = lane; i < n; i += 32) out[b0 + i] = to_item(s.items[b0 + i]);
  }
  __syncthreads();
  if (any_huge)
    for (uint32_t g = 0; g < n_big; ++g)
      if ((big[g] >> 16) > kWarpCell) rank_by_block(s.items + (big[g] & 0xFFFFu), big[g] >> 16, out + (big[g] & 0xFFFFu));
}

// Ranks m <= kRankItems items whose inv lies in [base, base + span]: spread over kCells equal ranges of inv, about one item per
// cell, then compared with the others of their cell.  `meanwhile` is run once all threads have passed a barrier.
template <class Meanwhile>
__device__ __forceinline__ void rank_buckets(RankShared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out, uint32_t keytop,
                                             Meanwhile&& meanwhile) {
  __shared__ uint32_t s_n_big, s_big[kRankItems / kCompareAll];  // cells beyond kCompareAll
  const int tid = threadIdx.x;
  // the first kHold candidates of a thread stay in registers between counting and placing
  constexpr int kHold = 8;
  u64 it[kHold];
#pragma unroll
  for (int u = 0; u < kHold; ++u)
    if ((uint32_t)tid + u * kRankThreads < m) it[u] = src[tid + u * kRankThreads];
  {
    uint4* cells = reinterpret_cast<uint4*>(s.zero);
    for (uint32_t i = tid; i < kCells / 4 + 1; i += kRankThreads) cells[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) s_n_big = 0;
  }
  __syncthreads();
  const int csh = span < kCells ? 0 : 32 - __clz(span) - (int)kCellBits;  // span >> csh below kCells
  const uint32_t top = keytop - base;
  auto cell_of_key = [&](uint32_t key) -> uint32_t {
    const uint32_t k = (top - key) >> csh;
    return k < kCells ? k : kCells - 1;
  };
#pragma unroll
  for (int u = 0; u < kHold; ++u)
    if ((uint32_t)tid + u * kRankThreads < m) atomicAdd(&s.cell[cell_of_key((uint32_t)(it[u] >> 32))], 1u);
  for (uint32_t i = tid + kHold * kRankThreads; i < m; i += kRankThreads) atomicAdd(&s.cell[cell_of_key((uint32_t)(src[i] >> 32))], 1u);
  __syncthreads();
  scan_cells(s.cell);
  auto put = [&](u64 item) { s.items[atomicAdd(&s.cell[cell_of_key((uint32_t)(item >> 32))], 1u)] = to_value(item); };
#pragma unroll
  for (int u = 0; u < kHold; ++u)
    if ((uint32_t)tid + u * kRankThreads < m) put(it[u]);
  for (uint32_t i = tid + kHold * kRankThreads; i < m; i += kRankThreads) put(src[i]);
  __syncthreads();
  meanwhile();
  for (uint32_t p = tid; p < m; p += kRankThreads) {
    const u64 v = s.items[p];
    uint32_t k = ((uint32_t)(v >> 32) - ~top) >> csh;
    k = k < kCells ? k : kCells - 1;
    const uint32_t e1 = s.cell[k], e0 = (&s.cell[k])[-1];  // the places have advanced to the cells' ends
    uint32_t rank = p;
    if (e1 - e0 > 1) {
      if (e1 - e0 > kCompareAll) {
        if (p == e0) s_big[atomicAdd(&s_n_big, 1u)] = e0 | (e1 - e0) << 16;
        continue;
      }
      rank = e0;
#pragma unroll 1
      for (uint32_t q = e0; q < e1; q += 2) {  // the one behind the cell's last is read, not counted
        const u64 a = s.items[q], b = s.items[q + 1];
        rank += (a < v ? 1u : 0u) + ((q + 1 < e1 && b < v) ? 1u : 0u);
      }
    }
    out[rank] = to_item(v);
  }
  __syncthreads();
  if (s_n_big) rank_big_cells(s, s_big, s_n_big, out);
}

// Tile t of a client: the buckets (sub-buckets after a partition) that start in [t window, (t + 1) window), at most the window
// plus one bucket; of a bucket that a block cannot hold the ranks that lie in the window, whether it starts there or before.
// 79 M candidates of 100 clients: 755 us, 1.7 TB/s of candidates in and out; bound by issue and by the barriers of a tile.
__global__ void __launch_bounds__(kRankThreads, 2)
k_rank(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L, const uint32_t* __restrict__ bin_start_all) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  RankShared& s = *reinterpret_cast<RankShared*>(s_raw);
  // per slot: ticket; first bucket at or behind the window's start and end; where those start; where the bucket before the first starts
  __shared__ uint32_t s_ticket[2], s_bucket[2][2], s_start[2][2], s_before[2];
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (rank_skips(hdr)) return;
  const uint32_t n = batch.n, tickets = hdr->rank_tiles * n, window = hdr->window;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const ClientRank* rank = reinterpret_cast<const ClientRank*>(ws + L.off_rank);
  auto start_of = [&](uint32_t c, const ClientRank& r, uint32_t i) -> uint32_t {
    return r.split ? reinterpret_cast<const uint32_t*>(ws + L.off_sub_start)[(size_t)c * (kRankSubs + 64) + i]
                   : coarse_start(r, bin_start_all + (size_t)c * CVLC_HIST_BINS, i);
  };
  // the buckets of ticket t into slot `to`, a 32-way search by one warp per end of the window (warps 0 and 1 call)
  auto search = [&](uint32_t t, uint32_t to) {
    if (t >= tickets) return;
    const uint32_t tile = t / n, c = t - tile * n;
    const ClientRank r = rank[c];
    const uint32_t n_buckets = r.split ? r.n_coarse << r.sub_bits : r.n_coarse;
    const u64 x = (u64)(tile + warp) * window;
    uint32_t lo = 0, hi = n_buckets;  // the answer lies in [lo, hi]
    while (lo < hi) {
      const uint32_t span = hi - lo;
      const uint32_t i = span <= 32 ? lo + lane : lo + (uint32_t)(((u64)span * lane) / 32);
      const bool behind = i >= hi || start_of(c, r, i) >= x;
      const unsigned hit = __ballot_sync(kFull, behind);
      const int first = hit ? __ffs(hit) - 1 : 32;  // probes before it start in front of x
      const uint32_t new_hi = first < 32 ? __shfl_sync(kFull, i, first) : hi;
      if (first > 0) lo = __shfl_sync(kFull, i, first - 1) + 1;
      hi = new_hi < hi ? new_hi : hi;
    }
    if (lane == 0) {
      s_bucket[to][warp] = lo;
      s_start[to][warp] = lo < n_buckets ? start_of(c, r, lo) : r.n;
      if (warp == 0) s_before[to] = lo > 0 ? start_of(c, r, lo - 1) : 0u;
    }
  };
  if (tid == 0) s_ticket[0] = atomicAdd(&hdr->rank_ticket, 1u);
  __syncthreads();
  if (warp < 2) search(s_ticket[0], 0);
  __syncthreads();
  for (uint32_t slot = 0;; slot ^= 1u) {
    const uint32_t t = s_ticket[slot];
    if (t >= tickets) return;
    if (tid == 0) s_ticket[slot ^ 1u] = atomicAdd(&hdr->rank_ticket, 1u);
    const uint32_t tile = t / n, c = t - tile * n;
    const ClientRank r = rank[c];
    const uint32_t sh = 19 + r.group - (r.split ? r.sub_bits : 0u);
    bool searched = false;
    auto next_search = [&]() {  // behind a barrier that follows the ticket
      if (!searched && warp < 2) search(s_ticket[slot ^ 1u], slot ^ 1u);
      searched = true;
    };
    const u64 x0 = (u64)tile * window, x1 = x0 + window;
    const u64* from = reinterpret_cast<const u64*>(ws + (r.split ? L.off_buf_b : L.off_buf_a)) + (size_t)c * L.capacity;
    u64* into = reinterpret_cast<u64*>(ws + L.off_buf_a) + (size_t)c * L.capacity;
    auto part_of = [&](uint32_t bucket, uint32_t first, uint32_t end) {  // the window's part of a large bucket
      const u64 lo = ((u64)~r.keytop + ((u64)bucket << sh)) << 32, end_high = (u64)~r.keytop + ((u64)(bucket + 1) << sh);
      const u64 hi = end_high >> 32 ? ~0ull : end_high << 32;  // the last bucket may reach below key 0
      const uint32_t a = x0 > first ? (uint32_t)(x0 - first) : 0u;
      const uint32_t b = x1 < end ? (uint32_t)(x1 - first) : end - first;
      rank_part(s, from + first, end - first, lo, hi, a, b, into + first);
    };
    uint32_t b_lo = s_bucket[slot][0], at = s_start[slot][0];
    const uint32_t b_end = s_bucket[slot][1], at_end = s_start[slot][1];
    if (x0 < r.n && r.split && b_lo > 0 && at > x0 && at - s_before[slot] > kRankItems) part_of(b_lo - 1, s_before[slot], at);
    // what is too large for one step ends with a large bucket: that bucket is a step of its own
    while (at < at_end) {
      uint32_t b_hi = b_end, to = at_end;
      if (at_end - at > kRankItems && b_hi - b_lo > 1) {
        --b_hi;
        to = start_of(c, r, b_hi);
      }
      if (to - at > kRankItems) {
        if (r.split) part_of(b_lo, at, to);
      } else if (to > at) {
        rank_buckets(s, from + at, to - at, b_lo << sh, (uint32_t)(((u64)b_hi << sh) - ((u64)b_lo << sh) - 1), into + at, r.keytop, next_search);
      }
      b_lo = b_hi;
      at = to;
    }
    if (!searched) {
      __syncthreads();
      next_search();
    }
    __syncthreads();
  }
}

cudaError_t launch_rank(Batch batch, const EncLayout& L, const unsigned char* plan_ws, unsigned char* ws, cudaStream_t st) {
  static bool attr_done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && !attr_done[dev]) {
    e = cudaFuncSetAttribute(k_rank, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RankShared));
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  auto blocks = [](uint64_t tiles, uint64_t most) -> unsigned { return (unsigned)(tiles < most ? tiles : most); };
  launch_kernel(kKRankSplit, k_rank_split, blocks((L.capacity + kSplitTile - 1) / kSplitTile * L.n, 2 * kNumSM), kRankThreads, kRankSubs * 4, st, true,
                batch, ws, L);
  const uint32_t* bin_start = reinterpret_cast<const uint32_t*>(plan_ws + plan_off_bin_start(L.n));
  launch_kernel(kKRank, k_rank, blocks((L.capacity + 1023) / 1024 * L.n, 2 * kNumSM), kRankThreads, sizeof(RankShared), st, true, batch, ws, L, bin_start);
  return cudaGetLastError();
}

}  // namespace cvlc
