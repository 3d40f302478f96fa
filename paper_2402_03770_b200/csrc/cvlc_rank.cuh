// Ranking of tiles of candidates in shared memory: what the ranking kernel and the kernel that works its left-overs off share.
#pragma once
#include "cvlc_common.cuh"
#include "cvlc_lookback.cuh"

namespace cvlc {

constexpr uint32_t kCellBits = 12, kCells = 1u << kCellBits;  // value ranges a tile is spread over before its items are compared
constexpr uint32_t kCompareAll = 48;    // a cell of up to this many items is ranked by comparing each with all,
constexpr uint32_t kWarpCell = 256;     // one of up to this many is ranked by one warp, a larger one by the block

typedef unsigned long long u64;

// Whether an earlier kernel of the call has reported an error.  Other blocks may set the word while this kernel runs or blocks of
// it start, so one thread reads it and the whole block takes the same branch: warps that part here would leave the others of their
// block at its barriers with work not done.
__device__ __forceinline__ bool block_sees_error(const int32_t* status) {
  __shared__ int s_err;
  if (threadIdx.x == 0) s_err = *reinterpret_cast<const volatile int32_t*>(status);
  __syncthreads();
  return s_err != 0;
}

template <uint32_t ITEMS>
struct RankSharedOf {
  u64 items[ITEMS + 2];       // values (see to_value): all distinct, ordered like the ranks
  uint32_t zero[4];           // cell[-1] = 0: where the first cell starts
  uint32_t cell[kCells];      // counts, then starts, then (after placing) ends of the cells
};
// What a block of the clusters ranks at most, and one of k_rank_rest of equal keys that they leave: a bin of kRankItems and some more.  The fullest bin
// of a spread-out update has about an eighth of the candidates, 0.131 of a normal distribution.  With 8192 in clusters, too, it was cut from 62,400
// records on: one client of 655,000 coordinates at 2.4 bits 49.4 us, 47.0 as kernels of their own, 39.1 with a block for such a bin; seven of them
// 54.0, 59.1 and 43.3.
constexpr uint32_t kRankHold = 9216;
typedef RankSharedOf<kRankHold> RankShared;

// A candidate as a value to rank: the key's complement in the high word, index << 1 | sign in the low word.
__device__ __forceinline__ u64 to_value(u64 item) {
  const uint32_t lo = (uint32_t)item;
  return ((u64)~(uint32_t)(item >> 32) << 32) | (u64)__funnelshift_l(lo, lo, 1);
}
__device__ __forceinline__ u64 to_item(u64 value) {
  const uint32_t lo = (uint32_t)value;
  return ((u64)~(uint32_t)(value >> 32) << 32) | (u64)__funnelshift_r(lo, lo, 1);
}

// f(i, src[i]) for the block's items, sixteen loads of a thread in flight
template <int THREADS, class F>
__device__ __forceinline__ void for_items(const u64* src, uint32_t n, F&& f) {
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 16 * THREADS) {
    u64 v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = i0 + u * THREADS < n ? src[i0 + u * THREADS] : 0ull;
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (i0 + u * THREADS < n) f(i0 + u * THREADS, v[u]);
  }
}

// exclusive scan of the cells in place by the whole block; returns the total
template <int THREADS, uint32_t CELLS = kCells>
__device__ __forceinline__ uint32_t scan_cells(uint32_t* cell) {
  __shared__ uint32_t s_warp[THREADS / 32];
  constexpr int kVec = CELLS / THREADS / 4;
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
  const uint32_t wt = lane < THREADS / 32 ? s_warp[lane] : 0u;
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
template <int THREADS>
__device__ __noinline__ void rank_by_block(u64* items, uint32_t n, u64* __restrict__ out) {
  bitonic_sort(items, n, threadIdx.x, THREADS, [] { __syncthreads(); });
  for (uint32_t i = threadIdx.x; i < n; i += THREADS) out[i] = to_item(items[i]);
  __syncthreads();
}

// The rank of v among the items of its cell, items[e0 .. e1)
__device__ __forceinline__ uint32_t rank_in_cell(const u64* items, u64 v, uint32_t e0, uint32_t e1) {
  uint32_t rank = e0;
#pragma unroll 1
  for (uint32_t q = e0; q < e1; q += 2) {  // the one behind the cell's last is read, not counted
    const u64 a = items[q], b = items[q + 1];
    rank += (a < v ? 1u : 0u) + ((q + 1 < e1 && b < v) ? 1u : 0u);
  }
  return rank;
}

// ---- cells that hold many equal keys and up to kOthers other items --------------------------
// The low words of the equal ones are spread over equal ranges between the least and the largest, grouped by range in the place of
// the high words, and compared with the others of their range.  The other items are set aside and compared with each other.
constexpr uint32_t kOthers = 32, kAside = 0xFFFFFFFFu;
struct Others {
  u64 value[kOthers];
  uint32_t place[kOthers];
  uint32_t n, below;  // how many; of those in front of the equal ones
};

// the key of most items, if there is one
__device__ __forceinline__ uint32_t frequent_key(const uint2* it, uint32_t n) {
  const uint32_t a = it[n / 4].y, b = it[n / 2].y, c = it[n / 4 * 3].y;
  return a == c ? a : b;
}
// sets item p aside; false: no room
__device__ __forceinline__ bool set_aside(Others& o, uint2* it, uint32_t p) {
  const uint32_t i = atomicAdd(&o.n, 1u);
  if (i >= kOthers) return false;
  o.value[i] = (u64)it[p].y << 32 | it[p].x;
  o.place[i] = p;
  it[p].x = kAside;
  return true;
}
__device__ __forceinline__ void put_back(const Others& o, uint2* it, uint32_t i) {
  if (i < (o.n < kOthers ? o.n : kOthers)) it[o.place[i]].x = (uint32_t)o.value[i];
}
// item i of those set aside, by one thread each: counts those in front of the equal ones, writes the item out
__device__ __forceinline__ void rank_other(Others& o, uint32_t i, uint32_t key, uint32_t equal, u64* out) {
  if (i >= o.n) return;
  const u64 v = o.value[i];
  uint32_t rank = v > ((u64)key << 32) ? equal : 0u;  // (one of the same key has the largest low word there is)
  if (rank == 0) atomicAdd(&o.below, 1u);
  for (uint32_t q = 0; q < o.n; ++q) rank += o.value[q] < v ? 1u : 0u;
  out[rank] = to_item(v);
}

// Ranks items[0 .. n), n <= kRankHold, and writes them out; by the whole block.  False, and nothing done, if too many keys differ or
// a range has too many items.
template <int THREADS, uint32_t BITS>
__device__ __noinline__ bool rank_equal(RankShared& s, u64* items, uint32_t n, u64* __restrict__ out) {
  __shared__ uint32_t s_least, s_most, s_no;
  __shared__ Others s_others;
  const int tid = threadIdx.x, lane = tid & 31;
  uint2* it = reinterpret_cast<uint2*>(items);
  const uint32_t key = frequent_key(it, n);
  if (tid == 0) {
    s_least = 0xFFFFFFFFu;
    s_most = s_no = s_others.n = s_others.below = 0;
  }
  {
    uint4* cells = reinterpret_cast<uint4*>(s.zero);
    for (uint32_t i = tid; i < (1u << BITS) / 4 + 1; i += THREADS) cells[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  uint32_t least = 0xFFFFFFFFu, most = 0;
#pragma unroll 4
  for (uint32_t p = tid; p < n; p += THREADS) {
    const uint2 v = it[p];
    if (v.y != key || v.x == kAside) {
      if (!set_aside(s_others, it, p)) s_no = 1;
      continue;
    }
    least = min(least, v.x);
    most = max(most, v.x);
  }
  least = __reduce_min_sync(kFull, least);
  most = __reduce_max_sync(kFull, most);
  if (lane == 0) {
    atomicMin(&s_least, least);
    atomicMax(&s_most, most);
  }
  __syncthreads();
  least = s_least;
  const uint32_t span = s_most > least ? s_most - least : 0u;
  const int sh = span < (1u << BITS) ? 0 : 32 - __clz(span) - (int)BITS;
  if (!s_no) {
    bool crowded = false;
    for (uint32_t p0 = tid; p0 < n; p0 += 4 * THREADS) {
      uint32_t x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = p0 + u * THREADS < n ? it[p0 + u * THREADS].x : kAside;
#pragma unroll
      for (int u = 0; u < 4; ++u) crowded |= x[u] != kAside && atomicAdd(&s.cell[(x[u] - least) >> sh], 1u) >= kCompareAll;
    }
    if (crowded) s_no = 1;
  }
  __syncthreads();
  if (s_no) {
    put_back(s_others, it, tid);
    __syncthreads();
    return false;
  }
  scan_cells<THREADS, 1u << BITS>(s.cell);
  const uint32_t equal = n - s_others.n;
  rank_other(s_others, tid, key, equal, out);
  for (uint32_t p0 = tid; p0 < n; p0 += 4 * THREADS) {
    uint32_t x[4], to[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = p0 + u * THREADS < n ? it[p0 + u * THREADS].x : kAside;
#pragma unroll
    for (int u = 0; u < 4; ++u) to[u] = x[u] != kAside ? atomicAdd(&s.cell[(x[u] - least) >> sh], 1u) : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (x[u] != kAside) it[to[u]].y = x[u];
  }
  __syncthreads();
  u64* __restrict__ to = out + s_others.below;
  for (uint32_t p = tid; p < equal; p += THREADS) {
    const uint32_t x = it[p].y, k = (x - least) >> sh, e1 = s.cell[k], e0 = (&s.cell[k])[-1];
    uint32_t rank = e0;
#pragma unroll 1
    for (uint32_t q = e0; q < e1; ++q) rank += it[q].y < x ? 1u : 0u;
    to[rank] = to_item((u64)key << 32 | x);
  }
  __syncthreads();
  return true;
}

// the same by one warp with kWarpCells ranges (one item at a time, us: fp16 values, 10 clients of 300,000 coordinates at 4 bits 69 -> 66, one of 600,000
// at 2.5 bits 67.8 -> 67.2, 20 of 1.2 M on a grid of 24 steps per deviation 205.7 -> 201.5)
constexpr uint32_t kWarpCellBits = 8, kWarpCells = 1u << kWarpCellBits;
template <int THREADS>
__device__ __forceinline__ bool rank_equal_by_warp(uint32_t* cell, u64* items, uint32_t n, u64* __restrict__ out) {
  static_assert(kWarpCells * (THREADS / 32) <= kCells && kWarpCells == 256, "the warps share the block's cells; eight per lane");
  __shared__ Others s_others[THREADS / 32];
  Others& others = s_others[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  uint2* it = reinterpret_cast<uint2*>(items);
  uint4* mine = reinterpret_cast<uint4*>(cell) + 2 * lane;
  mine[0] = mine[1] = make_uint4(0u, 0u, 0u, 0u);
  const uint32_t key = frequent_key(it, n);
  if (lane == 0) others.n = others.below = 0;
  __syncwarp();
  uint32_t least = 0xFFFFFFFFu, most = 0;
  bool no = false;
  for (uint32_t p0 = lane; p0 < n; p0 += 128) {  // four at a time, here and below: their loads and additions side by side
    uint2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = p0 + 32 * u < n ? it[p0 + 32 * u] : make_uint2(0xFFFFFFFEu, key);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (p0 + 32 * u >= n) continue;
      if (v[u].y != key || v[u].x == kAside) {
        no |= !set_aside(others, it, p0 + 32 * u);
        continue;
      }
      least = min(least, v[u].x);
      most = max(most, v[u].x);
    }
  }
  __syncwarp();
  least = __reduce_min_sync(kFull, least);
  most = __reduce_max_sync(kFull, most);
  const uint32_t span = most > least ? most - least : 0u;
  const int sh = span < kWarpCells ? 0 : 32 - __clz(span) - (int)kWarpCellBits;
  if (!__any_sync(kFull, no)) {
    for (uint32_t p0 = lane; p0 < n; p0 += 128) {
      uint32_t x[4], before[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = p0 + 32 * u < n ? it[p0 + 32 * u].x : kAside;
#pragma unroll
      for (int u = 0; u < 4; ++u) before[u] = x[u] != kAside ? atomicAdd(&cell[(x[u] - least) >> sh], 1u) : 0u;
#pragma unroll
      for (int u = 0; u < 4; ++u) no |= before[u] >= kCompareAll;
    }
  }
  if (__any_sync(kFull, no)) {
    put_back(others, it, lane);
    __syncwarp();
    return false;
  }
  __syncwarp();
  const uint4 c[2] = {mine[0], mine[1]};
  const uint32_t sum = c[0].x + c[0].y + c[0].z + c[0].w + c[1].x + c[1].y + c[1].z + c[1].w;
  uint32_t run = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, run, off);
    if (lane >= off) run += o;
  }
  run -= sum;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint4 e;
    e.x = run;
    e.y = e.x + c[i].x;
    e.z = e.y + c[i].y;
    e.w = e.z + c[i].z;
    run = e.w + c[i].w;
    mine[i] = e;
  }
  const uint32_t equal = n - others.n;
  rank_other(others, lane, key, equal, out);
  __syncwarp();
  for (uint32_t p0 = lane; p0 < n; p0 += 128) {
    uint32_t x[4], to[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = p0 + 32 * u < n ? it[p0 + 32 * u].x : kAside;
#pragma unroll
    for (int u = 0; u < 4; ++u) to[u] = x[u] != kAside ? atomicAdd(&cell[(x[u] - least) >> sh], 1u) : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (x[u] != kAside) it[to[u]].y = x[u];
  }
  __syncwarp();
  u64* __restrict__ to = out + others.below;
  for (uint32_t p = lane; p < equal; p += 32) {
    const uint32_t x = it[p].y, k = (x - least) >> sh, e0 = k ? cell[k - 1] : 0u, e1 = cell[k];
    uint32_t rank = e0;
#pragma unroll 1
    for (uint32_t q = e0; q < e1; ++q) rank += it[q].y < x ? 1u : 0u;
    to[rank] = to_item((u64)key << 32 | x);
  }
  __syncwarp();
  return true;
}

// Ranks the n <= kRankHold items of a cell of many keys and writes them out (in their place, too); by the whole block.  They are
// spread over equal ranges of (key, index) between the least and the largest of each.  False, and nothing done, if a range has too many.
template <int THREADS>
__device__ __noinline__ bool rank_spread(RankShared& s, const u64* at, uint32_t n, u64* out) {
  __shared__ uint32_t s_least[2], s_most[2], s_no;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 2) {
    s_least[tid] = 0xFFFFFFFFu;
    s_most[tid] = 0;
  }
  if (tid == 0) s_no = 0;
  {
    uint4* cells = reinterpret_cast<uint4*>(s.zero);
    for (uint32_t i = tid; i < kCells / 4 + 1; i += THREADS) cells[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  uint32_t least[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, most[2] = {0u, 0u};
  for_items<THREADS>(at, n, [&](uint32_t, u64 item) {
    const u64 v = to_value(item);
    least[0] = min(least[0], (uint32_t)v);
    most[0] = max(most[0], (uint32_t)v);
    least[1] = min(least[1], (uint32_t)(v >> 32));
    most[1] = max(most[1], (uint32_t)(v >> 32));
  });
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    least[h] = __reduce_min_sync(kFull, least[h]);
    most[h] = __reduce_max_sync(kFull, most[h]);
    if (lane == 0) {
      atomicMin(&s_least[h], least[h]);
      atomicMax(&s_most[h], most[h]);
    }
  }
  __syncthreads();
  const uint32_t lo0 = s_least[0], hi0 = s_least[1];
  const u64 width = (u64)(s_most[0] - lo0) + 1, largest = (u64)(s_most[1] - hi0) * width + (width - 1);
  const int sh = largest < kCells ? 0 : 64 - __clzll((long long)largest) - (int)kCellBits;
  auto cell_of = [&](u64 v) -> uint32_t { return (uint32_t)(((u64)((uint32_t)(v >> 32) - hi0) * width + ((uint32_t)v - lo0)) >> sh); };
  for_items<THREADS>(at, n, [&](uint32_t, u64 item) {
    if (atomicAdd(&s.cell[cell_of(to_value(item))], 1u) >= kCompareAll) s_no = 1;
  });
  __syncthreads();
  if (s_no) {
    __syncthreads();
    return false;
  }
  scan_cells<THREADS>(s.cell);
  for_items<THREADS>(at, n, [&](uint32_t, u64 item) {
    const u64 v = to_value(item);
    s.items[atomicAdd(&s.cell[cell_of(v)], 1u)] = v;
  });
  __syncthreads();
  for (uint32_t p = tid; p < n; p += THREADS) {
    const u64 v = s.items[p];
    const uint32_t k = cell_of(v);
    out[rank_in_cell(s.items, v, (&s.cell[k])[-1], s.cell[k])] = to_item(v);
  }
  __syncthreads();
  return true;
}

// Ranks n <= kRankHold items, most of them of one key or nearly equal, and writes them out (in their place, too); by the whole block
template <int THREADS>
__device__ __noinline__ void rank_cell(RankShared& s, const u64* at, uint32_t n, u64* out) {
  for (int attempt = 0; attempt < 3; ++attempt) {
    if (attempt != 1) {
      for_items<THREADS>(at, n, [&](uint32_t i, u64 item) { s.items[i] = to_value(item); });
      __syncthreads();
    }
    if (attempt == 0) {
      if (n <= kCells / 2 ? rank_equal<THREADS, kCellBits - 1>(s, s.items, n, out) : rank_equal<THREADS, kCellBits>(s, s.items, n, out)) return;
    } else if (attempt == 1 && rank_spread<THREADS>(s, at, n, out)) {
      return;
    }
  }
  rank_by_block<THREADS>(s.items, n, out);
}

// Ranks m <= kRankItems items whose inv lies in [base, base + span]: spread over kCells equal ranges of inv, about one item per
// cell, then compared with the others of their cell.  Cells of more than kCompareAll items are left to `later`, their items in any
// order in their place.  `meanwhile` is run once all threads have passed a barrier.
template <int THREADS, int HOLD = 8, class Shared, class Later, class Meanwhile>
__device__ __forceinline__ void rank_buckets(Shared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out, uint32_t keytop,
                                             Later&& later, Meanwhile&& meanwhile) {
  const int tid = threadIdx.x;
  // the first HOLD candidates of a thread stay in registers between counting and placing
  u64 it[HOLD];
#pragma unroll
  for (int u = 0; u < HOLD; ++u)
    if ((uint32_t)tid + u * THREADS < m) it[u] = src[tid + u * THREADS];
  {
    uint4* cells = reinterpret_cast<uint4*>(s.zero);
    for (uint32_t i = tid; i < kCells / 4 + 1; i += THREADS) cells[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();
  const int csh = span < kCells ? 0 : 32 - __clz(span) - (int)kCellBits;  // span >> csh below kCells
  const uint32_t top = keytop - base;
  auto cell_of_key = [&](uint32_t key) -> uint32_t {
    const uint32_t k = (top - key) >> csh;
    return k < kCells ? k : kCells - 1;
  };
#pragma unroll
  for (int u = 0; u < HOLD; ++u)
    if ((uint32_t)tid + u * THREADS < m) atomicAdd(&s.cell[cell_of_key((uint32_t)(it[u] >> 32))], 1u);
  for (uint32_t i = tid + HOLD * THREADS; i < m; i += THREADS) atomicAdd(&s.cell[cell_of_key((uint32_t)(src[i] >> 32))], 1u);
  __syncthreads();
  scan_cells<THREADS>(s.cell);
  auto put = [&](u64 item) { s.items[atomicAdd(&s.cell[cell_of_key((uint32_t)(item >> 32))], 1u)] = to_value(item); };
#pragma unroll
  for (int u = 0; u < HOLD; ++u)
    if ((uint32_t)tid + u * THREADS < m) put(it[u]);
  for (uint32_t i = tid + HOLD * THREADS; i < m; i += THREADS) put(src[i]);
  __syncthreads();
  meanwhile();
  for (uint32_t p = tid; p < m; p += THREADS) {
    const u64 v = s.items[p];
    uint32_t k = ((uint32_t)(v >> 32) - ~top) >> csh;
    k = k < kCells ? k : kCells - 1;
    const uint32_t e1 = s.cell[k], e0 = (&s.cell[k])[-1];  // the places have advanced to the cells' ends
    uint32_t rank = p;
    if (e1 - e0 > 1) {
      if (e1 - e0 > kCompareAll) {
        if (p == e0) later(out + e0, e1 - e0);
      } else {
        rank = rank_in_cell(s.items, v, e0, e1);
      }
    }
    out[rank] = to_item(v);
  }
  __syncthreads();
}

// A tile: the buckets (sub-buckets after a partition) of a client that start in [tile window, (tile + 1) window), at most the
// window plus one bucket.  The last may be one that a block cannot hold: it is on the list of large buckets and ranked from there.
// What a block needs to know of one is found by two warps and kept in shared memory.
struct RankTile {
  uint32_t ticket;
  uint32_t bucket[2], start[2];  // first bucket at or behind the window's start and end; where those start
  uint32_t sh, keytop;
  const u64* from;               // the client's candidates by buckets, and in order
  u64* into;
};

struct RankArgs {
  const ClientRank* rank;
  const uint32_t *sub_start, *bin_start;
  u64 *buf_a, *buf_b;
  ulonglong2* list[2];  // left over: cells for a warp; cells for a block and tiles of more than a block holds
  BigBucket* big;
  u64* piece;           // bucket of the round << 32 | piece of it
  u64* splitter;
  uint32_t *part_count, *part_start, *base;
  BigPart* part;
  size_t capacity, big_room, piece_room;  // the latter two per round
  uint32_t n, tickets, window, limit;
};
__device__ __forceinline__ RankArgs rank_args(unsigned char* ws, const EncLayout& L, const uint32_t* bin_start, const EncHeader* hdr, uint32_t n,
                                              uint32_t blocks, uint32_t window) {
  RankArgs a;
  a.rank = reinterpret_cast<const ClientRank*>(ws + L.off_rank);
  a.sub_start = reinterpret_cast<const uint32_t*>(ws + L.off_sub_start);
  a.bin_start = bin_start;
  a.buf_a = reinterpret_cast<u64*>(ws + L.off_buf_a);
  a.buf_b = reinterpret_cast<u64*>(ws + L.off_buf_b);
  a.list[0] = reinterpret_cast<ulonglong2*>(ws + L.off_list[0]);
  a.list[1] = reinterpret_cast<ulonglong2*>(ws + L.off_list[1]);
  a.big = reinterpret_cast<BigBucket*>(ws + L.off_big);
  a.piece = reinterpret_cast<u64*>(ws + L.off_piece);
  a.splitter = reinterpret_cast<u64*>(ws + L.off_splitter);
  a.part_count = reinterpret_cast<uint32_t*>(ws + L.off_part_count);
  a.part_start = reinterpret_cast<uint32_t*>(ws + L.off_part_start);
  a.base = reinterpret_cast<uint32_t*>(ws + L.off_base);
  a.part = reinterpret_cast<BigPart*>(ws + L.off_part);
  a.capacity = (size_t)L.capacity;
  a.big_room = (size_t)n * a.capacity / kRankItems + 1;
  a.piece_room = (size_t)n * a.capacity / kBigPiece + a.big_room;
  a.n = n;
  a.window = rank_window(hdr->most, n, blocks, window);
  a.tickets = (hdr->most + a.window - 1) / a.window * n;
  a.limit = hdr->limit;
  return a;
}
__device__ __forceinline__ uint32_t bucket_start(const RankArgs& a, uint32_t c, const ClientRank& r, uint32_t i) {
  return r.split ? a.sub_start[(size_t)c * (kRankSubs + 64) + i] : coarse_start(r, a.bin_start + (size_t)c * CVLC_HIST_BINS, i);
}
// the buckets of the tile's ticket, a 32-way search by one warp per end of the window (warps 0 and 1 call)
__device__ __forceinline__ void find_tile(RankTile& T, const RankArgs& a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (T.ticket >= a.tickets) return;
  const uint32_t tile = T.ticket / a.n, c = T.ticket - tile * a.n;
  const ClientRank r = a.rank[c];
  const uint32_t n_buckets = r.split ? r.n_coarse << r.sub_bits : r.n_coarse;
  const u64 x = (u64)(tile + warp) * a.window;
  uint32_t lo = 0, hi = n_buckets;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const uint32_t span = hi - lo;
    const uint32_t i = span <= 32 ? lo + lane : lo + (uint32_t)(((u64)span * lane) / 32);
    const bool behind = i >= hi || bucket_start(a, c, r, i) >= x;
    const unsigned hit = __ballot_sync(kFull, behind);
    const int first = hit ? __ffs(hit) - 1 : 32;  // probes before it start in front of x
    const uint32_t new_hi = first < 32 ? __shfl_sync(kFull, i, first) : hi;
    if (first > 0) lo = __shfl_sync(kFull, i, first - 1) + 1;
    hi = new_hi < hi ? new_hi : hi;
  }
  if (lane == 0) {
    T.bucket[warp] = lo;
    T.start[warp] = lo < n_buckets ? bucket_start(a, c, r, lo) : r.n;
    if (warp == 0) {
      T.sh = 19 + r.group - (r.split ? r.sub_bits : 0u);
      T.keytop = r.keytop;
      T.from = (r.split ? a.buf_b : a.buf_a) + (size_t)c * a.capacity;
      T.into = a.buf_a + (size_t)c * a.capacity;
    }
  }
}

// ---- buckets that a block cannot hold ---------------------------------------------------------
// Equal keys mostly: a layer's clipped values, updates that were rounded to 16 or 8 bits.  In rounds: a bucket's splitters are taken
// from a sample of its values, its pieces counted over the parts between them, the parts' places summed up by the block that
// counts the bucket's last piece, and the pieces placed there.  Parts that a block can hold are ranked; larger ones are the next
// round's buckets (a bucket of more than kBigParts parts).  Values are distinct, so equal keys are split by their indices and no
// distribution is special.  A step's items are drawn by ticket, and a block waits for the step before when no item of that is left: the
// blocks it waits for are running.
// Smaller ones are split by one block each, all steps at once (up to 8192 / 16384 / 32768 / 65536 candidates: 10 clients of 5 M
// coordinates in 16 bits 111 / 72 / 73 / 72 us, one of 100 M with every seventh layer on a grid 321 / 300 / 292 / 378).
// A candidate is read three times and moved twice, whatever the bucket's size, and not moved where its part is never sent.  Two
// blocks per SM: bound by the latencies of a piece (12 us for 8192 candidates, most of them the setting up) and of the steps one
// behind the other (68 us for one bucket of 100,000).  The kernel's time for 4 clients of 50 M coordinates in 16 bits (13.5 M
// candidates, buckets of 40,000): 324 us; 4 of 50 M on a grid of 24 steps per deviation: 338; one million equal keys in one client of
// 11.2 M: 108; 10 of 5 M with 250,000 equal keys each: 118.  With every tile ranking its window of a bucket, reading all of it, and
// digit passes over all candidates for buckets beyond 262,144: 1212, 2925, 308 and 1200.

__device__ __forceinline__ uint32_t big_parts(uint32_t m) { return m / kBigPart + 1 < kBigParts ? m / kBigPart + 1 : kBigParts; }
// where a bucket's entries in the tables of parts begin: of its own candidates' slots
__device__ __forceinline__ u64 big_slot(u64 pos) { return (pos + kBigSlot - 1) / kBigSlot; }
static_assert(kRankItems / kBigSlot - 1 > kRankItems / kBigPart + 1 && kBigPart > 2 * kBigSlot, "a bucket has a slot for every part");
static_assert(kBigParts <= kRankItems / 8 && 2 * kBigParts <= kCells, "splitters and counts in shared memory, eight samples for a part");

// a bucket that a block of the ranking cannot hold: its sort keys lie in [lo, end)
static __device__ __noinline__ void list_bucket(EncHeader* hdr, unsigned char* ws, const EncLayout& L, uint32_t c, uint32_t keytop, u64 lo, u64 end,
                                                uint32_t start, uint32_t m) {
  const u64 from = (u64)~keytop + lo, to = (u64)~keytop + end;  // the last bucket may reach below key 0
  const bool own = m <= kBigOwn;
  if (!own) atomicAdd(&hdr->big[0].slots, m / kBigSlot);
  const size_t row = own ? kBigOwnRow * ((size_t)L.n * L.capacity / kRankItems + 1) : 0;
  reinterpret_cast<BigBucket*>(ws + L.off_big)[row + atomicAdd(own ? &hdr->own_n : &hdr->big[0].n, 1u)] =
      BigBucket{(u64)c * L.capacity + start, from << 32, to >> 32 ? ~0ull : to << 32, ~0ull, m, big_parts(m), 0u, 0u};
}

// Waits (bounded) until *done reaches `want`.  False: the wait ran out.  By the whole block.
__device__ __forceinline__ bool block_waits(const uint32_t* done, uint32_t want, int32_t* status) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    int polls = 0;
    s_ok = 1;
    while (*reinterpret_cast<const volatile uint32_t*>(done) < want) {
      if (++polls > kMaxPolls) {
        set_status(status, CVLC_ERR_DEVICE_TIMEOUT);
        s_ok = 0;
        break;
      }
      __nanosleep(polls > 64 ? 256 : 32);
    }
    __threadfence();
  }
  __syncthreads();
  const bool ok = s_ok != 0;
  __syncthreads();
  return ok;
}
// counts an item of a step as finished, behind all the block's writes; by the whole block
__device__ __forceinline__ void block_done(uint32_t* done) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(done, 1u);
  }
}
// the next item of a step, the same for all threads of the block
__device__ __forceinline__ uint32_t block_takes(uint32_t* next) {
  __shared__ uint32_t s_item;
  __syncthreads();
  if (threadIdx.x == 0) s_item = atomicAdd(next, 1u);
  __syncthreads();
  return s_item;
}
// Candidates of a round's pieces: enough for some pieces a block, and the more the less the setting up of each counts
// (20 buckets of 1.2 M: the round's counting 120 us with pieces of 8192)
__device__ __forceinline__ uint32_t big_piece_size(const BigRound& R) {
  const uint32_t slots = *reinterpret_cast<const volatile uint32_t*>(&R.slots);
  uint32_t size = kBigPiece;
  while (size < 8 * kBigPiece && slots / (2 * size / kBigSlot) >= 4 * kNumSM) size *= 2;
  return size;
}
// a bucket as another block has left it
__device__ __forceinline__ BigBucket big_bucket(const RankArgs& a, int round, uint32_t i) {
  const volatile BigBucket* b = a.big + (size_t)round * a.big_room + i;
  return BigBucket{b->pos, b->from, b->to, b->last, b->m, b->parts, 0u, 0u};
}
__device__ __forceinline__ const u64* big_source(const RankArgs& a, int round, u64 pos) { return (round & 1 ? a.buf_a : a.buf_b) + pos; }
__device__ __forceinline__ u64* big_target(const RankArgs& a, int round, u64 pos) { return (round & 1 ? a.buf_b : a.buf_a) + pos; }

// A cell of up to kWarpCell items, whose values are `mine`, by one warp of the block; cell: kWarpCells counters of its own
template <int THREADS>
__device__ __forceinline__ void rank_values_by_warp(uint32_t* cell, u64* mine, uint32_t m, u64* at) {
  const int lane = threadIdx.x & 31;
  if (!rank_equal_by_warp<THREADS>(cell, mine, m, at)) {
    bitonic_sort(mine, m, lane, 32, [] { __syncwarp(); });
    for (uint32_t i = lane; i < m; i += 32) at[i] = to_item(mine[i]);
    __syncwarp();
  }
}
template <int THREADS>
__device__ __forceinline__ void rank_cell_by_warp(RankShared& s, u64* at, uint32_t m) {
  static_assert(kWarpCell * (THREADS / 32) <= kRankItems, "room for every warp's cell");
  u64* mine = s.items + (threadIdx.x >> 5) * kWarpCell;
  for (uint32_t i = threadIdx.x & 31; i < m; i += 32) mine[i] = to_value(at[i]);
  __syncwarp();
  rank_values_by_warp<THREADS>(s.cell + (threadIdx.x >> 5) * kWarpCells, mine, m, at);
}

// Ranks m <= kRankHold items in [base, base + span] of inv, but for the cells of more than kCompareAll, whose places and items go to `cells`; returns
// how many.  By the whole block.
template <int THREADS>
__device__ __forceinline__ uint32_t rank_but_cells(RankShared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out, uint32_t keytop,
                                                   uint32_t (&cells)[kRankHold / kCompareAll]) {
  __shared__ uint32_t s_n;
  if (threadIdx.x == 0) s_n = 0;
  rank_buckets<THREADS>(s, src, m, base, span, out, keytop,
                        [&](u64* where, uint32_t items) { cells[atomicAdd(&s_n, 1u)] = (uint32_t)(where - out) | items << 16; }, [] {});
  return s_n;
}
// ... with those cells, by the block one after the other.  (Those of up to 256 by its warps side by side, as in clusters: one client of 11.2 M
// coordinates in 255 steps 163.5 -> 167.6 us, on a grid of 24 steps per deviation 163.8 -> 169.7, one of 5 M 122.0 -> 126.5.)
template <int THREADS>
__device__ __noinline__ void rank_with_cells(RankShared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out, uint32_t keytop) {
  __shared__ uint32_t s_cell[kRankHold / kCompareAll];
  const uint32_t n = rank_but_cells<THREADS>(s, src, m, base, span, out, keytop, s_cell);
  for (uint32_t g = 0; g < n; ++g) {
    u64* at = out + (s_cell[g] & 0xFFFFu);
    rank_cell<THREADS>(s, at, s_cell[g] >> 16, at);
  }
  __syncthreads();
}
// ... by its warps; those that a warp cannot rank by k_rank_rest, by all its blocks.  The items are client c's from rank `start` on; they come from either
// buffer and go to the first.
template <int THREADS>
__device__ __noinline__ void rank_and_leave(RankShared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, uint32_t keytop, unsigned char* ws,
                                            const EncLayout& L, uint32_t c, uint32_t start) {
  __shared__ uint32_t s_cell[kRankHold / kCompareAll];
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  u64* buf_a = reinterpret_cast<u64*>(ws + L.off_buf_a);
  u64* out = buf_a + (size_t)c * L.capacity + start;
  ulonglong2* list = reinterpret_cast<ulonglong2*>(ws + L.off_list[1]);
  const uint32_t n = rank_but_cells<THREADS>(s, src, m, base, span, out, keytop, s_cell);
  for (uint32_t g = threadIdx.x >> 5; g < n; g += THREADS / 32) {
    const uint32_t first = s_cell[g] & 0xFFFFu, items = s_cell[g] >> 16;
    if (items <= kWarpCell) rank_values_by_warp<THREADS>(s.cell + (threadIdx.x >> 5) * kWarpCells, s.items + first, items, out + first);
    else if ((threadIdx.x & 31) == 0) list[atomicAdd(&hdr->list_n[1], 1u)] = make_ulonglong2((u64)(out + first - buf_a), items);
  }
  __syncthreads();
}

// Ranks n <= kRankItems items whose keys lie between two, the larger one first; by the whole block
template <int THREADS>
__device__ __forceinline__ void rank_keys(RankShared& s, const u64* src, uint32_t n, uint32_t first_key, uint32_t last_key, u64* out) {
  if (first_key == last_key) rank_cell<THREADS>(s, src, n, out);
  else rank_with_cells<THREADS>(s, src, n, 0u, first_key - last_key, out, first_key);
}

// What a block needs to find a value's part, the number of splitters not above it: the bucket's splitters in s.items, and, where the
// values between the first and the last of them are cut into equal cells, how many lie in the cells before each, in s.cell behind
// the parts' counts.  Equal keys differ by their indices, which are spread about evenly: one cell, one splitter or two.  (A search
// among all splitters, ten steps, took 1.6 times as long.)
constexpr uint32_t kBigCells = 2048;
static_assert(kBigRounds == 3, "the second round alone ends in the second buffer");
struct BigSearch {
  u64 first, last;    // splitters (of a bucket with at least two parts)
  int shift;          // bits of a cell
  uint32_t steps;     // of the search among a cell's splitters
};
static_assert(2 * kBigParts + kBigCells <= kCells, "the cells' place");
// ... brought into shared memory; the parts' counts are cleared
template <int THREADS>
__device__ __forceinline__ BigSearch big_prepare(RankShared& s, const RankArgs& a, const BigBucket& b) {
  __shared__ uint32_t s_most;
  const u64* splitter = a.splitter + big_slot(b.pos);
  const uint32_t n = b.parts - 1;
  uint32_t* cells = s.cell + 2 * kBigParts;
  for (uint32_t p = threadIdx.x; p < n; p += THREADS) s.items[p] = __ldcg(splitter + p);
  for (uint32_t p = threadIdx.x; p < kBigParts; p += THREADS) s.cell[p] = 0;
  for (uint32_t p = threadIdx.x; p < kBigCells; p += THREADS) cells[p] = 0;
  if (threadIdx.x == 0) s_most = 0;
  __syncthreads();
  BigSearch h;
  h.first = s.items[0];
  h.last = s.items[n - 1];
  const u64 span = h.last - h.first;
  h.shift = span < kBigCells ? 0 : 64 - __clzll((long long)span) - 11;  // span >> shift below kBigCells
  static_assert(kBigCells == 1u << 11, "bits of a cell's number");
  for (uint32_t p = threadIdx.x; p < n; p += THREADS) atomicMax(&s_most, atomicAdd(cells + (uint32_t)((s.items[p] - h.first) >> h.shift), 1u) + 1);
  __syncthreads();
  h.steps = 32 - __clz(s_most);
  scan_cells<THREADS, kBigCells>(cells);
  return h;
}
// f(part, value) for the values up to `last` of the piece of bucket b that begins at `first`
template <int THREADS, class F>
__device__ __forceinline__ void big_piece(const RankShared& s, const BigSearch& h, const BigBucket& b, const u64* src, uint32_t first, uint32_t size, u64 last,
                                          F&& f) {
  const uint32_t m = b.m - first < size ? b.m - first : size, n = b.parts - 1;
  const uint32_t* cells = s.cell + 2 * kBigParts;
  for (uint32_t i0 = threadIdx.x; i0 < m; i0 += 8 * THREADS) {  // eight at a time: their loads, then their searches side by side
    u64 v[8];
    uint32_t p[8], e[8];
    bool any = false;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = i0 + u * THREADS < m ? to_value(src[first + i0 + u * THREADS]) : ~0ull;
      any |= v[u] <= last;
    }
    if (!__any_sync(__activemask(), any)) continue;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const u64 in = v[u] < h.first ? h.first : (v[u] > h.last ? h.last : v[u]);
      const uint32_t c = (uint32_t)((in - h.first) >> h.shift);
      p[u] = cells[c];
      e[u] = c + 1 < kBigCells ? cells[c + 1] : n;
    }
    for (uint32_t step = 0; step < h.steps; ++step) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (p[u] < e[u]) {
          const uint32_t mid = (p[u] + e[u]) >> 1;
          if (s.items[mid] <= v[u]) p[u] = mid + 1;
          else e[u] = mid;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u * THREADS < m && v[u] <= last) f(p[u], v[u]);
  }
}

// Where the parts of bucket b, the i-th of the round, begin: their counts are in s.cell (at least kBigParts, zeros behind the last),
// which then holds the starts.  The parts go to their lists.
template <int THREADS>
__device__ __forceinline__ void big_bounds(RankShared& s, EncHeader* hdr, const RankArgs& a, int round, uint32_t i, const BigBucket& b) {
  const u64 slot = big_slot(b.pos);
  for (uint32_t p = kBigParts + threadIdx.x; p < 2 * kBigParts; p += THREADS) s.cell[p] = 0u;
  __syncthreads();
  scan_cells<THREADS, 2 * kBigParts>(s.cell);
  for (uint32_t p = threadIdx.x; p < b.parts; p += THREADS) {
    const uint32_t start = s.cell[p], m = (p + 1 < b.parts ? s.cell[p + 1] : b.m) - start;
    const bool sent = (b.pos + start) % a.capacity < a.limit;
    a.part_start[slot + p] = start;
    if (!sent && p && (b.pos + s.cell[p - 1]) % a.capacity < a.limit) a.big[(size_t)round * a.big_room + i].last = s.items[p - 1] - 1;
    if (m == 0 || !sent) continue;
    const u64 from = p ? s.items[p - 1] : b.from, to = p + 1 < b.parts ? s.items[p] : b.to;
    if (m > kRankItems && round + 1 < kBigRounds) {
      atomicAdd(&hdr->big[round + 1].slots, m / kBigSlot);
      a.big[(size_t)(round + 1) * a.big_room + atomicAdd(&hdr->big[round + 1].n, 1u)] = BigBucket{b.pos + start, from, to, ~0ull, m, big_parts(m), 0u, 0u};
    } else {
      a.part[atomicAdd(&hdr->part_n, 1u)] = BigPart{b.pos + start, m, round == 1 ? 1u : 0u, ~(uint32_t)(from >> 32), ~(uint32_t)((to - 1) >> 32)};
    }
  }
}

// Step 1: the splitters of a bucket.  A sample of 16 candidates for a part (256 at least), one from every equal stretch of the bucket at
// a scattered place of it, since neighbours lie there in the order of the update.  It is ranked where the bucket's parts will lie
// (8192 of equal keys sorted in shared memory instead: 165 us).
template <int THREADS>
__device__ __forceinline__ void big_splitters(RankShared& s, const RankArgs& a, const BigBucket& b, const u64* src, u64* sample) {
  uint32_t samples = 256;
  while (samples < kRankItems && samples < 16 * b.parts) samples <<= 1;
  for (uint32_t t = threadIdx.x; t < samples; t += THREADS) {
    const uint32_t at = (uint32_t)((u64)t * b.m / samples), width = (uint32_t)((u64)(t + 1) * b.m / samples) - at;
    sample[t] = src[at + (uint32_t)(((u64)(t * 2654435761u) * width) >> 32)];
  }
  __syncthreads();
  rank_keys<THREADS>(s, sample, samples, ~(uint32_t)(b.from >> 32), ~(uint32_t)((b.to - 1) >> 32), sample);
  const u64 slot = big_slot(b.pos);
  for (uint32_t p = threadIdx.x; p < b.parts; p += THREADS) {
    if (p) a.splitter[slot + p - 1] = to_value(sample[(u64)p * samples / b.parts]);
    a.part_count[slot + p] = 0;
  }
}
// ... of the round's buckets, and their pieces
template <int THREADS>
__device__ __noinline__ void big_sample(RankShared& s, EncHeader* hdr, const RankArgs& a, int round) {
  __shared__ uint32_t s_first;
  BigRound& R = hdr->big[round];
  const uint32_t piece_size = big_piece_size(R);
  const uint32_t n = *reinterpret_cast<const volatile uint32_t*>(&R.n);
  while (true) {
    const uint32_t i = block_takes(&R.next_sample);
    if (i >= n) return;
    const BigBucket b = big_bucket(a, round, i);
    big_splitters<THREADS>(s, a, b, big_source(a, round, b.pos), big_target(a, round, b.pos));
    const uint32_t pieces = (b.m + piece_size - 1) / piece_size;
    if (threadIdx.x == 0) s_first = atomicAdd(&R.pieces, pieces);
    __syncthreads();
    for (uint32_t p = threadIdx.x; p < pieces; p += THREADS) a.piece[(size_t)round * a.piece_room + s_first + p] = (u64)i << 32 | p;
    block_done(&R.done_sample);
  }
}
// Buckets of few pieces: all steps by one block, so that none of them waits for others
template <int THREADS>
__device__ __noinline__ void big_own(RankShared& s, EncHeader* hdr, const RankArgs& a) {
  const uint32_t n = hdr->own_n;  // written by the selection alone
  while (true) {
    const uint32_t i = block_takes(&hdr->own_next);
    if (i >= n) return;
    const BigBucket b = big_bucket(a, kBigOwnRow, i);
    const u64* src = big_source(a, 0, b.pos);
    u64* dst = big_target(a, 0, b.pos);
    big_splitters<THREADS>(s, a, b, src, dst);
    __syncthreads();
    const BigSearch h = big_prepare<THREADS>(s, a, b);
    big_piece<THREADS>(s, h, b, src, 0, b.m, ~0ull, [&](uint32_t p, u64) { atomicAdd(&s.cell[p], 1u); });
    __syncthreads();
    big_bounds<THREADS>(s, hdr, a, kBigOwnRow, i, b);
    __syncthreads();
    big_piece<THREADS>(s, h, b, src, 0, b.m, big_bucket(a, kBigOwnRow, i).last, [&](uint32_t p, u64 v) { dst[atomicAdd(&s.cell[p], 1u)] = to_item(v); });
    block_done(&hdr->own_done);
  }
}

// Steps 2 and 3: the round's pieces counted; behind a bucket's last piece where its parts begin, and the parts to their lists
template <int THREADS>
__device__ __noinline__ void big_count(RankShared& s, EncHeader* hdr, const RankArgs& a, int round) {
  __shared__ uint32_t s_last;
  BigRound& R = hdr->big[round];
  const uint32_t piece_size = big_piece_size(R);
  const uint32_t n = *reinterpret_cast<const volatile uint32_t*>(&R.pieces);
  while (true) {
    const uint32_t t = block_takes(&R.next_count);
    if (t >= n) return;
    const u64 piece = __ldcg(a.piece + (size_t)round * a.piece_room + t);
    const uint32_t i = (uint32_t)(piece >> 32);
    const BigBucket b = big_bucket(a, round, i);
    const u64 slot = big_slot(b.pos);
    const BigSearch h = big_prepare<THREADS>(s, a, b);
    big_piece<THREADS>(s, h, b, big_source(a, round, b.pos), (uint32_t)piece * piece_size, piece_size, ~0ull, [&](uint32_t p, u64) { atomicAdd(&s.cell[p], 1u); });
    __syncthreads();
    for (uint32_t p = threadIdx.x; p < b.parts; p += THREADS)
      if (s.cell[p]) a.base[(size_t)t * kBigParts + p] = atomicAdd(a.part_count + slot + p, s.cell[p]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&a.big[(size_t)round * a.big_room + i].counted, 1u) + 1 == (b.m + piece_size - 1) / piece_size;
    __syncthreads();
    if (!s_last) continue;
    __threadfence();
    for (uint32_t p = threadIdx.x; p < kBigParts; p += THREADS) s.cell[p] = p < b.parts ? __ldcg(a.part_count + slot + p) : 0u;
    big_bounds<THREADS>(s, hdr, a, round, i, b);
    block_done(&R.done_bounds);
  }
}

// Step 4: the round's pieces placed, but for what is never sent
template <int THREADS>
__device__ __noinline__ void big_place(RankShared& s, EncHeader* hdr, const RankArgs& a, int round) {
  BigRound& R = hdr->big[round];
  const uint32_t piece_size = big_piece_size(R);
  const uint32_t n = *reinterpret_cast<const volatile uint32_t*>(&R.pieces);
  while (true) {
    const uint32_t t = block_takes(&R.next_place);
    if (t >= n) return;
    const u64 piece = __ldcg(a.piece + (size_t)round * a.piece_room + t);
    const BigBucket b = big_bucket(a, round, (uint32_t)(piece >> 32));
    const u64 slot = big_slot(b.pos);
    const u64* src = big_source(a, round, b.pos);
    u64* dst = big_target(a, round, b.pos);
    const BigSearch h = big_prepare<THREADS>(s, a, b);
    for (uint32_t p = threadIdx.x; p < b.parts; p += THREADS)  // (of a part that the piece has nothing of the base is not read)
      s.cell[p] = __ldcg(a.part_start + slot + p) + __ldcg(a.base + (size_t)t * kBigParts + p);
    __syncthreads();
    big_piece<THREADS>(s, h, b, src, (uint32_t)piece * piece_size, piece_size, b.last, [&](uint32_t p, u64 v) {
      const uint32_t o = atomicAdd(&s.cell[p], 1u);
      if (o < b.m) dst[o] = to_item(v);
    });
    block_done(&R.done_place);
  }
}

// Step 5: the parts ranked, into the first buffer
template <int THREADS>
__device__ __noinline__ void big_rank(RankShared& s, EncHeader* hdr, const RankArgs& a) {
  const uint32_t n = *reinterpret_cast<const volatile uint32_t*>(&hdr->part_n);
  while (true) {
    const uint32_t i = block_takes(&hdr->part_next);
    if (i >= n) return;
    const volatile BigPart* v = a.part + i;
    const BigPart b{v->pos, v->n, v->in_b, v->first_key, v->last_key};
    const u64* src = (b.in_b ? a.buf_b : a.buf_a) + b.pos;
    u64* out = a.buf_a + b.pos;
    if (b.n > kRankItems) {  // the samples have missed: sorted where it lies
      for (uint32_t p = threadIdx.x; p < b.n; p += THREADS) out[p] = to_value(src[p]);
      __syncthreads();
      bitonic_sort(out, b.n, threadIdx.x, THREADS, [] { __syncthreads(); });
      for (uint32_t p = threadIdx.x; p < b.n; p += THREADS) out[p] = to_item(out[p]);
      __syncthreads();
    } else {
      rank_keys<THREADS>(s, src, b.n, b.first_key, b.last_key, out);
    }
  }
}

// the large buckets, from step 2 of the first round on; by the whole block
template <int THREADS>
__device__ __noinline__ void rank_big(RankShared& s, EncHeader* hdr, const RankArgs& a) {
  for (int round = 0; round < kBigRounds; ++round) {
    BigRound& R = hdr->big[round];
    const uint32_t n = *reinterpret_cast<const volatile uint32_t*>(&R.n);
    if (n == 0) break;
    if (round) big_sample<THREADS>(s, hdr, a, round);
    if (!block_waits(&R.done_sample, n, &hdr->status)) return;
    big_count<THREADS>(s, hdr, a, round);
    if (!block_waits(&R.done_bounds, n, &hdr->status)) return;
    big_place<THREADS>(s, hdr, a, round);
    if (!block_waits(&R.done_place, *reinterpret_cast<const volatile uint32_t*>(&R.pieces), &hdr->status)) return;
  }
  if (!block_waits(&hdr->own_done, hdr->own_n, &hdr->status)) return;
  big_rank<THREADS>(s, hdr, a);
}

// A tile of more than a block holds: its last bucket is a step of its own, or a large one, which is ranked from its list
template <int THREADS>
__device__ __noinline__ void rank_full_tile(RankShared& s, const RankTile& T, const RankArgs& a) {
  const uint32_t c = T.ticket % a.n;
  const ClientRank r = a.rank[c];
  uint32_t b_lo = T.bucket[0], at = T.start[0];
  const uint32_t b_end = T.bucket[1], at_end = T.start[1];
  while (at < at_end) {
    uint32_t b_hi = b_end, to = at_end;
    if (at_end - at > kRankItems && b_hi - b_lo > 1) {
      --b_hi;
      to = bucket_start(a, c, r, b_hi);
    }
    if (to > at && to - at <= kRankItems)
      rank_with_cells<THREADS>(s, T.from + at, to - at, b_lo << T.sh, (uint32_t)(((u64)b_hi << T.sh) - ((u64)b_lo << T.sh) - 1), T.into + at, r.keytop);
    b_lo = b_hi;
    at = to;
  }
}

// What the ranking has left over: cells of many equal or nearly equal keys (a layer's clipped outliers, values on a grid), whose
// items lie in any order in their place, tiles of more than a block holds, and buckets of more than that.  The blocks take an entry
// of the second list at a time, then their warps one of the first; the large buckets' splitters are looked for before that, so that
// few blocks wait for them.  Not among the tiles: there the calls cost registers and a block's other warps waited.  By spreading the
// indices instead of sorting them: 50 clients of 23.5 M, every seventh layer on a grid (3500 cells for a block, 1200 items each):
// ranking 784 us with sorting among the tiles, 500 with spreading, 303 + 143 here with blocks of 256 threads (20 clients: 87 us,
// with 512 threads 71).
template <int THREADS>
__device__ __noinline__ void rank_lists(RankShared& s, EncHeader* hdr, const RankArgs& a) {
  __shared__ RankTile s_tile;
  __shared__ uint32_t s_entry;
  const int tid = threadIdx.x, lane = tid & 31;
  __syncthreads();  // the arguments are there
  const bool big = (hdr->big[0].n | hdr->own_n) != 0;  // written by the selection alone
  if (big) {
    big_sample<THREADS>(s, hdr, a, 0);
    big_own<THREADS>(s, hdr, a);
  }
  while (true) {
    __syncthreads();
    if (tid == 0) s_entry = atomicAdd(&hdr->list_next[1], 1u);
    __syncthreads();
    if (s_entry >= hdr->list_n[1]) break;
    const ulonglong2 e = a.list[1][s_entry];
    const uint32_t m = (uint32_t)e.y;
    if (m != 0) {
      u64* at = a.buf_a + e.x;
      rank_cell<THREADS>(s, at, m, at);
    } else {
      if (tid == 0) s_tile.ticket = (uint32_t)e.x;
      __syncthreads();
      if (tid < 64) find_tile(s_tile, a);
      __syncthreads();
      rank_full_tile<THREADS>(s, s_tile, a);
    }
  }
  __syncthreads();
  while (true) {
    uint32_t g = 0;
    if (lane == 0) g = atomicAdd(&hdr->list_next[0], 1u);
    g = __shfl_sync(kFull, g, 0);
    if (g >= hdr->list_n[0]) break;
    const ulonglong2 e = a.list[0][g];
    rank_cell_by_warp<THREADS>(s, a.buf_a + e.x, (uint32_t)e.y);
  }
  if (!big) return;
  __syncthreads();
  rank_big<THREADS>(s, hdr, a);
}

}  // namespace cvlc
