// Ranking of tiles of candidates in shared memory: what the ranking kernel and the kernel that works its left-overs off share.
#pragma once
#include "cvlc_common.cuh"

namespace cvlc {

constexpr uint32_t kCellBits = 12, kCells = 1u << kCellBits;  // value ranges a tile is spread over before its items are compared
constexpr uint32_t kCompareAll = 48;    // a cell of up to this many items is ranked by comparing each with all,
constexpr uint32_t kWarpCell = 256;     // one of up to this many is ranked by one warp, a larger one by the block

typedef unsigned long long u64;

// Whether the call has failed or is not ranked by partition.  While blocks of the selection start, others of the same launch may
// write either word (an update that is not the plan's, a bucket too large for the partition), so one thread reads them and the
// block takes one branch: warps that part here would leave the others of their block at its barriers with work not done.
__device__ __forceinline__ bool rank_skips(const EncHeader* hdr) {
  __shared__ int s_skip;
  if (threadIdx.x == 0)
    s_skip = *reinterpret_cast<const volatile int32_t*>(&hdr->status) != 0 || *reinterpret_cast<const volatile uint32_t*>(&hdr->lsd) != kRankPartition;
  __syncthreads();
  return s_skip != 0;
}

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

// Ranks items[0 .. n), n <= kRankItems, and writes them out; by the whole block.  False, and nothing done, if too many keys differ or
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

// the same by one warp with kWarpCells ranges
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
  for (uint32_t p = lane; p < n; p += 32) {
    const uint2 v = it[p];
    if (v.y != key || v.x == kAside) {
      no |= !set_aside(others, it, p);
      continue;
    }
    least = min(least, v.x);
    most = max(most, v.x);
  }
  __syncwarp();
  least = __reduce_min_sync(kFull, least);
  most = __reduce_max_sync(kFull, most);
  const uint32_t span = most > least ? most - least : 0u;
  const int sh = span < kWarpCells ? 0 : 32 - __clz(span) - (int)kWarpCellBits;
  if (!__any_sync(kFull, no)) {
    for (uint32_t p = lane; p < n; p += 32) {
      const uint32_t x = it[p].x;
      if (x != kAside) no |= atomicAdd(&cell[(x - least) >> sh], 1u) >= kCompareAll;
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
  for (uint32_t p = lane; p < n; p += 32) {
    const uint32_t x = it[p].x;
    if (x != kAside) it[atomicAdd(&cell[(x - least) >> sh], 1u)].y = x;
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

// Ranks the n <= kRankItems items of a cell of many keys in their place; by the whole block.  They are spread over equal ranges of
// (key, index) between the least and the largest of each.  False, and nothing done, if a range has too many.
template <int THREADS>
__device__ __noinline__ bool rank_spread(RankShared& s, u64* at, uint32_t n) {
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
    at[rank_in_cell(s.items, v, (&s.cell[k])[-1], s.cell[k])] = to_item(v);
  }
  __syncthreads();
  return true;
}

// Ranks n <= kRankItems items, most of them of one key or nearly equal, in their place; by the whole block
template <int THREADS>
__device__ __noinline__ void rank_cell(RankShared& s, u64* at, uint32_t n) {
  for (int attempt = 0; attempt < 3; ++attempt) {
    if (attempt != 1) {
      for_items<THREADS>(at, n, [&](uint32_t i, u64 item) { s.items[i] = to_value(item); });
      __syncthreads();
    }
    if (attempt == 0) {
      if (n <= kCells / 2 ? rank_equal<THREADS, kCellBits - 1>(s, s.items, n, at) : rank_equal<THREADS, kCellBits>(s, s.items, n, at)) return;
    } else if (attempt == 1 && rank_spread<THREADS>(s, at, n)) {
      return;
    }
  }
  rank_by_block<THREADS>(s.items, n, at);
}

// Boundaries near ranks x[0] and x[1] of the m values of src, all in [lo, hi): a value and how many of src lie below it.  The range
// around a rank is narrowed until at most kCutRest values are left in it; the boundary is where that range starts.  A function of the
// set of values and the rank alone, so that neighbouring tiles agree on it.  As long as both ranks lie in one range, one pass over
// the values serves both: of equal keys two passes find both boundaries.
constexpr uint32_t kCutRest = kRankItems - kRankWindow;
struct Cut {
  u64 value;
  uint32_t below;
};
struct CutSearch {
  u64 lo, hi;
  uint32_t x, below;
  bool open;
};
template <int THREADS>
__device__ __noinline__ void cut_near(RankShared& s, const u64* __restrict__ src, uint32_t m, CutSearch& a, CutSearch& b) {
  __shared__ uint32_t s_cell[2], s_below[2], s_count[2];
  const int tid = threadIdx.x;
  for (int level = 0; level < 16 && (a.open || b.open); ++level) {  // 63 bits, 12 a level, each rank on its own at worst
    const u64 lo = a.open ? a.lo : b.lo, hi = a.open ? a.hi : b.hi;
    const bool for_a = a.open, for_b = b.open && b.lo == lo && b.hi == hi;
    if (lo >= hi) {
      if (for_a) a.open = false;
      if (for_b) b.open = false;
      continue;
    }
    const u64 span = hi - lo - 1;
    const int sh = span < kCells ? 0 : 64 - __clzll((long long)span) - (int)kCellBits;  // span >> sh below kCells
    for (uint32_t i = tid; i < kCells; i += THREADS) s.cell[i] = 0;
    if (tid < 2) s_cell[tid] = s_below[tid] = s_count[tid] = 0;
    __syncthreads();
    for_items<THREADS>(src, m, [&](uint32_t, u64 item) {
      const u64 v = to_value(item);
      if (v >= lo && v < hi) atomicAdd(&s.cell[(uint32_t)((v - lo) >> sh)], 1u);
    });
    __syncthreads();
    const uint32_t total = scan_cells<THREADS>(s.cell);
    // the last cell that starts at or below the rank
    for (uint32_t i = tid; i < kCells; i += THREADS) {
      const uint32_t first = s.cell[i], end = (i + 1 < kCells) ? s.cell[i + 1] : total;
      auto look = [&](const CutSearch& c, int e) {
        const uint32_t at = c.x - c.below;
        if (first <= at && at < end) {
          s_cell[e] = i;
          s_below[e] = first;
          s_count[e] = end - first;
        }
      };
      if (for_a) look(a, 0);
      if (for_b) look(b, 1);
    }
    __syncthreads();
    auto narrow = [&](CutSearch& c, int e) {
      c.lo = lo + ((u64)s_cell[e] << sh);
      c.hi = c.lo + (1ull << sh) < hi ? c.lo + (1ull << sh) : hi;
      c.below += s_below[e];
      if (s_count[e] <= kCutRest || sh == 0) c.open = false;
    };
    if (for_a) narrow(a, 0);
    if (for_b) narrow(b, 1);
    __syncthreads();
  }
}

// Ranks a .. b (about) of a bucket that a block cannot hold, m values in [lo, hi), are collected in their place: items that begin at
// out + below and whose values lie in [from, to).  src and out differ.
struct RankPart {
  u64 from, to;
  uint32_t below, n;
};
template <int THREADS>
__device__ __noinline__ RankPart collect_part(RankShared& s, const u64* __restrict__ src, uint32_t m, u64 lo, u64 hi, uint32_t a, uint32_t b,
                                              u64* __restrict__ out) {
  __shared__ uint32_t s_n;
  const int tid = threadIdx.x;
  CutSearch at_a{lo, hi, a, 0, a != 0}, at_b{lo, hi, b, 0, b < m};
  cut_near<THREADS>(s, src, m, at_a, at_b);
  const Cut from{at_a.lo, at_a.below}, to = b >= m ? Cut{hi, m} : Cut{at_b.lo, at_b.below};
  if (tid == 0) s_n = 0;
  __syncthreads();
  for_items<THREADS>(src, m, [&](uint32_t, u64 item) {
    const u64 v = to_value(item);
    if (v >= from.value && v < to.value) {
      const uint32_t p = atomicAdd(&s_n, 1u);
      if (p < kRankItems) out[from.below + p] = item;
    }
  });
  __syncthreads();
  const uint32_t got = s_n < kRankItems ? s_n : kRankItems;  // at most a window and kCutRest
  __syncthreads();
  return RankPart{from.value, to.value, from.below, got};
}

// Ranks m <= kRankItems items whose inv lies in [base, base + span]: spread over kCells equal ranges of inv, about one item per
// cell, then compared with the others of their cell.  Cells of more than kCompareAll items are left to `later`, their items in any
// order in their place.  `meanwhile` is run once all threads have passed a barrier.
template <int THREADS, class Later, class Meanwhile>
__device__ __forceinline__ void rank_buckets(RankShared& s, const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out, uint32_t keytop,
                                             Later&& later, Meanwhile&& meanwhile) {
  const int tid = threadIdx.x;
  // the first kHold candidates of a thread stay in registers between counting and placing
  constexpr int kHold = 8;
  u64 it[kHold];
#pragma unroll
  for (int u = 0; u < kHold; ++u)
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
  for (int u = 0; u < kHold; ++u)
    if ((uint32_t)tid + u * THREADS < m) atomicAdd(&s.cell[cell_of_key((uint32_t)(it[u] >> 32))], 1u);
  for (uint32_t i = tid + kHold * THREADS; i < m; i += THREADS) atomicAdd(&s.cell[cell_of_key((uint32_t)(src[i] >> 32))], 1u);
  __syncthreads();
  scan_cells<THREADS>(s.cell);
  auto put = [&](u64 item) { s.items[atomicAdd(&s.cell[cell_of_key((uint32_t)(item >> 32))], 1u)] = to_value(item); };
#pragma unroll
  for (int u = 0; u < kHold; ++u)
    if ((uint32_t)tid + u * THREADS < m) put(it[u]);
  for (uint32_t i = tid + kHold * THREADS; i < m; i += THREADS) put(src[i]);
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
// window plus one bucket; of a bucket that a block cannot hold the ranks that lie in the window, whether it starts there or before.
// What a block needs to know of one is found by two warps and kept in shared memory.
struct RankTile {
  uint32_t ticket;
  uint32_t bucket[2], start[2];  // first bucket at or behind the window's start and end; where those start
  uint32_t before;               // where the bucket before the first starts
  uint32_t sh, keytop;
  const u64* from;               // the client's candidates by buckets, and in order
  u64* into;
};

struct RankArgs {
  const ClientRank* rank;
  const uint32_t *sub_start, *bin_start;
  u64 *buf_a, *buf_b;
  ulonglong2* list[2];  // left over: cells for a warp; cells for a block and tiles with a bucket that a block cannot hold
  size_t capacity;
  uint32_t n, tickets, window;
};
__device__ __forceinline__ RankArgs rank_args(unsigned char* ws, const EncLayout& L, const uint32_t* bin_start, const EncHeader* hdr, uint32_t n) {
  RankArgs a;
  a.rank = reinterpret_cast<const ClientRank*>(ws + L.off_rank);
  a.sub_start = reinterpret_cast<const uint32_t*>(ws + L.off_sub_start);
  a.bin_start = bin_start;
  a.buf_a = reinterpret_cast<u64*>(ws + L.off_buf_a);
  a.buf_b = reinterpret_cast<u64*>(ws + L.off_buf_b);
  // Room: 512 entries for every 5120 candidates; at most one for every 49 of them, or one for every 257 and one per tile
  static_assert(kSortPasses * kDigits * 8 / 2 / 16 > kSortTile / kCompareAll + 1 + kSortTile / 1024 + 1, "the lists fit");
  a.list[0] = reinterpret_cast<ulonglong2*>(ws + L.off_sort_state);
  a.list[1] = a.list[0] + (size_t)n * L.sort_tiles_max * (kSortPasses * kDigits * 8 / 2 / 16);
  a.capacity = (size_t)L.capacity;
  a.n = n;
  a.tickets = hdr->rank_tiles * n;
  a.window = hdr->window;
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
      T.before = lo > 0 ? bucket_start(a, c, r, lo - 1) : 0u;
      T.sh = 19 + r.group - (r.split ? r.sub_bits : 0u);
      T.keytop = r.keytop;
      T.from = (r.split ? a.buf_b : a.buf_a) + (size_t)c * a.capacity;
      T.into = a.buf_a + (size_t)c * a.capacity;
    }
  }
}

// A tile with a bucket that a block cannot hold
template <int THREADS>
__device__ __noinline__ void rank_large(RankShared& s, const RankTile& T, const RankArgs& a) {
  __shared__ uint32_t s_n, s_big[kRankItems / kCompareAll];
  const uint32_t tile = T.ticket / a.n, c = T.ticket - tile * a.n;
  const ClientRank r = a.rank[c];
  const u64 x0 = (u64)tile * a.window, x1 = x0 + a.window;
  const uint32_t sh = T.sh;
  auto rank = [&](const u64* src, uint32_t m, uint32_t base, uint32_t span, u64* out) {
    if (threadIdx.x == 0) s_n = 0;
    rank_buckets<THREADS>(s, src, m, base, span, out, r.keytop,
                          [&](u64* where, uint32_t items) { s_big[atomicAdd(&s_n, 1u)] = (uint32_t)(where - out) | items << 16; }, [] {});
    const uint32_t n_big = s_n;
    for (uint32_t g = 0; g < n_big; ++g) rank_cell<THREADS>(s, out + (s_big[g] & 0xFFFFu), s_big[g] >> 16);
    __syncthreads();
  };
  auto part_of = [&](uint32_t bucket, uint32_t first, uint32_t end) {  // the window's part of a large bucket
    const u64 lo = ((u64)~r.keytop + ((u64)bucket << sh)) << 32, end_high = (u64)~r.keytop + ((u64)(bucket + 1) << sh);
    const u64 hi = end_high >> 32 ? ~0ull : end_high << 32;  // the last bucket may reach below key 0
    const uint32_t from = x0 > first ? (uint32_t)(x0 - first) : 0u;
    const uint32_t to = x1 < end ? (uint32_t)(x1 - first) : end - first;
    const RankPart p = collect_part<THREADS>(s, T.from + first, end - first, lo, hi, from, to, T.into + first);
    if (p.n == 0) return;
    const uint32_t base = (uint32_t)(p.from >> 32) - ~r.keytop, last = (uint32_t)((p.to - 1) >> 32) - ~r.keytop;
    u64* at = T.into + first + p.below;
    rank(at, p.n, base, last - base, at);
  };
  uint32_t b_lo = T.bucket[0], at = T.start[0];
  const uint32_t b_end = T.bucket[1], at_end = T.start[1];
  if (x0 < r.n && r.split && b_lo > 0 && at > x0 && at - T.before > kRankItems) part_of(b_lo - 1, T.before, at);
  // what is too large for one step ends with a large bucket: that bucket is a step of its own
  while (at < at_end) {
    uint32_t b_hi = b_end, to = at_end;
    if (at_end - at > kRankItems && b_hi - b_lo > 1) {
      --b_hi;
      to = bucket_start(a, c, r, b_hi);
    }
    if (to - at > kRankItems) {
      if (r.split) part_of(b_lo, at, to);
    } else if (to > at) {
      rank(T.from + at, to - at, b_lo << sh, (uint32_t)(((u64)b_hi << sh) - ((u64)b_lo << sh) - 1), T.into + at);
    }
    b_lo = b_hi;
    at = to;
  }
}

// What the ranking has left over: cells of many equal or nearly equal keys (a layer's clipped outliers, values on a grid), whose
// items lie in any order in their place, and tiles with a bucket that a block cannot hold.  The blocks take an entry of the
// second list at a time, then their warps one of the first.  Not among the tiles: there the calls cost registers and a block's
// other warps waited.  By spreading the indices instead of sorting them: 50 clients of 23.5 M, every seventh layer on a grid
// (3500 cells for a block, 1200 items each): ranking 784 us with sorting among the tiles, 500 with spreading, 303 + 143 here.
template <int THREADS>
__device__ __noinline__ void rank_lists(RankShared& s, EncHeader* hdr, const RankArgs a) {
  __shared__ RankArgs s_args;
  __shared__ RankTile s_tile;
  __shared__ uint32_t s_entry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_args = a;
  while (true) {
    __syncthreads();
    if (tid == 0) s_entry = atomicAdd(&hdr->list_next[1], 1u);
    __syncthreads();
    if (s_entry >= hdr->list_n[1]) break;
    const ulonglong2 e = s_args.list[1][s_entry];
    const uint32_t m = (uint32_t)e.y;
    if (m != 0) {
      u64* at = s_args.buf_a + e.x;
      rank_cell<THREADS>(s, at, m);
    } else {
      if (tid == 0) s_tile.ticket = (uint32_t)e.x;
      __syncthreads();
      if (tid < 64) find_tile(s_tile, s_args);
      __syncthreads();
      rank_large<THREADS>(s, s_tile, s_args);
    }
  }
  __syncthreads();
  static_assert(kWarpCell * (THREADS / 32) <= kRankItems, "room for every warp's cell");
  u64* mine = s.items + warp * kWarpCell;
  while (true) {
    uint32_t g = 0;
    if (lane == 0) g = atomicAdd(&hdr->list_next[0], 1u);
    g = __shfl_sync(kFull, g, 0);
    if (g >= hdr->list_n[0]) return;
    const ulonglong2 e = s_args.list[0][g];
    const uint32_t m = (uint32_t)e.y;
    u64* at = s_args.buf_a + e.x;
    for (uint32_t i = lane; i < m; i += 32) mine[i] = to_value(at[i]);
    __syncwarp();
    if (!rank_equal_by_warp<THREADS>(s.cell + warp * kWarpCells, mine, m, at)) {
      bitonic_sort(mine, m, lane, 32, [] { __syncwarp(); });
      for (uint32_t i = lane; i < m; i += 32) at[i] = to_item(mine[i]);
      __syncwarp();
    }
  }
}

}  // namespace cvlc
