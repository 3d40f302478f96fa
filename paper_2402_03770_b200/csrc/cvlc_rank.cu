// Ranking of the selected candidates by partition (Algorithm 1, step 15: |x| descending, ties by ascending index).
//
// The selection has left every client's candidates in coarse buckets, ranges of the sort key inv = keytop - key whose
// starts are known, in no particular order inside a bucket.  k_rank_split moves the candidates of a client with large
// buckets on into sub-buckets (the next bits of inv); k_rank then ranks whole buckets in shared memory by (inv, index) and
// writes them out in order; cells of equal keys and buckets beyond a block's shared memory are on lists that the kernel after
// it works off.  The order is total, so the result does not depend on how the candidates arrived.  Against a
// stable radix sort of the same keys (three passes of 9 bits) a candidate is moved once or twice instead of three times
// and costs one counting and one placing shared-memory atomic per move instead of a stable rank among the lanes of a warp.
#include "cvlc_rank.cuh"

namespace cvlc {

constexpr int kRankThreads = 512;

// (no candidate lies above keytop: the selection has checked that the update is the plan's)
__device__ __forceinline__ uint32_t inv_of(u64 item, uint32_t keytop) { return keytop - (uint32_t)(item >> 32); }

// ===================================================================================
// partition of the coarse buckets into sub-buckets
// ===================================================================================
// Tiles of kSplitTile consecutive candidates, held in registers.  A tile spans few coarse buckets, so its sub-buckets are a
// short range of counters: count, reserve each sub-bucket's room with one global atomic, place.  16 bytes per
// candidate; the stores are scattered 8 bytes at a time and merge in the L2.

constexpr int kSplitItems = 8;  // per thread
constexpr uint32_t kSplitTile = kRankThreads * kSplitItems;
static_assert(kSplitTile == kRankSplitTile, "tiles of the partition");
constexpr uint64_t kRankThree = 4 << 20;  // candidates of a batch, about, from which three blocks per SM are better than two

// THREE: three blocks per SM, the next tile asked into the L2 alone; else two, with the next tile's candidates on their way to registers.
// Three are better where the blocks have many tiles (two / three, us: 79 M candidates of 100 clients 321 / 296, 14 M of 24 46 / 40, 7 M
// of 24 24.7 / 21.5, 41 M of 50 178 / 172, 9 M of 10, about even: 54 / 55), two where they have one or two and its latency is all there is
// (2 M of 20 10.8 / 11.2, 0.9 M of one 8.1 / 10.0, 0.4 M of 10 7.9 / 9.4).
template <bool THREE>
__global__ void __launch_bounds__(kRankThreads, THREE ? 3 : 2)
k_rank_split(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L) {
  extern __shared__ uint32_t s_at[];  // [kRankSubs] counts, then next places
  __shared__ uint32_t s_next;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const uint32_t n = batch.n, tickets = (hdr->most_split + kRankSplitTile - 1) / kRankSplitTile * n;
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
  if (!THREE) request(t);
  while (t < tickets) {
    __syncthreads();  // everyone has read the ticket
    if (THREE) request(t);
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
    if (THREE && next < tickets) {  // a request per 128 bytes
      const uint32_t tile2 = next / n, c2 = next - tile2 * n, i = tile2 * kSplitTile + tid * 16;
      if (tid < kSplitTile / 16 && i < rank[c2].n) asm volatile("prefetch.global.L2 [%0];" ::"l"(buf_a + (size_t)c2 * L.capacity + i));
    }
    uint32_t* room = reinterpret_cast<uint32_t*>(ws + L.off_sub_pos) + (size_t)c * kRankSubs + s0;
    for (uint32_t i = tid; i < ns; i += kRankThreads) {
      const uint32_t v = s_at[i];
      if (v) s_at[i] = atomicAdd(room + i, v);
    }
    __syncthreads();
    u64 cur[kSplitItems];
#pragma unroll
    for (int u = 0; u < kSplitItems; ++u) cur[u] = it[u];
    if (!THREE) request(next);
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

// Tiles of buckets (RankTile), drawn by ticket; the next tile's buckets are searched for by two warps while the others compare.
// THREE: three blocks per SM, each with three quarters of the window.
// No calls and no per-client state in registers: 62 of them and no spills, 40 with THREE (with the crowded cells ranked here, 80 bytes of
// spills and waiting warps).  Bound by a tile's barriers and the latency of shared memory (two blocks issue 0.44 per scheduler and cycle), about
// 100 instructions per warp of candidates.  Two blocks and three, us: 79 M candidates of 100 clients 551 / 528 (and 41 for what is left over, see
// k_rank_rest), 41 M of 50, every seventh layer on a grid, 301 / 285 (and 113), 14 M of 24 92 / 86, 17 M of 20 in two calls 148 / 135; but whole
// calls of 5 clients of 600,000 coordinates 56.7 / 58.3, one of 11.2 M 87 / 88.  Half as many cells, or blocks of 256 threads with half the
// window, are within 5 %; twice the cells cost 20 % (clearing and scanning them), keeping an item's place from the counting 10 % (the atomic
// then returns a value); the next tile's candidates requested before the comparing: no gain, 2 us lost by 43,000 of ten clients.
template <bool THREE>
__global__ void __launch_bounds__(kRankThreads, THREE ? 3 : 2)
k_rank(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L, const uint32_t* __restrict__ bin_start_all, uint32_t blocks) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  typedef RankSharedOf<THREE ? kRankTile3 : kRankItems> Shared;
  Shared& s = *reinterpret_cast<Shared*>(s_raw);
  __shared__ RankTile s_tile[2];
  __shared__ RankArgs s_args;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const int tid = threadIdx.x;
  if (tid == 0) {
    s_args = rank_args(ws, L, bin_start_all, hdr, batch.n, blocks, THREE ? kRankWindow3 : kRankWindow);
    s_tile[0].ticket = atomicAdd(&hdr->rank_ticket, 1u);
  }
  __syncthreads();
  if (tid < 64) find_tile(s_tile[0], s_args);
  __syncthreads();
  for (uint32_t slot = 0;; slot ^= 1u) {
    const RankTile& T = s_tile[slot];
    if (T.ticket >= s_args.tickets) return;
    if (tid == 0) s_tile[slot ^ 1u].ticket = atomicAdd(&hdr->rank_ticket, 1u);
    const uint32_t at = T.start[0], m = T.start[1] - at;
    const bool large = m > (THREE ? kRankTile3 : kRankItems);
    auto leave = [&](uint32_t list, u64 what, uint32_t items) { s_args.list[list][atomicAdd(&hdr->list_n[list], 1u)] = make_ulonglong2(what, items); };
    if (!large && m != 0) {
      const uint32_t sh = T.sh, base = T.bucket[0] << sh;
      rank_buckets<kRankThreads, THREE ? 6 : 8>(s, T.from + at, m, base, (uint32_t)(((u64)T.bucket[1] << sh) - ((u64)T.bucket[0] << sh) - 1), T.into + at, T.keytop,
                                 [&](u64* where, uint32_t items) { leave(items > kWarpCell ? 1u : 0u, (u64)(where - s_args.buf_a), items); },
                                 [&]() {  // behind a barrier that follows the ticket
                                   if (tid < 64) find_tile(s_tile[slot ^ 1u], s_args);
                                 });
    } else {
      if (large && tid == 0) leave(1, T.ticket, 0);
      __syncthreads();
      if (tid < 64) find_tile(s_tile[slot ^ 1u], s_args);
    }
    __syncthreads();
  }
}

// What the ranking has left over (see rank_lists)
__global__ void __launch_bounds__(kRankThreads, 2)
k_rank_rest(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L, const uint32_t* __restrict__ bin_start_all, uint32_t blocks,
            uint32_t window) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ RankArgs s_args;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  if ((hdr->list_n[0] | hdr->list_n[1] | hdr->big[0].n | hdr->own_n) == 0) return;
  if (threadIdx.x == 0) s_args = rank_args(ws, L, bin_start_all, hdr, batch.n, blocks, window);
  rank_lists<kRankThreads>(*reinterpret_cast<RankShared*>(s_raw), hdr, s_args);
}

static cudaError_t rank_attributes() {
  static OncePerDevice once;
  return once_per_device(once, [] {
    cudaError_t e = allow_shared(k_rank<false>, sizeof(RankSharedOf<kRankItems>));
    if (e == cudaSuccess) e = allow_shared(k_rank<true>, sizeof(RankSharedOf<kRankTile3>));
    return e != cudaSuccess ? e : allow_shared(k_rank_rest, sizeof(RankShared));
  });
}
static unsigned blocks(uint64_t tiles, uint64_t most) { return (unsigned)(tiles < most ? tiles : most); }

cudaError_t launch_rank_rest(Batch batch, const EncLayout& L, const unsigned char* plan_ws, unsigned char* ws, unsigned sms, bool three, cudaStream_t st) {
  const cudaError_t e = rank_attributes();
  if (e != cudaSuccess) return e;
  launch_kernel(kKRankRest, k_rank_rest, blocks((L.capacity + kRankItems - 1) / kRankItems * L.n, 2 * sms), kRankThreads, sizeof(RankShared), st, true,
                batch, ws, L, reinterpret_cast<const uint32_t*>(plan_ws + plan_off_bin_start(L.n)), (three ? 3 : 2) * sms, three ? kRankWindow3 : kRankWindow);
  return cudaGetLastError();
}

cudaError_t launch_rank(Batch batch, const EncLayout& L, const unsigned char* plan_ws, unsigned char* ws, unsigned sms, uint64_t most, cudaStream_t st) {
  const cudaError_t e = rank_attributes();
  if (e != cudaSuccess) return e;
  const bool three = most * L.n >= kRankThree;
  launch_kernel(kKRankSplit, three ? k_rank_split<true> : k_rank_split<false>, blocks((L.capacity + kSplitTile - 1) / kSplitTile * L.n, (three ? 3 : 2) * sms),
                kRankThreads, kRankSubs * 4, st, true, batch, ws, L);
  const uint32_t* bin_start = reinterpret_cast<const uint32_t*>(plan_ws + plan_off_bin_start(L.n));
  launch_kernel(kKRank, three ? k_rank<true> : k_rank<false>, blocks((L.capacity + 1023) / 1024 * L.n, (three ? 3 : 2) * sms), kRankThreads,
                three ? sizeof(RankSharedOf<kRankTile3>) : sizeof(RankSharedOf<kRankItems>), st, true, batch, ws, L, bin_start, (three ? 3 : 2) * sms);
  return launch_rank_rest(batch, L, plan_ws, ws, sms, three, st);
}

}  // namespace cvlc
