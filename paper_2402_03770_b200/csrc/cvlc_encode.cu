// Encoding kernels (Algorithm 1, steps 15-17), batched over clients: top-k candidate selection by the
// plan's histogram threshold, into the buckets of the ranking by partition (cvlc_rank.cu) or, without the
// plan's workspace, in index order in front of a stable LSD radix ranking by |x|; the per-packet
// centroid distribution (PQ: minimum and maximum; QSGD: l2-norm), stochastic quantization with
// Philox4x32-10 (PQ or QSGD) and bit packing of (position ID, centroid ID) pairs into fixed-size packets
// (Fig. 2).
#include <string.h>

#include "cvlc_common.cuh"
#include "cvlc_lookback.cuh"
#include "cvlc_quant.cuh"
#include "cvlc_rank.cuh"

namespace cvlc {

// ===================================================================================
// K0  workspace reset, plan validation, sort-tile prefix over the clients
// ===================================================================================
// Where a plan comes from an earlier call; the planning front of cvlc_compress_batch does without (see EncFront).
// The grid zeroes the per-client counters, digit histograms and look-back states; block 0
// alone owns the 256-byte header and the sort-tile prefix (nobody else writes them).

// The bin that holds rank k and how many candidates there are from it on.  The plan's threshold was set before the lengths were tuned, for
// the most that could be sent; where the plan is complete, a tenth of its candidates are known not to be (8 clients of 1.2 M coordinates in
// the unframed format: 198 -> 192 us).  bin_start falls from bin to bin; eight places of the range are looked at together.
__device__ __forceinline__ uint2 sent_from(const cvlc_plan_t* plan, const uint32_t* __restrict__ bin_start) {
  const unsigned long long k = plan->k;
  const uint32_t thresh = plan->thresh_bin, n = (uint32_t)plan->n_candidates;
  if (k == 0 || k > n || thresh > plan->top_bin || plan->top_bin >= CVLC_HIST_BINS) return make_uint2(thresh, n);
  uint32_t lo = thresh, hi = plan->top_bin;  // the first bin with fewer than k candidates above it lies in [lo, hi]: none lies above the top
  while (lo < hi) {
    const uint32_t step = (hi - lo + 8) / 9;
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = bin_start[min(lo + i * step, hi)];
    uint32_t below = 0;  // places with k candidates or more above them
#pragma unroll
    for (int i = 0; i < 8; ++i) below += v[i] >= k ? 1u : 0u;
    const uint32_t new_hi = below < 8 ? min(lo + below * step, hi) : hi;
    if (below) lo = min(lo + (below - 1) * step, hi) + 1;
    hi = new_hi;
  }
  return make_uint2(lo, lo > thresh ? bin_start[lo - 1] : n);
}

template <int CAP>
__global__ void __launch_bounds__(256)
k_encode_init(unsigned char* ws, const __grid_constant__ BatchDesc<CAP> batch, const __grid_constant__ Shape shape,
              const __grid_constant__ EncLayout L, const unsigned char* plan_ws) {
  __shared__ unsigned long long s_total;
  __shared__ int s_bad, s_pass3;
  __shared__ uint32_t s_most, s_most_split;  // candidates of the largest client / of the largest one that needs the partition
  __shared__ uint32_t s_tiles[CVLC_MAX_BATCH];  // sort tiles of every client
  const uint32_t n = batch.n;
  const uint32_t limit = rank_limit(shape);
  pdl_enter();
  if (threadIdx.x == 0) {
    s_total = 0;
    s_bad = 0;
    s_pass3 = 0;
    s_most = s_most_split = 0;
  }
  // the plan's tables must have been made for this very batch: looked at only if the header says so
  const PlanWsHeader* ph = reinterpret_cast<const PlanWsHeader*>(plan_ws);
  const bool tables = ph && ph->magic == kPlanWsMagic && ph->n == n && ph->d == shape.d;
  __syncthreads();
  {
    unsigned long long t = 0;
    int pass3 = 0;
    const uint32_t* max_bin = tables ? reinterpret_cast<const uint32_t*>(plan_ws + plan_off_max_bin(n)) : nullptr;
    for (uint32_t c = threadIdx.x; c < n; c += blockDim.x) {  // the plans are read side by side, not one after the other
      const cvlc_plan_t* plan = batch.c[c].plan;
      const uint32_t tiles = sort_tiles_of(plan->n_candidates, L.capacity);
      s_tiles[c] = tiles;
      t += tiles;
      if (plan->top_bin + 1u - plan->thresh_bin > 256u) pass3 = 1;  // see top_digit_is_zero
      if (max_bin && blockIdx.x == 0) {
        const uint2 from = sent_from(plan, reinterpret_cast<const uint32_t*>(plan_ws + plan_off_bin_start(n)) + (size_t)c * CVLC_HIST_BINS);
        const ClientRank r = client_rank(from.x, plan->top_bin, from.y, max_bin[c], L.capacity, n);
        atomicMax(&s_most, r.n < limit ? r.n : limit);  // buckets from the limit on are not ranked
        if (r.split) atomicMax(&s_most_split, r.n);
        reinterpret_cast<ClientRank*>(ws + L.off_rank)[c] = r;
      }
    }
    if (t) atomicAdd(&s_total, t);
    if (pass3) atomicOr(&s_pass3, 1);
  }
  __syncthreads();
  const size_t gtid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t gstride = (size_t)gridDim.x * blockDim.x;
  auto zero = [&](size_t from, size_t to) {  // multiples of 256 bytes
    ulonglong2* p = reinterpret_cast<ulonglong2*>(ws + from);
    for (size_t i = gtid; i < (to - from) / 16; i += gstride) p[i] = make_ulonglong2(0ull, 0ull);
  };
  if (plan_ws) {
    zero(L.off_group_next, L.off_sub_start);  // counters of the selection and the partition
  } else {
    zero(L.off_ghist, L.off_sort_state);  // digit histograms, their scans, selection tile states
    // look-back states of the digit passes that will run (the fourth only if some client's keys span more than 2^27)
    const size_t per_pass = (size_t)s_total * kDigits;
    const int n_passes = s_pass3 ? kSortPasses : kSortPasses - 1;
    for (int p = 0; p < n_passes; ++p) {
      ulonglong2* st = reinterpret_cast<ulonglong2*>(reinterpret_cast<unsigned long long*>(ws + L.off_sort_state) +
                                                     (size_t)p * n * L.sort_tiles_max * kDigits);
      for (size_t i = gtid; i < per_pass / 2; i += gstride) st[i] = make_ulonglong2(0ull, 0ull);
    }
  }
  if (blockIdx.x != 0) return;

  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  uint32_t* prefix = reinterpret_cast<uint32_t*>(ws + L.off_sort_prefix);
  ClientDesc* desc = reinterpret_cast<ClientDesc*>(ws + L.off_desc);
  for (uint32_t c = threadIdx.x; c < n; c += blockDim.x) {
    desc[c] = batch.c[c];
    // Only what selection and ranking use is checked here (the code lengths may still be on their way on
    // another stream); the packing kernel checks the lengths.
    const cvlc_plan_t* plan = batch.c[c].plan;
    int bad = 0;
    if (plan->status != CVLC_OK)
      bad = plan->status;
    else if (plan->s != shape.s || plan->R != shape.R || plan->n_candidates == 0 || plan->n_candidates > shape.d ||
             plan->thresh_bin >= CVLC_HIST_BINS || plan->top_bin >= CVLC_HIST_BINS || plan->top_bin < plan->thresh_bin)
      bad = CVLC_ERR_PLAN_MISMATCH;
    else if (plan->n_candidates > L.capacity)
      bad = CVLC_ERR_WORKSPACE_TOO_SMALL;
    if (bad) atomicCAS(&s_bad, 0, bad);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0, mx = 0;
    for (uint32_t c = 0; c < n; ++c) {
      prefix[c] = run;
      const uint32_t t = s_tiles[c];
      run += t;
      if (t > mx) mx = t;
    }
    prefix[n] = run;
    if (plan_ws && !tables && !s_bad) s_bad = CVLC_ERR_PLAN_MISMATCH;
    hdr->max_sort_tiles = mx;
    hdr->status = s_bad;
    hdr->limit = limit;
    hdr->select_ticket = hdr->split_ticket = hdr->rank_ticket = 0;
    for (int p = 0; p < kSortPasses; ++p) hdr->sort_ticket[p] = 0;
    hdr->list_n[0] = hdr->list_n[1] = hdr->list_next[0] = hdr->list_next[1] = 0;
    for (int r = 0; r < kBigRounds; ++r) hdr->big[r] = BigRound{};
    hdr->own_n = hdr->own_next = hdr->own_done = hdr->part_n = hdr->part_next = 0;
    hdr->most = s_most;
    hdr->most_split = s_most_split;
  }
  // ranked by partition: the result is in the first buffer (the digit passes write a mask of their own)
  if (plan_ws)
    for (uint32_t c = threadIdx.x; c < n; c += blockDim.x) reinterpret_cast<uint32_t*>(ws + L.off_pass_mask)[c] = (1u << kSortPasses) - 1u;
}

// ===================================================================================
// K3  threshold selection + order-preserving compaction (single pass, decoupled look-back)
// ===================================================================================
// Emits (key << 32 | sign << 31 | index) for every coordinate whose histogram bin is at or
// above the plan's threshold bin, in ascending index order.  4 bytes read per coordinate.
// Tiles of 8192 coordinates are handed out by an atomic ticket (tile-major, clients interleaved:
// the tiles in flight at any time are a few consecutive tiles of every client), so every
// predecessor of a tile is running or done; the look-back reads 512 predecessors per step.
// Used when the plan's workspace is not available, in front of the digit passes.

__device__ __forceinline__ void select_lookback_tile(const Batch& batch, uint64_t d, unsigned char* ws, const EncLayout& L, uint64_t gt) {
  constexpr int THREADS = kSelectThreads;
  __shared__ unsigned long long s_warp_incl[THREADS / 32];
  __shared__ unsigned long long s_look_sum[THREADS / 32];
  __shared__ uint32_t s_look_flag[THREADS / 32];
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t tiles_per_client = select_tiles_of(d);
  {
    const uint64_t tile = gt / batch.n;
    const uint32_t c = (uint32_t)(gt - tile * batch.n);
    const float* __restrict__ x = batch.c[c].x;
    const cvlc_plan_t* __restrict__ plan = batch.c[c].plan;
    const float4* xv = reinterpret_cast<const float4*>(x);
    const uint32_t thresh = plan->thresh_bin << 19;
    unsigned long long* tile_state = reinterpret_cast<unsigned long long*>(ws + L.off_select_state) + (size_t)c * L.select_tiles;
    unsigned long long* __restrict__ out = reinterpret_cast<unsigned long long*>(ws + L.off_buf_a) + (size_t)c * L.capacity;
    const uint64_t base_vec = tile * (uint64_t)(THREADS * kSelectVecPerThread);

    uint32_t bits[kSelectVecPerThread][4];
    uint32_t mask[kSelectVecPerThread];
#pragma unroll
    for (int v = 0; v < kSelectVecPerThread; ++v) {
      const uint64_t vi = base_vec + (uint64_t)v * THREADS + tid;
      const uint64_t e0 = vi * 4;
      uint32_t valid = 0;
      if (e0 + 3 < d) {
        const float4 f = __ldg(xv + vi);
        bits[v][0] = __float_as_uint(f.x);
        bits[v][1] = __float_as_uint(f.y);
        bits[v][2] = __float_as_uint(f.z);
        bits[v][3] = __float_as_uint(f.w);
        valid = 0xF;
      } else {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          bits[v][cc] = 0;
          if (e0 + cc < d) {
            bits[v][cc] = __float_as_uint(x[e0 + cc]);
            valid |= 1u << cc;
          }
        }
      }
      uint32_t m = 0;
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) m |= (((bits[v][cc] & 0x7FFFFFFFu) >= thresh) ? 1u : 0u) << cc;
      mask[v] = m & valid;
    }
    // block scan of the four per-vector counts, packed 16 bits each (tile totals <= 2048)
    unsigned long long packed = 0;
#pragma unroll
    for (int v = 0; v < kSelectVecPerThread; ++v) packed |= (unsigned long long)__popc(mask[v]) << (16 * v);
    unsigned long long incl = packed;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned long long o = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) s_warp_incl[warp] = incl;
    __syncthreads();
    unsigned long long below = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
      const unsigned long long t = s_warp_incl[w];
      if (w < warp) below += t;
      tot += t;
    }
    const unsigned long long excl = below + incl - packed;  // per-vector exclusive counts over threads
    const uint32_t tile_total = (uint32_t)((tot & 0xFFFF) + ((tot >> 16) & 0xFFFF) + ((tot >> 32) & 0xFFFF) + (tot >> 48));

    // decoupled look-back: thread i inspects predecessor (tile - 1 - i) of this client
    if (tid == 0) st_relaxed(tile_state + tile, (tile == 0 ? kFlagPrefix : kFlagAgg) | tile_total);
    unsigned long long run = 0;
    if (tile > 0) {
      long long base = (long long)tile - 1;
      while (true) {
        const long long idx = base - tid;
        unsigned long long sv = kFlagPrefix;  // before tile 0: empty prefix
        if (idx >= 0) sv = wait_state(tile_state + idx, &hdr->status);
        const bool to = (sv == 0);
        const unsigned is_prefix = __ballot_sync(kFull, (sv & kFlagMask) == kFlagPrefix);
        unsigned long long val = sv & kValMask;
        if (is_prefix) {
          const int firstp = __ffs(is_prefix) - 1;
          if (lane > firstp) val = 0;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) val += __shfl_xor_sync(kFull, val, off);
        if (lane == 0) {
          s_look_sum[warp] = val;
          s_look_flag[warp] = is_prefix ? 1u : 0u;
        }
        const int any_to = __syncthreads_or(to);
        // the nearest warp (smallest distance) that saw a prefix ends the walk
        bool found = false;
        unsigned long long add = 0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) {
          if (!found) {
            add += s_look_sum[w];
            found = s_look_flag[w] != 0;
          }
        }
        run += add;
        __syncthreads();
        if (any_to || found) break;  // after a timeout the status is set and the results are void
        base -= THREADS;
      }
      if (tid == 0) st_relaxed(tile_state + tile, kFlagPrefix | (run + tile_total));
    }
    if (tid == 0 && tile == tiles_per_client - 1) {
      if (run + tile_total != plan->n_candidates) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);
    }
    unsigned long long vec_base = 0;
#pragma unroll
    for (int v = 0; v < kSelectVecPerThread; ++v) {
      unsigned long long o = run + vec_base + ((excl >> (16 * v)) & 0xFFFF);
      const uint64_t e0 = (base_vec + (uint64_t)v * THREADS + tid) * 4;
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        if (mask[v] & (1u << cc)) {
          const uint32_t b = bits[v][cc];
          const unsigned long long pair = ((unsigned long long)(b & 0x7FFFFFFFu) << 32) | (unsigned long long)(b & 0x80000000u) |
                                          (unsigned long long)(e0 + cc);
          if (o < L.capacity) out[o] = pair;
          ++o;
        }
      }
      vec_base += (tot >> (16 * v)) & 0xFFFF;
    }
    __syncthreads();  // the look-back scratch is reused by the next tile
  }
}

__global__ void __launch_bounds__(kSelectThreads)
k_select_lookback(const Batch batch, uint64_t d, unsigned char* ws, const __grid_constant__ EncLayout L) {
  __shared__ uint32_t s_tile;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const uint64_t total_tiles = select_tiles_of(d) * batch.n;
  while (true) {
    if (threadIdx.x == 0) s_tile = atomicAdd(&hdr->select_ticket, 1u);
    __syncthreads();
    const uint64_t gt = s_tile;
    if (gt >= total_tiles) break;
    __syncthreads();  // everyone has read the ticket
    select_lookback_tile(batch, d, ws, L, gt);
  }
}

// ===================================================================================
// K3' threshold selection into the buckets of the ranking (no order inside a bucket)
// ===================================================================================
// Groups of rows, every client with a counter of its own; a block keeps to one client while that has groups left, so that its
// counts of the client's sub-buckets go out once.  Its warps work on their own: they take groups (the first one without asking)
// and read the rows that hold a candidate (the histogram pass left the rows' maxima), 32 at a time, while the next 32 are copied
// to shared memory.  There every lane finds its row of 16 coordinates: their flags are one word.  In a step with few candidates
// a lane's loop runs over its own, in one with many every coordinate is stored or not; either way they are appended to the warp's
// buffer.  When that is full the warp counts its candidates per coarse bucket, reserves room in every bucket with one global
// addition and puts the candidates there; they are also counted per sub-bucket where the client needs the partition.  The block
// that completes a client turns those counts into offsets.
// Bound by instruction issue (0.60 per scheduler and cycle).  100 clients of 11.2 M coordinates, 7 % candidates: 622 us (from the bin
// of rank k on, 6 %: 568); 50 of 23.5 M, 3.5 %: 610; 10 of 100 M, 1 %: 210.  The copies go past the L1 (cp.async.cg): with loads into registers the warps were
// bound by the L1 lines that shared memory leaves for loads in flight (832, 943 and 377 us), and more warps made it worse; asking
// the L2 for 64 bytes instead of the 128 that it fetches by default takes 344 instead of 512 MB from DRAM for 8 of the second.
// (One buffer per block, emptied by all its warps together, left them waiting for one another: 860 us for the first.)

constexpr uint32_t kSelBuffer = 512;    // candidates in a warp's buffer: all of a step at least
constexpr int kSelVec = 4;              // 128-bit loads per lane and step
constexpr uint32_t kSelRows = 32;       // rows of a step
constexpr uint32_t kSelDense = 96;      // a step with this many candidates takes each coordinate in turn, one with fewer only its candidates
constexpr uint64_t kSelGiven = 2 << 20;  // rows of a batch (33 M coordinates) whose groups are all given out beforehand
constexpr int kSelStages = 2;           // steps in shared memory: the current one and those on their way
constexpr uint32_t kSelQueue = 256;     // rows a warp has found (ring)
struct SelWarp {
  unsigned long long items[kSelBuffer];
  float4 stage[kSelStages][kSelVec * 32];
  uint32_t cnt[kRankCoarse];            // counts, then next places (zero between)
  uint32_t queue[kSelQueue];
};
constexpr size_t kSelSmem = (kSelThreads / 32) * sizeof(SelWarp) + ((size_t)kRankCoarse + kRankSubs) * 4;
static_assert(kRowUnits == kSelVec && kSelRows - 1 + kSelPiece <= kSelQueue, "a row per lane and step; the ring holds a piece and a rest");
static_assert(kSelVec * 128 <= kSelBuffer && kSelSmem <= 227 * 1024, "shared memory");

// inclusive sums over the lanes
__device__ __forceinline__ uint32_t warp_inclusive(uint32_t v) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1)
    asm volatile("{.reg .pred p; .reg .b32 o; shfl.sync.up.b32 o|p, %0, %1, 0, 0xffffffff; @p add.u32 %0, %0, o;}" : "+r"(v) : "r"(off));
  return v;
}

// red.add of four fp32 counts at once: below 2^24 they are exact (see rank_shape)
__device__ __forceinline__ void add_counts4(float* p, uint32_t a, uint32_t b, uint32_t c, uint32_t e) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"((float)a), "f"((float)b), "f"((float)c), "f"((float)e) : "memory");
}

// ... and of four whole ones, kept out of the kernel's code (inlined it cost the selection 1.5 %)
__device__ __noinline__ void add_counts4_wide(float* p, uint4 v) {
  uint32_t* whole = reinterpret_cast<uint32_t*>(p);
  if (v.x) atomicAdd(whole, v.x);
  if (v.y) atomicAdd(whole + 1, v.y);
  if (v.z) atomicAdd(whole + 2, v.z);
  if (v.w) atomicAdd(whole + 3, v.w);
}

__global__ void __launch_bounds__(kSelThreads, 1)
k_select(const Batch batch, uint64_t d, const __grid_constant__ Partition part, const __grid_constant__ SelectGroups sg,
         const unsigned char* __restrict__ plan_ws, unsigned char* ws, const __grid_constant__ EncLayout L) {
  extern __shared__ __align__(16) unsigned char s_sel[];
  SelWarp& sw = reinterpret_cast<SelWarp*>(s_sel)[threadIdx.x >> 5];
  uint32_t* s_start = reinterpret_cast<uint32_t*>(s_sel + (kSelThreads / 32) * sizeof(SelWarp));  // [kRankCoarse] starts of the client's buckets
  uint32_t* s_sub = s_start + kRankCoarse;                                                        // [kRankSubs] candidates per sub-bucket
  __shared__ uint32_t s_client, s_taken, s_scan[kSelThreads / 32];
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t i = tid; i < kRankSubs / 4; i += kSelThreads) reinterpret_cast<uint4*>(s_sub)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (uint32_t i = lane; i < kRankCoarse; i += 32) sw.cnt[i] = 0;
  if (tid == 0) s_taken = 0;
  if (block_sees_error(&hdr->status)) return;
  const uint32_t n = batch.n;
  const uint32_t rows = (uint32_t)part.rows, held_rows = ((uint32_t)(d >> 2) + kRowUnits - 1) / kRowUnits;  // with coordinates
  const uint32_t groups = sg.groups;
  // A group's rows are spread over all that the groups of its size share, in runs of kSelRun (small groups) or pieces (larger ones), so
  // that all of them meet a layer that holds most of a client's candidates, where neighbouring rows made a group dense or empty: 24
  // clients of 3 M coordinates, blocks done after 69 to 119 us -> 69 to 95, whole calls 477 -> 449 us (4 bits), 321 -> 310 (QSGD, 2
  // bits); one of 11.2 M 94 -> 90; 100 of 11.2 M 3080 -> 3040.  (Runs in the larger groups too: 3054, and 50 of 23.5 M 2440 -> 2460.)
  const uint32_t small_row = (sg.count[0] * sg.pieces[0] + sg.count[1] * sg.pieces[1]) * kSelPiece, runs = (rows - small_row) / kSelRun;
  const uint32_t small_groups = groups - sg.count[0] - sg.count[1], last_group = (runs - 1) % small_groups;
  const uint32_t nvec = (uint32_t)(d >> 2);
  uint32_t* group_next = reinterpret_cast<uint32_t*>(ws + L.off_group_next);
  uint32_t* group_done = reinterpret_cast<uint32_t*>(ws + L.off_group_done);
  // Block b starts with client b n / grid; the first groups of a client go to the warps of the blocks that start with it, the rest
  // by its counter.  A small batch would wait for that: there the warps have three quarters of the groups without asking, and all
  // of them with few clients, whose blocks are as good as equally many, and in the smallest batches, where the last of them are not
  // worth a wait.  Whole calls with all and with three quarters, us: 4 clients of 3 M coordinates 113 and 121, 8 of 3 M 154 and 160;
  // 10 of 0.3 / 1.2 / 3 M 65 and 69 / 100 and 105 / 174 and 176, 24 of 0.3 / 1.2 M 86 and 90 / 159 and 160; 12 / 16 of 3 M 205 and 201
  // / 239 and 228, 40 of 1.2 M 235 and 226.
  const uint32_t home = blockIdx.x * n / gridDim.x;
  auto first_block = [&](uint32_t c) -> uint32_t { return (c * gridDim.x + n - 1) / n; };
  auto warps_of = [&](uint32_t c) -> uint32_t { return (first_block(c + 1) - first_block(c)) * (kSelThreads / 32); };
  auto rounds_of = [&](uint32_t warps) -> uint32_t {
    if (sg.count[0] + sg.count[1] || warps == 0) return 1;
    const uint32_t most = n <= 8 || part.total <= kSelGiven ? (groups + warps - 1) / warps : groups / 4 * 3 / warps;
    return most > 1 ? most : 1;
  };
  auto given = [&](uint32_t c) -> uint32_t { return warps_of(c) * rounds_of(warps_of(c)); };

  // the first client from `from` on that has groups left (n: none), found by all threads together
  auto find_client = [&](uint32_t from) -> uint32_t {
    if (tid == 0) s_client = 0xFFFFFFFFu;
    __syncthreads();
    for (uint32_t i = tid; i < n; i += kSelThreads) {
      const uint32_t c = from + i < n ? from + i : from + i - n;
      if (__ldcg(group_next + c) + given(c) < groups) {
        atomicMin(&s_client, i);
        break;
      }
    }
    __syncthreads();
    const uint32_t i = s_client;
    __syncthreads();
    return i == 0xFFFFFFFFu ? n : (from + i < n ? from + i : from + i - n);
  };

  for (uint32_t c = home, visit = 0;; ++visit) {
    if (visit) c = find_client(c);
    if (c >= n) return;
    const ClientRank r = reinterpret_cast<const ClientRank*>(ws + L.off_rank)[c];
    const float* __restrict__ x = batch.c[c].x;
    const float4* __restrict__ xv = reinterpret_cast<const float4*>(x);
    const uint16_t* __restrict__ row_max = reinterpret_cast<const uint16_t*>(plan_ws + plan_off_row_max(n)) + (size_t)c * rows;
    const uint32_t thresh_bin = r.thresh_bin, thresh = thresh_bin << 19, keytop = r.keytop;
    const float below_thresh = thresh ? __uint_as_float(thresh - 1u) : -1.0f;       // key >= thresh <=> |x| > below_thresh
    const uint32_t sh_coarse = 19 + r.group, sh_sub = sh_coarse - r.sub_bits;
    unsigned long long* __restrict__ out = reinterpret_cast<unsigned long long*>(ws + L.off_buf_a) + (size_t)c * L.capacity;
    uint32_t* fill = reinterpret_cast<uint32_t*>(ws + L.off_bin_fill) + (size_t)c * kRankCoarse;
    {
      const uint32_t* __restrict__ bin_start = reinterpret_cast<const uint32_t*>(plan_ws + plan_off_bin_start(n)) + (size_t)c * CVLC_HIST_BINS;
      for (uint32_t i = tid; i < r.n_coarse; i += kSelThreads) s_start[i] = coarse_start(r, bin_start, i);
    }
    auto inv_of = [&](uint32_t key) -> uint32_t { return keytop - (key < keytop ? key : keytop); };  // key >= thresh: inside the buckets
    uint32_t held = 0;  // candidates in the warp's buffer
    auto flush = [&]() {  // to their buckets
      bool above = false;
      for (uint32_t i = lane; i < held; i += 128) {  // four at a time: their loads, then their additions
        uint32_t key[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) key[u] = i + 32 * u < held ? (uint32_t)(sw.items[i + 32 * u] >> 32) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (i + 32 * u < held) {
            above |= key[u] > keytop;
            const uint32_t inv = inv_of(key[u]);
            atomicAdd(sw.cnt + (inv >> sh_coarse), 1u);
            if (r.split) atomicAdd(s_sub + (inv >> sh_sub), 1u);
          }
        }
      }
      if (above) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);  // the update is not the plan's
      __syncwarp();
      for (uint32_t i0 = lane; i0 < r.n_coarse; i0 += 128) {
        uint32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = (i0 + 32 * u < r.n_coarse) ? sw.cnt[i0 + 32 * u] : 0u;
        uint32_t at[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) at[u] = v[u] ? atomicAdd(fill + i0 + 32 * u, v[u]) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (v[u]) sw.cnt[i0 + 32 * u] = s_start[i0 + 32 * u] + at[u];
      }
      __syncwarp();
      for (uint32_t i = lane; i < held; i += 128) {
        unsigned long long item[4];
        uint32_t p[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) item[u] = i + 32 * u < held ? sw.items[i + 32 * u] : 0ull;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          p[u] = i + 32 * u < held ? atomicAdd(sw.cnt + (inv_of((uint32_t)(item[u] >> 32)) >> sh_coarse), 1u) : 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (p[u] < r.n) out[p[u]] = item[u];
      }
      __syncwarp();
      for (uint32_t i = lane; i < r.n_coarse; i += 32) sw.cnt[i] = 0;
      held = 0;
      __syncwarp();
    };

    __syncthreads();  // the buckets' starts are there
    // ---- the warp's groups, piece after piece: the maxima of the next two pieces are on their way, and so is the number of the
    // group after the last one asked for
    uint32_t taken = 0, group = 0, group2 = 0, piece = 0;
    const uint32_t warps = warps_of(c), dynamic = given(c);  // first group that goes by the counter
    uint32_t rounds = 0;                                     // groups to come without asking
    if (visit == 0) {
      group = warp * (warps / (kSelThreads / 32)) + (blockIdx.x - first_block(c));  // a dense layer goes to all blocks
      rounds = rounds_of(warps) - 1;
    } else {
      if (lane == 0) group = dynamic + atomicAdd(group_next + c, 1u);
      group = __shfl_sync(kFull, group, 0);
    }
    if (lane == 0 && rounds == 0) group2 = dynamic + atomicAdd(group_next + c, 1u);
    struct Piece {
      uint32_t row;  // lane: its four rows begin here; beyond the client's rows: none
      bool any, last;  // a piece at all; the one that holds the client's last rows
      uint2 maxima;  // of the lane's rows
    };
    auto next_piece = [&]() -> Piece {
      Piece p{rows, group < groups, false, make_uint2(0u, 0u)};
      if (!p.any) return p;
      uint32_t pieces = 1, g = group;
      if (g < sg.count[0]) {
        pieces = sg.pieces[0];
        p.row = (piece * sg.count[0] + g) * kSelPiece + 4 * (uint32_t)lane;
      } else if ((g -= sg.count[0]) < sg.count[1]) {
        pieces = sg.pieces[1];
        p.row = (sg.count[0] * sg.pieces[0] + piece * sg.count[1] + g) * kSelPiece + 4 * (uint32_t)lane;
      } else {
        g -= sg.count[1];
        const uint32_t run = (uint32_t)lane / (kSelRun / 4) * small_groups + g;
        if (4 * (uint32_t)lane < sg.small) p.row = small_row + run * kSelRun + 4 * ((uint32_t)lane % (kSelRun / 4));
        p.last = g == last_group;
      }
      ++piece;
      if (p.row < rows) p.maxima = __ldg(reinterpret_cast<const uint2*>(row_max + p.row));
      if (piece == pieces) {
        ++taken;
        piece = 0;
        group = rounds ? group + warps : __shfl_sync(kFull, group2, 0);
        if (rounds) --rounds;
        if (lane == 0 && rounds == 0 && group < groups) group2 = dynamic + atomicAdd(group_next + c, 1u);
      }
      return p;
    };
    Piece now = next_piece(), then = next_piece();
    uint32_t* queue = sw.queue;
    uint32_t head = 0, tail = 0;
    uint32_t slot = 0;                         // stage that the next step goes to
    bool ragged = false;                       // the last row has been listed
    uint32_t step_row[kSelStages], step_rows[kSelStages];  // per step, the oldest first: this lane's row; rows
    static_assert(kSelVec == 4, "a lane's 16 coordinates are a row");
    // Staging layout: float4 g of a step (in memory order) sits in slot g ^ ((g >> 3) & 3): what a warp's copies write (consecutive g)
    // and its loads (lane l reads 4 l .. 4 l + 3) are then both free of bank conflicts.
    const uint32_t stage0 = (uint32_t)__cvta_generic_to_shared(sw.stage[0]);
    auto request = [&](uint32_t& my_row) -> uint32_t {  // asks for the next rows that hold a candidate; returns how many there are
      while (tail - head < kSelRows && now.any) {
        const Piece p = now;
        now = then;
        then = next_piece();
        if (p.last && lane < (int)(d & 3)) {  // the client's ragged tail goes with its last piece: straight to its buckets
          const uint32_t b = __float_as_uint(x[(uint64_t)nvec * 4 + lane]), key = b & 0x7FFFFFFFu;
          if (key >= thresh) {
            if (key > keytop) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);
            const uint32_t inv = inv_of(key);
            const uint32_t p = s_start[inv >> sh_coarse] + atomicAdd(fill + (inv >> sh_coarse), 1u);
            if (r.split) atomicAdd(s_sub + (inv >> sh_sub), 1u);
            if (p < r.n) out[p] = ((unsigned long long)key << 32) | (unsigned long long)((b & 0x80000000u) | (nvec * 4 + (uint32_t)lane));
          }
        }
        // bins are 12 bits: the top bit of a half survives the subtraction where the row's bin reaches the threshold's
        uint32_t h01 = (p.maxima.x | 0x80008000u) - thresh_bin * 0x10001u, h23 = (p.maxima.y | 0x80008000u) - thresh_bin * 0x10001u;
        const uint32_t row = p.row;
        if (row + 4 > held_rows) {  // not all of the lane's rows are there
          h01 &= (row < held_rows ? 0x8000u : 0u) | (row + 1 < held_rows ? 0x80000000u : 0u);
          h23 &= (row + 2 < held_rows ? 0x8000u : 0u) | (row + 3 < held_rows ? 0x80000000u : 0u);
        }
        ragged |= p.last;
        if (!__any_sync(kFull, ((h01 | h23) & 0x80008000u) != 0)) continue;
        auto list = [&](bool hit, uint32_t which) {
          const unsigned hits = __ballot_sync(kFull, hit);
          if (hit) queue[(tail + __popc(hits & ((1u << lane) - 1u))) & (kSelQueue - 1)] = which;
          tail += __popc(hits);
        };
        list(h01 & 0x8000u, row);
        list(h01 & 0x80000000u, row + 1);
        list(h23 & 0x8000u, row + 2);
        list(h23 & 0x80000000u, row + 3);
        __syncwarp();
      }
      const uint32_t have = tail - head < kSelRows ? tail - head : kSelRows;
      my_row = queue[(head + lane) & (kSelQueue - 1)];
      const bool whole = have == kSelRows && !ragged;
#pragma unroll
      for (int v = 0; v < kSelVec; ++v) {  // four neighbouring lanes fetch a row
        const uint32_t i = 8 * v + (lane >> 2), g = v * 32 + lane;
        const uint32_t unit = __shfl_sync(kFull, my_row, i) * kRowUnits + (lane & 3);
        const uint32_t to = stage0 + (slot * (kSelVec * 32) + (g ^ ((g >> 3) & 3u))) * 16;
        if (whole) {
          asm volatile("cp.async.cg.shared.global.L2::64B [%0], [%1], 16;" ::"r"(to), "l"(xv + unit) : "memory");
        } else {
          const bool on = i < have && unit < nvec;  // else zeros: no candidates
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(xv + (on ? unit : 0u)), "r"(on ? 16 : 0) : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      slot = slot + 1 == kSelStages ? 0 : slot + 1;
      head += have;
      __syncwarp();
      return have;
    };
    const uint32_t ct = ((uint32_t)lane >> 1) & 3u;
    const uint32_t word_of = 15u ^ (ct << 2);
    uint32_t cur = 0;  // stage of the current step
#pragma unroll
    for (int i = 0; i + 1 < kSelStages; ++i) step_rows[i] = request(step_row[i]);
    while (step_rows[0]) {
      __syncwarp();  // the step before has been read
      step_rows[kSelStages - 1] = request(step_row[kSelStages - 1]);
      asm volatile("cp.async.wait_group %0;" ::"n"(kSelStages - 1) : "memory");
      __syncwarp();
      const float4* stage = sw.stage[cur];
      const uint32_t* words = reinterpret_cast<const uint32_t*>(stage) + 16 * lane;
      cur = cur + 1 == kSelStages ? 0 : cur + 1;
      const uint32_t first = step_row[0] * (4 * kRowUnits);
      uint32_t m = 0;  // flags of this lane's coordinates, lowest index in bit 15
      uint32_t bits[16];
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const float4 f = stage[4 * lane + (j ^ ct)];
        bits[4 * j] = __float_as_uint(f.x);
        bits[4 * j + 1] = __float_as_uint(f.y);
        bits[4 * j + 2] = __float_as_uint(f.z);
        bits[4 * j + 3] = __float_as_uint(f.w);
      }
#pragma unroll
      for (int j = 0; j < 16; ++j)  // the difference of two distinct floats never rounds to zero: its sign is the flag
        m = __funnelshift_l(__float_as_uint(__fsub_rn(below_thresh, fabsf(__uint_as_float(bits[j])))), m, 1);
      if (thresh == 0) {  // zeros are candidates: not those that stand for rows and coordinates there are not
        const uint32_t there = (uint32_t)lane < step_rows[0] ? nvec - (first >> 2) : 0u;  // units of the update from this lane's row on
        if (there < 4) m &= 0xFFFF0000u >> (4 * there);
      }
#pragma unroll
      for (int i = 0; i + 1 < kSelStages; ++i) {
        step_row[i] = step_row[i + 1];
        step_rows[i] = step_rows[i + 1];
      }
      const uint32_t cnt = __popc(m);
      const uint32_t incl = warp_inclusive(cnt);
      const uint32_t total = __shfl_sync(kFull, incl, 31);
      if (held + total > kSelBuffer) flush();
      unsigned long long* o = sw.items + held + incl - cnt;
      if (total >= kSelDense) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (m & (1u << (15 - j))) *o++ = ((unsigned long long)(bits[j] & 0x7FFFFFFFu) << 32) | (unsigned long long)((bits[j] & 0x80000000u) | (first + j));
      } else {
        while (m) {
          const int hb = 31 - __clz(m);  // highest flag = lowest index first
          m ^= 1u << hb;
          const uint32_t b = words[hb ^ word_of];
          *o++ = ((unsigned long long)(b & 0x7FFFFFFFu) << 32) | (unsigned long long)((b & 0x80000000u) | (first + 15 - hb));
        }
      }
      held += total;
    }
    __syncwarp();
    if (held) flush();
    if (lane == 0 && taken) atomicAdd(&s_taken, taken);
    __syncthreads();
    const uint32_t block_taken = s_taken;
    __syncthreads();
    if (block_taken == 0) continue;
    if (tid == 0) s_taken = 0;
    if (r.split) {
      float* count = reinterpret_cast<float*>(ws + L.off_sub_count) + (size_t)c * kRankSubs;
      const uint32_t n_sub4 = ((r.n_coarse << r.sub_bits) + 3) / 4;
      uint4* sub4 = reinterpret_cast<uint4*>(s_sub);
      for (uint32_t i = tid; i < n_sub4; i += kSelThreads) {
        const uint4 v = sub4[i];
        if (v.x | v.y | v.z | v.w) {
          if (r.wide) add_counts4_wide(count + 4 * i, v);
          else add_counts4(count + 4 * i, v.x, v.y, v.z, v.w);
          sub4[i] = make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_client = atomicAdd(group_done + c, block_taken) + block_taken;
    __syncthreads();
    if (s_client == groups) {
      __threadfence();
      // A thread has sixteen sub-buckets: their counts and the check of the coarse ones are read side by side, and one scan does.  A
      // client's end takes 2.7 us of 8192 sub-buckets (two rounds of eight, read behind the check: 6.5).
      constexpr uint32_t kMine = 16;
      static_assert(kSelThreads * kMine >= kRankSubs && kRankSubs % kMine == 0, "one scan");
      const uint32_t n_sub = r.split ? r.n_coarse << r.sub_bits : 0u, i0 = (uint32_t)tid * kMine;
      uint4 v4[kMine / 4];
      if (i0 < n_sub) {
        const uint4* count = reinterpret_cast<const uint4*>(ws + L.off_sub_count) + ((size_t)c * kRankSubs + i0) / 4;
#pragma unroll
        for (uint32_t e = 0; e < kMine / 4; ++e) v4[e] = __ldcg(count + e);
      } else {
#pragma unroll
        for (uint32_t e = 0; e < kMine / 4; ++e) v4[e] = make_uint4(0u, 0u, 0u, 0u);
      }
      // the update must be the one the plan was made from
      for (uint32_t i = tid; i < r.n_coarse; i += kSelThreads) {
        const uint32_t end = i + 1 < r.n_coarse ? s_start[i + 1] : r.n;
        if (__ldcg(fill + i) != end - s_start[i]) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);
      }
      if (r.split) {
        uint32_t* start = reinterpret_cast<uint32_t*>(ws + L.off_sub_start) + (size_t)c * (kRankSubs + 64);
        uint32_t* next = reinterpret_cast<uint32_t*>(ws + L.off_sub_pos) + (size_t)c * kRankSubs;
        uint32_t v[kMine], sum = 0;
#pragma unroll
        for (uint32_t e = 0; e < kMine; ++e) {
          const uint32_t w = e % 4 == 0 ? v4[e / 4].x : e % 4 == 1 ? v4[e / 4].y : e % 4 == 2 ? v4[e / 4].z : v4[e / 4].w;
          v[e] = r.wide ? w : (uint32_t)__uint_as_float(w);
          sum += v[e];
        }
        const uint32_t incl = warp_inclusive(sum);
        if (lane == 31) s_scan[warp] = incl;
        __syncthreads();
        const uint32_t of_warp = lane < kSelThreads / 32 ? s_scan[lane] : 0u;
        const uint32_t all = __reduce_add_sync(kFull, of_warp);
        uint32_t run = __reduce_add_sync(kFull, lane < warp ? of_warp : 0u) + incl - sum;
        if (i0 < n_sub) {  // behind the last sub-bucket there are none: the total
#pragma unroll
          for (uint32_t e = 0; e < kMine; e += 4) {
            uint4 at;
            at.x = run;
            at.y = at.x + v[e];
            at.z = at.y + v[e + 1];
            at.w = at.z + v[e + 2];
            run = at.w + v[e + 3];
            reinterpret_cast<uint4*>(start + i0)[e / 4] = at;
            reinterpret_cast<uint4*>(next + i0)[e / 4] = at;
            if (max(max(v[e], v[e + 1]), max(v[e + 2], v[e + 3])) > kRankItems) {
              const uint32_t from[4] = {at.x, at.y, at.z, at.w};
#pragma unroll
              for (uint32_t u = 0; u < 4; ++u)
                if (v[e + u] > kRankItems && from[u] < hdr->limit && from[u] + v[e + u] <= r.n) list_bucket(hdr, ws, L, c, keytop, (u64)(i0 + e + u) << sh_sub, (u64)(i0 + e + u + 1) << sh_sub, from[u], v[e + u]);
            }
          }
        }
        if (tid == 0 && n_sub % kMine == 0) start[n_sub] = all;  // else among the above
      }
    }
    __syncthreads();
  }
}

// With at most 256 histogram bins between the threshold and the top, keytop - key stays below 2^27 for every
// candidate: the fourth digit is zero throughout and neither counted nor ranked.
__device__ __forceinline__ bool top_digit_is_zero(const cvlc_plan_t* plan) { return plan->top_bin + 1u - plan->thresh_bin <= 256u; }

__device__ __forceinline__ uint32_t sort_digit(unsigned long long pair, int pass, uint32_t keytop) {
  const uint32_t key = (uint32_t)(pair >> 32);
  const uint32_t inv = key > keytop ? 0u : keytop - key;  // key > keytop only if the plan is not of this update
  return (inv >> (kDigitBits * pass)) & (kDigits - 1);
}

// ===================================================================================
// K4  stable LSD radix ranking of the candidates, |x| descending (ties keep ascending index)
// ===================================================================================
// Sort key = keytop - key, keytop = the largest key of the client's highest non-empty histogram
// bin, so the key only spans the bins between the threshold and the top: 19 + log2(#bins) bits.
// Digits of 9, 9, 9, 4 bits: one kernel counts all four for all clients, a small one scans the counts, then one
// single-pass kernel per digit (tiles handed out by ticket, tile-major with the clients interleaved;
// decoupled look-back per digit value).  A pass whose digit is the same for every candidate of a client
// (normally the fourth) is skipped for that client; which buffer holds its data after pass q follows from
// the mask of skipped passes.  Used where the plan's workspace is not at hand.
// 100 clients of 11.2 M coordinates at 2 bits (79 M candidates): 1525 us; 24 of 3 M at 4 bits: 285; 20 of 1.2 M: 112; one of 11.2 M: 95.
// As phases of one kernel that wait for one another 2185, 400, 165 and 117: the counting had the passes' occupancy, and a pass that
// no client needs its tickets.

// two adjacent look-back words in one 128-bit access (each 64-bit half is its own atomic access)
__device__ __forceinline__ void ld_relaxed2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_relaxed2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}

struct SortShared {
  uint32_t tile;                                        // ticket of the tile being worked on
  uint32_t next;                                        // the ticket after it (known once the tile's items are requested)
  uint32_t scan_w[kSortThreads / 32];                   // warp totals of the block scan
  __align__(16) uint16_t wc[kSortThreads / 32][kDigits];  // per warp and digit value: the count, then the first slot
                                                          // (lanes index it by digit value: the banks are as random as the digits)
  uint32_t gofs[kDigits];  // per digit value: (position in dst of the tile's first item of that value) - (its slot in the tile)
  uint32_t mm[kSortThreads / 32][kDigits];  // per warp and digit value: lanes of the current row holding it (zero between rows)
};

constexpr size_t kSortSharedBytes = (sizeof(SortShared) + 15) & ~(size_t)15;
constexpr size_t sort_smem_bytes(uint32_t n) { return kSortSharedBytes + (size_t)kSortTile * 8 + (4 * (size_t)n + 1) * 4; }

// One tile of one digit pass.  FULL: the tile holds kSortTile items (no bounds checks in the item loops).
// Thread t < 256 owns the digit values 2t and 2t + 1 in the counting, scan and look-back steps.
template <bool FULL, class Prefetch>
__device__ __forceinline__ void sort_tile(SortShared& sh, unsigned long long* __restrict__ s_items,
                                          const unsigned long long* __restrict__ src, unsigned long long* __restrict__ dst,
                                          unsigned long long* __restrict__ state, const unsigned long long* __restrict__ gbase,
                                          uint32_t tile, uint32_t count, uint32_t n32, uint32_t keytop, int shift,
                                          int32_t* status, uint32_t next, Prefetch&& prefetch_next) {
  constexpr int kWarps = kSortThreads / 32;
  constexpr int IT = kSortItemsPerThread;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lanemask_lt = (1u << lane) - 1u;
  const uint32_t wbase = (uint32_t)warp * (32 * IT) + lane;  // this thread's first item inside the tile

  unsigned long long item[IT];
  uint32_t rd[IT];  // digit value | rank among the warp's items of that value << 16
  {
    const unsigned long long* __restrict__ p = src + (size_t)tile * kSortTile + wbase;
#pragma unroll
    for (int i = 0; i < IT; ++i) item[i] = (FULL || wbase + i * 32 < count) ? __ldcg(p + i * 32) : ~0ull;  // written in this kernel: L2
  }
  if (tid == 0) sh.next = next;  // waits for the ticket counter's answer, behind the item requests
  // the look-back needs the digit values' first positions in dst: requested early, used late
  unsigned long long gb0 = 0, gb1 = 0;
  if (tid < kDigits / 2) {
    const ulonglong2 g = __ldcg(reinterpret_cast<const ulonglong2*>(gbase + 2 * tid));
    gb0 = g.x;
    gb1 = g.y;
  }
  // stable rank inside the warp, items in (i, lane) order.  The lanes of a row that hold the same digit value
  // find each other through a word of shared memory that each of them ORs its lane bit into (nine ballots cost
  // four times the issue slots, a match instruction one step per distinct value in the warp); all of them read
  // the warp's running count of the value, the highest lane then updates it and clears the word.
  uint32_t* mm = &sh.mm[warp][0];
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const bool valid = FULL || (wbase + i * 32 < count);
    const uint32_t key = (uint32_t)(item[i] >> 32);
    const uint32_t inv = keytop - (key < keytop ? key : keytop);  // key > keytop only if the plan is not of this update
    const uint32_t dig = (inv >> shift) & (kDigits - 1);
    if (valid) atomicOr(mm + dig, 1u << lane);
    __syncwarp();
    unsigned peers = 1u << lane;
    uint32_t pre = 0;
    if (valid) {
      peers = *reinterpret_cast<volatile uint32_t*>(mm + dig);
      pre = *reinterpret_cast<volatile uint16_t*>(&sh.wc[warp][dig]);
    }
    __syncwarp();
    rd[i] = dig | ((pre + __popc(peers & lanemask_lt)) << 16);
    if (valid && (peers >> lane) == 1u) {  // no peer in a higher lane
      sh.wc[warp][dig] = (uint16_t)(pre + __popc(peers));
      mm[dig] = 0u;
    }
    __syncwarp();
  }
  __syncthreads();
  prefetch_next(sh.next);

  // counts of the two digit values in every warp (a 32-bit word holds both), published as the tile's aggregate
  constexpr int kOwners = kDigits / 2;
  const bool owner = tid < kOwners;
  uint32_t* wc32 = reinterpret_cast<uint32_t*>(&sh.wc[0][0]);
  uint32_t tot0 = 0, tot1 = 0, incl = 0;
  unsigned long long* my_state = state + (size_t)tile * kDigits + 2 * (tid & (kOwners - 1));
  if (owner) {
    uint32_t p = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) p += wc32[w * (kDigits / 2) + tid];  // 16-bit lanes: no carry (<= kSortTile)
    tot0 = p & 0xFFFFu;
    tot1 = p >> 16;
    const unsigned long long f = (tile == 0) ? kFlagPrefix : kFlagAgg;
    st_relaxed2(my_state, f | tot0, f | tot1);
    // first slot of every digit value inside the tile: block scan in digit order
    incl = tot0 + tot1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) sh.scan_w[warp] = incl;
  }
  __syncthreads();
  if (owner) {
    uint32_t below = 0;
#pragma unroll
    for (int w = 0; w < kOwners / 32; ++w) {
      const uint32_t v = sh.scan_w[w];
      if (w < warp) below += v;
    }
    const uint32_t dstart0 = below + incl - (tot0 + tot1);
    const uint32_t dstart1 = dstart0 + tot0;
    // the counters become first slots: slot of (value, warp) = first slot of the value + items of earlier warps
    {
      uint32_t t = dstart0 | (dstart1 << 16);  // both running slots stay below 2^16
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t v = wc32[w * (kDigits / 2) + tid];
        wc32[w * (kDigits / 2) + tid] = t;
        t += v;
      }
    }
    // decoupled look-back over the client's earlier tiles, both digit values per step
    unsigned long long run0 = 0, run1 = 0;
    if (tile > 0) {
      constexpr int kWin = 4;  // predecessors requested together: one round trip for all of them
      bool open0 = true, open1 = true;
      for (long long t = (long long)tile - 1; t >= 0 && (open0 || open1); t -= kWin) {
        unsigned long long a[kWin], b[kWin];
#pragma unroll
        for (int j = 0; j < kWin; ++j) {
          a[j] = b[j] = kFlagPrefix;  // before the client's first tile: nothing, chain closed
          if (t - j >= 0) ld_relaxed2(state + (size_t)(t - j) * kDigits + 2 * tid, a[j], b[j]);
        }
#pragma unroll
        for (int j = 0; j < kWin; ++j) {
          if (!(open0 || open1)) break;
          int polls = 0;
          while ((a[j] & kFlagMask) == 0 || (b[j] & kFlagMask) == 0) {
            if (++polls > kMaxPolls) {
              set_status(status, CVLC_ERR_DEVICE_TIMEOUT);
              a[j] = b[j] = kFlagPrefix;  // give up: close both chains
              break;
            }
            if (polls > 64) __nanosleep(64);
            ld_relaxed2(state + (size_t)(t - j) * kDigits + 2 * tid, a[j], b[j]);
          }
          if (open0) {
            run0 += a[j] & kValMask;
            open0 = (a[j] & kFlagMask) != kFlagPrefix;
          }
          if (open1) {
            run1 += b[j] & kValMask;
            open1 = (b[j] & kFlagMask) != kFlagPrefix;
          }
        }
      }
      st_relaxed2(my_state, kFlagPrefix | (run0 + tot0), kFlagPrefix | (run1 + tot1));
    }
    sh.gofs[2 * tid] = (uint32_t)(gb0 + run0) - dstart0;
    sh.gofs[2 * tid + 1] = (uint32_t)(gb1 + run1) - dstart1;
  }
  __syncthreads();
  // the items go to shared memory in digit order, then out in runs of consecutive addresses
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (FULL || wbase + i * 32 < count) {
      const uint32_t dig = rd[i] & 0xFFFFu;
      s_items[(uint32_t)sh.wc[warp][dig] + (rd[i] >> 16)] = item[i];
    }
  }
  __syncthreads();
  if (FULL) {
#pragma unroll
    for (int j = 0; j < IT; ++j) {
      const uint32_t k = j * kSortThreads + tid;
      const unsigned long long it = s_items[k];
      const uint32_t key = (uint32_t)(it >> 32);
      const uint32_t inv = keytop - (key < keytop ? key : keytop);
      const uint32_t o = sh.gofs[(inv >> shift) & (kDigits - 1)] + k;
      if (o < n32) dst[o] = it;
    }
  } else {
    for (uint32_t k = tid; k < count; k += kSortThreads) {
      const unsigned long long it = s_items[k];
      const uint32_t key = (uint32_t)(it >> 32);
      const uint32_t inv = keytop - (key < keytop ? key : keytop);
      const uint32_t o = sh.gofs[(inv >> shift) & (kDigits - 1)] + k;
      if (o < n32) dst[o] = it;
    }
  }
}

// digit counts of all candidates: the clients' arrays are concatenated in units of sort tiles and cut into equal contiguous chunks,
// one per block; a block that crosses a client boundary merges its counts into that client's and starts afresh
__global__ void __launch_bounds__(256)
k_sort_hist(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L) {
  __shared__ uint32_t s_count[kSortPasses * kDigits];
  pdl_enter();
  const EncHeader* hdr = reinterpret_cast<const EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const uint32_t* prefix = reinterpret_cast<const uint32_t*>(ws + L.off_sort_prefix);
  for (int i = threadIdx.x; i < kSortPasses * kDigits; i += 256) s_count[i] = 0;
  __syncthreads();
  const uint32_t total_tiles = prefix[batch.n];
  const uint32_t chunk = (total_tiles + gridDim.x - 1) / gridDim.x;
  uint32_t t = blockIdx.x * chunk;
  const uint32_t t_end = (t + chunk < total_tiles) ? t + chunk : total_tiles;
  uint32_t c = 0;
  while (t < t_end) {
    while (prefix[c + 1] <= t) ++c;  // client of tile t (clients without tiles are passed over)
    const uint32_t seg_end = prefix[c + 1] < t_end ? prefix[c + 1] : t_end;
    const cvlc_plan_t* plan = batch.c[c].plan;
    const uint32_t keytop = sort_keytop(plan);
    const int n_count = top_digit_is_zero(plan) ? kSortPasses - 1 : kSortPasses;
    const unsigned long long* __restrict__ in = reinterpret_cast<const unsigned long long*>(ws + L.off_buf_a) + (size_t)c * L.capacity;
    const unsigned long long i0 = (unsigned long long)(t - prefix[c]) * kSortTile;
    unsigned long long i1 = (unsigned long long)(seg_end - prefix[c]) * kSortTile;
    if (i1 > plan->n_candidates) i1 = plan->n_candidates;
    for (unsigned long long i = i0 + threadIdx.x; i < i1; i += 256) {
      const unsigned long long pair = in[i];
#pragma unroll
      for (int p = 0; p < kSortPasses; ++p)
        if (p < n_count) atomicAdd(&s_count[p * kDigits + sort_digit(pair, p, keytop)], 1u);
    }
    __syncthreads();
    unsigned long long* ghist = reinterpret_cast<unsigned long long*>(ws + L.off_ghist) + (size_t)c * kSortPasses * kDigits;
    for (int i = threadIdx.x; i < kSortPasses * kDigits; i += 256) {
      const uint32_t v = s_count[i];
      s_count[i] = 0;
      if (v) atomicAdd(ghist + i, (unsigned long long)v);
    }
    __syncthreads();
    t = seg_end;
  }
}

// per client: exclusive scans of the four digit histograms and the mask of constant digits
__global__ void __launch_bounds__(kDigits)
k_sort_scan(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L) {
  __shared__ unsigned long long s_scan[kDigits / 32];
  pdl_enter();
  const EncHeader* hdr = reinterpret_cast<const EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const uint32_t c = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const cvlc_plan_t* plan = batch.c[c].plan;
  const unsigned long long* ghist = reinterpret_cast<const unsigned long long*>(ws + L.off_ghist) + (size_t)c * kSortPasses * kDigits;
  unsigned long long* gbase = reinterpret_cast<unsigned long long*>(ws + L.off_gbase) + (size_t)c * kSortPasses * kDigits;
  uint32_t mask = top_digit_is_zero(plan) ? 1u << (kSortPasses - 1) : 0u;  // not counted: known to be constant
  for (int p = 0; p < kSortPasses; ++p) {
    const unsigned long long cnt = ghist[p * kDigits + tid];
    if (__syncthreads_or(cnt == plan->n_candidates)) mask |= 1u << p;
    unsigned long long incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned long long o = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) s_scan[warp] = incl;
    __syncthreads();
    unsigned long long below = 0;
    for (int w = 0; w < warp; ++w) below += s_scan[w];
    gbase[p * kDigits + tid] = below + incl - cnt;
    __syncthreads();
  }
  if (tid == 0) reinterpret_cast<uint32_t*>(ws + L.off_pass_mask)[c] = mask;
}

__global__ void __launch_bounds__(kSortThreads, kSortMinBlocks)
k_sort_pass(const Batch batch, unsigned char* ws, const __grid_constant__ EncLayout L, int pass) {
  static_assert(kSortThreads * 2 == kDigits && kSortTile <= 0xFFFF, "two digit values per thread; 16-bit slots");
  extern __shared__ __align__(16) unsigned char s_raw[];
  SortShared& sh = *reinterpret_cast<SortShared*>(s_raw);
  unsigned long long* s_items = reinterpret_cast<unsigned long long*>(s_raw + kSortSharedBytes);  // [kSortTile] the tile's items in digit order
  uint32_t* s_prefix = reinterpret_cast<uint32_t*>(s_items + kSortTile);                         // [n + 1] first sort tile of every client
  uint32_t* s_ncand = s_prefix + (batch.n + 1);  // [n] candidates of the client
  uint32_t* s_keytop = s_ncand + batch.n;        // [n] top of its key range
  uint32_t* s_mask = s_keytop + batch.n;         // [n] its constant digits
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  if (block_sees_error(&hdr->status)) return;
  const int tid = threadIdx.x;
  const uint32_t n = batch.n;
  {
    const uint32_t* prefix = reinterpret_cast<const uint32_t*>(ws + L.off_sort_prefix);
    const uint32_t* pass_mask = reinterpret_cast<const uint32_t*>(ws + L.off_pass_mask);
    for (uint32_t i = tid; i <= n; i += kSortThreads) s_prefix[i] = prefix[i];
    uint32_t moves = 0;  // some client's digit is not constant
    for (uint32_t i = tid; i < n; i += kSortThreads) {
      const cvlc_plan_t* plan = batch.c[i].plan;
      s_ncand[i] = (uint32_t)plan->n_candidates;  // <= capacity < 2^32: checked by k_encode_init
      s_keytop[i] = sort_keytop(plan);
      s_mask[i] = pass_mask[i];
      moves |= ~s_mask[i] & (1u << pass);
    }
    if (!__syncthreads_or(moves)) return;
  }
  for (int i = tid; i < (kSortThreads / 32) * kDigits; i += kSortThreads) (&sh.mm[0][0])[i] = 0u;
  if (tid == 0) sh.tile = atomicAdd(&hdr->sort_ticket[pass], 1u);
  __syncthreads();
  const uint32_t tickets = hdr->max_sort_tiles * n;
  unsigned long long* state_all =
      reinterpret_cast<unsigned long long*>(ws + L.off_sort_state) + (size_t)pass * n * L.sort_tiles_max * kDigits;
  uint4* s_wc4 = reinterpret_cast<uint4*>(&sh.wc[0][0]);

  while (true) {
    const uint32_t gt = sh.tile;
    if (gt >= tickets) break;
    s_wc4[2 * tid] = make_uint4(0u, 0u, 0u, 0u);
    s_wc4[2 * tid + 1] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();  // everyone has read the ticket; the counters are clear
    // the next ticket is fetched while this tile is worked on
    uint32_t next = 0;
    if (tid == 0) next = atomicAdd(&hdr->sort_ticket[pass], 1u);
    // tile-major tickets with the clients interleaved: the tiles in flight are a few consecutive
    // tiles of every client, which keeps every look-back short
    const uint32_t tile = gt / n, c = gt - tile * n;
    const uint32_t mask = s_mask[c];
    auto source = [&](uint32_t cc) -> unsigned long long* {  // buffer holding client cc's items before this pass
      const int flips = __popc(~s_mask[cc] & ((1u << pass) - 1u));
      return reinterpret_cast<unsigned long long*>(ws + ((flips & 1) ? L.off_buf_b : L.off_buf_a)) + (size_t)cc * L.capacity;
    };
    if (tile < s_prefix[c + 1] - s_prefix[c] && !(mask & (1u << pass))) {  // else: no such tile, or a constant digit
      const uint32_t n32 = s_ncand[c];
      const uint32_t keytop = s_keytop[c];
      const int flips = __popc(~mask & ((1u << pass) - 1u));
      const unsigned long long* src = source(c);
      unsigned long long* dst =
          reinterpret_cast<unsigned long long*>(ws + ((flips & 1) ? L.off_buf_a : L.off_buf_b)) + (size_t)c * L.capacity;
      unsigned long long* state = state_all + (size_t)s_prefix[c] * kDigits;
      const unsigned long long* gbase = reinterpret_cast<const unsigned long long*>(ws + L.off_gbase) + ((size_t)c * kSortPasses + pass) * kDigits;
      const uint32_t tile_first = tile * (uint32_t)kSortTile;
      const uint32_t count = (n32 - tile_first < (uint32_t)kSortTile) ? n32 - tile_first : (uint32_t)kSortTile;
      // the next tile's items are asked into L2 while this one is ranked and written
      auto prefetch_next = [&](uint32_t nt) {
        if (nt >= tickets) return;
        const uint32_t t2 = nt / n, c2 = nt - t2 * n;
        for (uint32_t l = tid; l < (uint32_t)(kSortTile / 16); l += kSortThreads) {  // 128-byte lines of 16 items
          const uint32_t line = t2 * (uint32_t)(kSortTile / 16) + l;
          if (line * 16u < s_ncand[c2]) {
            const unsigned long long* p = source(c2) + (size_t)line * 16;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
          }
        }
      };
      if (count == (uint32_t)kSortTile)
        sort_tile<true>(sh, s_items, src, dst, state, gbase, tile, count, n32, keytop, kDigitBits * pass, &hdr->status, next, prefetch_next);
      else
        sort_tile<false>(sh, s_items, src, dst, state, gbase, tile, count, n32, keytop, kDigitBits * pass, &hdr->status, next, prefetch_next);
    }
    if (tid == 0) sh.tile = next;
    __syncthreads();
  }
}

// ===================================================================================
// K5  per-packet centroid distribution (PQ: min/max; QSGD: l2-norm), stochastic quantization, bit packing
// ===================================================================================
// One warp works through kPackGroup consecutive packets of one client, without block-wide barriers; where a batch has so few packets
// that most of the chip would stand idle, the block's four warps share one.  Packet r (longest codes first) holds ranks
// [Z, Z + cap(y_r)).  The packet is assembled in a shared-memory buffer: every record ORs its bits into the (at most three) 32-bit
// words it touches, then the words go out with consecutive addresses.  The ranked pairs are read twice from global memory
// (statistics, then quantization); the second read hits in cache.  A lane of a warp alone quantizes about twelve records of a packet
// one after the other, one of four warps three.

constexpr int kPackThreads = 128;
constexpr int kPackWarps = kPackThreads / 32;
constexpr int kPackGroup = 1;  // packets per warp (more of them amortise the length table but lengthen the tail)
// A block works on a packet where all of them are resident at a time (9 blocks per SM) and have records for its threads; with packets of
// 4.5 KB and more up to a half beyond that.  Block minus warp for a packet, whole encoding calls of one client, us, at 200 / 600 / 1000 /
// 1332 / 1500 / 1924 packets of 1500 bytes -1.8 / -0.8 / -0.1 / 0 / +1.2 / +2.1 (QSGD, whose norm is one lane's chain in both: -2.1 / -3.6
// / -2.0 / -1.4 / +2.7 / +1.9), of 752 bytes -0.7 / -0.9 / -0.2 / -1.1 / +2.0 / +2.1, of 256 bytes 0 / +0.1 / +0.4 / +0.8 / +2.0 / +2.1 (QSGD
// -0.8 / -0.3 / -0.6 / -0.9 / +1.9 / +2.0), of 32 bytes -0.2 / +0.8 / +0.2 / +0.1 / +2.1 / +2.1; at 1332 / 1700 / 1924 / 2300 packets of 3000
// bytes -1.1 / +0.9 / +0.3 / +0.1, of 4500 -7.2 / +0.1 / -3.8 / -1.4 (8 clients -6.3 / -4.9 / -5.1 / -3.5).  Between the two lines it
// also depends on the values: 1340 to 1920 packets of 1500 bytes, one and four clients, +1 to +7 for one Laplace distribution, -3.5 to 0 for
// layers of different scales; 8 and 24 clients -1.6 to +3.
inline bool pack_team(uint64_t packets, bool qsgd, uint32_t records, size_t packet_bytes) {
  return records >= (qsgd ? 48u : 128u) && packets <= (!qsgd && packet_bytes >= 4500 ? 13u : 9u) * (uint64_t)kNumSM;
}

template <int CAP, bool QSGD, int TEAM>
__global__ void __launch_bounds__(kPackThreads)
k_pack(const __grid_constant__ BatchDesc<CAP> batch, const __grid_constant__ Shape shape, unsigned char* ws,
       const __grid_constant__ EncLayout L, uint32_t warp_bytes, int write_residual) {
  [[maybe_unused]] __shared__ float s_team[2][TEAM];
  extern __shared__ __align__(16) unsigned char s_pack[];  // per packet at work: packet words; QSGD: then cap(1) squares
  static_assert(TEAM == 1 || TEAM == kPackWarps, "a warp or the block for a packet");
  constexpr uint32_t STEP = TEAM * 32;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(ws);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t at = TEAM == 1 ? lane : tid;  // thread of the packet's
  auto sync = [] {
    if constexpr (TEAM == 1) __syncwarp();
    else __syncthreads();
  };
  const uint32_t c = blockIdx.y;
  const ClientDesc& cd = batch.c[c];
  const cvlc_plan_t* __restrict__ plan = cd.plan;
  // packet -> its code length and first rank: lane l holds length 32 - l (longest first), below with the
  // inclusive sums of packets and of records up to and including that length
  const uint32_t yl = CVLC_MAX_CODE_BITS - lane;
  const uint32_t ny = plan->n_y[yl];
  const uint32_t capl = plan->cap[yl];
  const unsigned long long plan_k = plan->k, plan_candidates = plan->n_candidates;
  const uint32_t mask = reinterpret_cast<const uint32_t*>(ws + L.off_pass_mask)[c];
  if (block_sees_error(&hdr->status)) return;  // looked at behind the others' requests
  const uint32_t s = shape.s;
  const uint32_t H = shape.header_bits;
  const uint32_t n_words = shape.packet_bits / 32;
  unsigned char* s_mine = s_pack + (TEAM == 1 ? (size_t)warp * warp_bytes : 0);
  uint32_t* words = reinterpret_cast<uint32_t*>(s_mine);
  uint32_t* stream_words = reinterpret_cast<uint32_t*>(cd.stream);
  // error compensation: the encoder's input is memory + update and becomes the new memory, i.e. every sent
  // coordinate gives up what the parameter server will rebuild for it (its centroid value divided by B)
  float* __restrict__ residual = write_residual ? const_cast<float*>(cd.x) : nullptr;
  const PhiloxRoundKeys rk = philox_round_keys(cd.seed);

  const int flips = __popc(~mask & ((1u << kSortPasses) - 1u));
  const unsigned long long* __restrict__ sorted =
      reinterpret_cast<const unsigned long long*>(ws + ((flips & 1) ? L.off_buf_b : L.off_buf_a)) + (size_t)c * L.capacity;

  const unsigned long long nz = (unsigned long long)ny * capl;
  uint32_t cum = ny;
  unsigned long long zc = nz;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t a = __shfl_up_sync(kFull, cum, off);
    const unsigned long long b = __shfl_up_sync(kFull, zc, off);
    if (lane >= off) {
      cum += a;
      zc += b;
    }
  }
  {
    // the code lengths must fill the stream's R packets with k of the selected candidates (every warp of every
    // block of the client sees the same plan and takes the same branch)
    const uint32_t tot_packets = __shfl_sync(kFull, cum, 31);
    const unsigned long long tot_records = __shfl_sync(kFull, zc, 31);
    const bool qsgd_one_bit = QSGD && __shfl_sync(kFull, ny, 31) != 0;  // a one-bit QSGD code holds no level
    if (tot_packets != shape.R || tot_records != plan_k || tot_records == 0 || tot_records > plan_candidates ||
        tot_records > (unsigned long long)shape.R * shape.cap[1] || qsgd_one_bit) {
      if (blockIdx.x == 0 && tid == 0) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);
      return;
    }
  }

  for (int g = 0; g < kPackGroup; ++g) {
    const uint32_t r = (TEAM == 1 ? blockIdx.x * kPackWarps + warp : blockIdx.x) * kPackGroup + g;
    if (r >= shape.R) break;
    const unsigned hit = __ballot_sync(kFull, r < cum);
    if (hit == 0) break;
    const int src_lane = __ffs(hit) - 1;
    const uint32_t y = CVLC_MAX_CODE_BITS - (uint32_t)src_lane;
    const unsigned long long Z = __shfl_sync(kFull, (zc - nz) + (unsigned long long)(r - (cum - ny)) * capl, src_lane);
    const uint32_t P = __shfl_sync(kFull, capl, src_lane);
    for (uint32_t w = at; w < n_words; w += STEP) words[w] = 0u;
    sync();
    const uint32_t wd = s + y;
    const unsigned long long* __restrict__ seg = sorted + Z;
    float lo, hi;  // the header's two centroid fields
    // a record's bits, low bit first from packet bit H + j * wd
    const bool narrow = wd <= 32;  // a record then touches at most two words
    auto put = [&](uint32_t j, unsigned long long rec) {
      const uint32_t bitpos = H + j * wd;
      const uint32_t w = bitpos >> 5, sh = bitpos & 31u;
      if (narrow) {
        const uint32_t r32 = (uint32_t)rec;
        const uint32_t p0 = r32 << sh, p1 = __funnelshift_l(r32, 0u, sh);  // the bits that leave the first word
        if (p0) atomicOr(words + w, p0);
        if (p1) atomicOr(words + w + 1, p1);
        return;
      }
      const unsigned long long lo64 = rec << sh;
      const uint32_t p0 = (uint32_t)lo64, p1 = (uint32_t)(lo64 >> 32);
      const uint32_t p2 = sh ? (uint32_t)(rec >> (64 - sh)) : 0u;
      if (p0) atomicOr(words + w, p0);
      if (p1) atomicOr(words + w + 1, p1);
      if (p2) atomicOr(words + w + 2, p2);
    };

    if constexpr (QSGD) {
      // ---- QSGD: |x| against the packet's l2-norm; code = sign bit above a level of s_q = 2^(y-1) - 1 steps ----
      double* sqv = reinterpret_cast<double*>(s_mine + (((size_t)n_words * 4 + 8 + 15) & ~(size_t)15));
      for (uint32_t j = at; j < P; j += STEP) {
        const double a = (double)__uint_as_float((uint32_t)(seg[j] >> 32));
        sqv[j] = __dmul_rn(a, a);  // exact: 24 x 24 bits
      }
      sync();
      // the norm is defined with the squares added in rank order in double: one lane walks the chain
      float norm = 0.0f;
      if (at == 0) norm = qsgd_norm_of_squares(sqv, P);
      if constexpr (TEAM == 1) {
        norm = __shfl_sync(kFull, norm, 0);
      } else {
        if (at == 0) s_team[0][0] = norm;
        __syncthreads();
        norm = s_team[0][0];
      }
      lo = norm;
      hi = 0.0f;
      const uint32_t sq = (uint32_t)((1ull << (y - 1)) - 1ull);  // y >= 2: checked with the plan
      const double sqd = (double)sq;
      const double dn = (double)norm;
      const double scale = (norm > 0.0f) ? __ddiv_rn(sqd, dn) : 0.0;
      const float fscale = fast_scale(scale, y - 1);
      for (uint32_t j = at; j < P; j += STEP) {
        const unsigned long long pair = seg[j];
        const uint32_t key = (uint32_t)(pair >> 32);
        const uint32_t pid = (uint32_t)pair & 0x7FFFFFFFu;
        const uint32_t sign = key ? (((uint32_t)pair >> 31) & 1u) : 0u;  // -0 is stored as +0
        uint32_t level = 0;
        if (norm > 0.0f) {
          const uint32_t word = philox_coord(rk, cd.client_id, cd.round, pid);
          if (!fast_round(__uint_as_float(key), fscale, (float)sqd, word, level)) level = qsgd_quantize_slow(__uint_as_float(key), norm, sq, word);
        }
        const uint32_t code = (sign << (y - 1)) | level;
        put(j, (unsigned long long)pid | ((unsigned long long)code << s));
        if (residual) {
          const float mag = (float)__dmul_rn((double)level, __ddiv_rn(dn, sqd));
          const float v = sign ? -mag : mag;
          const float xv = __uint_as_float(key ? (key | ((uint32_t)pair & 0x80000000u)) : 0u);
          residual[pid] = __fsub_rn(xv, (float)__ddiv_rn((double)v, cd.scale_B));
        }
      }
    } else {
      // ---- PQ: minimum / maximum of the packet's signed values (its centroid distribution) ----
      float vmin = CUDART_INF_F, vmax = -CUDART_INF_F;
      for (uint32_t j = at; j < P; j += STEP) {
        const unsigned long long pair = seg[j];
        const uint32_t key = (uint32_t)(pair >> 32);
        const uint32_t b = key ? (key | ((uint32_t)pair & 0x80000000u)) : 0u;  // -0 is stored as +0
        const float v = __uint_as_float(b);
        vmin = fminf(vmin, v);
        vmax = fmaxf(vmax, v);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        vmin = fminf(vmin, __shfl_xor_sync(kFull, vmin, off));
        vmax = fmaxf(vmax, __shfl_xor_sync(kFull, vmax, off));
      }
      if constexpr (TEAM > 1) {
        if (lane == 0) {
          s_team[0][warp] = vmin;
          s_team[1][warp] = vmax;
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < TEAM; ++w) {
          vmin = fminf(vmin, s_team[0][w]);
          vmax = fmaxf(vmax, s_team[1][w]);
        }
      }
      lo = vmin;
      hi = vmax;

      // stochastic rounding onto the 2^y uniform centroids of [lo, hi]
      const double Lc = (double)((1ull << y) - 1ull);
      const double dlo = (double)lo;
      const double den = __dsub_rn((double)hi, dlo);
      const double scale = (hi != lo) ? __ddiv_rn(Lc, den) : 0.0;
      const float fscale = fast_scale(scale, y);
      const double cstep = (hi != lo) ? __ddiv_rn(den, Lc) : 0.0;  // distance of two centroids
      const bool plain = !residual && hi != lo;
      if (plain) {
        // the usual case, without a branch but for the rounding fp32 cannot tell; the next record is requested ahead
        const float fL = (float)Lc;
        unsigned long long next = at < P ? seg[at] : 0ull;
        uint32_t bitpos = H + at * wd;
        for (uint32_t j = at; j < P; j += STEP, bitpos += STEP * wd) {
          const unsigned long long pair = next;
          if (j + STEP < P) next = seg[j + STEP];
          const uint32_t key = (uint32_t)(pair >> 32), pid = (uint32_t)pair & 0x7FFFFFFFu;
          const float v = __uint_as_float(key | ((uint32_t)pair & 0x80000000u));
          const uint32_t word = philox_coord(rk, cd.client_id, cd.round, pid);
          uint32_t code;
          if (!fast_round(__fsub_rn(v, lo), fscale, fL, word, code)) code = pq_quantize_slow(v, lo, hi, y, word);
          const uint32_t r0 = pid | (code << s), sh = bitpos & 31u;
          uint32_t* w = words + (bitpos >> 5);
          atomicOr(w, r0 << sh);
          if (narrow) {
            atomicOr(w + 1, __funnelshift_l(r0, 0u, sh));  // zero behind the packet's last word
          } else {
            const uint32_t r1 = __funnelshift_l(code, 0u, s);
            atomicOr(w + 1, __funnelshift_l(r0, r1, sh));
            atomicOr(w + 2, __funnelshift_l(r1, 0u, sh));
          }
        }
      }
      for (uint32_t j = plain ? P : at; j < P; j += STEP) {
        const unsigned long long pair = seg[j];
        const uint32_t key = (uint32_t)(pair >> 32);
        const uint32_t pid = (uint32_t)pair & 0x7FFFFFFFu;
        const uint32_t b = key ? (key | ((uint32_t)pair & 0x80000000u)) : 0u;
        uint32_t code = 0;
        if (hi != lo) {
          const uint32_t word = philox_coord(rk, cd.client_id, cd.round, pid);
          if (!fast_round(__fsub_rn(__uint_as_float(b), lo), fscale, (float)Lc, word, code)) code = pq_quantize_slow(__uint_as_float(b), lo, hi, y, word);
        }
        put(j, (unsigned long long)pid | ((unsigned long long)code << s));
        if (residual) {
          const float v = (hi != lo) ? (float)__dadd_rn(dlo, __dmul_rn((double)code, cstep)) : lo;
          residual[pid] = __fsub_rn(__uint_as_float(b), (float)__ddiv_rn((double)v, cd.scale_B));
        }
      }
    }  // PQ

    // packet header {s, y, lo, hi} in bits 0..79 (bits 80..H-1 stay zero)
    if (at == 0) {
      const uint32_t blo = __float_as_uint(lo), bhi = __float_as_uint(hi);
      atomicOr(words + 0, s | (y << 8) | (blo << 16));
      atomicOr(words + 1, (blo >> 16) | (bhi << 16));
      atomicOr(words + 2, bhi >> 16);
    }
    sync();
    uint32_t* pkt = stream_words + CVLC_STREAM_HEADER_BYTES / 4 + (size_t)r * n_words;
    for (uint32_t w = at; w < n_words; w += STEP) pkt[w] = words[w];
    sync();  // the word buffer is reused by the next packet
  }

  // global header (64 bytes), written once per client
  if (blockIdx.x == 0 && tid < 16) {
    uint32_t v = 0;
    const unsigned long long Bbits = (unsigned long long)__double_as_longlong(cd.scale_B);
    const unsigned long long k = plan->k;
    switch (tid) {
      case 0: v = CVLC_STREAM_MAGIC; break;
      case 1: v = 1u | (shape.quantizer << 16) | (s << 24); break;
      case 2: v = (uint32_t)shape.d; break;
      case 3: v = (uint32_t)(shape.d >> 32); break;
      case 4: v = shape.R; break;
      case 5: v = shape.packet_bits; break;
      case 6: v = shape.header_bits; break;
      case 7: v = cd.client_id; break;
      case 8: v = (uint32_t)cd.seed; break;
      case 9: v = (uint32_t)(cd.seed >> 32); break;
      case 10: v = cd.round; break;
      case 11: v = 0; break;
      case 12: v = (uint32_t)Bbits; break;
      case 13: v = (uint32_t)(Bbits >> 32); break;
      case 14: v = (uint32_t)k; break;
      default: v = (uint32_t)(k >> 32); break;
    }
    stream_words[tid] = v;
  }
}

// ===================================================================================
// launcher
// ===================================================================================

template <int CAP>
static void launch_init_t(const ClientDesc* clients, uint32_t n, const Shape& shape, const EncLayout& L, const unsigned char* plan_ws,
                          unsigned char* w, cudaStream_t st) {
  BatchDesc<CAP> batch;
  batch.n = n;
  batch.pad = 0;
  memcpy(batch.c, clients, (size_t)n * sizeof(ClientDesc));
  launch_kernel(kKEncodeInit, k_encode_init<CAP>, 2 * kNumSM, 256, 0, st, false, w, batch, shape, L, plan_ws);
}

// What the largest packets take is allowed to every form of the kernel beforehand.  (Asked for where a launch has more than 48 KB of its
// own, that line would have to count the kernel's static shared memory too.)
template <int CAP>
static cudaError_t pack_attributes() {
  cudaError_t e = allow_shared(k_pack<CAP, false, 1>, kPackSharedMax);
  if (e == cudaSuccess) e = allow_shared(k_pack<CAP, false, kPackWarps>, kPackSharedMax);
  if (e == cudaSuccess) e = allow_shared(k_pack<CAP, true, 1>, kPackSharedMax);
  return e != cudaSuccess ? e : allow_shared(k_pack<CAP, true, kPackWarps>, kPackSharedMax);
}

template <int CAP>
static cudaError_t launch_pack_t(const ClientDesc* clients, uint32_t n, const Shape& shape, const EncLayout& L, unsigned char* w, size_t warp_bytes,
                                 int write_residual, cudaStream_t st, bool overlap) {
  const bool qsgd = shape.quantizer == CVLC_QUANT_QSGD;
  const bool team = pack_team((uint64_t)shape.R * n, qsgd, shape.cap[1], shape.packet_bits / 8);
  auto kernel = team ? (qsgd ? k_pack<CAP, true, kPackWarps> : k_pack<CAP, false, kPackWarps>) : (qsgd ? k_pack<CAP, true, 1> : k_pack<CAP, false, 1>);
  const uint32_t at_work = team ? 1 : kPackWarps;  // packets of a block
  BatchDesc<CAP> batch;
  batch.n = n;
  batch.pad = 0;
  memcpy(batch.c, clients, (size_t)n * sizeof(ClientDesc));
  const unsigned grid = (shape.R + at_work * kPackGroup - 1) / (at_work * kPackGroup);
  launch_kernel(kKPack, kernel, dim3(grid, n), kPackThreads, warp_bytes * at_work, st, overlap, batch, shape, w, L, (uint32_t)warp_bytes, write_residual);
  return cudaGetLastError();
}

cudaError_t launch_pack(const ClientDesc* clients, uint32_t n, const Shape& shape, uint64_t capacity, void* ws, cudaStream_t st, bool overlap,
                        int write_residual) {
  const EncLayout L = enc_layout(shape.d, n, capacity);
  unsigned char* w = static_cast<unsigned char*>(ws);
  // packet words and two more; QSGD: and the squares of a packet's values
  const size_t pack_warp = (((size_t)shape.packet_bits / 8 + 8 + 15) & ~(size_t)15) + (shape.quantizer == CVLC_QUANT_QSGD ? (size_t)shape.cap[1] * 8 : 0);
  if (n <= (uint32_t)kSmallBatch) return launch_pack_t<kSmallBatch>(clients, n, shape, L, w, pack_warp, write_residual, st, overlap);
  if (n <= (uint32_t)kMediumBatch) return launch_pack_t<kMediumBatch>(clients, n, shape, L, w, pack_warp, write_residual, st, overlap);
  return launch_pack_t<kLargeBatch>(clients, n, shape, L, w, pack_warp, write_residual, st, overlap);
}

cudaError_t launch_encode(const ClientDesc* clients, uint32_t n, const Shape& shape, uint64_t capacity,
                          const void* plan_ws, void* ws, cudaStream_t st, bool prepared, bool behind_wait, cudaEvent_t wait_before_pack,
                          int write_residual, bool ranked) {
  static OncePerDevice once;
  cudaError_t e = once_per_device(once, [] {
    cudaError_t e = allow_shared(k_select, kSelSmem);
    if (e == cudaSuccess) e = allow_shared(k_sort_pass, sort_smem_bytes(CVLC_MAX_BATCH));
    if (e == cudaSuccess) e = pack_attributes<kSmallBatch>();
    if (e == cudaSuccess) e = pack_attributes<kMediumBatch>();
    return e != cudaSuccess ? e : pack_attributes<kLargeBatch>();
  });
  if (e != cudaSuccess) return e;
  const EncLayout L = enc_layout(shape.d, n, capacity);
  if (enc_lists_end(L) > L.off_buf_a) return cudaErrorInvalidValue;
  unsigned char* w = static_cast<unsigned char*>(ws);
  if (ranked) {
    e = launch_rank_rest(Batch{nullptr, n}, L, static_cast<const unsigned char*>(plan_ws), w, kNumSM, false, st);
    return e != cudaSuccess ? e : launch_pack(clients, n, shape, capacity, ws, st, true, write_residual);
  }
  const Partition part = make_partition(shape.d, n);
  const unsigned sms = wait_before_pack && tune_place(shape.d, n) == kTuneRoomLeft ? kNumSM - n : kNumSM;
  const unsigned char* pws = static_cast<const unsigned char*>(plan_ws);
  Batch batch{reinterpret_cast<const ClientDesc*>(w + L.off_desc), n};
  if (prepared) batch.c = reinterpret_cast<const ClientDesc*>(pws + plan_off_desc(n));
  else if (n <= (uint32_t)kSmallBatch) launch_init_t<kSmallBatch>(clients, n, shape, L, pws, w, st);
  else if (n <= (uint32_t)kMediumBatch) launch_init_t<kMediumBatch>(clients, n, shape, L, pws, w, st);
  else launch_init_t<kLargeBatch>(clients, n, shape, L, pws, w, st);
  if (pws) {
    const SelectGroups sg = select_groups(part, n);  // here: its divisions in every warp took a microsecond
    const uint64_t want = (uint64_t)sg.groups * n;
    const unsigned grid = (unsigned)(want < (uint64_t)sms ? want : sms);
    launch_kernel(kKSelect, k_select, grid, kSelThreads, kSelSmem, st, !behind_wait, batch, shape.d, part, sg, pws, w, L);
    const uint64_t most = (uint64_t)shape.R * shape.cap[1];
    e = launch_rank(batch, L, pws, w, sms, most < shape.d ? most : shape.d, st);
    if (e != cudaSuccess) return e;
  } else {
    const uint64_t want = select_tiles_of(shape.d) * n;
    const unsigned grid = (unsigned)(want < (uint64_t)(4 * kNumSM) ? want : 4 * kNumSM);
    launch_kernel(kKSelectLookback, k_select_lookback, grid, kSelectThreads, 0, st, true, batch, shape.d, w, L);
    const uint64_t tiles = L.sort_tiles_max * n;
    auto blocks = [&](uint64_t most) -> unsigned { return (unsigned)(tiles < most ? tiles : most); };
    launch_kernel(kKSort, k_sort_hist, blocks(8 * kNumSM), 256, 0, st, true, batch, w, L);
    launch_kernel(kKSort, k_sort_scan, n, kDigits, 0, st, true, batch, w, L);
    for (int pass = 0; pass < kSortPasses; ++pass)
      launch_kernel(kKSort, k_sort_pass, blocks(kSortMinBlocks * kNumSM), kSortThreads, sort_smem_bytes(n), st, true, batch, w, L, pass);
  }
  if (wait_before_pack) {
    const cudaError_t ew = cudaStreamWaitEvent(st, wait_before_pack, 0);
    if (ew != cudaSuccess) return ew;
  }
  if (write_residual == kPackNone) return cudaGetLastError();  // the caller goes on from the ranked records
  return launch_pack(clients, n, shape, capacity, ws, st, wait_before_pack == nullptr, write_residual);
}

// memory <- memory + update in fp32, for every client of a batch (the first step of a round with error compensation)
struct EcPair {
  float* memory;
  const float* update;
};
template <int CAP>
struct EcBatch {
  uint32_t n, pad;
  EcPair c[CAP];
};

template <int CAP>
__global__ void __launch_bounds__(256)
k_ec_accumulate(const __grid_constant__ EcBatch<CAP> batch, uint64_t d) {
  pdl_enter();
  const uint64_t nvec = d >> 2;
  const uint64_t per_client = nvec + 1;  // float4 units and one unit for the ragged tail
  const uint64_t total = per_client * batch.n;
  for (uint64_t g = (uint64_t)blockIdx.x * 256 + threadIdx.x; g < total; g += (uint64_t)gridDim.x * 256) {
    const uint32_t c = (uint32_t)(g / per_client);
    const uint64_t v = g - (uint64_t)c * per_client;
    float* m = batch.c[c].memory;
    const float* u = batch.c[c].update;
    if (v < nvec) {
      float4 a = reinterpret_cast<float4*>(m)[v];
      const float4 b = __ldg(reinterpret_cast<const float4*>(u) + v);
      a.x = __fadd_rn(a.x, b.x);
      a.y = __fadd_rn(a.y, b.y);
      a.z = __fadd_rn(a.z, b.z);
      a.w = __fadd_rn(a.w, b.w);
      reinterpret_cast<float4*>(m)[v] = a;
    } else {
      for (uint64_t i = nvec << 2; i < d; ++i) m[i] = __fadd_rn(m[i], u[i]);
    }
  }
}

template <int CAP>
static void launch_ec_t(float* const* memory, const float* const* update, uint32_t n, uint64_t d, cudaStream_t st) {
  EcBatch<CAP> batch;
  batch.n = n;
  batch.pad = 0;
  for (uint32_t i = 0; i < n; ++i) {
    batch.c[i].memory = memory[i];
    batch.c[i].update = update[i];
  }
  const uint64_t want = (((d >> 2) + 1) * n + 255) / 256;
  const unsigned grid = (unsigned)(want < (uint64_t)(8 * kNumSM) ? want : 8 * kNumSM);
  launch_kernel(kKEcAccumulate, k_ec_accumulate<CAP>, grid, 256, 0, st, false, batch, d);
}

cudaError_t launch_ec_accumulate(float* const* memory, const float* const* update, uint32_t n, uint64_t d, cudaStream_t st) {
  if (n <= (uint32_t)kMediumBatch) launch_ec_t<kMediumBatch>(memory, update, n, d, st);
  else launch_ec_t<kLargeBatch>(memory, update, n, d, st);
  return cudaGetLastError();
}

// The bounded wait of the look-back scans, run on a word nobody publishes: after max_polls polls it gives up,
// reports DEVICE_TIMEOUT and the kernel returns.
__global__ void k_selftest_wait(const unsigned long long* word, int32_t* status, int max_polls) {
  wait_state(word, status, max_polls);
}

cudaError_t launch_selftest_wait(unsigned long long* word, int32_t* status, uint32_t max_polls, cudaStream_t st) {
  { LaunchScope ls(kKSelftest, st); k_selftest_wait<<<1, 32, 0, st>>>(word, status, (int)max_polls); }
  return cudaGetLastError();
}

}  // namespace cvlc
