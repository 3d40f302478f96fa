// Unframed stream (version 2): the records of every packet without the packet frame.
//
// Section IV-C gives every packet one code length and a fixed size because a real network needs a header per
// packet; Proposition 1 itself only groups the top-k coordinates by code length.  Here the groups of the plan are
// kept (block r holds the records of packet r, longest codes first, with that packet's centroid distribution, so
// the plan and its error bound are unchanged), but a block is exactly as long as its records need: no s / y_r
// fields (a table of n_y and cap(y) in the stream header tells which block has which length), no padding, and the
// position IDs of a block are sorted and sent as differences in a Golomb-Rice code.  Records therefore have
// different lengths: bit offsets come from an exclusive prefix sum of the per-record code lengths, inside a block
// by warp scans, across the blocks of a client by a decoupled look-back.
//
// Layout (little-endian, bit i of the body = bit i mod 32 of its 32-bit word i / 32):
//   bytes 0..63    the global header of version 1 with version = 2
//   64..195        n_y[0..32] (uint32): blocks per code length;   196..327  cap[0..32]: records per block
//   328..335       total bits of the body (uint64);   336..  directory: R x uint64 bit offsets of the blocks
//   body           blocks in descending code length: lo (32), hi (32) [PQ min, max; QSGD norm, 0], then the block's
//                  records in ascending position: Rice(position - previous position - 1; previous = -1 at the start
//                  of a block) then the centroid ID (y bits).  Rice parameter m = floor(log2(d / P)); a value v
//                  goes out as v >> m one-bits, a zero bit, the low m bits.
//   size           336 + 8 R + 8 * ceil(total bits / 64) bytes
#include "cvlc_common.cuh"
#include "cvlc_lookback.cuh"
#include "cvlc_quant.cuh"

namespace cvlc {

constexpr int kUfThreads = 128;
constexpr int kUfWarps = kUfThreads / 32;
constexpr size_t kUfSharedMax = 200 * 1024;
constexpr uint32_t kUfCellBits = 9, kUfCells = 1u << kUfCellBits;  // position ranges a block's records are sorted by

// every byte of the output buffers starts at zero: block boundaries share words (they are OR-ed in) and the
// stream ends with zero padding
__global__ void __launch_bounds__(256)
k_uf_clear(const Batch batch, size_t words16, unsigned char* uf_ws, size_t ws_words) {
  pdl_enter();
  const size_t gtid = (size_t)blockIdx.x * 256 + threadIdx.x, gstride = (size_t)gridDim.x * 256;
  const size_t total = words16 * batch.n;
  for (size_t i = gtid; i < total; i += gstride) {
    const uint32_t c = (uint32_t)(i / words16);
    reinterpret_cast<uint4*>(batch.c[c].stream)[i - (size_t)c * words16] = make_uint4(0u, 0u, 0u, 0u);
  }
  for (size_t i = gtid; i < ws_words; i += gstride) reinterpret_cast<uint32_t*>(uf_ws)[i] = 0u;
}

__device__ __forceinline__ void or_bits(uint32_t* img, uint32_t pos, unsigned long long value) {  // up to 64 bits at bit pos
  const uint32_t w = pos >> 5, sh = pos & 31u;
  const unsigned long long lo64 = value << sh;
  const uint32_t p0 = (uint32_t)lo64, p1 = (uint32_t)(lo64 >> 32);
  const uint32_t p2 = sh ? (uint32_t)(value >> (64 - sh)) : 0u;
  if (p0) atomicOr(img + w, p0);
  if (p1) atomicOr(img + w + 1, p1);
  if (p2) atomicOr(img + w + 2, p2);
}

__device__ __forceinline__ void or_ones(uint32_t* img, uint32_t pos, uint32_t count) {  // `count` one-bits from bit pos
  while (count) {
    const uint32_t sh = pos & 31u;
    const uint32_t nb = (32u - sh < count) ? 32u - sh : count;
    const uint32_t mask = (nb == 32u) ? 0xFFFFFFFFu : (((1u << nb) - 1u) << sh);
    atomicOr(img + (pos >> 5), mask);
    pos += nb;
    count -= nb;
  }
}

// A thread block writes one block of records, or each of its four warps writes one.  They are handed out by a per-client ticket, so every
// earlier one of the client is being written or done when a team looks back for its bit offset.  A block of records takes 13 KB of shared
// memory (1500-byte packets): with a warp each an SM holds 16 warps, and the kernel is the chain of one; a thread block each finishes
// sooner wherever all of them are resident at a time.  Short ones are over before four warps' barriers pay: there many warps do it.
// Between events, a warp and a thread block each, us: 8 clients of 1.2 M coordinates at 2 bits in packets of 1500 / 1000 / 512 / 128 / 24 bytes
// 37 and 31 / 34 and 36 / 36 and 50 / 76 and 130 / 320 and 614; one client of 0.3 M 31 and 18 / 27 and 18 / 21 and 17 / 23 and 19 / 25 and
// 31; 4 of 0.6 M in packets of 512 / 376 / 256 bytes (1171, 1595, 2343 blocks) 25 and 22 / 25 and 22 / 28 and 30.  For twelve thread blocks on
// an SM (40 registers) a few words are spilled; with nine 8 clients of 1.2 M take 35.4 instead of 29.1, with sixteen 31.2.
constexpr uint64_t kUfTeamBlocks = 12 * kNumSM;   // blocks of records up to which all are resident, a thread block each
constexpr uint32_t kUfTeamRecords = 16;           // of a block, at least
constexpr size_t kUfTeamBytes = 11 * 1024;        // shared memory of one from which on an SM holds fewer than 20 warps
inline bool uf_team(uint64_t blocks, uint32_t records, size_t bytes) {
  return (blocks <= kUfTeamBlocks && records >= kUfTeamRecords) || bytes > kUfTeamBytes;
}

template <bool QSGD, int TEAM>
__global__ void __launch_bounds__(kUfThreads, TEAM == 1 ? 8 : 12)
k_pack_unframed(const Batch batch, const __grid_constant__ Shape shape, unsigned char* enc_ws,
                const __grid_constant__ EncLayout L, unsigned char* uf_ws, uint32_t P_max, uint32_t img_words, uint32_t team_bytes,
                unsigned long long* __restrict__ sizes_out) {
  extern __shared__ __align__(16) unsigned char s_uf[];  // per block of records
  __shared__ int s_err;
  // across the warps of a team
  [[maybe_unused]] __shared__ uint32_t s_ticket, s_low[TEAM], s_high[TEAM], s_full[TEAM], s_sum[TEAM], s_len[2][TEAM];
  [[maybe_unused]] __shared__ float s_lo[TEAM], s_hi[TEAM];
  [[maybe_unused]] __shared__ unsigned long long s_run;
  static_assert(TEAM == 1 || TEAM == kUfWarps, "a warp or the thread block for a block of records");
  constexpr uint32_t STEP = TEAM * 32;
  pdl_enter();
  EncHeader* hdr = reinterpret_cast<EncHeader*>(enc_ws);
  const uint32_t c = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tid = TEAM == 1 ? (uint32_t)lane : threadIdx.x;  // thread of the team
  auto sync = [] {
    if constexpr (TEAM == 1) __syncwarp();
    else __syncthreads();
  };
  uint32_t* ticket = reinterpret_cast<uint32_t*>(uf_ws + uf_off_ticket()) + c;
  if (threadIdx.x == 0) {
    s_err = *reinterpret_cast<const volatile int32_t*>(&hdr->status);
    if (TEAM > 1) s_ticket = atomicAdd(ticket, 1u);
  }
  __syncthreads();
  if (s_err != 0) return;
  const ClientDesc cd = batch.c[c];
  const cvlc_plan_t* __restrict__ plan = cd.plan;
  const uint32_t R = shape.R;
  unsigned long long* rec = reinterpret_cast<unsigned long long*>(s_uf + (TEAM == 1 ? (size_t)warp * team_bytes : 0));  // [P_max] position << 32 | value bits
  unsigned long long* by_cell = rec + P_max;                                // [P_max] the records by their cells
  double* sqv = reinterpret_cast<double*>(by_cell);                         // QSGD: before that the squares of the values
  uint32_t* cell = reinterpret_cast<uint32_t*>(by_cell + P_max);            // [kUfCells]
  uint32_t* img = cell + kUfCells;                                          // [img_words + 2] the block's bits
  unsigned long long* state = reinterpret_cast<unsigned long long*>(uf_ws + uf_off_state(batch.n)) + (size_t)c * R;
  uint32_t* stream_words = reinterpret_cast<uint32_t*>(cd.stream);
  uint32_t* body = stream_words + uf_head_bytes(R) / 4;

  const uint32_t mask = reinterpret_cast<const uint32_t*>(enc_ws + L.off_pass_mask)[c];
  const int flips = __popc(~mask & ((1u << kSortPasses) - 1u));
  const unsigned long long* __restrict__ sorted =
      reinterpret_cast<const unsigned long long*>(enc_ws + ((flips & 1) ? L.off_buf_b : L.off_buf_a)) + (size_t)c * L.capacity;

  // block -> its code length and first rank: lane l holds length 32 - l with the inclusive sums of blocks and records
  const uint32_t yl = CVLC_MAX_CODE_BITS - lane;
  const uint32_t ny = plan->n_y[yl];
  const uint32_t capl = plan->cap[yl];
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
    const uint32_t tot_blocks = __shfl_sync(kFull, cum, 31);
    const unsigned long long tot_records = __shfl_sync(kFull, zc, 31);
    const bool qsgd_one_bit = QSGD && __shfl_sync(kFull, ny, 31) != 0;
    if (tot_blocks != R || tot_records != plan->k || tot_records == 0 || tot_records > plan->n_candidates ||
        tot_records > (unsigned long long)shape.R * shape.cap[1] || qsgd_one_bit) {
      if (blockIdx.x == 0 && threadIdx.x == 0) set_status(&hdr->status, CVLC_ERR_PLAN_MISMATCH);
      return;
    }
  }

  uint32_t r;
  if constexpr (TEAM == 1) {
    r = 0;
    if (lane == 0) r = atomicAdd(ticket, 1u);
    r = __shfl_sync(kFull, r, 0);
    if (r >= R) return;
  } else {
    r = s_ticket;  // below R: the client has R thread blocks
  }
  const unsigned hit = __ballot_sync(kFull, r < cum);
  const int src_lane = __ffs(hit) - 1;
  const uint32_t y = CVLC_MAX_CODE_BITS - (uint32_t)src_lane;
  const unsigned long long Z = __shfl_sync(kFull, (zc - nz) + (unsigned long long)(r - (cum - ny)) * capl, src_lane);
  const uint32_t P = __shfl_sync(kFull, capl, src_lane);
  const uint32_t m = uf_rice_param(shape.d, P);
  const unsigned long long* __restrict__ seg = sorted + Z;
  const PhiloxRoundKeys rk = philox_round_keys(cd.seed);

  // ---- the block's records and its centroid distribution (over the records in rank order, as for a packet)
  float vmin = CUDART_INF_F, vmax = -CUDART_INF_F;
  uint32_t pmin = 0xFFFFFFFFu, pmax = 0u;
  for (uint32_t j = tid; j < P; j += STEP) {
    const unsigned long long pair = seg[j];
    const uint32_t key = (uint32_t)(pair >> 32), pid = (uint32_t)pair & 0x7FFFFFFFu;
    const uint32_t b = key ? (key | ((uint32_t)pair & 0x80000000u)) : 0u;  // -0 is stored as +0
    if constexpr (QSGD) {
      const double a = (double)__uint_as_float(key);
      sqv[j] = __dmul_rn(a, a);
    } else {
      const float v = __uint_as_float(b);
      vmin = fminf(vmin, v);
      vmax = fmaxf(vmax, v);
    }
    pmin = pid < pmin ? pid : pmin;
    pmax = pid > pmax ? pid : pmax;
    rec[j] = ((unsigned long long)pid << 32) | b;
  }
  pmin = __reduce_min_sync(kFull, pmin);
  pmax = __reduce_max_sync(kFull, pmax);
  if constexpr (!QSGD) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      vmin = fminf(vmin, __shfl_xor_sync(kFull, vmin, off));
      vmax = fmaxf(vmax, __shfl_xor_sync(kFull, vmax, off));
    }
  }
  if (TEAM > 1 && lane == 0) {
    s_low[warp] = pmin;
    s_high[warp] = pmax;
    s_lo[warp] = vmin;
    s_hi[warp] = vmax;
  }
  for (uint32_t i = tid; i < kUfCells; i += STEP) cell[i] = 0u;
  for (uint32_t w = tid; w < img_words + 2; w += STEP) img[w] = 0u;
  sync();
  if constexpr (TEAM > 1) {
#pragma unroll
    for (int w = 0; w < TEAM; ++w) {
      pmin = min(pmin, s_low[w]);
      pmax = max(pmax, s_high[w]);
    }
  }
  float lo, hi;
  if constexpr (QSGD) {
    lo = 0.0f;
    if (tid == 0) lo = qsgd_norm_of_squares(sqv, P);
    if constexpr (TEAM == 1) {
      lo = __shfl_sync(kFull, lo, 0);
    } else {
      if (tid == 0) s_lo[0] = lo;
      sync();
      lo = s_lo[0];
    }
    hi = 0.0f;
  } else {
    lo = vmin;
    hi = vmax;
    if constexpr (TEAM > 1) {
#pragma unroll
      for (int w = 0; w < TEAM; ++w) {
        lo = fminf(lo, s_lo[w]);
        hi = fmaxf(hi, s_hi[w]);
      }
    }
  }

  // ---- ascending position: the records are spread over kUfCells equal ranges of the block's positions, a few in each, and
  // compared with the others of their cell.  Where the positions crowd into few cells, a bitonic network sorts them instead.
  const uint32_t csh = (pmax - pmin) < kUfCells ? 0u : 32u - __clz(pmax - pmin) - kUfCellBits;  // (pmax - pmin) >> csh < kUfCells
  for (uint32_t j = tid; j < P; j += STEP) atomicAdd(cell + (((uint32_t)(rec[j] >> 32) - pmin) >> csh), 1u);
  sync();
  uint32_t fullest;
  {
    constexpr uint32_t kMine = kUfCells / STEP / 4;  // a thread's cells, by fours
    uint4* mine = reinterpret_cast<uint4*>(cell) + tid * kMine;
    uint4 v[kMine];
    uint32_t sum = 0;
    fullest = 0;
#pragma unroll
    for (uint32_t i = 0; i < kMine; ++i) {
      v[i] = mine[i];
      sum += v[i].x + v[i].y + v[i].z + v[i].w;
      fullest = max(fullest, max(max(v[i].x, v[i].y), max(v[i].z, v[i].w)));
    }
    fullest = __reduce_max_sync(kFull, fullest);
    uint32_t run = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, run, off);
      if (lane >= off) run += o;
    }
    if constexpr (TEAM > 1) {
      if (lane == 31) {
        s_sum[warp] = run;
        s_full[warp] = fullest;
      }
      sync();
    }
    run -= sum;
    if constexpr (TEAM > 1) {
#pragma unroll
      for (int w = 0; w < TEAM; ++w) {
        if (w < warp) run += s_sum[w];
        fullest = max(fullest, s_full[w]);
      }
    }
#pragma unroll
    for (uint32_t i = 0; i < kMine; ++i) {
      mine[i] = make_uint4(run, run + v[i].x, run + v[i].x + v[i].y, run + v[i].x + v[i].y + v[i].z);
      run += v[i].x + v[i].y + v[i].z + v[i].w;
    }
  }
  sync();
  if (fullest <= 64) {
    for (uint32_t j = tid; j < P; j += STEP) {
      const unsigned long long e = rec[j];
      by_cell[atomicAdd(cell + (((uint32_t)(e >> 32) - pmin) >> csh), 1u)] = e;
    }
    sync();
    for (uint32_t j = tid; j < P; j += STEP) {
      const unsigned long long e = by_cell[j];
      const uint32_t k = ((uint32_t)(e >> 32) - pmin) >> csh;
      const uint32_t q0 = k ? cell[k - 1] : 0u, q1 = cell[k];  // the places have advanced to the cells' ends
      uint32_t rank = q0;
      for (uint32_t q = q0; q < q1; ++q) rank += by_cell[q] < e ? 1u : 0u;
      rec[rank] = e;
    }
    sync();
  } else {
    // comparators that all point the same way: places behind the last record need none
    uint32_t size = 2;
    while (size < P) size <<= 1;
    for (uint32_t k = 2; k <= size; k <<= 1) {
      for (uint32_t jj = k >> 1; jj > 0; jj >>= 1) {
        const uint32_t flip = (jj == k >> 1) ? k - 1 : jj;  // first step of a merge: against the mirror image
        for (uint32_t t = tid; t < size / 2; t += STEP) {
          const uint32_t i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1)), p = i ^ flip;
          if (p < P) {
            const unsigned long long x = rec[i], z = rec[p];
            if (x > z) {
              rec[i] = z;
              rec[p] = x;
            }
          }
        }
        sync();
      }
    }
  }

  // ---- records, one a thread at a time: code, length, offset by a scan, bits OR-ed into the block's image
  if (tid == 0) {
    img[0] = __float_as_uint(lo);
    img[1] = __float_as_uint(hi);
  }
  sync();
  const double Lc = (double)((1ull << y) - 1ull);
  const double dlo = (double)lo;
  const double den = __dsub_rn((double)hi, dlo);
  const double pq_scale = (hi != lo) ? __ddiv_rn(Lc, den) : 0.0;
  const uint32_t sq = QSGD ? (uint32_t)((1ull << (y - 1)) - 1ull) : 0u;
  const double sqd = (double)sq, dn = (double)lo;
  const double q_scale = (QSGD && lo > 0.0f) ? __ddiv_rn(sqd, dn) : 0.0;
  const float fscale = QSGD ? fast_scale(q_scale, y - 1) : fast_scale(pq_scale, y);
  uint32_t carry = 64;
  for (uint32_t base = 0; base < P; base += STEP) {
    const uint32_t j = base + tid;
    const bool valid = j < P;
    uint32_t len = 0, quo = 0;
    unsigned long long tail = 0;
    if (valid) {
      const unsigned long long e = rec[j];
      const uint32_t pid = (uint32_t)(e >> 32), b = (uint32_t)e;
      const uint32_t prev = j ? (uint32_t)(rec[j - 1] >> 32) + 1u : 0u;
      const uint32_t delta = pid - prev;
      quo = delta >> m;
      uint32_t code = 0;
      const uint32_t word = philox_coord(rk, cd.client_id, cd.round, pid);
      if constexpr (QSGD) {
        const uint32_t key = b & 0x7FFFFFFFu;
        uint32_t level = 0;
        if (lo > 0.0f && !fast_round(__uint_as_float(key), fscale, (float)sqd, word, level))
          level = qsgd_quantize_level((double)__uint_as_float(key), dn, sqd, sq, q_scale, unit_of(word));
        code = ((key ? (b >> 31) : 0u) << (y - 1)) | level;
      } else if (hi != lo) {
        if (!fast_round(__fsub_rn(__uint_as_float(b), lo), fscale, (float)Lc, word, code))
          code = pq_quantize(__dsub_rn((double)__uint_as_float(b), dlo), den, Lc, pq_scale, unit_of(word));
      }
      // after the unary part: the zero bit, the low m bits of the difference, the centroid ID
      tail = ((unsigned long long)(delta & ((1u << m) - 1u)) << 1) | ((unsigned long long)code << (1 + m));
      len = quo + 1u + m + y;
    }
    uint32_t incl = len;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += o;
    }
    uint32_t pos = carry + incl - len;
    if constexpr (TEAM == 1) {
      carry += __shfl_sync(kFull, incl, 31);
    } else {
      uint32_t* sums = s_len[(base / STEP) & 1];  // the last but one's have been read: a barrier lies between
      if (lane == 31) sums[warp] = incl;
      sync();
#pragma unroll
      for (int w = 0; w < TEAM; ++w) {
        if (w < warp) pos += sums[w];
        carry += sums[w];
      }
    }
    if (valid) {
      or_ones(img, pos, quo);
      or_bits(img, pos + quo, tail);
    }
  }
  sync();
  const uint32_t block_bits = carry;

  // ---- bit offset of the block: decoupled look-back over the client's earlier blocks, 32 at a time, by one warp
  if (tid == 0) st_relaxed(state + r, (r == 0 ? kFlagPrefix : kFlagAgg) | block_bits);
  unsigned long long run = 0;
  if (r > 0 && (TEAM == 1 || warp == 0)) {
    long long top = (long long)r - 1;
    while (true) {
      const long long idx = top - lane;
      unsigned long long sv = kFlagPrefix;  // before the client's first block: nothing
      if (idx >= 0) {
        sv = wait_state(state + idx, &hdr->status);
        if (sv == 0) sv = kFlagPrefix;  // gave up (status set): close the chain, the results are void
      }
      const unsigned is_prefix = __ballot_sync(kFull, (sv & kFlagMask) == kFlagPrefix);
      unsigned long long val = sv & kValMask;
      if (is_prefix && lane > __ffs(is_prefix) - 1) val = 0;  // everything behind the nearest prefix is inside it
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) val += __shfl_xor_sync(kFull, val, off);
      run += val;
      if (is_prefix) break;
      top -= 32;
    }
    if (lane == 0) {
      st_relaxed(state + r, kFlagPrefix | (run + block_bits));
      if (TEAM > 1) s_run = run;
    }
  }
  if constexpr (TEAM > 1) {
    sync();
    if (r > 0) run = s_run;
  }

  // ---- the image goes out shifted to its bit offset; the first and the last word are shared with the neighbours
  {
    const uint32_t shift = (uint32_t)(run & 31ull);
    const size_t w0 = (size_t)(run >> 5);
    const uint32_t n_out = (shift + block_bits + 31) >> 5;
    for (uint32_t ow = tid; ow < n_out; ow += STEP) {
      uint32_t v = img[ow] << shift;  // img has two zero words behind its last used one
      if (shift && ow) v |= img[ow - 1] >> (32 - shift);
      if (ow == 0 || ow == n_out - 1) {
        if (v) atomicOr(body + w0 + ow, v);
      } else {
        body[w0 + ow] = v;
      }
    }
    if (tid == 0) {
      unsigned long long* dir = reinterpret_cast<unsigned long long*>(cd.stream + kUfDirectory);
      dir[r] = run;
      if (r == R - 1) {
        const unsigned long long total = run + block_bits;
        *reinterpret_cast<unsigned long long*>(cd.stream + kUfTotalBits) = total;
        if (sizes_out) sizes_out[c] = uf_head_bytes(R) + ((total + 63) / 64) * 8;
      }
    }
  }

  // ---- stream header and the tables of lengths, by the first warp of the team that wrote block 0
  if (r == 0 && (TEAM == 1 || warp == 0)) {
    if (lane < 16) {
      uint32_t v = 0;
      const unsigned long long Bbits = (unsigned long long)__double_as_longlong(cd.scale_B);
      const unsigned long long k = plan->k;
      switch (lane) {
        case 0: v = CVLC_STREAM_MAGIC; break;
        case 1: v = 2u | (shape.quantizer << 16) | (shape.s << 24); break;
        case 2: v = (uint32_t)shape.d; break;
        case 3: v = (uint32_t)(shape.d >> 32); break;
        case 4: v = R; break;
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
      stream_words[lane] = v;
    }
    uint32_t* tab = stream_words + kUfTables / 4;
    tab[lane] = plan->n_y[lane];
    tab[33 + lane] = plan->cap[lane];
    if (lane == 0) {
      tab[32] = plan->n_y[32];
      tab[33 + 32] = plan->cap[32];
    }
  }
}

cudaError_t launch_pack_unframed(uint32_t n, const Shape& shape, uint64_t capacity,
                                 size_t stream_capacity, void* enc_ws, void* uf_ws, unsigned long long* sizes_out, cudaStream_t st) {
  static OncePerDevice once;
  const cudaError_t e = once_per_device(once, [] {
    cudaError_t e = allow_shared(k_pack_unframed<false, 1>, kUfSharedMax);
    if (e == cudaSuccess) e = allow_shared(k_pack_unframed<true, 1>, kUfSharedMax);
    if (e == cudaSuccess) e = allow_shared(k_pack_unframed<false, kUfWarps>, kUfSharedMax);
    return e != cudaSuccess ? e : allow_shared(k_pack_unframed<true, kUfWarps>, kUfSharedMax);
  });
  if (e != cudaSuccess) return e;
  const EncLayout L = enc_layout(shape.d, n, capacity);
  // the encoder has left the descriptors in its workspace
  const Batch batch{reinterpret_cast<const ClientDesc*>(static_cast<unsigned char*>(enc_ws) + L.off_desc), n};
  const bool qsgd = shape.quantizer == CVLC_QUANT_QSGD;
  // the largest block: cap of the shortest admissible length
  const uint32_t y_lo = qsgd ? 2u : 1u;
  const uint32_t P_max = shape.cap[y_lo];
  // bits of a block: 64 of header, per record 1 + m + y, fewer than 2 P one-bits of unary parts in all
  uint64_t bits = 0;
  for (uint32_t y = y_lo; y <= shape.max_code_bits; ++y) {
    const uint64_t b = 64 + (uint64_t)shape.cap[y] * (1 + uf_rice_param(shape.d, shape.cap[y]) + y) + 2 * (uint64_t)shape.cap[y];
    if (b > bits) bits = b;
  }
  const uint32_t img_words = (uint32_t)((bits + 31) / 32);
  const size_t block_bytes = (size_t)P_max * 16 + ((((size_t)img_words + 2 + kUfCells) * 4 + 15) & ~(size_t)15);
  launch_kernel(kKZeroWords, k_uf_clear, 4 * kNumSM, 256, 0, st, true, batch, stream_capacity / 16, static_cast<unsigned char*>(uf_ws),
                uf_ws_bytes(n, shape.R) / 4);
  const bool team = uf_team((uint64_t)shape.R * n, P_max, block_bytes);
  auto kernel = team ? (qsgd ? k_pack_unframed<true, kUfWarps> : k_pack_unframed<false, kUfWarps>)
                     : (qsgd ? k_pack_unframed<true, 1> : k_pack_unframed<false, 1>);
  const uint32_t at_work = team ? 1 : kUfWarps;  // blocks of records of a thread block
  launch_kernel(kKPackUnframed, kernel, dim3((shape.R + at_work - 1) / at_work, n), kUfThreads, block_bytes * at_work, st, true, batch, shape,
                static_cast<unsigned char*>(enc_ws), L, static_cast<unsigned char*>(uf_ws), P_max, img_words, (uint32_t)block_bytes, sizes_out);
  return cudaGetLastError();
}

// ===================================================================================
// parameter server: decode + dequantize + weighted scatter-accumulate of unframed streams
// ===================================================================================

constexpr int kUfPrepThreads = 1024;

// validates the headers and tables, derives the per-client coefficients and the prefix of block counts (block 0); meanwhile the other
// blocks write the accumulator's zeros, which depend on nothing
__global__ void __launch_bounds__(kUfPrepThreads)
k_uf_decode_prepare(const uint8_t* const* __restrict__ streams, const uint64_t* __restrict__ stream_bytes,
                    const float* __restrict__ weights, uint32_t n, double weight_total, uint64_t d, uint32_t s, unsigned char* ws,
                    float* __restrict__ zero_out) {
  __shared__ double s_part[kUfPrepThreads / 32];
  __shared__ uint32_t s_cnt[kUfPrepThreads / 32];
  __shared__ double s_W;
  __shared__ uint32_t s_carry;
  int32_t* status = reinterpret_cast<int32_t*>(ws + kDecWsStatus);
  float* coef = reinterpret_cast<float*>(ws + kDecWsCoef);
  uint32_t* prefix = reinterpret_cast<uint32_t*>(ws + dec_off_prefix(n));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_enter();
  if (blockIdx.x > 0) {
    zero_fill(zero_out, d, (uint64_t)(blockIdx.x - 1) * kUfPrepThreads + tid, (uint64_t)(gridDim.x - 1) * kUfPrepThreads);
    return;
  }
  if (tid == 0) {
    *status = 0;
    s_carry = 0;
  }
  double wsum = 0.0;
  for (uint32_t i = tid; i < n; i += kUfPrepThreads) wsum += (double)weights[i];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) wsum += __shfl_xor_sync(kFull, wsum, off);
  if (lane == 0) s_part[warp] = wsum;
  __syncthreads();
  if (tid == 0) {
    double W = 0.0;
    for (int w = 0; w < kUfPrepThreads / 32; ++w) W += s_part[w];
    s_W = (weight_total != 0.0) ? weight_total : W;
  }
  __syncthreads();
  const double W = s_W;
  if (tid == 0 && !(W > 0.0)) set_status(status, CVLC_ERR_INVALID_ARG);
  for (uint32_t base = 0; base < n; base += kUfPrepThreads) {
    const uint32_t i = base + tid;
    uint32_t R = 0;
    if (i < n) {
      const uint8_t* st = streams[i];
      const uint64_t nbytes = stream_bytes[i];
      bool ok = (st != nullptr) && ((reinterpret_cast<uintptr_t>(st) & 15) == 0) && nbytes >= kUfDirectory;
      if (ok) {
        const uint32_t* hw = reinterpret_cast<const uint32_t*>(st);
        const uint32_t magic = hw[0], ver_q_s = hw[1];
        const uint64_t sd = (uint64_t)hw[2] | ((uint64_t)hw[3] << 32);
        const uint32_t sR = hw[4], pb = hw[5], hb = hw[6];
        const double B = __longlong_as_double((long long)((uint64_t)hw[12] | ((uint64_t)hw[13] << 32)));
        const uint32_t quantizer = (ver_q_s >> 16) & 0xFF;
        ok = (magic == CVLC_STREAM_MAGIC) && ((ver_q_s & 0xFFFF) == 2) && (quantizer <= CVLC_QUANT_QSGD) && ((ver_q_s >> 24) == s) &&
             (sd == d) && (pb != 0) && ((pb & 31) == 0) && (hb >= 80) && (hb < pb) && (B >= 1.0) && (B < 1e300) &&
             (nbytes >= uf_head_bytes(sR));
        if (ok) {
          const uint32_t* tab = hw + kUfTables / 4;
          unsigned long long blocks = 0;
          for (uint32_t y = 0; y <= CVLC_MAX_CODE_BITS; ++y) {
            const uint32_t ny = tab[y], cp = tab[33 + y];
            blocks += ny;
            if (ny && (y == 0 || cp == 0 || cp > kUfMaxRecords || (quantizer == CVLC_QUANT_QSGD && y < 2))) ok = false;
          }
          const unsigned long long total = *reinterpret_cast<const unsigned long long*>(st + kUfTotalBits);
          ok = ok && blocks == sR && uf_head_bytes(sR) + ((total + 63) / 64) * 8 == nbytes;
        }
        if (ok) {
          R = sR;
          const float wi = weights[i];
          if (!(wi > 0.0f) || __float_as_uint(wi) >= 0x7F800000u) set_status(status, CVLC_ERR_INVALID_ARG);
          coef[i] = (float)((double)wi / (W * B));
        }
      }
      if (!ok) {
        set_status(status, CVLC_ERR_BAD_STREAM);
        coef[i] = 0.0f;
      }
    }
    uint32_t incl = R;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) s_cnt[warp] = incl;
    __syncthreads();
    uint32_t below = s_carry;
    for (int w = 0; w < warp; ++w) below += s_cnt[w];
    if (i < n) prefix[i] = below + incl - R;
    __syncthreads();
    if (tid == kUfPrepThreads - 1) s_carry = below + incl;
    __syncthreads();
  }
  if (tid == 0) prefix[n] = s_carry;
}

// 64 bits of the body from bit pos on (zero beyond its last word)
__device__ __forceinline__ unsigned long long uf_peek(const uint32_t* __restrict__ body, unsigned long long n_words, unsigned long long pos) {
  const unsigned long long w = pos >> 5;
  const uint32_t sh = (uint32_t)(pos & 31ull);
  const unsigned long long a = (w < n_words) ? __ldg(body + w) : 0u, b = (w + 1 < n_words) ? __ldg(body + w + 1) : 0u;
  unsigned long long v = (a | (b << 32)) >> sh;
  if (sh) {
    const unsigned long long c2 = (w + 2 < n_words) ? __ldg(body + w + 2) : 0u;
    v |= c2 << (64 - sh);
  }
  return v;
}

constexpr int kUfDecThreads = 128;
constexpr int kUfDecWarps = kUfDecThreads / 32;
constexpr uint32_t kUfStage = 288;    // words of a block staged at a time
constexpr uint32_t kUfChunk = 512;    // records whose starts are found before the warp takes them apart
constexpr uint32_t kUfSteps = 16;     // records that are followed between two looks at what was met
struct UfDecWarp {
  alignas(16) uint8_t len[kUfStage * 32 + 256];  // length of a record that starts at this bit of the stage; zeros behind it
  uint32_t bits[kUfStage + 4];                   // the block's words from the current stage on (four words of zeros behind them)
  uint16_t start[kUfChunk + kUfSteps];           // first bit of every record, and the one behind the last
};

// One warp per block.  The unary parts make finding the records sequential; to keep the chain short, the lanes first work out how
// long a record would be from every bit of a staged piece on (four bits by one multiplication from a table of their 16 patterns), and
// one lane then only adds lengths up: a load from shared memory and an addition per record, with a look every 16 records at whether the
// piece has ended or a unary part was too long for the table (updates with layers that send nothing have some; they are counted out word by
// word).  The warp then takes 32 records at a time apart, sums their differences by a scan, dequantizes and accumulates.
// 8 clients of 1.2 M coordinates at 2 bits (1600 blocks of about 400 records): 57 us with the checks in the chain (117 cycles a record) and
// a new piece behind every long unary part, 24 us here.  (Four warps per block, each following a quarter of the piece from 64 entries at once:
// 86 us; only a lone client gains by it.)
__global__ void __launch_bounds__(kUfDecThreads)
k_decode_unframed(const uint8_t* const* __restrict__ streams, uint32_t n, uint64_t d, float* __restrict__ out, unsigned char* ws) {
  extern __shared__ uint32_t s_dec[];  // [n + 1] block prefix
  __shared__ UfDecWarp s_warp[kUfDecWarps];
  __shared__ uint2 s_nibble[16];  // of four bits: ones from each bit on (a byte each), and whether they go on above the fourth
  __shared__ int s_err;
  pdl_enter();
  int32_t* status = reinterpret_cast<int32_t*>(ws + kDecWsStatus);
  const float* coef = reinterpret_cast<const float*>(ws + kDecWsCoef);
  const uint32_t* prefix = reinterpret_cast<const uint32_t*>(ws + dec_off_prefix(n));
  if (threadIdx.x == 0) s_err = *reinterpret_cast<const volatile int32_t*>(status);
  for (uint32_t i = threadIdx.x; i <= n; i += kUfDecThreads) s_dec[i] = prefix[i];
  if (threadIdx.x < 16) {
    uint2 v = make_uint2(0u, 0u);
    for (int e = 0; e < 4; ++e) {
      const uint32_t ones = (uint32_t)__ffs((int)~(threadIdx.x >> e)) - 1u;  // at most 4 - e
      v.x |= ones << (8 * e);
      v.y |= (ones == 4u - e ? 1u : 0u) << (8 * e);
    }
    s_nibble[threadIdx.x] = v;
  }
  __syncthreads();
  if (s_err != 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  UfDecWarp& sw = s_warp[warp];
  for (uint32_t i = lane; i < 64; i += 32) reinterpret_cast<uint32_t*>(sw.len + kUfStage * 32)[i] = 0u;
  const uint32_t total = s_dec[n];
  const uint32_t warps_total = gridDim.x * kUfDecWarps;
  for (uint32_t g = blockIdx.x * kUfDecWarps + warp; g < total; g += warps_total) {
    uint32_t lo_c = 0, hi_c = n;
    while (hi_c - lo_c > 1) {
      const uint32_t mid = (lo_c + hi_c) >> 1;
      if (s_dec[mid] <= g) lo_c = mid; else hi_c = mid;
    }
    const uint32_t c = lo_c, r = g - s_dec[c];
    const uint8_t* st = streams[c];
    const uint32_t* hw = reinterpret_cast<const uint32_t*>(st);
    const uint32_t R = hw[4], quantizer = (hw[1] >> 16) & 0xFF;
    const uint32_t* tab = hw + kUfTables / 4;
    // the block's length: lane l holds length 32 - l and the inclusive count of blocks down to it
    const uint32_t ny = tab[CVLC_MAX_CODE_BITS - lane], cp = tab[33 + CVLC_MAX_CODE_BITS - lane];
    uint32_t cum = ny;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t a = __shfl_up_sync(kFull, cum, off);
      if (lane >= off) cum += a;
    }
    const unsigned hit = __ballot_sync(kFull, r < cum);
    const int src_lane = __ffs(hit) - 1;  // the tables add up to R: checked by the prepare kernel
    const uint32_t y = CVLC_MAX_CODE_BITS - (uint32_t)src_lane;
    const uint32_t P = __shfl_sync(kFull, cp, src_lane);
    const uint32_t m = uf_rice_param(d, P);
    const unsigned long long total_bits = *reinterpret_cast<const unsigned long long*>(st + kUfTotalBits);
    const unsigned long long n_words = ((total_bits + 63) / 64) * 2;
    const uint32_t* body = hw + uf_head_bytes(R) / 4;
    const unsigned long long* dir = reinterpret_cast<const unsigned long long*>(st + kUfDirectory);
    unsigned long long pos = dir[r];
    // blocks follow one another without gaps: this one ends where the directory says the next one starts
    const unsigned long long next = (r + 1 < R) ? dir[r + 1] : total_bits;
    const bool qsgd = quantizer == CVLC_QUANT_QSGD;
    bool bad = pos + 64 > total_bits || pos + 64 < pos || next > total_bits;
    float lo = 0.f, hi = 0.f;
    if (!bad) {
      const unsigned long long h = uf_peek(body, n_words, pos);
      lo = __uint_as_float((uint32_t)h);
      hi = __uint_as_float((uint32_t)(h >> 32));
      pos += 64;
      if (qsgd && __float_as_uint(lo) >= 0x7F800000u) bad = true;
      if (!qsgd && ((__float_as_uint(lo) & 0x7FFFFFFFu) >= 0x7F800000u || (__float_as_uint(hi) & 0x7FFFFFFFu) >= 0x7F800000u || lo > hi)) bad = true;
    }
    const uint32_t level_mask = qsgd ? (uint32_t)((1ull << (y - 1)) - 1ull) : 0u;
    const double dlo = qsgd ? 0.0 : (double)lo;
    const double step = qsgd ? __ddiv_rn((double)lo, (double)level_mask)
                             : ((hi == lo) ? 0.0 : __ddiv_rn(__dsub_rn((double)hi, dlo), (double)((1ull << y) - 1ull)));
    const float cf = coef[c];
    const unsigned long long code_mask = (1ull << y) - 1ull, low_mask = (1ull << m) - 1ull;
    const uint32_t tail_bits = 1 + m + y;
    uint32_t done = 0;                 // records walked
    unsigned long long prev = 0;       // smallest position the next record may have
    while (!bad && done < P) {
      const unsigned long long w0 = pos >> 5;  // stage from the word that holds the next bit
      __syncwarp();                            // the previous stage and records have been read
      for (uint32_t i = lane; i < kUfStage + 4; i += 32) sw.bits[i] = (i < kUfStage && w0 + i < n_words) ? __ldg(body + w0 + i) : 0u;
      __syncwarp();
      const unsigned long long base = w0 << 5;
      const uint32_t first = (uint32_t)(pos - base);
      const uint32_t last = (uint32_t)(next > base ? (next - base < kUfStage * 32ull ? next - base : kUfStage * 32ull) : 0ull);  // the piece's end
      // The length of a record that started at any bit of the stage (128 and more: its unary part leaves the next word), every
      // lane a word of bits at a time, from the top bits down; then one lane follows the lengths from record to record.
      for (uint32_t i = lane; 32 * i < last; i += 32) {
        const uint32_t x0 = sw.bits[i], x1 = sw.bits[i + 1];
        uint32_t run = x1 == 0xFFFFFFFFu ? 128u : (uint32_t)__ffs((int)~x1) - 1u;
        uint32_t packed[8];
#pragma unroll
        for (int q = 7; q >= 0; --q) {
          const uint2 v = s_nibble[(x0 >> (4 * q)) & 15u];
          const uint32_t runs = v.y * run + v.x;
          run = runs & 0xFFu;
          packed[q] = runs + tail_bits * 0x01010101u;
        }
        uint4* len4 = reinterpret_cast<uint4*>(sw.len) + 2 * i;
        len4[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        len4[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
      }
      __syncwarp();
      const uint32_t want = P - done < kUfChunk ? P - done : kUfChunk;
      uint32_t found = 0;  // starts written down, and the one behind them
      if (lane == 0) {
        uint32_t p = first;
        while (found < want && p < last) {
          const uint32_t from = p;
          uint32_t seen = 0;
#pragma unroll
          for (uint32_t u = 0; u < kUfSteps; ++u) {
            const uint32_t l = sw.len[p];
            sw.start[found + u] = (uint16_t)p;
            seen |= l;
            p += l;
          }
          found += kUfSteps;
          if (seen < 128u) continue;
          found -= kUfSteps;  // once more, up to the long one
          p = from;
          while (sw.len[p] < 128u) {
            sw.start[found++] = (uint16_t)p;
            p += sw.len[p];
          }
          if (p >= last) break;
          uint32_t w = p >> 5, ones = ~sw.bits[w] >> (p & 31u);
          uint32_t zero = p + (ones ? (uint32_t)__ffs((int)ones) - 1u : 32u - (p & 31u));  // where its unary part ends
          while (ones == 0 && zero < last) {
            ones = ~sw.bits[++w];
            zero += ones ? (uint32_t)__ffs((int)ones) - 1u : 32u;
          }
          if (zero + tail_bits > last || found >= want) break;  // not whole in the piece: the next one begins with it
          sw.start[found++] = (uint16_t)p;
          p = zero + tail_bits;
        }
        sw.start[found] = (uint16_t)p;
      }
      found = __shfl_sync(kFull, found, 0);
      __syncwarp();
      // a record that is whole inside the piece
      auto whole = [&](uint32_t j) -> bool { return j < found && sw.start[j] < last && sw.start[j + 1] <= last; };
      auto accumulate = [&](uint32_t pid, uint32_t code) {
        float v;
        if (qsgd) {
          const float mag = (float)__dmul_rn((double)(code & level_mask), step);
          v = ((code >> (y - 1)) & 1u) ? -mag : mag;
        } else {
          v = (float)__dadd_rn(dlo, __dmul_rn((double)code, step));
        }
        atomicAdd(out + pid, cf * v);
      };
      if (!whole(0)) {
        // a record longer than a stage (the unary parts of a block add up to less than two bits per record, so only a malformed
        // or extremely sparse block has one): walked in global memory, by all lanes alike
        unsigned long long q = pos, quo = 0;
        while (true) {
          const unsigned long long v = uf_peek(body, n_words, q);
          const int ones = (~v == 0ull) ? 64 : __ffsll((long long)~v) - 1;
          quo += ones;
          q += ones;
          if (ones < 64 || q >= total_bits) break;
        }
        const unsigned long long v = uf_peek(body, n_words, q + 1);
        const unsigned long long pid = prev + ((quo << m) | (v & low_mask));
        bad = q + tail_bits > total_bits || (quo >> 32) != 0 || pid >= d;
        if (bad) break;
        if (lane == 0) accumulate((uint32_t)pid, (uint32_t)((v >> m) & code_mask));
        prev = pid + 1;
        pos = q + tail_bits;
        done += 1;
        continue;
      }
      uint32_t count = 0;
      for (uint32_t j0 = 0; j0 < want; j0 += 32) {
        const unsigned there = __ballot_sync(kFull, j0 + lane < want && whole(j0 + lane));
        const uint32_t here = there == kFull ? 32u : (uint32_t)__ffs((int)~there) - 1u;  // up to the first that is not
        const bool on = (uint32_t)lane < here;
        unsigned long long gap = 0;  // this record's distance from the first place behind the one before it, plus one
        uint32_t code = 0;
        if (on) {
          const uint32_t begin = sw.start[j0 + lane], end = sw.start[j0 + lane + 1];
          const uint32_t q = end - tail_bits + 1;  // behind the unary part and its stop bit
          const uint32_t w = q >> 5, sh = q & 31u;
          const uint32_t x0 = sw.bits[w], x1 = sw.bits[w + 1], x2 = sw.bits[w + 2];
          const unsigned long long v = (unsigned long long)__funnelshift_r(x0, x1, sh) | ((unsigned long long)__funnelshift_r(x1, x2, sh) << 32);
          gap = (((unsigned long long)(q - 1 - begin) << m) | (v & low_mask)) + 1;
          code = (uint32_t)((v >> m) & code_mask);
        }
        unsigned long long incl = gap;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const unsigned long long o = __shfl_up_sync(kFull, incl, off);
          if (lane >= off) incl += o;
        }
        const unsigned long long pid = prev + incl - 1;
        bad = __any_sync(kFull, on && pid >= d);
        if (bad) break;
        if (on) accumulate((uint32_t)pid, code);
        prev += __shfl_sync(kFull, incl, 31);
        count += here;
        if (here < 32) break;
      }
      if (bad) break;
      pos = base + sw.start[count];
      done += count;
    }
    if ((bad || pos != next) && lane == 0) set_status(status, CVLC_ERR_BAD_STREAM);
  }
}

cudaError_t launch_decode_unframed(const uint8_t* const* streams, const uint64_t* stream_bytes, const float* weights,
                                   uint32_t n, double weight_total, uint64_t d, uint32_t s, float* out, int accumulate,
                                   void* ws, cudaStream_t st) {
  unsigned char* w = static_cast<unsigned char*>(ws);
  launch_kernel(kKDecodePrepare, k_uf_decode_prepare, 1 + (accumulate ? 0 : fill_grid(d, kUfPrepThreads, 2 * kNumSM)), kUfPrepThreads, 0, st, false,
                streams, stream_bytes, weights, n, weight_total, d, s, w, out);
  const size_t prefix_bytes = ((size_t)n + 1) * 4;
  if (prefix_bytes + sizeof(UfDecWarp) * kUfDecWarps > 47 * 1024) {  // hundreds of clients: the most of any call, another thread's too
    const cudaError_t e = allow_shared(k_decode_unframed, ((size_t)CVLC_MAX_CLIENTS_PER_CALL + 1) * 4);
    if (e != cudaSuccess) return e;
  }
  launch_kernel(kKDecodeUnframed, k_decode_unframed, 4 * kNumSM, kUfDecThreads, prefix_bytes, st, true, streams, n, d, out, w);
  return cudaGetLastError();
}

}  // namespace cvlc
