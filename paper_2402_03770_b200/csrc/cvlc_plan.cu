// Planning kernels: magnitude histogram (Algorithm 1, step 1) with the selection threshold, the exponent fit of
// Definition 1, and the code-length tuning by atomic operations on Eq. (5) (Algorithm 1 steps 2-14), one CTA per
// client or, in larger batches, per distinct (exponent, scale).
//
// The planner's floating point is IEEE binary64 with every multiply and add
// rounded separately (the *_rn intrinsics keep the compiler from contracting
// them), in a fixed order, so that its decisions do not depend on the machine.
#include <cooperative_groups.h>
#include <string.h>

#include "cvlc_common.cuh"
#include "cvlc_rank.cuh"

namespace cvlc {

// ===================================================================================
// Series arithmetic of the planner
// ===================================================================================

// log2 of a positive normal double: v = m 2^e, m folded into (sqrt(1/2), sqrt(2)],
// ln m = 2 atanh(t) with t = (m-1)/(m+1), odd series up to t^25.
__device__ __forceinline__ double series_log2(double v) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  int e = (int)((bits >> 52) & 0x7FF) - 1023;
  double m = __longlong_as_double((long long)((bits & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
  if (m > 1.4142135623730951) {
    m = __dmul_rn(m, 0.5);
    e += 1;
  }
  const double t = __ddiv_rn(__dsub_rn(m, 1.0), __dadd_rn(m, 1.0));
  const double q = __dmul_rn(t, t);
  double p = 1.0 / 25.0;
#pragma unroll
  for (int j = 11; j >= 0; --j) p = __dadd_rn(__dmul_rn(p, q), 1.0 / (double)(2 * j + 1));
  const double ln_m = __dmul_rn(__dmul_rn(2.0, t), p);
  return __dadd_rn((double)e, __dmul_rn(ln_m, 1.4426950408889634));
}

// u / j for a small positive integer j, correctly rounded, from the rounded reciprocal:
// q0 = RN(u * rcp), r = u - j*q0 (exact in one fused operation: it is a small multiple
// of ulp(q0)), q1 = RN(q0 + r*rcp).  q0 + r*rcp differs from u/j by less than 2^-52 ulp,
// while u/j, a quotient by an integer below 2^5, is either representable or at least
// 1/(2j) ulp away from every rounding boundary, so q1 = RN(u/j).
__device__ __forceinline__ double div_small_int(double u, int j) {
  const double rcp = 1.0 / (double)j;  // folded at compile time when j is constant
  const double q0 = __dmul_rn(u, rcp);
  const double r = __fma_rn(-(double)j, q0, u);
  return __fma_rn(r, rcp, q0);
}

// 2^v for |v| <= 1000: v = n + r with |r| <= 1/2, e^(r ln 2) as the degree-20 Taylor
// polynomial in Horner form p = 1 + (u/j) p, then n added to the exponent field.
__device__ __forceinline__ double series_exp2(double v) {
  const double n = floor(__dadd_rn(v, 0.5));
  const double r = __dsub_rn(v, n);
  const double u = __dmul_rn(r, 0.6931471805599453);
  // u / j for j = 1 .. 20: a division by an odd j is done once, the even ones are its exact halvings
  // (RN(u / 2j) = RN(u / j) / 2: scaling by two commutes with rounding; u is zero or far above the subnormals)
  double uj[21];
  uj[1] = u;
#pragma unroll
  for (int j = 3; j <= 19; j += 2) uj[j] = div_small_int(u, j);
#pragma unroll
  for (int j = 2; j <= 20; j += 2) uj[j] = __dmul_rn(uj[j / 2], 0.5);
  double p = 1.0;
#pragma unroll
  for (int j = 20; j >= 1; --j) p = __dadd_rn(1.0, __dmul_rn(uj[j], p));
  const long long ni = (long long)n;
  return __longlong_as_double(__double_as_longlong(p) + ni * (1ll << 52));
}

__device__ __forceinline__ double series_powr(double a, double beta) { return series_exp2(__dmul_rn(beta, series_log2(a))); }

// share of ||U||^2 in the top Z ranks under Definition 1: ((Z+1)^beta - 1) / (d^beta - 1)
__device__ __forceinline__ double energy_E(uint64_t Z, double beta, double D) {
  return __ddiv_rn(__dsub_rn(series_powr((double)(Z + 1), beta), 1.0), D);
}

// ===================================================================================
// K2  planner: threshold and bins' starts by the histogram's blocks, exponent fit and length tuning
// ===================================================================================

constexpr int kPlanThreads = 512;  // of the blocks that work on one client's histogram: that of the histogram, the fit's, the tuning's
constexpr int kPlanBins = CVLC_HIST_BINS / kPlanThreads;
constexpr size_t kSurvivalBytes = (CVLC_HIST_BINS + 4) * 4;  // survival counts in shared memory
// The tuning kernel settles neighbouring lengths with one warp and looks at all pairs with all but one (see FastLane below); all of its
// warps fit the exponent and evaluate what is left to the series arithmetic.
constexpr int kTuneThreads = 512;
constexpr int kTuneWarps = kTuneThreads / 32;
constexpr int kPlanItems = 1024;
constexpr int kPairSlots = (496 + kTuneThreads - 1) / kTuneThreads;  // pairs of a sweep a thread looks at

// scratch of the length-tuning loop (the tuning kernel's dynamic shared memory)
constexpr int kMaxBatchOps = 32;  // atomic operations evaluated together
struct PlanOp {                   // one atomic operation of a batch
  int i, j;                       // candidate indices, i > j
  uint32_t X, na0;                // packets shared by the pair; current count of length i
  uint32_t lo, hi;                // bisection interval
  int m;                          // lengths a trial must evaluate (used lengths <= i, plus i and j)
  int levels;                     // bisection levels evaluated in this round (0: waits)
  int item_base, eval_base;       // first (evaluation, slot) item / first evaluation of this operation
  double F_final;                 // F at the end of the bisection
  unsigned char slot_lane[32];    // those lengths, longest first
};
struct PlanSolver {
  double Fpre[33];                // running sum of F after length l (index 32: nothing yet)
  double Eab[33];                 // energy of the nearest used length at or above l
  unsigned long long Wc[32];      // ranks covered by lengths >= l, current counts
  unsigned used;                  // lengths with a positive count
  double Ev[kPlanItems];          // trial energies, one per item
  double Fv[kPlanItems];          // trial objective values, one per evaluation
  uint32_t tv[kPlanItems];        // trial split of every evaluation (0xFFFFFFFF: not needed)
  PlanOp op[kMaxBatchOps];
  int item_end[kMaxBatchOps];     // exclusive end of every operation's items / evaluations in this round
  int eval_end[kMaxBatchOps];
  int n_ops, n_items, n_evals, unfinished;
  int next_i, next_j, moved;      // where the sweep resumes after the batch
  uint32_t col_warp[32];          // batch collection: warp totals of the (operations, items) scan
  int col_nops, col_last, col_first_left;  // operations taken; thread of the last one; thread of the first one left over
  unsigned char ea[kPlanItems];   // operation of every evaluation
};

struct PlanShared {
  uint32_t n[32];
  double D;
};

// candidate lengths of one client and their coefficients (Eq. (5)): g(y) > 0 (the paper's B > (Q+1)/2) and not dominated
struct PlanTab {
  uint64_t d;
  uint32_t s, R, nY, y_min, fixed_y;
  uint32_t Y[32];     // candidate lengths, ascending
  uint32_t capY[32];  // cap(Y[i])
  double gY[32];      // g(Y[i]) = 1 - (Q/B^2 + (1 - 1/B)^2)
  double QY[32];      // PQ error factor Q(Y[i]) = cap / (2^y - 1)^2
};

// by one full warp, lane = length - 1
__device__ __forceinline__ void build_plan_tab(PlanTab& T, const Shape& shape, double B, int lane) {
  const uint32_t y = lane + 1;
  const bool in_range = y <= shape.max_code_bits;
  const uint32_t cap_y = in_range ? shape.cap[y] : 0u;
  double Q;  // error factor of cap(y) values at y bits (Appendix, case study)
  if (shape.quantizer == CVLC_QUANT_QSGD) {
    // min(P / s_q^2, sqrt(P) / s_q), s_q = 2^(y-1) - 1 levels beside the sign bit; one bit holds no level
    const double sq = (double)((1ull << (y - 1)) - 1ull);
    const double Q1 = __ddiv_rn((double)cap_y, __dmul_rn(sq, sq));
    const double Q2 = __ddiv_rn(__dsqrt_rn((double)cap_y), sq);
    Q = (y < 2) ? CUDART_INF : ((Q1 < Q2) ? Q1 : Q2);
  } else {
    const double L = (double)((1ull << y) - 1ull);  // PQ: P / (2^y - 1)^2
    Q = __ddiv_rn((double)cap_y, __dmul_rn(L, L));
  }
  const double one_m = __dsub_rn(1.0, __ddiv_rn(1.0, B));
  const double g = __dsub_rn(1.0, __dadd_rn(__ddiv_rn(Q, __dmul_rn(B, B)), __dmul_rn(one_m, one_m)));
  unsigned member;  // bit y - 1: length y is a candidate
  uint32_t y_min;
  if (shape.fixed_y) {
    y_min = shape.fixed_y;
    member = 1u << (shape.fixed_y - 1);
  } else {
    const unsigned pos = __ballot_sync(kFull, in_range && g > 0.0);
    y_min = pos ? (uint32_t)__ffs(pos) : 1u;  // the host has checked that one exists
    const uint32_t cap_next = __shfl_down_sync(kFull, cap_y, 1);
    const bool keep = in_range && y >= y_min && (y == shape.max_code_bits || cap_y > cap_next);
    member = __ballot_sync(kFull, keep);
  }
  if (member & (1u << lane)) {
    const int i = __popc(member & ((1u << lane) - 1u));
    T.Y[i] = y;
    T.capY[i] = cap_y;
    T.gY[i] = g;
    T.QY[i] = Q;
  }
  if (lane == 0) {
    T.d = shape.d;
    T.s = shape.s;
    T.R = shape.R;
    T.nY = (uint32_t)__popc(member);
    T.y_min = y_min;
    T.fixed_y = shape.fixed_y;
  }
}
// zeroes two ranges of the workspace and leaves the clients' descriptors in it
template <int CAP>
__global__ void __launch_bounds__(256)
k_zero_words(const __grid_constant__ BatchDesc<CAP> batch, ClientDesc* desc, uint4* p, size_t n16, uint4* q, size_t m16) {
  pdl_enter();
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = first; i < batch.n; i += stride) desc[i] = batch.c[i];
  for (size_t i = first; i < n16; i += stride) p[i] = make_uint4(0u, 0u, 0u, 0u);
  for (size_t i = first; i < m16; i += stride) q[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ---- what a client's histogram gives, by a block of kPlanThreads threads ------------------------
// Survival counts N_j = #{bin >= j} into N[0 .. 4096] (they add up to d <= 2^31); ends with a barrier.
// h: the thread's kPlanBins bins.
__device__ __forceinline__ void survival_of(const uint32_t (&h)[kPlanBins], uint32_t* N) {
  __shared__ uint32_t s_warp[kPlanThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t sum = 0;
#pragma unroll
  for (int i = 0; i < kPlanBins; ++i) sum += h[i];
  uint32_t incl = sum;  // from the top bin down: of this lane and those above
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_down_sync(kFull, incl, off);
    if (lane + off < 32) incl += o;
  }
  if (lane == 0) s_warp[warp] = incl;
  __syncthreads();
  uint32_t run = incl - sum + __reduce_add_sync(kFull, lane > warp && lane < kPlanThreads / 32 ? s_warp[lane] : 0u);
#pragma unroll
  for (int i = kPlanBins - 4; i >= 0; i -= 4) {
    uint4 v;
    v.w = run + h[i + 3];
    v.z = v.w + h[i + 2];
    v.y = v.z + h[i + 1];
    v.x = v.y + h[i];
    run = v.x;
    reinterpret_cast<uint4*>(N)[(kPlanBins * tid + i) / 4] = v;
  }
  if (tid == 0) N[CVLC_HIST_BINS] = 0;
  __syncthreads();
}
__device__ __forceinline__ void survival_counts(const unsigned long long* hist, uint32_t* N) {
  uint32_t h[kPlanBins];
#pragma unroll
  for (int i = 0; i < kPlanBins; i += 2) {
    const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(hist) + (kPlanBins * threadIdx.x + i) / 2);
    h[i] = (uint32_t)v.x;
    h[i + 1] = (uint32_t)v.y;
  }
  survival_of(h, N);
}

// The selection threshold.  The number of transmitted coordinates k is not known before the lengths are tuned, but it never exceeds
// k_sel = R * cap(shortest candidate length) (every packet at the shortest code; with a fixed length, exactly R * cap(y)), so the
// selection keeps every coordinate down to the bin that holds rank min(k_sel, d): a superset of the top k whose first k ranks are
// the top k.  Written to the plan (may be null); where every candidate bin starts among the client's candidates (from the top bin down) to
// bin_start (may be null).  Ends with a barrier.
struct Threshold {
  uint32_t bin, top, n, fullest;  // threshold's bin, highest bin, candidates, those in the fullest bin
};
__device__ __forceinline__ Threshold client_threshold(const uint32_t* N, const Shape& shape, uint32_t cap0, cvlc_plan_t* plan, uint32_t* bin_start) {
  __shared__ Threshold s_t;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) s_t.fullest = 0;
  const unsigned long long most = (unsigned long long)shape.R * cap0;
  const uint32_t k_sel = (uint32_t)(most < shape.d ? most : shape.d);
  __syncthreads();
  const int first = kPlanBins * (tid & ~31);
  if (N[first] > 0 && N[first + 32 * kPlanBins] < k_sel) {  // most warps' bins hold no candidates
    uint32_t fullest = 0;
#pragma unroll
    for (int i = 0; i < kPlanBins; ++i) {
      const int j = first + 32 * i + lane;
      const uint32_t at = N[j], next = N[j + 1];  // from this bin on, in the bins above it
      if (at > 0 && next < k_sel) {               // a candidate's bin
        if (at >= k_sel) {
          s_t.bin = (uint32_t)j;
          s_t.n = at;
        }
        fullest = max(fullest, at - next);
        if (next == 0) s_t.top = (uint32_t)j;
        if (bin_start) bin_start[j] = next;
      }
    }
    fullest = __reduce_max_sync(kFull, fullest);
    if (lane == 0) atomicMax(&s_t.fullest, fullest);
  }
  __syncthreads();
  const Threshold t = s_t;
  if (tid == 0 && plan) {
    plan->status = CVLC_OK;
    plan->s = shape.s;
    plan->R = shape.R;
    plan->thresh_bin = t.bin;
    plan->top_bin = t.top;
    plan->n_candidates = t.n;
  }
  return t;
}

// The power law of Definition 1 (Algorithm 1, step 1): alpha and its quantised value, known to all threads.  Ends with a barrier.
constexpr size_t kFitPoints = 4096;  // at most, filled up with zeros to whole groups
constexpr uint32_t kFitGroup = 16;
struct FitScratch {
  double sum_of[4][kFitPoints + 2 * kFitGroup];  // X, Y, X X, X Y of the points
  uint16_t bin[kFitPoints];
};
// `meanwhile` is run by the warps but the first while that adds up.
template <class Meanwhile>
__device__ __forceinline__ double2 client_fit(const uint32_t* N, FitScratch& F, const Shape& shape, Meanwhile&& meanwhile) {
  __shared__ uint32_t s_warp[kPlanThreads / 32];
  __shared__ double2 s_alpha;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (shape.fixed_y) return make_double2(-1.0, -1.0);
  // ---- fit points: non-empty normal bins in the upper half of the ranks ----------
  uint32_t flags = 0;
  uint32_t at = N[kPlanBins * tid];
#pragma unroll
  for (int i = 0; i < kPlanBins; ++i) {
    const int j = kPlanBins * tid + i;
    const uint32_t next = N[j + 1];
    if (j >= 16 && j <= 4079 && at > next && at <= shape.d / 2) flags |= 1u << i;
    at = next;
  }
  const uint32_t cnt = __popc(flags);
  uint32_t incl = cnt;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  const uint32_t wt = lane < kPlanThreads / 32 ? s_warp[lane] : 0u;
  const uint32_t np = __reduce_add_sync(kFull, wt);
  uint32_t pos = __reduce_add_sync(kFull, lane < warp ? wt : 0u) + incl - cnt;
  for (; flags; flags &= flags - 1) F.bin[pos++] = (uint16_t)(kPlanBins * tid + __ffs(flags) - 1);
  __syncthreads();
  // the logarithms, spread over the threads: those of a point in two neighbouring warps
  for (uint32_t q = tid; q < 2 * ((np + 31) & ~31u); q += kPlanThreads) {
    const uint32_t i = (q >> 6) * 32 + lane;
    if (i >= np) continue;
    const int j = F.bin[i];
    const bool is_x = (q & 32) == 0;
    const double l = series_log2(is_x ? (double)N[j] : __dadd_rn(1.0, (double)(j & 15) / 16.0));
    F.sum_of[is_x ? 0 : 1][i] = is_x ? l : __dadd_rn((double)((j >> 4) - 127), l);
  }
  __syncthreads();
  const uint32_t filled = (np + kFitGroup - 1) / kFitGroup * kFitGroup + kFitGroup;  // one group more: read ahead, not added
  for (uint32_t i = tid; i < filled; i += kPlanThreads) {
    const double X = i < np ? F.sum_of[0][i] : 0.0, Y = i < np ? F.sum_of[1][i] : 0.0;
    if (i >= np) F.sum_of[0][i] = F.sum_of[1][i] = 0.0;
    F.sum_of[2][i] = __dmul_rn(X, X);
    F.sum_of[3][i] = __dmul_rn(X, Y);
  }
  __syncthreads();
  // ---- least squares of log2|U{l}| on log2 l, sums in ascending bin order: four lanes, one sum each ----------
  if (warp == 0) {
    double acc = 0.0;
    const double2* A = reinterpret_cast<const double2*>(F.sum_of[lane & 3]);
    double2 t[kFitGroup / 2], next[kFitGroup / 2];
#pragma unroll
    for (uint32_t u = 0; u < kFitGroup / 2; ++u) t[u] = A[u];
    for (uint32_t i = kFitGroup; i < filled; i += kFitGroup) {
#pragma unroll
      for (uint32_t u = 0; u < kFitGroup / 2; ++u) next[u] = A[i / 2 + u];
#pragma unroll
      for (uint32_t u = 0; u < kFitGroup / 2; ++u) {
        acc = __dadd_rn(acc, t[u].x);
        acc = __dadd_rn(acc, t[u].y);
        t[u] = next[u];
      }
    }
    const double n = (double)np;
    const double Sx = __shfl_sync(kFull, acc, 0), Sy = __shfl_sync(kFull, acc, 1), Sxx = __shfl_sync(kFull, acc, 2), Sxy = __shfl_sync(kFull, acc, 3);
    const double den = __dsub_rn(__dmul_rn(n, Sxx), __dmul_rn(Sx, Sx));
    double a;
    if (n < 2.0 || !(den > 0.0))
      a = -1.0;
    else
      a = __ddiv_rn(__dsub_rn(__dmul_rn(n, Sxy), __dmul_rn(Sx, Sy)), den);
    double aq = __dmul_rn(floor(__dadd_rn(__dmul_rn(a, 256.0), 0.5)), 1.0 / 256.0);
    if (aq < -4.0) aq = -4.0;
    if (aq > -1.0 / 256.0) aq = -1.0 / 256.0;
    if (aq == -0.5) aq = -0.5 - 1.0 / 256.0;  // beta = 0 would make d^beta - 1 vanish
    if (lane == 0) s_alpha = make_double2(a, aq);
  } else {
    meanwhile();
  }
  __syncthreads();
  return s_alpha;
}

// the plan's fields that the fit gives, by all threads
__device__ __forceinline__ void write_fit(cvlc_plan_t* plan, double2 alpha, const PlanTab& T, const Shape& shape) {
  const int tid = threadIdx.x;
  if (tid == 32) {
    plan->y_min = T.y_min;
    plan->n_lengths = T.nY;
    plan->alpha = alpha.x;
    plan->alpha_q = alpha.y;
    plan->beta = __dadd_rn(__dmul_rn(2.0, alpha.y), 1.0);
  }
  if (tid <= CVLC_MAX_CODE_BITS) plan->cap[tid] = shape.cap[tid];
}

// What is known with a client's threshold, by one thread: the headers and, for an encoder in the same call, the client's buckets
__device__ __forceinline__ void write_client(uint32_t c, uint32_t n, cvlc_plan_t* plan, const Threshold& t, uint32_t nonfinite, const Shape& shape,
                                             unsigned char* ws, const EncFront& enc) {
  PlanWsHeader* hdr = reinterpret_cast<PlanWsHeader*>(ws);
  EncHeader* eh = reinterpret_cast<EncHeader*>(enc.ws);
  if (nonfinite) {
    plan->status = CVLC_ERR_NONFINITE_INPUT;
    set_status(&hdr->status, CVLC_ERR_NONFINITE_INPUT);
  }
  reinterpret_cast<uint32_t*>(ws + plan_off_max_bin(n))[c] = t.fullest;
  if (c == 0) {
    hdr->n = n;
    hdr->d = shape.d;
    hdr->magic = kPlanWsMagic;
  }
  if (enc.ws) {
    if (nonfinite) set_status(&eh->status, CVLC_ERR_NONFINITE_INPUT);
    else if (t.n > enc.L.capacity) set_status(&eh->status, CVLC_ERR_WORKSPACE_TOO_SMALL);
    const uint32_t limit = rank_limit(shape);
    const ClientRank r = client_rank(t.bin, t.top, t.n, t.fullest, enc.L.capacity, n);
    reinterpret_cast<ClientRank*>(enc.ws + enc.L.off_rank)[c] = r;
    reinterpret_cast<uint32_t*>(enc.ws + enc.L.off_pass_mask)[c] = (1u << kSortPasses) - 1u;  // ranked by partition: the result is in the first buffer
    add_client(eh, r, limit);
    if (c == 0) eh->limit = limit;
  }
}

// What the last block of a client's histogram does: the client's threshold, the bins' starts and the above
__device__ __noinline__ void finish_client(uint32_t c, const Batch& batch, const Shape& shape, unsigned char* ws, const EncFront& enc, uint32_t* N) {
  const uint32_t n = batch.n;
  cvlc_plan_t* plan = batch.c[c].plan;
  const uint32_t cap0 = batch.c[c].cap0;
  const uint32_t nonfinite = __ldcg(reinterpret_cast<const uint32_t*>(ws + plan_off_flags(n)) + c);
  survival_counts(reinterpret_cast<const unsigned long long*>(ws + kPlanWsHist) + (size_t)c * CVLC_HIST_BINS, N);
  const Threshold t = client_threshold(N, shape, cap0, plan, reinterpret_cast<uint32_t*>(ws + plan_off_bin_start(n)) + (size_t)c * CVLC_HIST_BINS);
  if (threadIdx.x == 0) write_client(c, n, plan, t, nonfinite, shape, ws, enc);
}

// ===================================================================================
// K1  magnitude histogram: h[key >> 19], key = bits(|x|); HBM-bound, 4 bytes / coordinate
// ===================================================================================

constexpr int kHistThreads = kStreamThreads;
constexpr int kHistSub = 2;  // shared sub-histograms per block (32 KB)

// The clients' rows form one concatenated array that is cut into equal contiguous chunks, one or two
// per block, so the load is even whatever the number of clients; a block that crosses a client
// boundary merges its shared histogram into that client's global one and starts afresh.

// In small batches, whose blocks have one client each, the block that completes a client's histogram works out its threshold and
// the bins' starts.  As kernels of their own, one block per client behind the exponent fit and one behind that for the encoder's
// workspace, they stood between histogram and selection for 16 us; here it is 4 (20 clients of 1.2 M coordinates, whole call and
// aggregation: 161 -> 150 us; 24 of 3 M 498 -> 487).  In large batches a block would have to finish up to four clients one after the
// other at the end (100 clients of 11.2 M: 23 us): there a kernel of one block per client does it (k_plan_threshold).
static_assert(kHistThreads == kPlanThreads && kSurvivalBytes <= kHistSub * CVLC_HIST_BINS * 4, "finish_client runs in the histogram's blocks");

// An addition in front of which the block's writes before the last barrier are visible, and behind which those are that others
// published in this way
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}

// counts the four magnitude keys of a float4; returns the largest of them
__device__ __forceinline__ uint32_t hist_add4(uint32_t* my, const float4 a) {
  const uint32_t k0 = __float_as_uint(a.x) & 0x7FFFFFFFu, k1 = __float_as_uint(a.y) & 0x7FFFFFFFu;
  const uint32_t k2 = __float_as_uint(a.z) & 0x7FFFFFFFu, k3 = __float_as_uint(a.w) & 0x7FFFFFFFu;
  atomicAdd(my + (k0 >> 19), 1u);
  atomicAdd(my + (k1 >> 19), 1u);
  atomicAdd(my + (k2 >> 19), 1u);
  atomicAdd(my + (k3 >> 19), 1u);
  const uint32_t m01 = k0 > k1 ? k0 : k1, m23 = k2 > k3 ? k2 : k3;
  return m01 > m23 ? m01 : m23;
}

__device__ __forceinline__ uint32_t largest_key(const float4& a) {
  return max(max(__float_as_uint(a.x) & 0x7FFFFFFFu, __float_as_uint(a.y) & 0x7FFFFFFFu), max(__float_as_uint(a.z) & 0x7FFFFFFFu, __float_as_uint(a.w) & 0x7FFFFFFFu));
}

__global__ void __launch_bounds__(kHistThreads, 3)
k_hist(const Batch batch, const __grid_constant__ Shape shape, const __grid_constant__ Partition part, unsigned char* ws,
       const __grid_constant__ EncFront enc, int finish) {
  extern __shared__ __align__(16) uint32_t sh_hist[];  // [kHistSub][4096]
  const uint64_t d = shape.d;
  unsigned long long* hist_all = reinterpret_cast<unsigned long long*>(ws + kPlanWsHist);
  uint32_t* nonfinite_all = reinterpret_cast<uint32_t*>(ws + plan_off_flags(batch.n));
  uint16_t* row_max_all = reinterpret_cast<uint16_t*>(ws + plan_off_row_max(batch.n));
  pdl_enter();
  for (int i = threadIdx.x; i < kHistSub * CVLC_HIST_BINS; i += kHistThreads) sh_hist[i] = 0;
  __syncthreads();
  uint32_t* my = sh_hist + ((threadIdx.x >> 5) & (kHistSub - 1)) * CVLC_HIST_BINS;
  const int lane = threadIdx.x & 31;

  const uint64_t nvec = d >> 2;
  for (uint32_t q = blockIdx.x; q < part.n_chunks; q += gridDim.x) {
  uint64_t pos, end;
  if (part.per_client) {
    const uint32_t c = q / part.per_client;
    pos = c * part.rows + (uint64_t)(q - c * part.per_client) * part.chunk;
    end = (c + 1) * part.rows;
  } else {
    pos = (uint64_t)q * part.chunk;
    end = part.total;
  }
  if (pos + part.chunk < end) end = pos + part.chunk;

  while (pos < end) {
    const uint64_t c = part.per_client ? q / part.per_client : pos / part.rows;
    const uint64_t seg_end = ((c + 1) * part.rows < end) ? (c + 1) * part.rows : end;
    const uint64_t u0 = (pos - c * part.rows) * kRowUnits, u1 = (seg_end - c * part.rows) * kRowUnits;  // units of the client
    const float* __restrict__ x = batch.c[c].x;
    const float4* xv = reinterpret_cast<const float4*>(x);
    const uint64_t v1 = (u1 < nvec) ? u1 : nvec;  // float4 units of this segment: [u0, v1)
    uint16_t* __restrict__ row_max = row_max_all + c * part.rows;
    static_assert(kRowUnits == 4, "a row is held by four neighbouring lanes");
    uint32_t top = 0;
    uint64_t v = u0 + threadIdx.x;
    // four independent 128-bit loads in flight per thread; the loop condition is the same for the lanes of a warp
    for (; (v - lane) + 31 + 3 * kHistThreads < v1; v += 4 * kHistThreads) {
      float4 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = __ldg(xv + v + u * kHistThreads);
      uint32_t m[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        m[u] = hist_add4(my, a[u]);
        top = m[u] > top ? m[u] : top;
      }
      // The rows' maxima of the four loads, two bins to a word: the first exchange leaves an even lane with loads 0 and 1, an odd
      // lane with 2 and 3, the second completes the rows; each lane then stores one of its row's four.
      const uint32_t w01 = m[0] >> 19 | (m[1] >> 3 & 0xFFFF0000u), w23 = m[2] >> 19 | (m[3] >> 3 & 0xFFFF0000u);
      uint32_t w = __vmaxu2(lane & 1 ? w23 : w01, __shfl_xor_sync(0xFFFFFFFFu, lane & 1 ? w01 : w23, 1));
      w = __vmaxu2(w, __shfl_xor_sync(0xFFFFFFFFu, w, 2));
      const uint32_t load = ((lane & 1) << 1) | (lane >> 1 & 1);
      row_max[(v + load * kHistThreads) / kRowUnits] = (uint16_t)(lane & 2 ? w >> 16 : w);
    }
    for (; v - lane < v1; v += kHistThreads) {  // rows that may end inside the warp
      const bool on = v < v1;
      uint32_t m = on ? hist_add4(my, __ldg(xv + v)) : 0u;
      top = m > top ? m : top;
      m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
      m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, 2));
      if (lane % kRowUnits == 0 && on) row_max[v / kRowUnits] = (uint16_t)(m >> 19);
    }
    // ragged tail of the client (d not a multiple of 4)
    if (seg_end == (c + 1) * part.rows && threadIdx.x < (d & 3)) {
      const uint32_t k0 = __float_as_uint(x[(nvec << 2) + threadIdx.x]) & 0x7FFFFFFFu;
      top = k0 > top ? k0 : top;
      atomicAdd(my + (k0 >> 19), 1u);
    }
    if (top >= 0x7F800000u) atomicOr(nonfinite_all + c, 1u);  // a key of exponent 255: Inf or NaN
    __syncthreads();
    unsigned long long* __restrict__ hist = hist_all + (size_t)c * CVLC_HIST_BINS;
    for (int b = threadIdx.x; b < CVLC_HIST_BINS; b += kHistThreads) {
      uint32_t cnt = 0;
#pragma unroll
      for (int sub = 0; sub < kHistSub; ++sub) {
        cnt += sh_hist[sub * CVLC_HIST_BINS + b];
        sh_hist[sub * CVLC_HIST_BINS + b] = 0;
      }
      if (cnt) atomicAdd(hist + b, (unsigned long long)cnt);
    }
    __syncthreads();
    pos = seg_end;
  }
  }
  if (finish && part.per_client) {
    __shared__ bool s_complete;
    const uint32_t c = blockIdx.x / part.per_client, begin = (blockIdx.x - c * part.per_client) * (uint32_t)part.chunk;
    const uint32_t left = (uint32_t)part.rows - begin, rows = left < (uint32_t)part.chunk ? left : (uint32_t)part.chunk;
    uint32_t* rows_done = reinterpret_cast<uint32_t*>(ws + plan_off_rows_done(batch.n));
    if (threadIdx.x == 0) s_complete = add_acq_rel(rows_done + c, rows) + rows == (uint32_t)part.rows;
    __syncthreads();
    if (s_complete) finish_client(c, batch, shape, ws, enc, sh_hist);
  }
}

__global__ void __launch_bounds__(kPlanThreads)
k_plan_threshold(const Batch batch, const __grid_constant__ Shape shape, unsigned char* ws, const __grid_constant__ EncFront enc) {
  __shared__ __align__(16) uint32_t N[kSurvivalBytes / 4];
  pdl_enter();
  finish_client(blockIdx.x, batch, shape, ws, enc, N);
}

// K2a  per client: exponent fit and tuning key, where the tuning is shared by clients of one key.  What the threshold bin comes from:
enum FitThreshold {
  kThresholdThere,    // the histogram's last blocks have worked it out
  kThresholdFinish,   // finish_client, here
  kThresholdOutside,  // a histogram from outside: the bin alone
};
__global__ void __launch_bounds__(kPlanThreads, 1)
k_plan_fit(const unsigned long long* __restrict__ hist_all, const uint32_t* __restrict__ nonfinite_all, const Batch batch,
           const __grid_constant__ Shape shape, unsigned char* ws, const __grid_constant__ EncFront enc, FitThreshold threshold) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* N = reinterpret_cast<uint32_t*>(smem_raw);
  pdl_enter();
  const uint32_t c = blockIdx.x;
  const uint32_t nonfinite = nonfinite_all[c];
  cvlc_plan_t* plan = batch.c[c].plan;
  int32_t* ws_status = reinterpret_cast<int32_t*>(ws);
  const int tid = threadIdx.x, lane = tid & 31;
  if (nonfinite & 2u) {  // a histogram from outside whose counts do not add up to d (its tuning key stays zero: no tuning)
    if (tid == 0) {
      plan->status = CVLC_ERR_INVALID_ARG;
      set_status(ws_status, CVLC_ERR_INVALID_ARG);
    }
    return;
  }
  const double B = batch.c[c].scale_B;
  __shared__ PlanTab T;
  if (threshold == kThresholdFinish) finish_client(c, batch, shape, ws, enc, N);
  else survival_counts(hist_all + (size_t)c * CVLC_HIST_BINS, N);
  auto beside_fit = [&]() {
    if (tid >= kPlanThreads - 32) build_plan_tab(T, shape, B, lane);
  };
  const double2 alpha = client_fit(N, *reinterpret_cast<FitScratch*>(smem_raw + kSurvivalBytes), shape, beside_fit);
  if (shape.fixed_y) {
    beside_fit();
    __syncthreads();
  }
  write_fit(plan, alpha, T, shape);
  if (threshold == kThresholdOutside) {
    client_threshold(N, shape, batch.c[c].cap0, plan, nullptr);
    if (tid == 0 && nonfinite) {
      plan->status = CVLC_ERR_NONFINITE_INPUT;
      set_status(ws_status, CVLC_ERR_NONFINITE_INPUT);
    }
  }
  if (tid == 0) {
    // clients with the same quantised exponent and the same scale get the same lengths
    unsigned long long* key = reinterpret_cast<unsigned long long*>(ws + plan_off_keys(batch.n)) + 2 * (size_t)c;
    key[0] = (unsigned long long)__double_as_longlong(alpha.y);
    key[1] = (unsigned long long)__double_as_longlong(B);
  }
}

// ---- atomic operations decided without the series arithmetic -----------------------------------
// An atomic operation on the lengths i > j looks for the first split t with F(t + 1) <= F(t), F evaluated in the
// series arithmetic.  Over the reals F(t) = sum_l h_l E(W_l(t)) with h_l = g_l - g_(l-1) >= 0 over the candidate
// lengths (Eq. (5) summed by parts: a length without packets adds nothing), W_l linear in t and E concave, so the
// differences F(t + 1) - F(t) fall with t.  A difference whose size exceeds `guard` has the same sign in the series
// arithmetic, and by concavity so has every difference on the far side of it: two differences around the answer, each
// beyond the guard, settle the whole bisection, and with it the comparison of the new split with the current one.
// The guard covers the rounding of both sides.  E(W) = (p - 1) / D with p = (W + 1)^beta <= max(1, D + 1): a power is
// within about 5e-15 of its value in either arithmetic (log2 of up to 31 rounded to 1.8e-15 twice, the polynomial's
// roundings), the weights h_l add up to at most 1, the ordered sum of 32 terms adds 4e-15, twice: below
// 3e-14 (1 + 1 / |D|); the guard is 7 times that.  Differences around an optimum are 1e-11 and more for the usual
// budgets; an operation that meets a smaller one is left to the series arithmetic (steep power laws: most are).
//
// What is left is latency, about four cycles for every instruction of a lone warp, so the steps are few and short.  A packet moved
// from length j to length i > j gives the covers of the lengths between them (and i) cap_i ranks and takes delta = cap_j - cap_i
// from those up to j.  The latter is little next to their size a = W + 1, so that their part of the difference is four terms of a
// Taylor series in delta, with coefficients that are prefix sums over the lengths of h / D a^(beta - k), the same for all pairs; the
// former are worked out as they are.  Both directions of all neighbouring pairs are then one evaluation by one warp (lane = i), and
// those of all pairs one per row (lane = j, a row per warp).  Where an operation on neighbours moves to follows from the condition
// that the derivative vanishes, solved for a_i (the other covers hardly change); with the half step between difference and
// derivative that is at most one packet from the answer.  The move is made, and the evaluation of the sweep's next operations
// tells whether it was the right one.  Moves between other pairs (none after the neighbours are settled, in all the usual cases) are
// left to the series arithmetic.
// Measured, exponent fit and tuning together: one ResNet-18-sized client (12 moves, 23 evaluations of about 1200 cycles, a check of
// all pairs of 3500) 68 -> 37 us, a client of 100,000 coordinates 25 -> 19, one of 300,000 of ten 30 -> 21, against an operation
// per warp, 16 of them in step, and moves searched for by trial splits (35 steps of checks of 1400 cycles each, 27 of trials).
constexpr double kTuneGuard = 0x1p-42;
// Nearly every sign already shows in fp32, where the terms of a difference are worked out as
// h / D a^beta ((1 + x)^beta - 1), x = step / a, without cancellation inside a term.  A term is good to 3e-6 of itself
// (for |beta| <= 1; the argument of a^beta is split so that its rounding stays below 1e-7, see fast_power; the growth
// factor where its logarithm leaves the series: 2.5e-6), a sum of terms of one sign to 5e-7 more, the series' first term to 2e-6, its
// remainder is bounded where it is used: a difference beyond kTuneRel (1 + |beta|) of its parts' sizes has a certain sign, and the
// rest is looked at in fp64.
constexpr float kTuneRel = 0x1p-17f;
constexpr int kTuneTries = 8;  // corrections of a guess by one packet

// the state of one warp: one candidate length per lane
struct FastLane {
  double h;                 // weight of E(W) in F (0 beyond the last length)
  float hD, u, af, ra;      // h / D, h / D a^beta, a, 1 / a
  uint32_t a;               // W + 1, W = ranks covered down to this lane's length
  uint32_t n, cap;          // packets and records per packet of this lane's length
  float M1, M2, M3, M4;     // prefix sums over the lengths up to this one of h / D a^(beta - k)
};
struct FastShared {
  int4 result[2];           // of the operations on neighbours: cursor, whether something has moved, sweeps
  uint4 lane_a[32], lane_b[32];  // a warp's state for the others: n, a, M1, M2; M3, M4
  int key[kTuneWarps];      // first operation that is not known to stay, per warp
  int code;
};
struct FastConst {
  double beta, inv_D, guard;
  float fbeta, frel, fguard;
  float b1, b2, b3, b4;     // binomial coefficients of beta
  float b51;                // size of the fifth against the first
};

__device__ __forceinline__ float fast_lg2(float v) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float fast_ex2(float v) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float fast_rcp(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
// a^beta, beta a multiple of 1/128 below 8 in size: beta times the exponent of a is exact, its whole part goes to the
// result's exponent, and only a number below 5 is rounded before the exponential
__device__ __forceinline__ float fast_power(float af, float beta) {
  const uint32_t bits = __float_as_uint(af) - 0x3F3504F3u;        // mantissa into [sqrt(1/2), sqrt(2))
  const float e = (float)((int)bits >> 23);
  const float m = __uint_as_float((bits & 0x007FFFFFu) + 0x3F3504F3u);
  const float be = beta * e, whole = rintf(be);
  const float r = fast_ex2((be - whole) + beta * fast_lg2(m));
  const float w = fmaxf(whole, -100.0f);                           // below 2^-100: nothing next to the guard
  return r * __uint_as_float((uint32_t)((int)w + 127) << 23);
}
// (b1 / b0)^beta - 1, step = b1 - b0, r0 = 1 / b0
__device__ __forceinline__ float fast_growth(float b0, float b1, float step, float r0, float beta) {
  const float s = step * fast_rcp(b0 + b1), q = s * s;              // ln(b1 / b0) = 2 atanh(s)
  const float series = 2.0f * s * fmaf(q, fmaf(q, fmaf(q, 1.0f / 7, 1.0f / 5), 1.0f / 3), 1.0f);
  const float ln = fabsf(s) <= 0.1f ? series : 0.693147181f * fast_lg2(b1 * r0);
  const float z = beta * ln;
  const float e = z * fmaf(z, fmaf(z, fmaf(z, fmaf(z, fmaf(z, 1.0f / 720, 1.0f / 120), 1.0f / 24), 1.0f / 6), 0.5f), 1.0f);
  return fabsf(z) < 0.25f ? e : fast_ex2(1.44269504f * z) - 1.0f;
}

// Signs of F(t + 1) - F(t) and F(t) - F(t - 1) from fp64 powers, by a whole warp; 0: too close to tell.  `on` / `back`: whether there
// is such a split; at = covers plus one at t, step = what they gain for a packet
__device__ __noinline__ int2 fast_signs64(double h, double at, double step, bool on, bool back, double beta, double inv_D, double guard) {
  double p[3];
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    const double a = k == 0 ? at : (k == 1 ? at + step : at - step);
    p[k] = (k == 1 && !on) || (k == 2 && !back) ? 0.0 : exp2(beta * log2(a));
  }
  double up = h * (p[1] - p[0]), down = h * (p[0] - p[2]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    up += __shfl_xor_sync(kFull, up, off);
    down += __shfl_xor_sync(kFull, down, off);
  }
  up *= inv_D;
  down *= inv_D;
  return make_int2(up > guard ? 1 : (up < -guard ? -1 : 0), down > guard ? 1 : (down < -guard ? -1 : 0));
}
// K2b  exponent fit and code-length tuning, one CTA per client.  Where every client has an SM to itself (hist or survival counts given) it fits and
// tunes for itself.  In larger batches, whose blocks take SMs from the selection beside them, the fit has been a kernel before and
// only the first client of every tuning key does the work.
__device__ __forceinline__ void tune_client(uint32_t c, const Batch& batch, const Shape& shape, unsigned char* ws,
                                            const unsigned long long* __restrict__ hist_all, const uint32_t* survival, unsigned char* smem_raw) {
  __shared__ PlanShared S;
  __shared__ PlanTab T;
  __shared__ FastShared FS;
  __shared__ uint32_t s_leader;
  __shared__ uint32_t s_ny[CVLC_MAX_CODE_BITS + 1];
  __shared__ double s_single[CVLC_MAX_CODE_BITS];
  const unsigned long long* keys = reinterpret_cast<const unsigned long long*>(ws + plan_off_keys(batch.n));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  unsigned long long key0, key1;
  cvlc_plan_t* const my_plan = batch.c[c].plan;
  // beside the fit: the table of lengths; the logarithms of the single-length plans' covers (lane = length - 1) and of d
  auto beside_fit = [&]() {
    if (warp == kTuneWarps - 1) build_plan_tab(T, shape, batch.c[c].scale_B, lane);
    if (warp == 1) s_single[lane] = series_log2((double)((uint64_t)shape.R * shape.cap[lane + 1] + 1));
    if (tid == 64) S.D = series_log2((double)shape.d);
  };
  double2 alpha = make_double2(0.0, 0.0);
  const bool own = hist_all || survival;
  if (own) {
    const double B = batch.c[c].scale_B;
    const uint32_t* N = survival;
    if (!survival) {
      survival_counts(hist_all + (size_t)c * CVLC_HIST_BINS, reinterpret_cast<uint32_t*>(smem_raw));
      N = reinterpret_cast<const uint32_t*>(smem_raw);
    }
    alpha = client_fit(N, *reinterpret_cast<FitScratch*>(smem_raw + kSurvivalBytes), shape, beside_fit);
    key0 = (unsigned long long)__double_as_longlong(alpha.y);
    key1 = (unsigned long long)__double_as_longlong(B);
  } else {
    key0 = keys[2 * (size_t)c];
    key1 = keys[2 * (size_t)c + 1];
    if (key1 == 0ull) return;  // no key: the fit refused this client's histogram
    if (tid == 0) s_leader = c;
    __syncthreads();
    for (uint32_t i = tid; i < c; i += kTuneThreads)
      if (keys[2 * (size_t)i] == key0 && keys[2 * (size_t)i + 1] == key1) atomicMin(&s_leader, i);
    __syncthreads();
    if (s_leader != c) return;  // an earlier client of the batch tunes for this key and writes the result to all that share it
  }

  const double beta = __dadd_rn(__dmul_rn(2.0, __longlong_as_double((long long)key0)), 1.0);
  if (!own || shape.fixed_y) {  // a fixed length has no fit to stand beside
    beside_fit();
    __syncthreads();
  }
  if (warp == 1) s_single[lane] = series_exp2(__dmul_rn(beta, s_single[lane]));
  if (tid == 64) S.D = __dsub_rn(series_exp2(__dmul_rn(beta, S.D)), 1.0);
  if (warp == 3) S.n[lane] = 0;
  __syncthreads();
  const double D = S.D;
  const int nY = (int)T.nY;
  const uint32_t my_cap = (lane < nY) ? T.capY[lane] : 0u;

  // ---- objective bookkeeping -----------------------------------------------------------
  // F(n) = 1 - gamma of Eq. (5) is a running sum over the used lengths, longest first:
  // F += g_l * (E(W_l) - E(W_prev)), W_l = ranks covered down to and including length l.
  // For the current counts the kernel keeps, per candidate index l: the running sum after
  // length l (Q.Fpre) and the energy of the nearest used length at or above l (Q.Eab).  An
  // atomic operation on the lengths i > j leaves everything above i untouched, so a trial split
  // only needs E for the used lengths at or below i and continues the running sum from
  // Q.Fpre[i + 1]: the same operations in the same order as a full evaluation, on a fraction of
  // the lanes.
  PlanSolver& Q = *reinterpret_cast<PlanSolver*>(smem_raw);

  auto refresh_warp = [&]() {  // by one warp
    const uint32_t my_n = (lane < nY) ? S.n[lane] : 0u;
    uint64_t W = (uint64_t)my_n * my_cap;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint64_t o = __shfl_down_sync(kFull, W, off);
      if (lane + off < 32) W += o;
    }
    const double E = (my_n > 0) ? energy_E(W, beta, D) : 0.0;
    const unsigned used = __ballot_sync(kFull, my_n > 0);
    // the terms side by side, their sum in the order of the lengths
    const unsigned above = lane < 31 ? used & (kFull << (lane + 1)) : 0u;
    const double Eup = __shfl_sync(kFull, E, above ? __ffs(above) - 1 : 0);
    const double Eprev = above ? Eup : 0.0;
    const double term = (my_n > 0) ? __dmul_rn(T.gY[lane], __dsub_rn(E, Eprev)) : 0.0;
    double F = 0.0, Fmine = 0.0;
    for (unsigned rest = used; rest;) {
      const int l = 31 - __clz(rest);
      rest ^= 1u << l;
      F = __dadd_rn(F, __shfl_sync(kFull, term, l));
      if (lane <= l) Fmine = F;
    }
    Q.Wc[lane] = W;
    Q.Fpre[lane] = Fmine;
    Q.Eab[lane] = (my_n > 0) ? E : Eprev;
    if (lane == 0) {
      Q.used = used;
      Q.Fpre[32] = 0.0;
      Q.Eab[32] = 0.0;
    }
  };
  auto refresh_state = [&]() {  // all threads; ends with a barrier
    if (warp == 0) refresh_warp();
    __syncthreads();
  };

  if (T.fixed_y != 0) {
    if (tid == 0) S.n[0] = T.R;
    __syncthreads();
    refresh_state();
  } else {
    // ---- equal packets: best admissible single-length plan, ties to the longer code ----
    if (warp == 0) {
      const uint64_t W = (uint64_t)T.R * my_cap;
      // one term: F = 0 + g * (E - 0), E = (power - 1) / D
      const bool on = lane < nY && W <= T.d;
      const double F = on ? __dmul_rn(T.gY[lane], __ddiv_rn(__dsub_rn(s_single[T.Y[lane] - 1], 1.0), D)) : -CUDART_INF;
      double most = F;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_xor_sync(kFull, most, off);
        if (o > most) most = o;
      }
      const unsigned best = __ballot_sync(kFull, on && F == most);
      if (lane == (best ? 31 - __clz(best) : 0)) S.n[lane] = T.R;  // the host has checked that a plan is admissible
    }
    __syncthreads();

    // ---- atomic operations (Section IV-C) on pairs of lengths until nothing moves ----
    // An atomic operation bisects the split of X = n_i + n_j packets between the lengths i > j
    // for the first t with F(t+1) <= F(t) and moves there if that is strictly better.  Most
    // operations of a sweep change nothing, so consecutive operations are evaluated together as
    // if none of them moved; the first one (in sweep order) that does move is applied, the later
    // ones of the batch are dropped and the sweep resumes right after it: exactly the sequential
    // result.  Per round every unfinished operation gets as many bisection levels as the block's
    // 1024 (evaluation, length) items allow: evaluation e = 2q, 2q+1 of an operation is
    // F(mid+1), F(mid) of node q+1 of its decision tree (heap order: child 2h after
    // "F(mid+1) <= F(mid)", child 2h+1 after "F(mid+1) > F(mid)").
    auto next_pair = [&](int phase, int& i, int& j) {  // sweep order; i = 0 marks the end
      if (phase == 0) {
        --i;
        j = i - 1;
      } else if (j > 0) {
        --j;
      } else {
        --i;
        j = i - 1;
      }
    };
    // ---- the operations that the concavity of F settles (see FastLane above) -----------------
    const bool fast = (uint64_t)T.R * T.capY[0] <= T.d;  // no trial can send more than d coordinates (F = -infinity)
    FastConst fc;
    fc.beta = beta;
    fc.inv_D = 1.0 / D;
    fc.guard = kTuneGuard * (1.0 + fabs(fc.inv_D));
    fc.fbeta = (float)beta;
    fc.frel = kTuneRel * (1.0f + fabsf(fc.fbeta));
    fc.fguard = (float)fc.guard * 1.0001f;
    fc.b1 = fc.fbeta;
    fc.b2 = fc.b1 * (fc.fbeta - 1.0f) * 0.5f;
    fc.b3 = fc.b2 * (fc.fbeta - 2.0f) * (1.0f / 3);
    fc.b4 = fc.b3 * (fc.fbeta - 3.0f) * 0.25f;
    fc.b51 = fabsf((fc.fbeta - 1.0f) * (fc.fbeta - 2.0f) * (fc.fbeta - 3.0f) * (fc.fbeta - 4.0f)) * (1.001f / 120);
    FastLane fl;  // warp 0's throughout, the others' while all pairs are looked at
    fl.cap = my_cap;
    fl.h = (lane < nY) ? T.gY[lane] - (lane ? T.gY[lane - 1] : 0.0) : 0.0;
    fl.hD = (float)(fl.h * fc.inv_D);
    bool stale = true;  // the bookkeeping of the series arithmetic is behind the counts
    int turns = 0;
    auto set_cover = [&]() {  // what follows from a
      fl.af = (float)fl.a;
      fl.ra = fast_rcp(fl.af);
      fl.u = fl.hD * fast_power(fl.af, fc.fbeta);
    };
    auto set_sums = [&]() {
      float M1 = fl.u * fl.ra, M2 = M1 * fl.ra, M3 = M2 * fl.ra, M4 = M3 * fl.ra;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float o1 = __shfl_up_sync(kFull, M1, off), o2 = __shfl_up_sync(kFull, M2, off);
        const float o3 = __shfl_up_sync(kFull, M3, off), o4 = __shfl_up_sync(kFull, M4, off);
        if (lane >= off) {
          M1 += o1;
          M2 += o2;
          M3 += o3;
          M4 += o4;
        }
      }
      fl.M1 = M1;
      fl.M2 = M2;
      fl.M3 = M3;
      fl.M4 = M4;
    };
    auto load_counts = [&]() {  // the counts of S.n into the warp's copy
      fl.n = S.n[lane];
      uint32_t W = fl.n * my_cap;  // at most d in all
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_down_sync(kFull, W, off);
        if (lane + off < 32) W += o;
      }
      fl.a = W + 1u;
      set_cover();
    };
    // ranks that this lane's cover W gains for every packet moved from length j to length i > j
    auto cover_step = [&](int i, int j) -> int {
      const int ci = (int)__shfl_sync(kFull, fl.cap, i), cj = (int)__shfl_sync(kFull, fl.cap, j);
      return lane > i ? 0 : (lane > j ? ci : ci - cj);
    };
    // What an operation does by its two differences, rise = sign of F(t + 1) - F(t) and came = sign of F(t) - F(t - 1): 0 stays,
    // 1 more packets of the longer code, 2 fewer, 3 too close to tell
    auto op_code = [](int rise, int came) -> int { return (rise < 0 && came > 0) ? 0 : rise > 0 ? 1 : came < 0 ? 2 : 3; };
    // The same for this lane's pair of ni and nj packets: gu, gd = what the lengths between contribute if a packet is moved to the
    // longer code and back; S1 .. S4 the sums over those up to j, x = delta / a_j the largest relative step among them, whose fifth
    // term bounds the series' remainder
    auto lane_code = [&](float gu, float gd, float delta, float S1, float S2, float S3, float S4, float x, uint32_t ni, uint32_t nj) -> int {
      const float d2 = delta * delta;
      const float t1 = fc.b1 * delta * S1, odd = fmaf(fc.b3 * d2 * delta, S3, t1), even = d2 * fmaf(fc.b4 * d2, S4, fc.b2 * S2);
      const float up = gu + (even - odd), back = gd + (even + odd);
      const float size = fabsf(t1), left = size * fc.b51 * (x * x) * (x * x);
      const float away = fast_ex2((fc.fbeta - 5.0f) * fast_lg2(1.0f - x));  // the remainder's growth towards smaller a
      const float up_err = fmaf(fc.frel, fabsf(gu) + size, fmaf(left, away, fc.fguard));
      const float back_err = fmaf(fc.frel, fabsf(gd) + size, left + fc.fguard);
      int rise = (x < 0.5f && fabsf(up) > up_err) ? (up > 0.0f ? 1 : -1) : 0;
      int came = (x < 0.5f && fabsf(back) > back_err) ? (back > 0.0f ? -1 : 1) : 0;
      if (nj == 0) rise = -1;
      if (ni == 0) came = 1;
      return op_code(rise, came);
    };
    // the same in fp64, by a whole warp
    auto exact_code = [&](int i, int j) -> int {
      const uint32_t ni = __shfl_sync(kFull, fl.n, i), nj = __shfl_sync(kFull, fl.n, j);
      const int step = cover_step(i, j);
      const int2 sign = fast_signs64(fl.h, (double)fl.a, (double)step, nj != 0, ni != 0, fc.beta, fc.inv_D, fc.guard);
      return op_code(nj == 0 ? -1 : sign.x, ni == 0 ? 1 : sign.y);
    };
    // moves length i's packets from the pair (i, i - 1) of X packets to t
    auto put_split = [&](int i, uint32_t ni, uint32_t X, uint32_t t) {
      const int step = cover_step(i, i - 1);
      if (lane == i) fl.n = t;
      if (lane == i - 1) fl.n = X - t;
      fl.a += (t - ni) * (uint32_t)step;
      set_cover();
    };
    // Walks a sweep over neighbours from the pair (ci, ci - 1) on, by one warp; ends with ci = 0 behind its last operation, or with ci
    // on one that only the series arithmetic can decide.
    auto fast_sweep = [&](int& ci, int& moved) {
      int i = 0;                            // the operation whose move is still to be confirmed (0: none)
      uint32_t old = 0, X = 0, t = 0, lo = 0, hi = 0;
      int tries = 0;
      while (true) {
        set_sums();
        // lane i: the pair (i, i - 1)
        int mine;
        {
          const float S1 = __shfl_up_sync(kFull, fl.M1, 1), S2 = __shfl_up_sync(kFull, fl.M2, 1), S3 = __shfl_up_sync(kFull, fl.M3, 1), S4 = __shfl_up_sync(kFull, fl.M4, 1);
          const uint32_t nj = __shfl_up_sync(kFull, fl.n, 1), capj = __shfl_up_sync(kFull, fl.cap, 1);
          const float raj = __shfl_up_sync(kFull, fl.ra, 1);
          const float give = (float)fl.cap, delta = (float)capj - give;
          const float gu = fl.u * fast_growth(fl.af, fl.af + give, give, fl.ra, fc.fbeta);
          const float gd = fl.n > 0 ? fl.u * fast_growth(fl.af, (float)(fl.a - fl.cap), -give, fl.ra, fc.fbeta) : 0.0f;
          mine = lane_code(gu, gd, delta, S1, S2, S3, S4, delta * raj, fl.n, nj);
          if (lane == 0 || (fl.n | nj) == 0) mine = 0;
        }
        if (i) {  // was the move the right one?
          int code = __shfl_sync(kFull, mine, i);
          if (code == 3) code = exact_code(i, i - 1);
          const uint32_t next = code == 1 ? t + 1 : t - 1;
          if (code) {
            if (code == 3 || ++tries > kTuneTries || next - lo > hi - lo) {  // back to where it was
              put_split(i, t, X, old);
              ci = i;
              return;
            }
            put_split(i, t, X, next);
            t = next;
            continue;
          }
          moved = 1;
          ci = i - 1;
          i = 0;
        }
        int code = 0;
        for (unsigned flagged = __ballot_sync(kFull, mine != 0 && lane <= ci); flagged && code == 0;) {  // in the order of the sweep
          i = 31 - __clz(flagged);
          flagged ^= 1u << i;
          code = __shfl_sync(kFull, mine, i);
          if (code == 3) code = exact_code(i, i - 1);
        }
        if (code == 0) {
          ci = 0;
          return;
        }
        ci = i;
        if (code == 3) return;
        old = __shfl_sync(kFull, fl.n, i);
        X = old + __shfl_sync(kFull, fl.n, i - 1);
        lo = (code == 1) ? old + 1 : 0u;  // the answer lies in [lo, hi]
        hi = (code == 1) ? X : old - 1;
        {
          const float give = (float)__shfl_sync(kFull, fl.cap, i), delta = (float)__shfl_sync(kFull, fl.cap, i - 1) - give;
          const float S1 = __shfl_sync(kFull, fl.M1, i - 1), S2 = __shfl_sync(kFull, fl.M2, i - 1), ai = __shfl_sync(kFull, fl.af, i);
          const float inv_give = fast_rcp(give), per = fast_rcp(fc.fbeta - 1.0f);
          const float base = fast_lg2(delta * S1 * fast_rcp(__shfl_sync(kFull, fl.hD, i) * give));
          const float drift = (1.0f - fc.fbeta) * delta * S2 * fast_rcp(S1);
          float by = 0.0f;
#pragma unroll
          for (int k = 0; k < 2; ++k) {  // delta S1(t) = h_i / D cap_i a_i(t)^(beta - 1)
            const float a_new = fast_ex2(per * (base + fast_lg2(fmaxf(fmaf(drift, by, 1.0f), 1e-3f))));
            by = fminf(fmaxf((a_new - ai) * inv_give, -(float)old), (float)(X - old));
          }
          t = (uint32_t)fminf(fmaxf(ceilf((float)old + by - 0.5f), (float)lo), (float)hi);
          t = t < lo ? lo : (t > hi ? hi : t);
        }
        tries = 0;
        put_split(i, old, X, t);
      }
    };
    // the neighbours' sweeps until one of them is quiet (ci = 0), or up to an operation for the series arithmetic; by warp 0
    auto fast_neighbours = [&](int& ci, int& moved, int& sweep) {
      while (true) {
        fast_sweep(ci, moved);
        if (ci >= 1) break;
        if (!moved || ++sweep == 256) break;
        moved = 0;
        ci = nY - 1;
      }
      S.n[lane] = fl.n;
    };
    // All pairs from the cursor on, by all warps: leaves the cursor on the first operation that moves or that fp64 cannot tell, or
    // ci = 0.  Warp 0's state is the current one; the last warp meanwhile brings the series' bookkeeping up to date.
    auto fast_all_pairs = [&](int& ci, int& cj) {
      if (warp == 0) {
        set_sums();
        FS.lane_a[lane] = make_uint4(fl.n, fl.a, __float_as_uint(fl.M1), __float_as_uint(fl.M2));
        FS.lane_b[lane] = make_uint4(__float_as_uint(fl.M3), __float_as_uint(fl.M4), __float_as_uint(fl.u), 0u);
      }
      __syncthreads();
      if (warp != 0) {
        const uint4 v = FS.lane_a[lane], w = FS.lane_b[lane];
        fl.n = v.x;
        fl.a = v.y;
        fl.M1 = __uint_as_float(v.z);
        fl.M2 = __uint_as_float(v.w);
        fl.M3 = __uint_as_float(w.x);
        fl.M4 = __uint_as_float(w.y);
        fl.u = __uint_as_float(w.z);
        fl.af = (float)fl.a;
        fl.ra = fast_rcp(fl.af);
      }
      const unsigned used = __ballot_sync(kFull, fl.n > 0);
      while (ci >= 1) {
        int key = 0;
        if (warp == kTuneWarps - 1) {
          if (stale) refresh_warp();
        } else {
          for (int row = ci - warp; row >= 1 && key == 0; row -= kTuneWarps - 1) {  // a row i per warp, lane j: the pairs (i, j)
            const uint32_t ni = __shfl_sync(kFull, fl.n, row);
            if (ni == 0 && (used & ((1u << row) - 1u)) == 0) continue;
            const uint32_t cap_i = __shfl_sync(kFull, fl.cap, row);
            const float give = (float)cap_i;
            float gu = lane <= row ? fl.u * fast_growth(fl.af, fl.af + give, give, fl.ra, fc.fbeta) : 0.0f, gd = 0.0f;
            if (ni > 0 && lane <= row) gd = fl.u * fast_growth(fl.af, (float)(fl.a - cap_i), -give, fl.ra, fc.fbeta);
            // summed from the row's length down to the one above this lane's
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
              const float o1 = __shfl_down_sync(kFull, gu, off), o2 = __shfl_down_sync(kFull, gd, off);
              if (lane + off < 32) {
                gu += o1;
                gd += o2;
              }
            }
            gu = __shfl_down_sync(kFull, gu, 1);
            gd = __shfl_down_sync(kFull, gd, 1);
            const float delta = (float)fl.cap - give;
            int mine = lane_code(gu, gd, delta, fl.M1, fl.M2, fl.M3, fl.M4, delta * fl.ra, ni, fl.n);
            if (lane >= row || (row == ci && lane > cj) || (ni | fl.n) == 0) mine = 0;
            const unsigned flagged = __ballot_sync(kFull, mine != 0);
            if (flagged) {
              const int col = 31 - __clz(flagged);
              key = (row << 16) | (col << 8) | __shfl_sync(kFull, mine, col);
            }
          }
        }
        if (lane == 0) FS.key[warp] = key;
        __syncthreads();
        stale = false;
        key = __reduce_max_sync(kFull, lane < kTuneWarps ? FS.key[lane] : 0);
        ci = key >> 16;
        cj = (key >> 8) & 0xFF;
        if ((key & 0xFF) != 3) return;
        if (warp == 0) {
          const int code = exact_code(ci, cj);
          if (lane == 0) FS.code = code;
        }
        __syncthreads();
        if (FS.code != 0) return;
        next_pair(1, ci, cj);
      }
    };
    // One batch of operations from the cursor on in the series arithmetic (see above), by all warps
    auto series_batch = [&](int phase, int& ci, int& cj, int& moved) {
            if (stale) {
              __syncthreads();
              refresh_state();
              stale = false;
            }
            // ---- collect a batch: thread t looks at the t-th pair of the sweep from the cursor on (at most
            // 31 + 465 pairs).  The batch is the first pairs, in sweep order, that share packets (X > 0), up to
            // kMaxBatchOps of them and as long as two evaluations of each fit the block: a prefix of the flagged
            // pairs, found with one block scan of (operations, items) packed in a word.
            {
              auto pair_at = [&](int t, int& i, int& j) -> bool {
                if (t < 0) return false;
                if (phase == 0) {
                  i = ci - t;
                  j = i - 1;
                  return i >= 1;
                }
                const int first = cj + 1;  // rest of the cursor's row: j = cj .. 0
                if (t < first) {
                  i = ci;
                  j = cj - t;
                  return true;
                }
                const int rest = (ci - 1) * ci / 2;  // rows ci - 1 .. 1, row r holding the pairs (r, r-1) .. (r, 0)
                const int tp = t - first;
                if (tp >= rest) return false;
                const int u = rest - 1 - tp;  // counted upwards from pair (1, 0)
                int r = 1;
                while ((r * (r + 1)) / 2 <= u) ++r;
                i = r;
                j = u - (r - 1) * r / 2;
                return true;
              };
              // a thread looks at the pairs t = tid, tid + kTuneThreads, ...; the scan runs over t in order
              const unsigned used = Q.used;
              if (tid == 0) {
                Q.col_nops = 0;
                Q.col_last = -1;
                Q.col_first_left = 0x7FFFFFFF;
              }
              uint32_t carry = 0;
#pragma unroll
              for (int slot = 0; slot < kPairSlots; ++slot) {
                const int t = slot * kTuneThreads + tid;
                int pi = 0, pj = 0;
                const bool valid = pair_at(t, pi, pj);
                uint32_t X = 0;
                unsigned need = 0;
                int m = 0;
                if (valid) {
                  X = S.n[pi] + S.n[pj];
                  if (X > 0) {
                    need = (used | (1u << pi) | (1u << pj)) & (0xFFFFFFFFu >> (31 - pi));
                    m = __popc(need);
                  }
                }
                const bool flag = valid && X > 0;
                uint32_t incl = flag ? ((1u << 16) | (uint32_t)(2 * m)) : 0u;  // items stay below 2^16: 496 pairs of at most 64
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                  const uint32_t o = __shfl_up_sync(kFull, incl, off);
                  if (lane >= off) incl += o;
                }
                if (lane == 31) Q.col_warp[warp] = incl;
                __syncthreads();
                {
                  const uint32_t wt = (lane < kTuneThreads / 32) ? Q.col_warp[lane] : 0u;
                  uint32_t wi = wt;
#pragma unroll
                  for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t o = __shfl_up_sync(kFull, wi, off);
                    if (lane >= off) wi += o;
                  }
                  incl += carry + __shfl_sync(kFull, wi - wt, warp);
                  carry += __shfl_sync(kFull, wi, 31);
                }
                const int rank = (int)(incl >> 16) - 1;
                const bool taken = flag && rank < kMaxBatchOps && (incl & 0xFFFFu) <= (uint32_t)kPlanItems;
                if (taken) {
                  PlanOp& o = Q.op[rank];
                  o.i = pi; o.j = pj; o.X = X; o.na0 = S.n[pi]; o.lo = 0; o.hi = X; o.m = m; o.F_final = 0.0;
                  for (unsigned rest_bits = need; rest_bits;) {  // the lengths a trial evaluates, longest first
                    const int l = 31 - __clz(rest_bits);
                    rest_bits ^= 1u << l;
                    o.slot_lane[l == 31 ? 0 : __popc(need >> (l + 1))] = (unsigned char)l;
                  }
                  atomicMax(&Q.col_nops, rank + 1);
                  atomicMax(&Q.col_last, t);
                } else if (flag) {
                  atomicMin(&Q.col_first_left, t);
                }
                if (slot + 1 < kPairSlots) __syncthreads();  // the warp totals are reused by the next slot
              }
              __syncthreads();
              const int n_ops = Q.col_nops;
              // the sweep resumes after the last operation of a full batch, else at the first pair left over
              const int resume = (n_ops == kMaxBatchOps) ? Q.col_last + 1
                                                         : (Q.col_first_left != 0x7FFFFFFF ? Q.col_first_left : -1);
              int bi = 0, bj = 0;
              if (!pair_at(resume, bi, bj)) bi = bj = 0;
              if (tid == 0) {
                Q.n_ops = n_ops;
                Q.next_i = bi;
                Q.next_j = bj;
                Q.moved = 0;
                Q.unfinished = n_ops;
              }
              ci = bi;
              cj = bj;
              if (n_ops == 0) {  // the rest of the sweep had nothing to split
                __syncthreads();  // the collection's scratch is reset by the next one
                return;
              }
            }
            __syncthreads();
            const int n_ops = Q.n_ops;
            const double F_cur = Q.Fpre[0];
            // ---- rounds until every operation of the batch has finished its bisection
            // level assignment (warp 0, lane = operation), before the first round and right after every tree walk:
            // the planner is bound by the FP64 throughput
            // of its SM, and every extra level evaluated ahead doubles the work, so all operations get
            // the same small depth: the largest one whose items fit the block
            auto assign_levels = [&]() {
                const bool mine = lane < n_ops;
                const uint32_t span = (mine && Q.op[lane].lo < Q.op[lane].hi) ? Q.op[lane].hi - Q.op[lane].lo : 0u;
                const int need_levels = span ? 32 - __clz(span) : 0;  // a bisection of s points takes at most floor(log2 s) + 1 steps
                const int m_op = mine ? Q.op[lane].m : 0;
                // items of the whole batch at every candidate depth: nine reductions side by side (one after the
                // other they are nine chains of five dependent shuffles, as long as the energy evaluation itself)
                int items_at[9];
#pragma unroll
                for (int cand = 1; cand <= 9; ++cand) {
                  const int lvc = need_levels < cand ? need_levels : cand;
                  items_at[cand - 1] = lvc ? 2 * ((1 << lvc) - 1) * m_op : 0;
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
                  for (int q = 0; q < 9; ++q) items_at[q] += __shfl_xor_sync(kFull, items_at[q], off);
                }
                int depth = 0;
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                  if (items_at[q] <= kPlanItems && depth == q) depth = q + 1;  // the sums grow with the depth
                }
                const int lv = need_levels < depth ? need_levels : depth;
                const int ne = lv ? 2 * ((1 << lv) - 1) : 0;
                int items_incl = ne * m_op, evals_incl = ne;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                  const int a1 = __shfl_up_sync(kFull, items_incl, off), a2 = __shfl_up_sync(kFull, evals_incl, off);
                  if (lane >= off) {
                    items_incl += a1;
                    evals_incl += a2;
                  }
                }
                if (mine) {
                  Q.op[lane].levels = lv;
                  Q.op[lane].item_base = items_incl - ne * m_op;
                  Q.op[lane].eval_base = evals_incl - ne;
                }
                Q.item_end[lane] = items_incl;
                Q.eval_end[lane] = evals_incl;
                const unsigned unfinished = __ballot_sync(kFull, need_levels > 0);
                if (lane == 31) {
                  Q.n_items = items_incl;
                  Q.n_evals = evals_incl;
                  Q.unfinished = __popc(unfinished);
                }
                          };
            if (warp == 0) assign_levels();
            while (true) {
              __syncthreads();
              if (Q.unfinished == 0) break;
              // phase 1: energies, one thread per (operation, evaluation, slot)
              for (int vt = tid; vt < Q.n_items; vt += kTuneThreads) {
                int a = -1, e = 0, sl = 0;
                uint32_t t = 0xFFFFFFFFu;
                // the operation whose item range holds this item: first a with vt < item_end[a]
                int lo_a = 0, hi_a = 31;
                while (lo_a < hi_a) {
                  const int mid = (lo_a + hi_a) >> 1;
                  if (vt < Q.item_end[mid]) hi_a = mid; else lo_a = mid + 1;
                }
                a = lo_a;
                const PlanOp& o = Q.op[a];
                const int rel = vt - o.item_base;
                e = rel / o.m;
                sl = rel - e * o.m;
                const int hnode = (e >> 1) + 1;
                const int depth = 31 - __clz(hnode);
                uint32_t l3 = o.lo, h3 = o.hi;
                bool open = true;
                for (int b = depth - 1; b >= 0; --b) {
                  if (!(l3 < h3)) { open = false; break; }
                  const uint32_t mid = l3 + (h3 - l3) / 2;
                  if ((hnode >> b) & 1) l3 = mid + 1; else h3 = mid;
                }
                if (open && l3 < h3) {
                  t = l3 + (h3 - l3) / 2 + ((e & 1) ? 0u : 1u);
                  const int l = o.slot_lane[sl];
                  // ranks down to length l with the pair's packets re-split: the current cover, minus the
                  // pair's current share, plus the trial's
                  uint64_t W = Q.Wc[l] - (uint64_t)S.n[o.i] * T.capY[o.i] + (uint64_t)t * T.capY[o.i];
                  if (l <= o.j) W = W - (uint64_t)S.n[o.j] * T.capY[o.j] + (uint64_t)(o.X - t) * T.capY[o.j];
                  Q.Ev[vt] = energy_E(W, beta, D);
                }
                if (sl == 0) {
                  Q.tv[o.eval_base + e] = t;
                  Q.ea[o.eval_base + e] = (unsigned char)a;
                }
              }
              __syncthreads();
              // phase 2: one thread per evaluation continues the running sum below length i with the terms
              // g_l * (E_l - E_prev) in the order of the lengths; only the lengths i and j can be unused in a trial
              // (no term, and the next term's E_prev skips them).  The terms do not depend on the sum, so they are
              // worked out four at a time ahead of the ordered additions.
              for (int vt = tid; vt < Q.n_evals; vt += kTuneThreads) {
                const PlanOp& o = Q.op[Q.ea[vt]];
                const uint32_t tt = Q.tv[vt];
                if (tt != 0xFFFFFFFFu) {
                  const int ee = vt - o.eval_base;
                  const double* Ez = Q.Ev + o.item_base + ee * o.m;
                  double F = Q.Fpre[o.i + 1];
                  double Eprev = Q.Eab[o.i + 1];
                  for (int z0 = 0; z0 < o.m; z0 += 4) {
                    double term4[4];
                    bool on4[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                      const int z = z0 + q;
                      on4[q] = false;
                      term4[q] = 0.0;
                      if (z < o.m) {
                        const int l = o.slot_lane[z];
                        const uint32_t nn = (l == o.i) ? tt : (l == o.j) ? (o.X - tt) : 1u;
                        if (nn > 0) {
                          const double Ec = Ez[z];
                          on4[q] = true;
                          term4[q] = __dmul_rn(T.gY[l], __dsub_rn(Ec, Eprev));
                          Eprev = Ec;
                        }
                      }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                      if (on4[q]) F = __dadd_rn(F, term4[q]);
                  }
                  const uint64_t Wtot = Q.Wc[0] - (uint64_t)S.n[o.i] * T.capY[o.i] - (uint64_t)S.n[o.j] * T.capY[o.j] +
                                        (uint64_t)tt * T.capY[o.i] + (uint64_t)(o.X - tt) * T.capY[o.j];
                  Q.Fv[vt] = (Wtot > T.d) ? -CUDART_INF : F;
                }
              }
              __syncthreads();
              // phase 4: one thread per operation walks its decision tree
              if (tid < n_ops) {
                PlanOp& o = Q.op[tid];
                if (o.levels > 0) {
                  uint32_t lo = o.lo, hi = o.hi;
                  double Ff = o.F_final;
                  int hnode = 1;
                  for (int level = 0; level < o.levels && lo < hi; ++level) {
                    const uint32_t mid = lo + (hi - lo) / 2;
                    const double F1 = Q.Fv[o.eval_base + 2 * (hnode - 1)], F0 = Q.Fv[o.eval_base + 2 * (hnode - 1) + 1];
                    if (F1 > F0) {
                      lo = mid + 1;
                      Ff = F1;
                      hnode = 2 * hnode + 1;
                    } else {
                      hi = mid;
                      Ff = F0;
                      hnode = 2 * hnode;
                    }
                  }
                  o.lo = lo;
                  o.hi = hi;
                  o.F_final = Ff;
                }
              }
              if (warp == 0) {  // the lanes that walked the trees own the same operations in the level assignment
                __syncwarp();
                assign_levels();
              }
            }
            // ---- the first operation of the batch that improves F is applied; the sweep resumes after it
            if (tid == 0) {
              for (int a = 0; a < n_ops; ++a) {
                const PlanOp& o = Q.op[a];
                if (o.lo != o.na0 && o.F_final > F_cur) {
                  S.n[o.i] = o.lo;
                  S.n[o.j] = o.X - o.lo;
                  int ri = o.i, rj = o.j;
                  next_pair(phase, ri, rj);
                  Q.next_i = ri;
                  Q.next_j = rj;
                  Q.moved = 1;
                  break;
                }
              }
            }
            __syncthreads();
            ci = Q.next_i;
            cj = Q.next_j;
            if (Q.moved) {
              moved = 1;
              refresh_state();
              if (fast && warp == 0) load_counts();
            } else {
              __syncthreads();
            }
    };
    if (fast && warp == 0) load_counts();
    for (int round = 0; round < 64; ++round) {
      // neighbouring lengths until quiet
      int ci = nY - 1, cj = nY - 2, moved = 0;  // cursor of the sweep
      for (int sweep = 0; ci >= 1 || sweep == 0;) {
        if (fast) {
          if (warp == 0) {
            fast_neighbours(ci, moved, sweep);
            if (lane == 0) FS.result[turns & 1] = make_int4(ci, moved, sweep, 0);
          }
          __syncthreads();
          const int4 r = FS.result[turns++ & 1];
          ci = r.x;
          cj = ci - 1;
          moved = r.y;
          sweep = r.z;
          stale = true;
          if (ci < 1) break;
        }
        series_batch(0, ci, cj, moved);
        if (ci < 1) {
          if (!moved || ++sweep == 256) break;
          moved = 0;
          ci = nY - 1;
          cj = nY - 2;
        }
      }
      // every pair once
      ci = nY - 1;
      cj = nY - 2;
      moved = 0;
      while (ci >= 1) {
        if (fast) fast_all_pairs(ci, cj);
        if (ci >= 1) series_batch(1, ci, cj, moved);
      }
      if (!moved) break;
    }
    if (stale) {
      __syncthreads();
      refresh_state();
    }
  }

  // ---- outputs, to this client and to the later ones that share its tuning key -------------------
  if (own) write_fit(my_plan, alpha, T, shape);
  if (tid <= CVLC_MAX_CODE_BITS) s_ny[tid] = 0;
  __syncthreads();
  if (tid < nY) s_ny[T.Y[tid]] = S.n[tid];
  const uint32_t my_n = lane < nY ? S.n[lane] : 0u;
  const unsigned long long k = __reduce_add_sync(kFull, my_n * my_cap);  // at most d
  double Qmax = my_n > 0 ? T.QY[lane] : 0.0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_xor_sync(kFull, Qmax, off);
    if (o > Qmax) Qmax = o;
  }
  __syncthreads();
  for (uint32_t i = c + warp; i < (own ? c + 1 : batch.n); i += kTuneWarps) {
    if (i != c && (keys[2 * (size_t)i] != key0 || keys[2 * (size_t)i + 1] != key1)) continue;
    cvlc_plan_t* __restrict__ dst = i == c ? my_plan : batch.c[i].plan;
    dst->n_y[lane] = s_ny[lane];
    if (lane == 0) {
      dst->n_y[CVLC_MAX_CODE_BITS] = s_ny[CVLC_MAX_CODE_BITS];
      dst->k = k;
      dst->gamma = __dsub_rn(1.0, Q.Fpre[0]);
      dst->B_next = __dadd_rn(1.0, Qmax);
    }
  }
}

__global__ void __launch_bounds__(kTuneThreads, 1)
k_plan_tune(const Batch batch, const __grid_constant__ Shape shape, unsigned char* ws, const unsigned long long* __restrict__ hist_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_enter();
  tune_client(blockIdx.x, batch, shape, ws, hist_all, nullptr, smem_raw);
}

// ===================================================================================
// K1-K4 of few small clients: a cluster of blocks per client
// ===================================================================================
// Every block but the last keeps its share of the update in shared memory and counts its bins.  The counts are exchanged through the cluster's
// shared memory: every block then has the client's histogram and, for each bin, how many of its values are in the blocks before it, so that it
// knows the place of each of its candidates by bin, without an addition in global memory.  They go there (the L2), and behind a third
// barrier those blocks rank a share each, in whole bins, while the last one, which needs the histogram alone, has been fitting the exponent and
// tuning the lengths.  (With a share of the update for that one too the tuning began 3 to 5 us later: one client of 100,000 coordinates whose
// magnitudes fall as rank^-1.3 38.6 -> 37.0 us, ten of 300,000 at 0.4 bits 45.3 -> 41.3, a normal distribution 34.5 -> 31.0; one of 600,000 at 2.5
// bits, where the ranking is what the cluster ends with, 37.1 -> 37.4.)  A share may be more than a block keeps; the rest is read again.  Bins of more
// than a block holds are cut again (see cut_bins); cells of more than 256 equal or nearly equal keys are left to k_rank_rest, whose blocks work
// them off side by side.
// Bound by latencies: of 17 us for one client of 100,000 coordinates and 20 for ten of 300,000 the tuning takes the last 10.  As kernels
// of their own (zeros, histogram, selection, partition, ranking, what that leaves over, and the tuning on another stream between two
// events) the steps took 30 and 39; whole calls 36.9 -> 26.5 us, 56.7 -> 45.2 with the aggregation.

struct ClusterShared {
  uint32_t own[CVLC_HIST_BINS + 4];  // the block's counts; then the client's survival counts
  uint32_t total[CVLC_HIST_BINS];    // the client's
  uint32_t place[CVLC_HIST_BINS];    // those of the blocks before it; then next places
};
constexpr size_t kFitSmem = kSurvivalBytes + sizeof(FitScratch);
constexpr size_t kTuneSmem = sizeof(PlanSolver) > kFitSmem ? sizeof(PlanSolver) : kFitSmem;  // one after the other
constexpr size_t kClusterSmem = sizeof(ClusterShared) + (size_t)kClusterUnits * 16;
// Units of a share beyond those that a block keeps, for each of its threads: a share is a seventh or a fifteenth of what eight or sixteen blocks keep
constexpr uint32_t kClusterOver = 3;
static_assert(kClusterOver * kPlanThreads >= kClusterUnits / 7 + kRowUnits, "a share");
static_assert(kTuneSmem <= (size_t)kClusterUnits * 16 && sizeof(RankShared) <= (size_t)kClusterUnits * 16 && sizeof(ClusterShared) % 16 == 0 &&
              kClusterSmem <= 216 * 1024, "shared memory");

// One more in counters of a table for each of the lanes' values that is on: what was in them before.  One addition where all of the warp's go to
// one counter (which takes one a cycle), or all of a lane's.
template <int V>
__device__ __forceinline__ void add_all(uint32_t* table, const bool (&on)[V], const uint32_t (&i)[V], uint32_t (&at)[V]) {
  bool all = true;
#pragma unroll
  for (int u = 0; u < V; ++u) all = all && on[u] && i[u] == i[0];
  const uint32_t lane = threadIdx.x & 31, first = __shfl_sync(kFull, i[0], 0);
  if (__all_sync(kFull, all && i[0] == first)) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(table + first, 32u * V);
    at[0] = __shfl_sync(kFull, base, 0) + lane;
#pragma unroll
    for (uint32_t u = 1; u < V; ++u) at[u] = at[0] + 32 * u;
  } else if (all) {
    at[0] = atomicAdd(table + i[0], (uint32_t)V);
#pragma unroll
    for (uint32_t u = 1; u < V; ++u) at[u] = at[0] + u;
  } else {
#pragma unroll
    for (int u = 0; u < V; ++u) at[u] = on[u] ? atomicAdd(table + i[u], 1u) : 0u;
  }
}

// A block's candidates to their places where a bin holds many
__device__ __noinline__ void put_crowded(uint32_t* place, uint32_t thresh_bin, const float4* data, uint32_t units, uint32_t u0, unsigned long long* by_bin) {
  for (uint32_t i0 = 0; i0 < units; i0 += kPlanThreads) {
    const uint32_t i = i0 + threadIdx.x;
    const float4 a = i < units ? data[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t v[4] = {__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(a.z), __float_as_uint(a.w)};
    uint32_t bin[4], at[4];
    bool on[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      bin[u] = (v[u] & 0x7FFFFFFFu) >> 19;
      on[u] = i < units && bin[u] >= thresh_bin;
    }
    add_all(place, on, bin, at);
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u)
      if (on[u]) by_bin[at[u]] = ((unsigned long long)(v[u] & 0x7FFFFFFFu) << 32) | (unsigned long long)((v[u] & 0x80000000u) | (4 * (u0 + i) + u));
  }
}

// ---- bins of more candidates than a block ranks: values crowded in a bin, repeated ones, zeros --------------------------------
// Cut by all ranking blocks of the cluster, beside the tuning: every block counts a share of such a bin's candidates by the next nine bits of (key,
// index), the counts are added up in global memory, and the candidates go to the places of their parts.  Parts that are still too large
// are cut again; after the third cut a part is what 4096 neighbouring coordinates have of one key.
// A cut is a chain of latencies: reading, counting and moving 1 to 5 us each, two waits of the blocks for one another 1.5 each.  Left to k_rank_rest, as large
// buckets of other batches are, such bins came behind the tuning and took 45 to 120 us there.  Whole calls, as kernels of their own / left to
// k_rank_rest / cut, us: 36,000 candidates spread over one bin, ten clients of 300,000 coordinates 57 / 107 / 47; on eight values 74 / 125 / 66;
// signs only, one of 600,000 107 / 120 / 79, ten of 300,000 181 / 143 / 81; 5 % of one magnitude, one of 600,000 104 / 106 / 65; 98 % zeros, one of
// 320,000 101 / 101 / 91.  But one client of 600,000 in 16 bits (fp16, 59,500 records) 59 / 84 / 67: 15 blocks rank where 296 did.
constexpr uint32_t kCutParts = 512, kCutRanges = 8, kCuts = 3, kCutTable = kCutRanges * kCutParts;
static_assert(kCutParts == kPlanThreads && kCutParts == 16 * 32 && kCutTable <= CVLC_HIST_BINS && kCutRanges <= kPlanThreads / 32, "one part per thread");
static_assert((kRankItems + 1) * kCutRanges > kClusterCandidates, "room for all ranges that begin with a rank that may be sent");
static_assert(2 * kCutTable <= kRankSubs, "the tables' place");
static_assert(16 * 4 * kClusterUnits + 3 < 1u << 20, "bits of an index");
struct Cut {
  uint32_t n;                   // ranges that are cut
  uint32_t prefix[kCutRanges];  // their bits of (key's complement, index), those that follow say the part
  uint32_t start[kCutRanges], size[kCutRanges];
  uint32_t part[kCutRanges];    // their parts of the cut before (of the first cut: bins)
  bool in_a;                    // their candidates lie in the first buffer and go to the second
};
__device__ __forceinline__ uint32_t cut_part(u64 item, uint32_t cut) {
  const uint32_t inv_key = ~(uint32_t)(item >> 32);
  return cut == 0 ? (inv_key >> 10) & 511u : cut == 1 ? (inv_key >> 1) & 511u : (inv_key & 1u) << 8 | ((uint32_t)item & 0x7FFFFFFFu) >> 12;
}
// keytop - key where part `part` of range r begins
__device__ __forceinline__ uint32_t cut_inv(const Cut& C, uint32_t cut, uint32_t r, uint32_t part, uint32_t keytop) {
  const uint32_t inv_key = cut == 2 ? (C.prefix[r] << 1) + (part >> 8) : ((C.prefix[r] << 9) + part) << (cut == 0 ? 10 : 1);
  return inv_key - (0x7FFFFFFFu - keytop);
}
// what the parts of a cut hold, and the ranks that they begin with; the first are zero when the cutting begins
__device__ __forceinline__ uint32_t* cut_totals(unsigned char* ws, const EncLayout& L, uint32_t c, uint32_t cut) {
  return cut < 2 ? reinterpret_cast<uint32_t*>(ws + L.off_sub_start) + (size_t)c * (kRankSubs + 64) + cut * kCutTable
                 : reinterpret_cast<uint32_t*>(ws + L.off_sub_pos) + (size_t)c * kRankSubs;
}
__device__ __forceinline__ uint32_t* cut_starts(unsigned char* ws, const EncLayout& L, uint32_t c, uint32_t cut) {
  return cut < 2 ? reinterpret_cast<uint32_t*>(ws + L.off_sub_count) + (size_t)c * kRankSubs + cut * kCutTable
                 : reinterpret_cast<uint32_t*>(ws + L.off_sub_pos) + (size_t)c * kRankSubs + kCutTable;
}
// the ranking blocks' turns behind one another
__device__ __forceinline__ uint32_t* cut_turns(unsigned char* ws, const EncLayout& L, uint32_t c) { return reinterpret_cast<uint32_t*>(ws + L.off_group_done) + c; }

// f(items, which of them are there), kCutHold of src[lo .. hi) a thread at a time, by whole warps
constexpr int kCutHold = 8;
template <class F>
__device__ __forceinline__ void by_eights(const u64* src, uint32_t lo, uint32_t hi, F&& f) {
  for (uint32_t i0 = lo; i0 < hi; i0 += kCutHold * kPlanThreads) {
    const uint32_t first = i0 + kCutHold * (threadIdx.x & ~31u) + (threadIdx.x & 31u);  // a warp's are neighbours
    u64 v[kCutHold];
    bool on[kCutHold];
#pragma unroll
    for (uint32_t u = 0; u < kCutHold; ++u) {
      on[u] = first + 32 * u < hi;
      v[u] = on[u] ? __ldcg(src + first + 32 * u) : 0ull;
    }
    f(v, on);
  }
}

// By the ranking blocks of the cluster, q of `blocks`; N: the client's survival counts; table: of kCutTable counters.  False: a wait has run out.
__device__ __noinline__ bool cut_bins(uint32_t* table, const uint32_t* N, Cut* cuts, const Threshold& t, uint32_t limit, unsigned char* ws, const EncLayout& L,
                                      uint32_t c, uint32_t q, uint32_t blocks, u64* buf_a, u64* buf_b) {
  __shared__ uint32_t s_found[kCutRanges][kCutRanges][3], s_n[kCutRanges];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int32_t* status = &reinterpret_cast<EncHeader*>(ws)->status;
  uint32_t* turns = cut_turns(ws, L, c);
  uint32_t turn = 0;
  if (warp == 0) {
    uint32_t n = 0;
    for (int b0 = (int)t.top; b0 >= (int)t.bin; b0 -= 32) {
      const int b = b0 - lane;
      const uint32_t m = b >= (int)t.bin ? N[b] - N[b + 1] : 0u;
      const unsigned large = __ballot_sync(kFull, m > kRankHold);
      const uint32_t at = n + __popc(large & ((1u << lane) - 1u));
      if (m > kRankHold && at < kCutRanges) {
        cuts[0].prefix[at] = 4095u - (uint32_t)b;
        cuts[0].start[at] = N[b + 1];
        cuts[0].size[at] = m;
        cuts[0].part[at] = (uint32_t)b;
      }
      n += __popc(large);
    }
    if (lane == 0) {
      cuts[0].n = min(n, kCutRanges);
      cuts[0].in_a = false;
    }
  }
  for (uint32_t cut = 0; cut < kCuts; ++cut) {
    const Cut& C = cuts[cut];
    __syncthreads();
    const uint32_t n = C.n;
    if (n == 0) break;
    for (uint32_t i = tid; i < n * kCutParts; i += kPlanThreads) table[i] = 0;
    __syncthreads();
    const u64* src = C.in_a ? buf_a : buf_b;
    u64* dst = C.in_a ? buf_b : buf_a;
    uint32_t* totals = cut_totals(ws, L, c, cut);
    // f(items, which there are, their entries of the table, their places) of the block's share of the ranges
    auto share = [&](auto&& f) {
      for (uint32_t r = 0; r < n; ++r) {
        const uint32_t m = C.size[r];
        by_eights(src + C.start[r], m * q / blocks, m * (q + 1) / blocks, [&](const u64 (&v)[kCutHold], bool (&on)[kCutHold]) {
          uint32_t e[kCutHold], at[kCutHold];
#pragma unroll
          for (int u = 0; u < kCutHold; ++u) e[u] = r * kCutParts + cut_part(v[u], cut);
          f(v, on, e, at);
        });
      }
    };
    share([&](const u64 (&)[kCutHold], bool (&on)[kCutHold], const uint32_t (&e)[kCutHold], uint32_t (&at)[kCutHold]) { add_all(table, on, e, at); });
    __syncthreads();
    for (uint32_t i = tid; i < n * kCutParts; i += kPlanThreads) table[i] = table[i] ? atomicAdd(totals + i, table[i]) : 0u;
    block_done(turns);
    if (!block_waits(turns, ++turn * blocks, status)) return false;
    if (warp < (int)n) {  // a warp per range, a lane for 16 parts
      uint32_t v[16], sum = 0;
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const uint4 w = __ldcg(reinterpret_cast<const uint4*>(totals + warp * kCutParts + lane * 16 + i));
        v[i] = w.x;
        v[i + 1] = w.y;
        v[i + 2] = w.z;
        v[i + 3] = w.w;
        sum += w.x + w.y + w.z + w.w;
      }
      uint32_t at = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(kFull, at, off);
        if (lane >= off) at += o;
      }
      at += C.start[warp] - sum;
      uint32_t found = 0;
      uint32_t* starts = cut_starts(ws, L, c, cut) + warp * kCutParts + lane * 16;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint32_t part = lane * 16 + i;
        const bool again = v[i] > kRankItems && at < limit && cut + 1 < kCuts;
        const unsigned all = __ballot_sync(kFull, again);
        const uint32_t k = found + __popc(all & ((1u << lane) - 1u));
        if (again && k < kCutRanges) {
          s_found[warp][k][0] = part;
          s_found[warp][k][1] = at;
          s_found[warp][k][2] = v[i];
        }
        found += __popc(all);
        uint32_t* mine = table + warp * kCutParts + part;
        *mine = at < limit ? *mine + at : 0x80000000u;  // not moved where it is never sent
        if (q == 0) starts[i] = at;
        at += v[i];
      }
      if (lane == 0) s_n[warp] = min(found, kCutRanges);
    }
    __syncthreads();
    if (tid == 0 && cut + 1 < kCuts) {
      Cut& next = cuts[cut + 1];
      uint32_t m = 0;
      bool whole = true;  // a range is one part
      for (uint32_t r = 0; r < n; ++r) {
        whole = whole && s_n[r] == 1 && s_found[r][0][2] == C.size[r] && m < kCutRanges;
        for (uint32_t k = 0; k < s_n[r] && m < kCutRanges; ++k, ++m) {
          next.prefix[m] = C.prefix[r] << 9 | s_found[r][k][0];
          next.start[m] = s_found[r][k][1];
          next.size[m] = s_found[r][k][2];
          next.part[m] = r * kCutParts + s_found[r][k][0];
        }
      }
      next.n = m;
      next.in_a = whole ? C.in_a : !C.in_a;
    }
    __syncthreads();
    if (cut + 1 < kCuts && cuts[cut + 1].in_a == C.in_a) continue;  // they stay where they are
    share([&](const u64 (&v)[kCutHold], bool (&on)[kCutHold], const uint32_t (&e)[kCutHold], uint32_t (&at)[kCutHold]) {
#pragma unroll
      for (int u = 0; u < kCutHold; ++u) on[u] = on[u] && table[e[u]] < 0x80000000u;
      add_all(table, on, e, at);
#pragma unroll
      for (int u = 0; u < kCutHold; ++u)
        if (on[u]) dst[at[u]] = v[u];
    });
    block_done(turns);
    if (!block_waits(turns, ++turn * blocks, status)) return false;
  }
  return true;
}

// The parts whose candidates begin with the ranks [first, end), as many of a range as a block holds at a time; by the whole block
__device__ __noinline__ void rank_parts(RankShared& s, const Cut* cuts, unsigned char* ws, const EncLayout& L, uint32_t c, uint32_t keytop,
                                        u64* buf_a, u64* buf_b, uint32_t first, uint32_t end) {
  __shared__ uint32_t s_start[kCutParts + 1];
  const uint32_t tid = threadIdx.x;
  for (uint32_t cut = 0; cut < kCuts && cuts[cut].n; ++cut) {
    const Cut& C = cuts[cut];
    const u64* src = C.in_a ? buf_b : buf_a;
    for (uint32_t r = 0; r < C.n; ++r) {
      if (C.start[r] >= end || C.start[r] + C.size[r] <= first) continue;
      __syncthreads();
      s_start[tid] = __ldcg(cut_starts(ws, L, c, cut) + r * kCutParts + tid);
      if (tid == 0) s_start[kCutParts] = C.start[r] + C.size[r];
      __syncthreads();
      uint32_t i = __syncthreads_count(s_start[tid] < first);
      while (i < kCutParts && s_start[i] < end) {
        uint32_t stop = cut == 2 && i < kCutParts / 2 ? kCutParts / 2 : kCutParts;  // (one key at a time)
        if (cut + 1 < kCuts)  // those that have been cut again lie between
          for (uint32_t k = 0; k < cuts[cut + 1].n; ++k) {
            const uint32_t part = cuts[cut + 1].part[k] - r * kCutParts;
            if (part >= i && part < stop) stop = part;
          }
        if (stop == i) {
          ++i;
          continue;
        }
        const uint32_t at = s_start[i];
        const uint32_t fit = __syncthreads_count(tid >= i && tid < stop && s_start[tid] < end && s_start[tid + 1] - at <= kRankItems);
        const uint32_t behind = i + fit, m = s_start[behind] - at;  // one at least: what does not fit has been cut again
        const uint32_t inv = cut_inv(C, cut, r, i, keytop), inv_end = cut_inv(C, cut, r, behind, keytop);
        if (m && cut == 2) {
          rank_cell<kPlanThreads>(s, src + at, m, buf_a + at);
        } else if (m) {
          rank_and_leave<kPlanThreads>(s, src + at, m, inv, inv_end - inv - 1, keytop, ws, L, c, at);
        }
        i = behind;
      }
    }
  }
}

// first: the call's first kernel (one client): it clears the headers
template <int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kPlanThreads, 1)
k_client(const __grid_constant__ BatchDesc<kMediumBatch> batch, const __grid_constant__ Shape shape, uint32_t rows, int first, unsigned char* ws,
         const __grid_constant__ EncFront enc) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ClusterShared& S = *reinterpret_cast<ClusterShared*>(smem_raw);
  unsigned char* rest = smem_raw + sizeof(ClusterShared);
  float4* data = reinterpret_cast<float4*>(rest);
  __shared__ int s_bin[2];
  __shared__ Cut s_cut[kCuts];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t c = blockIdx.x / CL, q = blockIdx.x % CL, n = batch.n;
  for (int i = tid; i < CVLC_HIST_BINS; i += kPlanThreads) S.own[i] = 0;
  __syncthreads();
  pdl_enter();
  const ClientDesc& cd = batch.c[c];
  if (q == 0) {
    if (tid == 0) reinterpret_cast<ClientDesc*>(ws + plan_off_desc(n))[c] = cd;
    if (first) {
      if (tid < 64) reinterpret_cast<uint32_t*>(ws)[tid] = 0;
      else if (tid < 128) reinterpret_cast<uint32_t*>(enc.ws)[tid - 64] = 0;
    }
    if (tid == 128) reinterpret_cast<uint32_t*>(ws + plan_off_flags(n))[c] = 0;
  }
  // ---- the block's rows: kept, counted, their maxima written
  const float* __restrict__ x = cd.x;
  const float4* xv = reinterpret_cast<const float4*>(x);
  const uint32_t nvec = (uint32_t)(shape.d >> 2), slice = (rows + CL - 2) / (CL - 1) * kRowUnits;
  const uint32_t u0 = min(q * slice, nvec), units = q < CL - 1 ? min(u0 + slice, nvec) - u0 : 0u;
  uint16_t* __restrict__ row_max = reinterpret_cast<uint16_t*>(ws + plan_off_row_max(n)) + (size_t)c * rows;
  uint32_t top = 0, tail = 0, zeros = 0;
  const bool has_tail = q == CL - 2 && tid < (int)(shape.d & 3);
  if (has_tail) tail = __float_as_uint(x[4 * (size_t)nvec + tid]);
  constexpr int kLoads = 8;
  for (uint32_t i0 = 0; i0 < units; i0 += kLoads * kPlanThreads) {
    float4 a[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u)
      if (i0 + u * kPlanThreads + tid < units) a[u] = __ldg(xv + u0 + i0 + u * kPlanThreads + tid);
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const uint32_t i = i0 + u * kPlanThreads + tid;
      if (i0 + u * kPlanThreads < units) {
        const bool on = i < units;
        uint32_t m = 0;
        if (on) {
          if (i < kClusterUnits) data[i] = a[u];
          m = largest_key(a[u]);
          if (m == 0) zeros += 4;  // a counter takes one addition a cycle
          else hist_add4(S.own, a[u]);
        }
        top = max(top, m);
        m = max(m, __shfl_xor_sync(kFull, m, 1));
        m = max(m, __shfl_xor_sync(kFull, m, 2));
        if (lane % kRowUnits == 0 && on) row_max[(u0 + i) / kRowUnits] = (uint16_t)(m >> 19);
      }
    }
  }
  zeros = __reduce_add_sync(kFull, zeros);
  if (lane == 0 && zeros) atomicAdd(S.own, zeros);
  if (has_tail) {
    top = max(top, tail & 0x7FFFFFFFu);
    atomicAdd(S.own + ((tail & 0x7FFFFFFFu) >> 19), 1u);
  }
  cluster.sync();
  // ---- the client's counts, and those of the blocks before each, a share of the bins by every block
  uint32_t* flag = reinterpret_cast<uint32_t*>(ws + plan_off_flags(n)) + c;
  if (top >= 0x7F800000u) atomicOr(flag, 1u);  // a key of exponent 255: Inf or NaN
  for (uint32_t b = q * kPlanThreads + tid; b < CVLC_HIST_BINS; b += CL * kPlanThreads) {
    uint32_t v[CL], run = 0;
#pragma unroll
    for (int r = 0; r < CL; ++r) v[r] = cluster.map_shared_rank(S.own, r)[b];
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      cluster.map_shared_rank(S.place, r)[b] = run;
      run += v[r];
    }
#pragma unroll
    for (int r = 0; r < CL; ++r) cluster.map_shared_rank(S.total, r)[b] = run;
    (reinterpret_cast<unsigned long long*>(ws + kPlanWsHist) + (size_t)c * CVLC_HIST_BINS)[b] = run;
  }
  cluster.sync();
  const uint32_t nonfinite = __ldcg(flag);
  uint32_t* N = S.own;
  {
    uint32_t h[kPlanBins];
#pragma unroll
    for (int i = 0; i < kPlanBins; i += 4) {
      const uint4 v = reinterpret_cast<const uint4*>(S.total)[(kPlanBins * tid + i) / 4];
      h[i] = v.x;
      h[i + 1] = v.y;
      h[i + 2] = v.z;
      h[i + 3] = v.w;
    }
    survival_of(h, N);
  }
  const Threshold t = client_threshold(N, shape, cd.cap0, q == 0 ? cd.plan : nullptr,
                                       q == 0 ? reinterpret_cast<uint32_t*>(ws + plan_off_bin_start(n)) + (size_t)c * CVLC_HIST_BINS : nullptr);
  if (q == 0 && tid == 0) write_client(c, n, cd.plan, t, nonfinite, shape, ws, enc);
  const EncLayout& L = enc.L;
  const bool go = !nonfinite && t.n <= L.capacity, crowded = t.fullest > kRankHold;
  const uint32_t limit = shape.R * cd.cap0;  // ranks from here on are not sent (see by_clusters)
  unsigned long long* by_bin = reinterpret_cast<unsigned long long*>(enc.ws + L.off_buf_b) + (size_t)c * L.capacity;
  // ---- the candidates to their bins
  if (go && q < CL - 1) {
    for (uint32_t b = t.bin + tid; b <= t.top; b += kPlanThreads) S.place[b] += N[b + 1];
    __syncthreads();
    const uint32_t thresh = t.bin << 19;
    auto put = [&](uint32_t b, uint32_t index) {
      const uint32_t key = b & 0x7FFFFFFFu;
      if (key >= thresh) by_bin[atomicAdd(S.place + (key >> 19), 1u)] = ((unsigned long long)key << 32) | (unsigned long long)((b & 0x80000000u) | index);
    };
    auto put4 = [&](const float4 a, uint32_t at) {  // (by value: one load, ahead of the additions)
      put(__float_as_uint(a.x), at);
      put(__float_as_uint(a.y), at + 1);
      put(__float_as_uint(a.z), at + 2);
      put(__float_as_uint(a.w), at + 3);
    };
    const uint32_t kept = min(units, kClusterUnits);
    if (crowded) {
      put_crowded(S.place, t.bin, data, kept, u0, by_bin);
      put_crowded(S.place, t.bin, xv + u0 + kept, units - kept, u0 + kept, by_bin);
      for (uint32_t i = q * kPlanThreads + tid; i < kCuts * kCutTable; i += (CL - 1) * kPlanThreads) cut_totals(enc.ws, L, c, i / kCutTable)[i % kCutTable] = 0;
      if (q == 0 && tid == 0) *cut_turns(enc.ws, L, c) = 0;
    } else {
      float4 over[kClusterOver];  // on their way while the others go
#pragma unroll
      for (uint32_t u = 0; u < kClusterOver; ++u)
        if (kept + u * kPlanThreads + tid < units) over[u] = __ldg(xv + u0 + kept + u * kPlanThreads + tid);
#pragma unroll 4
      for (uint32_t i = tid; i < kept; i += kPlanThreads) put4(data[i], 4 * (u0 + i));
#pragma unroll
      for (uint32_t u = 0; u < kClusterOver; ++u)
        if (kept + u * kPlanThreads + tid < units) put4(over[u], 4 * (u0 + kept + u * kPlanThreads + tid));
    }
    if (has_tail) put(tail, 4 * nvec + tid);
  }
  cg::cluster_group::arrival_token token = cluster.barrier_arrive();
  if (q == CL - 1) {
    const Batch all{reinterpret_cast<const ClientDesc*>(ws + plan_off_desc(n)), n};
    tune_client(c, all, shape, ws, nullptr, N, rest);
    cluster.barrier_wait(std::move(token));
    return;
  }
  // ---- the bins whose candidates begin in the block's share of the ranks
  const uint32_t ranked = min(t.n, limit);
  const uint32_t share = (ranked + CL - 2) / (CL - 1);
  if (tid < 2) s_bin[tid] = (int)t.bin - 1;
  __syncthreads();
  for (uint32_t b = t.bin + tid; b <= t.top; b += kPlanThreads) {
#pragma unroll
    for (int end = 0; end < 2; ++end) {
      const uint32_t first = (q + end) * share;
      if (N[b + 1] >= first && (b == t.top || N[b + 2] < first)) s_bin[end] = (int)b;
    }
  }
  __syncthreads();
  const int last = s_bin[1];
  cluster.barrier_wait(std::move(token));
  if (!go) return;
  unsigned long long* out = reinterpret_cast<unsigned long long*>(enc.ws + L.off_buf_a) + (size_t)c * L.capacity;
  if (crowded && !cut_bins(S.total, N, s_cut, t, limit, enc.ws, L, c, q, CL - 1, out, by_bin)) return;
  const uint32_t keytop = sort_keytop(t.top);
  for (int hi = s_bin[0]; hi > last;) {  // bins (lo, hi], as many as a block holds
    const uint32_t at = N[hi + 1];
    if (at >= ranked) break;
    int lo = last;
    if (N[last + 1] - at > kRankItems) {  // not all of them; hundreds may be empty (98 % zeros: 30 us one after the other)
      int below = last;
      lo = hi - 1;
      while (lo - below > 1) {
        const int mid = (lo + below) >> 1;
        if (N[mid + 1] - at <= kRankItems) lo = mid;
        else below = mid;
      }
    }
    const uint32_t m = N[lo + 1] - at;
    const u64 inv = (u64)((int)t.top - hi) << 19, end = (u64)((int)t.top - lo) << 19;
    if (m && m <= kRankHold)  // else it is one bin, which has been cut
      rank_and_leave<kPlanThreads>(*reinterpret_cast<RankShared*>(rest), by_bin + at, m, (uint32_t)inv, (uint32_t)(end - inv - 1), keytop, enc.ws, L, c, at);
    hi = lo;
  }
  if (crowded)
    rank_parts(*reinterpret_cast<RankShared*>(rest), s_cut, enc.ws, L, c, keytop, out, by_bin, q * share,
               min((q + 1) * share, ranked));
}

// ===================================================================================
// launchers
// ===================================================================================

static cudaError_t plan_attributes() {
  static OncePerDevice once;
  return once_per_device(once, [] {
    cudaError_t e = allow_shared(k_hist, kHistSub * CVLC_HIST_BINS * 4);
    if (e == cudaSuccess) e = allow_shared(k_plan_fit, kFitSmem);
    if (e == cudaSuccess) e = allow_shared(k_client<8>, kClusterSmem);
    if (e == cudaSuccess) e = allow_shared(k_client<16>, kClusterSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_client<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e != cudaSuccess ? e : allow_shared(k_plan_tune, kTuneSmem);
  });
}

// the start of a planning call: the descriptors into the workspace, `bytes` from its start and `more` from `at` on zeroed
// (multiples of 256 bytes)
template <int CAP>
static void launch_zero_t(const ClientDesc* clients, uint32_t n, unsigned char* w, size_t bytes, unsigned char* at, size_t more,
                          cudaStream_t st) {
  BatchDesc<CAP> batch;
  batch.n = n;
  batch.pad = 0;
  memcpy(batch.c, clients, (size_t)n * sizeof(ClientDesc));
  const size_t want = (bytes + more) / 16 / 256 + 1;
  const unsigned grid = (unsigned)(want < (size_t)(4 * kNumSM) ? want : 4 * kNumSM);
  launch_kernel(kKZeroWords, k_zero_words<CAP>, grid, 256, 0, st, false, batch, reinterpret_cast<ClientDesc*>(w + plan_off_desc(n)),
                reinterpret_cast<uint4*>(w), bytes / 16, reinterpret_cast<uint4*>(at), more / 16);
}
static Batch launch_zero(const ClientDesc* clients, uint32_t n, unsigned char* w, size_t bytes, unsigned char* at, size_t more, cudaStream_t st) {
  if (n <= (uint32_t)kSmallBatch) launch_zero_t<kSmallBatch>(clients, n, w, bytes, at, more, st);
  else if (n <= (uint32_t)kMediumBatch) launch_zero_t<kMediumBatch>(clients, n, w, bytes, at, more, st);
  else launch_zero_t<kLargeBatch>(clients, n, w, bytes, at, more, st);
  return Batch{reinterpret_cast<const ClientDesc*>(w + plan_off_desc(n)), n};
}

// Whether every client has an SM for its tuning and then fits and tunes for itself, or one tunes for all that share a key
static bool own_tuning(uint32_t n, TunePlace place) { return n <= (place == kTuneAlone ? (uint32_t)kNumSM : kTuneRoom); }

static void launch_fit(const Batch& batch, const Shape& shape, unsigned char* w, const EncFront& enc, FitThreshold threshold, cudaStream_t st, bool overlap) {
  launch_kernel(kKPlanFit, k_plan_fit, batch.n, kPlanThreads, kFitSmem, st, overlap, reinterpret_cast<const unsigned long long*>(w + kPlanWsHist),
                reinterpret_cast<const uint32_t*>(w + plan_off_flags(batch.n)), batch, shape, w, enc, threshold);
}

// histogram of every client
static cudaError_t launch_hist(const ClientDesc* clients, uint32_t n, const Shape& shape, unsigned char* w, const Partition& part, const EncFront& enc,
                               bool finish, Batch* batch, cudaStream_t st) {
  const cudaError_t e = plan_attributes();
  if (e != cudaSuccess) return e;
  // header, histograms, flags, counters and tuning keys start at zero (and so does the encoder's workspace up to what its selection
  // writes in full); the rest is written in full by the kernels that follow
  *batch = launch_zero(clients, n, w, plan_off_desc(n), enc.ws, enc.ws ? enc.L.off_sub_start : 0, st);
  // the resident blocks share the concatenated updates evenly
  launch_kernel(kKHist, k_hist, part.grid, kHistThreads, kHistSub * CVLC_HIST_BINS * 4, st, true, *batch, shape, part, w, enc, finish ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_plan_front(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, const EncFront& enc, TunePlace place, cudaStream_t st) {
  unsigned char* w = static_cast<unsigned char*>(ws);
  const Partition part = make_partition(shape.d, n);
  Batch batch;
  const cudaError_t e = launch_hist(clients, n, shape, w, part, enc, true, &batch, st);
  if (e != cudaSuccess) return e;
  if (place != kTuneBehind && !own_tuning(n, place))
    launch_fit(batch, shape, w, enc, part.per_client ? kThresholdThere : kThresholdFinish, st, true);
  else if (!part.per_client)
    launch_kernel(kKPlanThreshold, k_plan_threshold, n, kPlanThreads, 0, st, true, batch, shape, w, enc);
  return cudaGetLastError();
}

// Asked once per device.  The shared memory of a block has to be allowed before.
bool clusters_run(uint32_t blocks) {
  static std::atomic<int> known[64][2];  // 1: they do, 2: they don't
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || plan_attributes() != cudaSuccess) return false;
  std::atomic<int>& answer = known[dev][blocks == 16];
  if (answer.load(std::memory_order_acquire) == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks;
    cfg.blockDim = kPlanThreads;
    cfg.dynamicSmemBytes = kClusterSmem;
    int n = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, blocks == 16 ? k_client<16> : k_client<8>, &cfg);
    if (e != cudaSuccess) (void)cudaGetLastError();  // it is no launch's
    answer.store(e == cudaSuccess && n > 0 ? 1 : 2, std::memory_order_release);
  }
  return answer.load(std::memory_order_acquire) == 1;
}

cudaError_t launch_clients(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, const EncFront& enc, cudaStream_t st) {
  unsigned char* w = static_cast<unsigned char*>(ws);
  const cudaError_t e = plan_attributes();
  if (e != cudaSuccess) return e;
  BatchDesc<kMediumBatch> batch;
  batch.n = n;
  batch.pad = 0;
  memcpy(batch.c, clients, (size_t)n * sizeof(ClientDesc));
  const uint32_t rows = (uint32_t)make_partition(shape.d, n).rows;
  if (n > 1) launch_zero(clients, n, w, 256, enc.ws, 256, st);
  const uint32_t blocks = cluster_blocks(rows, n);
  launch_kernel(kKClient, blocks == 16 ? k_client<16> : k_client<8>, blocks * n, kPlanThreads, kClusterSmem, st, n > 1, batch, shape, rows, n > 1 ? 0 : 1, w, enc);
  return cudaGetLastError();
}

cudaError_t launch_plan_back(uint32_t n, const Shape& shape, void* ws, TunePlace place, cudaStream_t st, bool overlap) {
  unsigned char* w = static_cast<unsigned char*>(ws);
  const Batch batch{reinterpret_cast<const ClientDesc*>(w + plan_off_desc(n)), n};
  const bool own = own_tuning(n, place);
  if (place == kTuneBehind && !own) {
    launch_fit(batch, shape, w, EncFront{}, kThresholdThere, st, overlap);
    overlap = true;
  }
  launch_kernel(kKPlanTune, k_plan_tune, n, kTuneThreads, kTuneSmem, st, overlap, batch, shape, w,
                own ? reinterpret_cast<const unsigned long long*>(w + kPlanWsHist) : nullptr);
  return cudaGetLastError();
}

cudaError_t launch_plan(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, cudaStream_t st) {
  const cudaError_t e = launch_plan_front(clients, n, shape, ws, EncFront{}, kTuneAlone, st);
  return e != cudaSuccess ? e : launch_plan_back(n, shape, ws, kTuneAlone, st, true);
}

// The histograms alone: what a client sends when the parameter server plans for it.  The workspace header stays unmarked, so an
// encode call cannot take it for one that holds a plan's tables.
cudaError_t launch_histogram(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws,
                             unsigned long long* hist_out, cudaStream_t st) {
  unsigned char* w = static_cast<unsigned char*>(ws);
  Batch batch;
  const cudaError_t e = launch_hist(clients, n, shape, w, make_partition(shape.d, n), EncFront{}, false, &batch, st);
  return e != cudaSuccess ? e : cudaMemcpyAsync(hist_out, w + kPlanWsHist, (size_t)n * CVLC_HIST_BINS * 8, cudaMemcpyDeviceToDevice, st);
}

// Checks histograms that come from outside: flag bit 0 = a value of exponent 255 (Inf, NaN),
// bit 1 = the counts do not add up to d.
__global__ void __launch_bounds__(256)
k_hist_check(const unsigned long long* __restrict__ hist_all, uint64_t d, uint32_t* __restrict__ flags) {
  __shared__ unsigned long long s_sum[8];
  __shared__ uint32_t s_nonfinite;
  pdl_enter();
  const unsigned long long* hist = hist_all + (size_t)blockIdx.x * CVLC_HIST_BINS;
  if (threadIdx.x == 0) s_nonfinite = 0;
  __syncthreads();
  unsigned long long sum = 0;
  for (int j = threadIdx.x; j < CVLC_HIST_BINS; j += 256) {
    const unsigned long long h = hist[j];
    sum += h;
    if (j >= (int)(0x7F800000u >> 19) && h != 0) s_nonfinite = 1u;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    for (int w = 0; w < 8; ++w) tot += s_sum[w];
    flags[blockIdx.x] = s_nonfinite | ((tot != d) ? 2u : 0u);
  }
}

cudaError_t launch_plan_from_hist(const ClientDesc* clients, uint32_t n, const Shape& shape,
                                  const unsigned long long* hist, void* ws, cudaStream_t st) {
  const cudaError_t e = plan_attributes();
  if (e != cudaSuccess) return e;
  unsigned char* w = static_cast<unsigned char*>(ws);
  uint32_t* flags = reinterpret_cast<uint32_t*>(w + plan_off_flags(n));
  // status word, header and tuning keys start at zero: the header stays unmarked, so an encode call cannot take this
  // workspace for one that holds the rows' maxima
  const Batch batch = launch_zero(clients, n, w, kPlanWsHist, w + plan_off_keys(n), plan_off_desc(n) - plan_off_keys(n), st);
  launch_kernel(kKHistCheck, k_hist_check, n, 256, 0, st, true, hist, shape.d, flags);
  launch_kernel(kKPlanFit, k_plan_fit, n, kPlanThreads, kFitSmem, st, true, hist, flags, batch, shape, w, EncFront{}, kThresholdOutside);
  launch_kernel(kKPlanTune, k_plan_tune, n, kTuneThreads, kTuneSmem, st, true, batch, shape, w, static_cast<const unsigned long long*>(nullptr));
  return cudaGetLastError();
}

// ===================================================================================
// Problem P2 with real-valued packet sizes (Section IV-C; Algorithm 1 steps 2-14 with the equidistant
// search over k of Section IV-D): a plan only, for comparing its error bound with the integer-length rule
// ===================================================================================
// One warp per value of k.  For that k the packets start equal and are re-split two consecutive ones at a time,
// r = 2 .. R in order (each re-split sees the previous one: the sweep is sequential by definition); a re-split
// minimises Eq. (7), strongly convex in the split (Lemma 2), by bracketing: the 32 lanes evaluate 32 equidistant
// splits of the bracket, the bracket shrinks to the neighbours of the best one, eight times.  All arithmetic is
// binary64 with separately rounded operations in a fixed order, so the result does not depend on the machine.

struct LiteralArgs {
  double bH, s, B, P_min, P_max, tol, alpha_q;
  unsigned long long k_lo, k_hi, d;
  uint32_t R, n_k, max_sweeps, quantizer;
};

// the bracket of Eq. (5) for a packet of P records at the length the packet constraint leaves: y = (b - H) / P - s
__device__ __forceinline__ double literal_cost(double P, const LiteralArgs& a) {
  const double y = __dsub_rn(__ddiv_rn(a.bH, P), a.s);
  double Q;
  if (a.quantizer == CVLC_QUANT_QSGD) {
    const double sq = __dsub_rn(series_exp2(__dsub_rn(y, 1.0)), 1.0);
    const double Q1 = __ddiv_rn(P, __dmul_rn(sq, sq));
    const double Q2 = __ddiv_rn(__dsqrt_rn(P), sq);
    Q = (Q1 < Q2) ? Q1 : Q2;
  } else {
    const double L = __dsub_rn(series_exp2(y), 1.0);
    Q = __ddiv_rn(P, __dmul_rn(L, L));
  }
  const double one_m = __dsub_rn(1.0, __ddiv_rn(1.0, a.B));
  return __dadd_rn(__ddiv_rn(Q, __dmul_rn(a.B, a.B)), __dmul_rn(one_m, one_m));
}

__device__ __forceinline__ double literal_energy(double Z, double beta, double D) {
  return __ddiv_rn(__dsub_rn(series_powr(__dadd_rn(Z, 1.0), beta), 1.0), D);
}

// Eq. (7) as a function of p = P_r: X = P_{r-1} + P_r, Z0 = Z_{r-2}, Z2 = Z_r
__device__ __forceinline__ double literal_pair_f(double p, double X, double Z0, double Z2, const LiteralArgs& a, double beta, double D) {
  const double Em = literal_energy(__dadd_rn(Z0, __dsub_rn(X, p)), beta, D);
  const double hi_part = __dmul_rn(literal_cost(p, a), __dsub_rn(literal_energy(Z2, beta, D), Em));
  const double lo_part = __dmul_rn(literal_cost(__dsub_rn(X, p), a), __dsub_rn(Em, literal_energy(Z0, beta, D)));
  return __dadd_rn(hi_part, lo_part);
}

__global__ void __launch_bounds__(32)
k_plan_literal(const __grid_constant__ LiteralArgs a, unsigned long long* __restrict__ k_grid, double* __restrict__ gamma_of_k,
               uint32_t* __restrict__ sweeps_of_k, double* __restrict__ P_all) {
  extern __shared__ double lit_smem[];  // P[R], Z[R + 1]
  double* P = lit_smem;
  double* Z = lit_smem + a.R;
  const int lane = threadIdx.x;
  const uint32_t ik = blockIdx.x, R = a.R;
  const double beta = __dadd_rn(__dmul_rn(2.0, a.alpha_q), 1.0);
  const double D = __dsub_rn(series_powr((double)a.d, beta), 1.0);
  // equidistant values of k; the product stays below 2^64 (n_k <= 4096, k <= 2^31 * 2^31 is never reached: k <= d)
  const unsigned long long k = (a.n_k == 1) ? a.k_lo : a.k_lo + ((unsigned long long)ik * (a.k_hi - a.k_lo)) / (a.n_k - 1);
  const double P0 = __ddiv_rn((double)k, (double)R);
  for (uint32_t r = lane; r < R; r += 32) P[r] = P0;
  __syncwarp();
  uint32_t sweep = 0;
  for (; sweep < a.max_sweeps; ++sweep) {
    if (lane == 0) {
      double z = 0.0;
      Z[0] = 0.0;
      for (uint32_t r = 0; r < R; ++r) {
        z = __dadd_rn(z, P[r]);
        Z[r + 1] = z;
      }
    }
    __syncwarp();
    double moved = 0.0;
    for (uint32_t r = 1; r < R; ++r) {
      const double Pr = P[r];
      const double X = __dadd_rn(P[r - 1], Pr), Z0 = Z[r - 1], Z2 = Z[r + 1];
      double lo = __ddiv_rn(X, 2.0), hi = __dsub_rn(X, a.P_min);
      if (lo < a.P_min) lo = a.P_min;
      const double lo2 = __dsub_rn(X, a.P_max);
      if (lo < lo2) lo = lo2;
      if (hi > a.P_max) hi = a.P_max;
      if (!(lo < hi)) continue;
      double best_x = lo;
      for (int round = 0; round < 8; ++round) {
        const double step = __ddiv_rn(__dsub_rn(hi, lo), 31.0);
        const double xj = (lane == 31) ? hi : __dadd_rn(lo, __dmul_rn((double)lane, step));
        double f = literal_pair_f(xj, X, Z0, Z2, a, beta, D);
        int j = lane;
        // the first of the smallest values
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const double fo = __shfl_xor_sync(kFull, f, off);
          const int jo = __shfl_xor_sync(kFull, j, off);
          if (fo < f || (fo == f && jo < j)) {
            f = fo;
            j = jo;
          }
        }
        const double nlo = (j == 0) ? lo : __dadd_rn(lo, __dmul_rn((double)(j - 1), step));
        const double nhi = (j >= 30) ? hi : __dadd_rn(lo, __dmul_rn((double)(j + 1), step));
        best_x = (j == 31) ? hi : __dadd_rn(lo, __dmul_rn((double)j, step));
        lo = nlo;
        hi = nhi;
      }
      // lanes 0 and 1 evaluate the new and the current split
      const double fe = literal_pair_f(lane == 0 ? best_x : Pr, X, Z0, Z2, a, beta, D);
      const double f_new = __shfl_sync(kFull, fe, 0), f_old = __shfl_sync(kFull, fe, 1);
      if (f_new < f_old) {
        const double delta = fabs(__dsub_rn(best_x, Pr));
        if (delta > moved) moved = delta;
        if (lane == 0) {
          const double Pm = __dsub_rn(X, best_x);
          P[r - 1] = Pm;
          P[r] = best_x;
          Z[r] = __dadd_rn(Z0, Pm);
        }
      }
      __syncwarp();
    }
    if (!(moved > a.tol)) {
      ++sweep;
      break;
    }
  }
  // Eq. (5) at these packet sizes: the terms side by side, their sum in packet order
  if (lane == 0) {
    double z = 0.0;
    Z[0] = 0.0;
    for (uint32_t r = 0; r < R; ++r) {
      z = __dadd_rn(z, P[r]);
      Z[r + 1] = z;
    }
  }
  __syncwarp();
  double* P_out = P_all + (size_t)ik * R;
  double* term = P_out;  // the terms borrow the output slots; the packet sizes follow once the sum is taken
  for (uint32_t r = lane; r < R; r += 32) {
    const double Eprev = (r == 0) ? 0.0 : literal_energy(Z[r], beta, D);
    const double Ecur = literal_energy(Z[r + 1], beta, D);
    term[r] = __dmul_rn(literal_cost(P[r], a), __dsub_rn(Ecur, Eprev));
  }
  __syncwarp();
  if (lane == 0) {
    double gamma = __dsub_rn(1.0, literal_energy(Z[R], beta, D));
    for (uint32_t r = 0; r < R; ++r) gamma = __dadd_rn(gamma, term[r]);
    gamma_of_k[ik] = gamma;
    k_grid[ik] = k;
    sweeps_of_k[ik] = sweep;
  }
  __syncwarp();
  for (uint32_t r = lane; r < R; r += 32) P_out[r] = P[r];
}

// the value of k with the smallest error bound (the first one on ties) and its packet sizes
__global__ void __launch_bounds__(256)
k_plan_literal_pick(const __grid_constant__ LiteralArgs a, const unsigned long long* __restrict__ k_grid,
                    const double* __restrict__ gamma_of_k, const uint32_t* __restrict__ sweeps_of_k,
                    const double* __restrict__ P_all, cvlc_literal_plan_t* __restrict__ out, double* __restrict__ P_star) {
  __shared__ uint32_t s_best;
  if (threadIdx.x == 0) {
    uint32_t best = 0;
    for (uint32_t i = 1; i < a.n_k; ++i)
      if (gamma_of_k[i] < gamma_of_k[best]) best = i;
    s_best = best;
    out->status = CVLC_OK;
    out->R = a.R;
    out->n_k = a.n_k;
    out->sweeps = sweeps_of_k[best];
    out->k_star = k_grid[best];
    out->gamma_star = gamma_of_k[best];
    out->alpha_q = a.alpha_q;
    out->beta = __dadd_rn(__dmul_rn(2.0, a.alpha_q), 1.0);
  }
  __syncthreads();
  if (P_star)
    for (uint32_t r = threadIdx.x; r < a.R; r += 256) P_star[r] = P_all[(size_t)s_best * a.R + r];
}

cudaError_t launch_plan_literal(const cvlc_params& p, double alpha_q, uint32_t s, uint32_t R, uint32_t n_k, uint32_t max_sweeps,
                                unsigned long long k_lo, unsigned long long k_hi, double P_min, double P_max, double tol,
                                cvlc_literal_plan_t* out, double* P_star, void* ws, cudaStream_t st) {
  LiteralArgs a;
  a.bH = (double)(p.packet_bits - p.header_bits);
  a.s = (double)s;
  a.B = p.scale_B;
  a.P_min = P_min;
  a.P_max = P_max;
  a.tol = tol;
  a.alpha_q = alpha_q;
  a.k_lo = k_lo;
  a.k_hi = k_hi;
  a.d = p.d;
  a.R = R;
  a.n_k = n_k;
  a.max_sweeps = max_sweeps;
  a.quantizer = p.quantizer;
  unsigned char* w = static_cast<unsigned char*>(ws);
  unsigned long long* k_grid = reinterpret_cast<unsigned long long*>(w + literal_off_k(n_k));
  double* gamma_of_k = reinterpret_cast<double*>(w + literal_off_gamma(n_k));
  uint32_t* sweeps_of_k = reinterpret_cast<uint32_t*>(w + literal_off_sweeps(n_k));
  double* P_all = reinterpret_cast<double*>(w + literal_off_P(n_k));
  {
    LaunchScope ls(kKPlanLiteral, st);
    k_plan_literal<<<n_k, 32, (2 * (size_t)R + 1) * 8, st>>>(a, k_grid, gamma_of_k, sweeps_of_k, P_all);
  }
  {
    LaunchScope ls(kKPlanLiteral, st);
    k_plan_literal_pick<<<1, 256, 0, st>>>(a, k_grid, gamma_of_k, sweeps_of_k, P_all, out, P_star);
  }
  return cudaGetLastError();
}

// ---- diagnostics ---------------------------------------------------------------------

__global__ void k_selftest_philox(uint64_t seed, uint32_t client_id, uint32_t round, uint64_t first, uint64_t n, uint32_t* out) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t c = first + i;
    const uint4 r = philox4x32_10(make_uint4((uint32_t)c, (uint32_t)(c >> 32), client_id, round),
                                  make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    out[4 * i + 0] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
  }
}

__global__ void k_selftest_math(const double* in, uint64_t n, double* l2, double* e2, double* dv, double* dr) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const double v = in[i];
    if (l2) l2[i] = (v > 0.0) ? series_log2(v) : 0.0;
    if (e2) e2[i] = (fabs(v) <= 1000.0) ? series_exp2(v) : 0.0;
    if (dv && dr) {
      for (int j = 1; j <= 20; ++j) {
        dv[i * 20 + j - 1] = div_small_int(v, j);
        dr[i * 20 + j - 1] = __ddiv_rn(v, (double)j);
      }
    }
  }
}

cudaError_t launch_selftest_philox(uint64_t seed, uint32_t client_id, uint32_t round, uint64_t first, uint64_t n,
                                   uint32_t* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  { LaunchScope ls(kKSelftest, st); k_selftest_philox<<<kNumSM, 256, 0, st>>>(seed, client_id, round, first, n, out); }
  return cudaGetLastError();
}

cudaError_t launch_selftest_math(const double* in, uint64_t n, double* l2, double* e2, double* dv, double* dr,
                                 cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  { LaunchScope ls(kKSelftest, st); k_selftest_math<<<kNumSM, 256, 0, st>>>(in, n, l2, e2, dv, dr); }
  return cudaGetLastError();
}

}  // namespace cvlc
