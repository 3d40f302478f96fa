// Internal declarations shared by the libcvlc translation units (sm_100a).
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <atomic>

#include "../../include/cvlc.h"

namespace cvlc {

constexpr int kNumSM = 148;  // B200: grids are sized in multiples of this

#ifdef __CUDACC__
#define CVLC_HD __host__ __device__
#else
#define CVLC_HD
#endif

CVLC_HD constexpr size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// ---- a batch of clients -------------------------------------------------------------
// Every kernel of the plan / encode path works on a batch of clients that share the problem
// shape (d, budget, packet and header size, candidate lengths) and differ in their update,
// scale and Philox identifiers.  The per-client descriptors travel as a kernel parameter of
// the first kernel of a call (no host-to-device copy), which leaves them in the workspace for
// the others: a launch with 24 KB of parameters costs the host about 3 us more than one without.
// That first kernel is instantiated for three descriptor capacities, and so is the packing kernel, which keeps the
// descriptors as a parameter: read from there, a client's Philox keys stay in uniform registers (530 us instead of 560
// for 100 ResNet-18-sized clients).

struct ClientDesc {
  const float* x;      // the update, d fp32
  cvlc_plan_t* plan;   // written by the plan kernels, read by the encode kernels
  uint8_t* stream;     // encode output (unused while planning)
  uint64_t seed;       // Philox key
  double scale_B;      // B of the scaling operation
  uint32_t client_id;  // Philox counter word 2
  uint32_t round;      // Philox counter word 3
  uint32_t cap0;       // planning: records of a packet at the shortest candidate length
  uint32_t pad;
};

constexpr int kSmallBatch = 4;
constexpr int kMediumBatch = 40;
constexpr int kLargeBatch = CVLC_MAX_BATCH;

template <int CAP>
struct BatchDesc {
  uint32_t n;
  uint32_t pad;
  ClientDesc c[CAP];
};
// the descriptors as the other kernels see them: in the workspace
struct Batch {
  const ClientDesc* c;
  uint32_t n;
};

struct Shape {
  uint64_t d;
  uint32_t s, R;
  uint32_t packet_bits, header_bits, quantizer, max_code_bits;
  uint32_t fixed_y;  // 0 = tune the lengths; otherwise every packet at this length
  uint32_t pad;
  uint32_t cap[CVLC_MAX_CODE_BITS + 1];  // records per packet per code length
};

constexpr unsigned kFull = 0xFFFFFFFFu;  // all lanes of a warp

// ---- workspace layouts (byte offsets; every region 256-byte aligned) ----------

// The float4 units of an update are grouped into rows of kRowUnits (16 coordinates, 64 bytes: what a DRAM access moves).  The
// histogram kernel streams the clients' rows as one concatenated array cut into equal contiguous chunks and leaves the bin of
// every row's largest key; the selection reads only the rows that hold a candidate (a bin at or above the threshold's).  With
// rows of 64 coordinates most of a spread-out update was read again (83 % at 3 % candidates, now 42 %).  The ragged tail of an
// update (d % 4 coordinates) goes with its last row.
constexpr int kStreamThreads = 512;
constexpr int kRowUnits = 4;
struct Partition {
  uint64_t rows;      // per client, rounded up to a multiple of 16 (the last ones may be empty)
  uint64_t total;     // rows * n
  uint64_t chunk;     // rows per chunk of the histogram kernel
  uint32_t n_chunks;
  uint32_t grid;      // its blocks
  uint32_t per_client;  // chunks of a client where they are cut from each client on its own; 0: from the concatenated rows
};
CVLC_HD inline Partition make_partition(uint64_t d, uint32_t n) {
  Partition P;
  P.rows = (((d >> 2) + kRowUnits - 1) / kRowUnits + 15) & ~(uint64_t)15;
  if (P.rows == 0) P.rows = 16;
  P.total = P.rows * n;
  // Three blocks per SM finish a small batch sooner (20 clients of 1.2 M coordinates: 26.6 instead of 28.2 us, 10 of 3 M 30.1 and 32.9, 10
  // of 8 M 65.7 and 68.9); at 100 M coordinates the two are even, and a large one streams faster with two, which also leave the
  // selection behind them more to find in the L2 (whole calls: 150 M 251 and 247 us, 280 M 421 and 394, 600 M 775 and 739).
  const uint64_t most = P.total <= (8u << 20) ? 3 * kNumSM : 2 * kNumSM;
  uint64_t grid = (P.total + 255) / 256;
  if (grid > most) grid = most;
  P.grid = (uint32_t)grid;
  P.per_client = 0;
  const uint64_t of_client = grid / n;
  if (P.total <= (8u << 20) && of_client * n * 16 >= grid * 15) {
    // a chunk then has one client: one merge per block, and the clients are finished by as many blocks (see finish_client)
    P.chunk = ((P.rows + of_client - 1) / of_client + 15) & ~(uint64_t)15;
    P.per_client = (uint32_t)((P.rows + P.chunk - 1) / P.chunk);
    P.n_chunks = P.grid = P.per_client * n;
    return P;
  }
  // two chunks per block where that leaves each a megabyte and more: every chunk ends with a merge into a client's histogram
  // (with two of 64 KB and more 10 clients of 5 M coordinates take 53 us)
  const uint64_t n_chunks = P.total / (2 * grid) >= 16384 ? 2 * grid : grid;
  P.chunk = ((P.total + n_chunks - 1) / n_chunks + 15) & ~(uint64_t)15;
  P.n_chunks = (uint32_t)((P.total + P.chunk - 1) / P.chunk);
  return P;
}

// plan workspace:
//   [0] PlanWsHeader | [256] uint64 hist[n][4096] | uint32 nonfinite[n] | uint32 rows_done[n] | uint64 tune_key[n][2]
//   | ClientDesc[n] | uint32 bin_start[n][4096] | uint32 max_bin[n] | uint16 row_max[n][rows]
// rows_done: rows in the client's histogram, where the block that completes it works out the threshold and the bins' starts.
// bin_start: candidates of the client in the bins above this one; max_bin: candidates in its fullest bin.
// tune_key = (bits of alpha_q, bits of scale_B): clients of a batch with equal keys have the same code lengths; in a large batch
// the first of them runs the length tuning and writes the result to all.
struct PlanWsHeader {
  int32_t status;   // byte 0
  uint32_t n;       // clients of the batch the workspace was filled for
  uint64_t d;
  uint32_t pad;
  uint32_t magic;   // set when the bins' tables and the rows' maxima are valid
};
constexpr uint32_t kPlanWsMagic = 0x53454743u;
constexpr size_t kPlanWsHist = 256;
CVLC_HD constexpr size_t plan_off_flags(uint32_t n) { return kPlanWsHist + (size_t)n * CVLC_HIST_BINS * 8; }
CVLC_HD constexpr size_t plan_off_rows_done(uint32_t n) { return plan_off_flags(n) + (size_t)n * 4; }
CVLC_HD constexpr size_t plan_off_keys(uint32_t n) { return align256(plan_off_rows_done(n) + (size_t)n * 4); }
CVLC_HD constexpr size_t plan_off_desc(uint32_t n) { return align256(plan_off_keys(n) + (size_t)n * 16); }
CVLC_HD constexpr size_t plan_off_bin_start(uint32_t n) { return align256(plan_off_desc(n) + (size_t)n * sizeof(ClientDesc)); }
CVLC_HD constexpr size_t plan_off_max_bin(uint32_t n) { return align256(plan_off_bin_start(n) + (size_t)n * CVLC_HIST_BINS * 4); }
CVLC_HD constexpr size_t plan_off_row_max(uint32_t n) { return align256(plan_off_max_bin(n) + (size_t)n * 4); }
CVLC_HD inline size_t plan_ws_bytes(const Partition& P, uint32_t n) { return align256(plan_off_row_max(n) + (size_t)P.total * 2); }

// One round of splitting large buckets (see rank_big): counters of its lists and of what has been taken and finished
constexpr int kBigRounds = 3;
struct BigRound {
  uint32_t n, pieces, slots;                        // buckets, pieces of them, their candidates in units of kBigSlot
  uint32_t next_sample, next_count, next_place;     // taken
  uint32_t done_sample, done_bounds, done_place;    // finished
};

// encode workspace header (first 256 bytes), written at the start of a call
struct EncHeader {
  int32_t status;           // byte 0
  uint32_t limit;           // ranks from here on are never sent
  uint32_t select_ticket;   // tile tickets of the look-back selection
  uint32_t split_ticket, rank_ticket;  // tile tickets of the partition and of the final ranking
  uint32_t most;            // candidates of the largest client, as far as they are ranked
  uint32_t most_split;      // candidates of the largest client that needs the partition
  uint32_t list_n[2], list_next[2];  // entries of the ranking's lists (of cells for a warp and for a block) and of them taken
  BigRound big[kBigRounds];
  uint32_t own_n, own_next, own_done;  // large buckets that a block splits by itself, of them taken, finished
  uint32_t part_n, part_next;  // parts of large buckets to rank, and of them taken
  uint32_t sort_ticket[4];  // tile tickets of the digit passes
  uint32_t max_sort_tiles;  // largest per-client tile count of this batch
};
static_assert(sizeof(EncHeader) <= 256, "the header's place");

constexpr int kSelectThreads = 512;
constexpr int kSelectVecPerThread = 4;  // float4 loads per thread per tile of the look-back selection
constexpr int kSelectTile = kSelectThreads * kSelectVecPerThread * 4;  // 8192 coordinates
CVLC_HD constexpr uint64_t select_tiles_of(uint64_t d) { return (d + kSelectTile - 1) / kSelectTile; }

constexpr int kSortThreads = 256;
constexpr int kSortItemsPerThread = 20;  // 128 registers per thread hold a tile without spilling: two blocks per SM
constexpr int kSortMinBlocks = 2;
constexpr int kSortTile = kSortThreads * kSortItemsPerThread;  // 5120 pairs
constexpr int kSortPasses = 4;                                 // digits of 9,9,9,4 bits
constexpr int kDigitBits = 9;
constexpr int kDigits = 1 << kDigitBits;                       // 512 digit values

// Ranking by partition.  The sort key of a candidate is inv = keytop - key, keytop the largest key of the client's top bin,
// so that histogram bins (and groups of them) are ranges of inv whose counts the planner knows: the selection writes every
// candidate straight into its coarse bucket, in any order.  A bucket that a block can hold is then ranked in shared memory
// by (inv, index); where coarse buckets are larger, a partition by the next bits of inv comes in between, with the
// sub-buckets' counts taken by the selection.
constexpr uint32_t kRankCoarse = 256;      // coarse buckets of a client
constexpr uint32_t kRankSubs = 8192;       // sub-buckets of a client
constexpr uint32_t kRankItems = 8192;      // candidates a block of the final ranking holds
constexpr uint32_t kRankBucket = 4096;     // largest coarse bucket that is ranked without a partition
// Candidates of a tile of the final ranking, but for its last bucket, where an SM has two or three blocks
constexpr uint32_t kRankWindow = 4096, kRankWindow3 = 3072;
constexpr uint32_t kRankTile3 = kRankWindow3 + kRankBucket;  // with the last bucket: what one of three holds
constexpr uint32_t kRankSplitTile = 4096;  // candidates of a tile of the partition
constexpr uint64_t kRankOneRound = 2ull * kNumSM * kRankSplitTile;  // candidates of a batch up to which a block of the partition has one tile
struct ClientRank {
  uint32_t n;          // candidates
  uint32_t keytop;     // largest key of the top bin
  uint32_t group;      // a coarse bucket holds 2^group histogram bins
  uint32_t n_coarse;
  uint32_t sub_bits;   // a coarse bucket holds 2^sub_bits sub-buckets
  uint32_t split;      // 1: coarse buckets are partitioned into sub-buckets
  uint32_t top_bin;
  uint32_t wide;       // 1: sub-buckets are counted in whole numbers, their counts may be beyond fp32's
  uint32_t thresh_bin; // lowest bin of the candidates: the plan's or, where k is known, the one that holds rank k
  uint32_t pad[3];
};
// The buckets of a client with nb bins between threshold and top, the fullest of them holding max_bin candidates, in a batch of `all`
// candidates.  As few sub-buckets as let a window and one of them fit a block if a bin's candidates spread evenly over it (every one that
// a block meets costs the selection a global addition); four times as many while a client then has at most 512, or 2048 where the
// partition's blocks have one tile each, since they often lie at one end of it: error compensation leaves the memories crowded below the
// threshold, in buckets that no block holds (10 clients of 5 M coordinates, up to 512 / 2048, us: 40th round 234 / 233, 150th 261 / 239,
// 400th 278 / 252), and even tiles are ranked sooner (as few as fit / up to 512: 20 of 1.2 M 121 / 119, 100 of 1.2 M 423 / 415).  Not up to
// 2048 beyond that: a partition that fills the chip then writes its 4096 candidates at a time to places of two each (512 / 2048: 300 of 3 M
// 2133 / 2184, 24 of 3 M at 4 bits 400 / 407, 20 of 1.2 M 115.1 / 116.1; only 40 of 5 M with error compensation, 400th round, gain,
// 842 / 811).  Nor in the smallest batches, whose selection and partition are the additions' latency (one of 1.2 M 47.9 / 49.0).  No
// distribution is excluded: sub-buckets that a block cannot hold are split by their own values (see rank_big), zeros among them where more
// coordinates are sent than are not zero.  (Digit passes for a batch with such a client, as phases of one kernel, took it from 844 to
// 1110 us for one of 11.2 M coordinates, 97 % zeros, and from 1636 to 3100 for 10 of 5 M, 95 % zeros.)
CVLC_HD inline void rank_shape(uint32_t nb, uint32_t max_bin, uint64_t all, ClientRank* r) {
  uint32_t g = 0;
  while (((nb - 1) >> g) + 1 > kRankCoarse) ++g;
  r->group = g;
  r->n_coarse = ((nb - 1) >> g) + 1;
  const uint64_t fullest = (uint64_t)max_bin << g;
  r->split = fullest > kRankBucket ? 1u : 0u;
  uint32_t k = 0;
  while ((fullest >> k) > kRankItems - kRankWindow && (r->n_coarse << (k + 1)) <= kRankSubs && k < 16) ++k;
  const uint32_t most = all <= kRankOneRound && all > kRankOneRound / 4 ? 2048 : 512;
  for (int more = 0; r->split && more < 2 && (r->n_coarse << (k + 1)) <= most && k < 16; ++more) ++k;
  r->sub_bits = k;
  r->wide = fullest >= (1u << 24) ? 1u : 0u;
}
// Groups of rows that the warps of the selection take one at a time by a client's counter: three quarters of a client in large
// groups, three quarters of the rest in groups a quarter as large, the last ones small, so that a block's warps finish about
// together.  A counter answers about every 20 ns, so the fewer clients share the rows the larger are the groups (10 clients of
// 100 M coordinates: 486 us with large groups of 4 pieces, 228 us with 25); with many clients small ones share out the dense
// layers better (100 of 11.2 M: 880 us with 24 pieces, 674 us with 4).  A large group is at most an eighth of a warp's share of
// the batch; a small batch is spread over all warps.
constexpr int kSelThreads = 608;
constexpr uint32_t kSelPiece = 128;  // rows whose maxima a warp loads at once (64 bits per lane)
constexpr uint32_t kSelRun = 16;     // neighbouring rows of a small group: their maxima are a sector of 32 bytes
struct SelectGroups {
  uint32_t pieces[2], count[2];  // large and middle groups: pieces in one, how many
  uint32_t small, groups;        // rows of a small group; all groups
};
CVLC_HD inline SelectGroups select_groups(const Partition& P, uint32_t n) {
  const uint64_t per_warp = P.total / ((uint64_t)kNumSM * (kSelThreads / 32));
  SelectGroups G;
  const uint32_t want = 256 / n < 4 ? 4u : (256 / n > 32 ? 32u : 256 / n);
  uint64_t pieces = per_warp / (8 * kSelPiece), left = P.rows;
  if (pieces > want) pieces = want;
  for (int l = 0; l < 2; ++l, pieces /= 4) {
    G.pieces[l] = (uint32_t)pieces;
    G.count[l] = pieces > 1 ? (uint32_t)(left * 3 / 4 / (pieces * kSelPiece)) : 0u;
    left -= G.count[l] * pieces * kSelPiece;
  }
  G.small = per_warp < kSelPiece ? 32u : kSelPiece;
  G.groups = G.count[0] + G.count[1] + (uint32_t)((left + G.small - 1) / G.small);
  return G;
}

struct EncLayout {
  uint32_t n;
  uint64_t capacity;             // candidate slots per client
  uint64_t select_tiles;         // per client, of the look-back selection
  uint64_t sort_tiles_max;       // per client
  size_t off_rank;               // ClientRank[n]
  size_t off_sort_prefix;        // uint32[n + 1]: first sort tile of every client
  size_t off_pass_mask;          // uint32[n]: digit passes that are constant for the client
  size_t off_desc;               // ClientDesc[n]
  size_t off_group_next;         // uint32[n]: next group of rows of the client
  size_t off_group_done;         // uint32[n]: groups whose candidates are in place
  size_t off_bin_fill;           // uint32[n][kRankCoarse]: candidates placed in every coarse bucket
  size_t off_sub_count;          // float[n][kRankSubs]
  size_t off_sub_start;          // uint32[n][kRankSubs + 64]: exclusive prefix, then the client's candidates
  size_t off_sub_pos;            // uint32[n][kRankSubs]: next free place
  size_t off_ghist;              // uint64[n][4][512] digit histograms
  size_t off_gbase;              // uint64[n][4][512] their exclusive scans
  size_t off_select_state;       // uint64[n][select_tiles]
  size_t off_sort_state;         // uint64[4][n * sort_tiles_max][512]
  // ranked by partition, in the place of the digit passes' states (see RankArgs):
  size_t off_list[2];            // cells left over for a warp and for a block
  size_t off_big;                // buckets that a block cannot hold, per round, and those that one block splits
  size_t off_piece;              // pieces of them, per round
  size_t off_splitter, off_part_count, off_part_start;  // per bucket: the values its parts begin with, what they hold, where they begin
  size_t off_base;               // per piece and part: what earlier pieces have of the part
  size_t off_part;               // parts to rank
  size_t off_buf_a, off_buf_b;   // uint64[n][capacity]
  size_t total;
};

// A bucket that a block cannot hold, a piece of one, and a part of one that a block can hold (see rank_big)
constexpr uint32_t kBigPart = 3072;   // candidates of a part, about
constexpr uint32_t kBigParts = 1024;  // most parts of a bucket in one round
constexpr uint32_t kBigPiece = 8192;  // candidates of a piece at least
constexpr uint32_t kBigOwn = 32768;   // a bucket of up to this many is split by one block,
constexpr int kBigOwnRow = kBigRounds;  // and stands in a row of its own behind those of the rounds
constexpr uint32_t kBigSlot = 1024;   // candidates per entry of the tables of parts
struct BigBucket {
  uint64_t pos;         // where it begins among all clients' candidates
  uint64_t from, to;    // its values lie in [from, to)
  uint64_t last;        // larger values are never sent
  uint32_t m, parts;
  uint32_t counted, pad;  // pieces counted
};
struct BigPart {
  uint64_t pos;
  uint32_t n, in_b;               // in_b: it lies in the second buffer
  uint32_t first_key, last_key;   // its keys lie between them, the larger one first
};

static inline EncLayout enc_layout(uint64_t d, uint32_t n, uint64_t capacity) {
  EncLayout L;
  L.n = n;
  L.capacity = capacity;
  L.select_tiles = select_tiles_of(d);
  L.sort_tiles_max = (capacity + kSortTile - 1) / kSortTile;
  L.off_rank = 256;
  L.off_sort_prefix = align256(L.off_rank + (size_t)n * sizeof(ClientRank));
  L.off_pass_mask = align256(L.off_sort_prefix + ((size_t)n + 1) * 4);
  L.off_desc = align256(L.off_pass_mask + (size_t)n * 4);
  L.off_group_next = align256(L.off_desc + (size_t)n * sizeof(ClientDesc));
  L.off_group_done = align256(L.off_group_next + (size_t)n * 4);
  L.off_bin_fill = align256(L.off_group_done + (size_t)n * 4);
  L.off_sub_count = align256(L.off_bin_fill + (size_t)n * kRankCoarse * 4);
  L.off_sub_start = align256(L.off_sub_count + (size_t)n * kRankSubs * 4);
  L.off_sub_pos = align256(L.off_sub_start + (size_t)n * (kRankSubs + 64) * 4);
  L.off_ghist = align256(L.off_sub_pos + (size_t)n * kRankSubs * 4);
  L.off_gbase = align256(L.off_ghist + (size_t)n * kSortPasses * kDigits * 8);
  L.off_select_state = align256(L.off_gbase + (size_t)n * kSortPasses * kDigits * 8);
  L.off_sort_state = align256(L.off_select_state + (size_t)n * L.select_tiles * 8);
  L.off_buf_a = align256(L.off_sort_state + (size_t)kSortPasses * n * L.sort_tiles_max * kDigits * 8);
  L.off_buf_b = align256(L.off_buf_a + (size_t)n * capacity * 8);
  L.total = align256(L.off_buf_b + (size_t)n * capacity * 8);
  // The lists, in the place of the digit passes' states.  Cells: at most one for every 49 candidates, and one for every 257 and one
  // per tile of at least 1024.  A large bucket has more than kRankItems candidates and at most one part for every kBigPart and one.
  const size_t all = (size_t)n * capacity, buckets = all / kRankItems + 1;
  L.off_list[0] = L.off_sort_state;
  L.off_list[1] = L.off_list[0] + align256((all / 49 + 1) * 16);
  L.off_big = L.off_list[1] + align256((all / 257 + all / 1024 + n + 1) * 16);
  L.off_piece = L.off_big + align256(buckets * (kBigRounds + 1) * sizeof(BigBucket));
  L.off_splitter = L.off_piece + align256((all / kBigPiece + buckets) * kBigRounds * 8);
  L.off_part_count = L.off_splitter + align256((all / kBigSlot + 1) * 8);
  L.off_part_start = L.off_part_count + align256((all / kBigSlot + 1) * 4);
  L.off_base = L.off_part_start + align256((all / kBigSlot + 1) * 4);
  L.off_part = L.off_base + (all / kBigPiece + buckets) * kBigParts * 4;
  return L;
}
// behind the last list; never behind the states' end, off_buf_a (a state takes 16 KB for up to 5120 candidates)
static inline size_t enc_lists_end(const EncLayout& L) {
  const size_t all = (size_t)L.n * L.capacity;
  return L.off_part + (all / kBigPart + all / kRankItems + 1) * kBigRounds * sizeof(BigPart);
}

// decode workspace
constexpr size_t kDecWsStatus = 0;     // int32 status
constexpr size_t kDecWsTotalPkts = 8;  // uint32 total packets
constexpr size_t kDecWsCoef = 256;     // float[n]
CVLC_HD constexpr size_t dec_off_prefix(uint32_t n) { return align256(kDecWsCoef + (size_t)n * 4); }  // uint32[n+1]
CVLC_HD constexpr size_t dec_off_meta(uint32_t n) { return align256(dec_off_prefix(n) + ((size_t)n + 1) * 4); }
// per client: packet_bits, header_bits (uint32 each)
CVLC_HD constexpr size_t dec_ws_bytes(uint32_t n) { return align256(dec_off_meta(n) + (size_t)n * 8); }

// ---- launch accounting and optional per-kernel timing ------------------------------

enum KernelId {
  kKZeroWords = 0, kKClient, kKHist, kKPlanThreshold, kKPlanFit, kKPlanTune, kKEncodeInit, kKSelect, kKSelectLookback, kKRankSplit, kKRank,
  kKRankRest, kKSort, kKPack, kKDecodePrepare, kKFillZero, kKPrefetchL2, kKDecode, kKNoallocStatus, kKSelftest, kKHistCheck, kKApply,
  kKPlanLiteral, kKEcAccumulate, kKPackUnframed, kKDecodeUnframed, kNumKernelIds
};

// Called around every kernel launch.  Counts launches; when a kernel has been selected with
// cvlc_profile_select, records a CUDA event pair on the launching stream around it: launch_begin
// returns the pair's number, or -1.
int launch_begin(int kernel_id, cudaStream_t st);
void launch_end(int kernel_id, int pair, cudaStream_t st);

struct LaunchScope {
  int id, pair;
  cudaStream_t st;
  LaunchScope(int id_, cudaStream_t st_) : id(id_), pair(launch_begin(id_, st_)), st(st_) {}
  ~LaunchScope() { launch_end(id, pair, st); }
};

// Something to be done once on every device (kernel attributes), asked for by every call.  Several threads may get to it
// together and then all do it, to the same effect.
struct OncePerDevice {
  std::atomic<bool> done[64];
};
template <class F>
inline cudaError_t once_per_device(OncePerDevice& once, F&& f) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < 64;
  if (known && once.done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  e = f();
  if (e == cudaSuccess && known) once.done[dev].store(true, std::memory_order_release);
  return e;
}
template <class K>
inline cudaError_t allow_shared(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

#ifdef __CUDACC__
// Every kernel of the plan / encode / decode path but the first of a call is launched with programmatic stream serialization: it is
// set up while the kernel before it drains, and pdl_enter(), the first thing every thread does, waits until that kernel is complete and its
// writes are visible.  Nothing is read or written before that.  This takes about 2 us off every kernel boundary (one small
// client, 12 kernels: 101 -> 78 us a pass; 100 ResNet-18 clients: 3.89 -> 3.87 ms).  No kernel lets its successor in before
// its own blocks have left (griddepcontrol.launch_dependents): blocks that move in early gather on the SMs that happen to be
// free, and the successor then runs on part of the chip (error compensation 314 -> 361 us, the large round 3.87 -> 4.00 ms).
// The attribute leaves the order behind the kernel before it on the stream to pdl_enter(), and waiting for that kernel alone is enough
// only where it has waited for its own predecessor.  Ours have.  What precedes the first kernel of a call is the caller's: a kernel
// launched in the same way that does not wait may end before the work in front of it.  So the first kernel of a call is an ordinary
// launch, behind all that the stream holds, and so is one behind a wait on another stream's event.  That costs 2 us a call in a stream
// of small calls (4 clients of 0.4 M coordinates, compressed and aggregated: 65 -> 70 us), nothing where the GPU waits for the host.
template <class... Params, class... Args>
inline void launch_kernel(int id, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool overlap, Args&&... args) {
  LaunchScope ls(id, st);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);  // the error stays in cudaGetLastError
}
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

// ---- launchers (one per translation unit) ---------------------------------------

// What the planning front prepares for the encoder of the same call (ws = nullptr: nothing): its workspace's header, the clients'
// shapes of the ranking, the counters of selection and partition at zero
struct EncFront {
  unsigned char* ws;
  EncLayout L;
};

// Where the length tuning runs, one block per client that tunes.  Beside selection and ranking, whose blocks fill an SM each, its place
// matters:
//  - They leave it its SMs where the clients are few and the selection short: blocks behind a tuning block would start when that ends
//    (after 25 to 80 us, 67 us into a selection of 120), and the kernel ends with them.  Not for long selections, where blocks that start
//    late still find work: the SMs given away cost the clients times the length of the selection.  Whole calls with room and without, us:
//    24 clients of 0.3 M coordinates 90 and 100, 32 of 0.3 / 1.2 / 3 M 98 and 111 / 195 and 203 / 385 and 390, 40 of 0.3 / 1.2 / 3 M 107
//    and 117 / 239 and 226 / 475 and 441; 10 of 13 / 20 / 40 M 319 and 346 / 434 and 467 / 816 and 820, 20 of 6 / 12 M 309 and 315 / 548
//    and 514.
//  - Else it must be ahead of the selection to find an SM before that ends.  That costs the selection's start: the exponent fit of more
//    than kTuneRoom clients comes first (10 us), then an event.  Behind the selection a tuning of a few hundred us, which steep power
//    laws need, ends behind the ranking.  Whole calls ahead and behind, us, for one normal distribution / for magnitudes that fall as
//    rank^-1.3: 10 clients of 40 M 566 and 567 / 1537 and 1672, 20 of 12 M 534 and 526 / 1627 and 1751, 100 of 11.2 M 2937 and 2928 / 3093 and
//    3904, 60 of 3 M 438 and 430 / 621 and 731; but 40 of 1.2 M 212 and 192 / 435 and 486, 100 of 0.3 M 124 and 105 / 132 and 131 (rank^-1.8:
//    404 and 446), 33 of 0.3 M 72 and 61 / 80 and 83 (382 and 393).  So short selections with more clients than there is room for, which
//    is a loss of up to a tenth for steep laws, and one of up to a sixth avoided for all others, have it behind.
enum TunePlace { kTuneAlone, kTuneRoomLeft, kTuneAhead, kTuneBehind };
constexpr uint32_t kTuneRoom = 32;
constexpr uint64_t kTuneRoomRows = 192 << 20;  // times clients
constexpr uint64_t kShortSelectRows = 8 << 20;
inline TunePlace tune_place(uint64_t d, uint32_t n) {
  const uint64_t rows = make_partition(d, n).total;
  if (n <= kTuneRoom && n * rows <= kTuneRoomRows) return kTuneRoomLeft;
  return n <= kTuneRoom || rows > kShortSelectRows ? kTuneAhead : kTuneBehind;
}
// Planning is launched in two parts.  The front (histogram, rows' maxima, selection threshold, the bins' starts) is all the
// selection and ranking kernels need; the back (exponent fit, unless it is done ahead of the selection, and length tuning) is only needed by
// the packing kernel, so it may run on another stream than they do.
cudaError_t launch_plan_front(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, const EncFront& enc, TunePlace place, cudaStream_t st);
// overlap: nothing but the front precedes the back on its stream (no wait for an event)
cudaError_t launch_plan_back(uint32_t n, const Shape& shape, void* ws, TunePlace place, cudaStream_t st, bool overlap);
cudaError_t launch_plan(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, cudaStream_t st);
// Few small clients: planning, selection and ranking by a cluster of blocks per client (see k_client).  All clusters run at a time, every block
// keeps most of its share of the coordinates in shared memory, and there is room for all bins that can be too large for a block (see kCutRanges).  The
// kernels of their own and this, close to the limit of 65,536 records, us: 1 / 7 clients of 320,000 coordinates at 4 bits (52,600 records) 44 and 31 / 54
// and 35, 12 of 320,000 at 2.8 (36,700) 58 and 41, 12 of 240,000 at 4 (41,400) 58 and 43, 3 of 600,000 at 2.7 (64,300) 51 and 40, 1 / 7 of 655,000 at 2.4
// (62,400) 48 and 39 / 59 and 43.
constexpr uint32_t kClusterUnits = 10240;  // float4 units that a block keeps at most
constexpr uint64_t kClusterCandidates = 65536;
// Blocks of a client's cluster; 0: too many clients or coordinates.  Clusters that run at a time, a block on an SM
// (cudaOccupancyMaxActiveClusters): 15 of eight blocks, 7 of sixteen.  Sixteen exchange more counts, eight read and rank longer; calls at 1 bit a
// coordinate, eight and sixteen, us: one client of 100,000 coordinates 26.8 each, of 200,000 27.3 and 27.6, of 240,000 28.9 and 28.4, of 320,000 30.9 and
// 28.9, seven of 200,000 29.0 and 31.0, of 240,000 31.0 each, of 320,000 33.1 and 31.0; at 4 bits one of 320,000 41.2 and 30.9.  Beyond that the kernels of
// their own and sixteen: one of 340,000 43.5 and 28.9, three of 450,000 47.7 and 34.4, seven of 650,000 52.7 and 41.3.
inline uint32_t cluster_blocks(uint64_t rows, uint32_t n) {
  const uint64_t of_block = kClusterUnits / kRowUnits;
  if (n <= 7 && rows > 6 * of_block && rows <= 16 * of_block) return 16;
  return n <= 15 && rows <= 8 * of_block ? 8 : 0;
}
bool clusters_run(uint32_t blocks);  // on the current device: a part of a GPU may have too few SMs side by side
inline bool by_clusters(const Shape& shape, uint32_t n, uint32_t cap0) {  // cap0: the largest of the clients'
  const uint32_t blocks = cluster_blocks(make_partition(shape.d, n).rows, n);
  return blocks != 0 && (uint64_t)shape.R * cap0 <= kClusterCandidates && clusters_run(blocks);
}
cudaError_t launch_clients(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws, const EncFront& enc, cudaStream_t st);
cudaError_t launch_histogram(const ClientDesc* clients, uint32_t n, const Shape& shape, void* ws,
                             unsigned long long* hist_out, cudaStream_t st);
cudaError_t launch_plan_from_hist(const ClientDesc* clients, uint32_t n, const Shape& shape,
                                  const unsigned long long* hist, void* ws, cudaStream_t st);
// workspace of cvlc_plan_literal: per value of k its value, its error bound, its sweeps and its packet sizes
CVLC_HD constexpr size_t literal_off_k(uint32_t) { return 256; }
CVLC_HD constexpr size_t literal_off_gamma(uint32_t n_k) { return align256(literal_off_k(n_k) + (size_t)n_k * 8); }
CVLC_HD constexpr size_t literal_off_sweeps(uint32_t n_k) { return align256(literal_off_gamma(n_k) + (size_t)n_k * 8); }
CVLC_HD constexpr size_t literal_off_P(uint32_t n_k) { return align256(literal_off_sweeps(n_k) + (size_t)n_k * 4); }
CVLC_HD constexpr size_t literal_ws_bytes(uint32_t n_k, uint32_t R) { return align256(literal_off_P(n_k) + (size_t)n_k * R * 8); }
constexpr uint32_t kLiteralMaxR = 2048;   // packet sizes and their running sums of one k live in shared memory
constexpr uint32_t kLiteralMaxK = 4096;
cudaError_t launch_plan_literal(const cvlc_params& p, double alpha_q, uint32_t s, uint32_t R, uint32_t n_k, uint32_t max_sweeps,
                                unsigned long long k_lo, unsigned long long k_hi, double P_min, double P_max, double tol,
                                cvlc_literal_plan_t* out, double* P_star, void* ws, cudaStream_t st);
cudaError_t launch_apply(float* model, const float* agg, uint64_t d, const void* dec_ws, cudaStream_t st);
// ranking by partition (after the selection); most: candidates of a client that can be sent
cudaError_t launch_rank(Batch batch, const EncLayout& L, const unsigned char* plan_ws, unsigned char* ws, unsigned sms, uint64_t most, cudaStream_t st);
// its last kernel alone: the large buckets that are on the lists
cudaError_t launch_rank_rest(Batch batch, const EncLayout& L, const unsigned char* plan_ws, unsigned char* ws, unsigned sms, bool three, cudaStream_t st);
// wait_before_pack: an event the stream waits for right before the packing kernel (the length tuning on
// another stream), or nullptr
// write_residual: kPackFramed = packets only; kPackResidual = the packing kernel also turns the encoder's input into
// the error-compensation memory (the input buffers are written: every sent coordinate loses what the parameter
// server rebuilds for it); kPackNone = selection and ranking only (launch_pack or the unframed writer follows)
constexpr int kPackFramed = 0, kPackResidual = 1, kPackNone = 2;
constexpr size_t kPackSharedMax = 200 * 1024;  // shared memory of four packets at work, at most
// ranked: planned, selected and ranked by launch_clients on the same stream
// prepared: the planning front of the same call has prepared the workspace (see EncFront) and precedes it on the stream; behind_wait:
// and a wait for another stream's event lies between
cudaError_t launch_encode(const ClientDesc* clients, uint32_t n, const Shape& shape, uint64_t capacity,
                          const void* plan_ws, void* ws, cudaStream_t st, bool prepared, bool behind_wait, cudaEvent_t wait_before_pack,
                          int write_residual, bool ranked = false);
// the packing alone, behind selection and ranking; overlap: they directly precede it on the stream
cudaError_t launch_pack(const ClientDesc* clients, uint32_t n, const Shape& shape, uint64_t capacity, void* ws, cudaStream_t st, bool overlap,
                        int write_residual);
cudaError_t launch_ec_accumulate(float* const* memory, const float* const* update, uint32_t n, uint64_t d, cudaStream_t st);
// unframed stream (version 2)
constexpr uint32_t kUfMaxRecords = 2048;  // records of a block (they are sorted and assembled in shared memory)
constexpr size_t kUfTables = 64, kUfTotalBits = 64 + 264, kUfDirectory = 64 + 264 + 8;
CVLC_HD constexpr size_t uf_head_bytes(uint32_t R) { return kUfDirectory + (size_t)R * 8; }
CVLC_HD constexpr size_t uf_off_ticket() { return 256; }
CVLC_HD constexpr size_t uf_off_state(uint32_t n) { return align256(uf_off_ticket() + (size_t)n * 4); }
CVLC_HD constexpr size_t uf_ws_bytes(uint32_t n, uint32_t R) { return align256(uf_off_state(n) + (size_t)n * R * 8); }
CVLC_HD inline uint32_t uf_rice_param(uint64_t d, uint32_t P) {  // floor(log2(d / P)), 0 when d < 2 P
  uint64_t g = d / (uint64_t)P;
  uint32_t m = 0;
  while (g >= 2) {
    g >>= 1;
    ++m;
  }
  return m;
}
cudaError_t launch_pack_unframed(uint32_t n, const Shape& shape, uint64_t capacity,
                                 size_t stream_capacity, void* enc_ws, void* uf_ws, unsigned long long* sizes_out, cudaStream_t st);
cudaError_t launch_decode_unframed(const uint8_t* const* streams, const uint64_t* stream_bytes, const float* weights,
                                   uint32_t n, double weight_total, uint64_t d, uint32_t s, float* out, int accumulate,
                                   void* ws, cudaStream_t st);
cudaError_t launch_selftest_wait(unsigned long long* word, int32_t* status, uint32_t max_polls, cudaStream_t st);
cudaError_t launch_decode(const uint8_t* const* streams, const uint64_t* stream_bytes, const float* weights,
                          uint32_t n, double weight_total, uint64_t d, uint32_t s, float* out, int accumulate,
                          void* ws, cudaStream_t st);
cudaError_t launch_selftest_philox(uint64_t seed, uint32_t client_id, uint32_t round, uint64_t first, uint64_t n,
                                   uint32_t* out, cudaStream_t st);
cudaError_t launch_selftest_math(const double* in, uint64_t n, double* l2, double* e2, double* dv, double* dr,
                                 cudaStream_t st);

// ---- device helpers ---------------------------------------------------------------

#ifdef __CUDACC__

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32->64
// multiplies with the constants 0xD2511F53 / 0xCD9E8D57, key bumped by the Weyl
// constants 0x9E3779B9 / 0xBB67AE85 after every round.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x, p1 = (unsigned long long)0xCD9E8D57u * c.z;
    const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0, hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// random word of one coordinate: counter (coord lo, coord hi, client, round), key = seed
__device__ __forceinline__ uint32_t philox_coord(uint64_t seed, uint32_t client_id, uint32_t round, uint64_t coord) {
  const uint4 r = philox4x32_10(make_uint4((uint32_t)coord, (uint32_t)(coord >> 32), client_id, round),
                                make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  return r.x;
}

// The same word with the ten round keys worked out once per client instead of once per coordinate.
struct PhiloxRoundKeys {
  uint32_t x[10], y[10];
};
__device__ __forceinline__ PhiloxRoundKeys philox_round_keys(uint64_t seed) {
  PhiloxRoundKeys rk;
  uint32_t kx = (uint32_t)seed, ky = (uint32_t)(seed >> 32);
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    rk.x[i] = kx;
    rk.y[i] = ky;
    kx += 0x9E3779B9u;
    ky += 0xBB67AE85u;
  }
  return rk;
}
__device__ __forceinline__ uint32_t philox_coord(const PhiloxRoundKeys& rk, uint32_t client_id, uint32_t round, uint32_t coord) {
  uint4 c = make_uint4(coord, 0u, client_id, round);  // coordinates are below 2^32: counter word 1 is zero
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const unsigned long long p0 = (unsigned long long)0xD2511F53u * c.x, p1 = (unsigned long long)0xCD9E8D57u * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ rk.x[i], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ rk.y[i], (uint32_t)p0);
  }
  return c.x;
}

__device__ __forceinline__ uint32_t sort_keytop(uint32_t top_bin) { return ((top_bin + 1u) << 19) - 1u; }
__device__ __forceinline__ uint32_t sort_keytop(const cvlc_plan_t* plan) { return sort_keytop(plan->top_bin); }
// candidates of a client in the coarse buckets before bucket i (bins from the top down)
__device__ __forceinline__ uint32_t coarse_start(const ClientRank& r, const uint32_t* bin_start, uint32_t i) {
  return i < r.n_coarse ? bin_start[r.top_bin - (i << r.group)] : r.n;
}

__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  // first error wins
  atomicCAS(status, 0, code);
}

__device__ __forceinline__ uint32_t sort_tiles_of(unsigned long long n_candidates, unsigned long long capacity) {
  const unsigned long long nc = n_candidates < capacity ? n_candidates : capacity;
  return (uint32_t)((nc + kSortTile - 1) / kSortTile);
}

// ranks from here on are never sent, whatever the lengths
CVLC_HD inline uint32_t rank_limit(const Shape& shape) {
  const unsigned long long most_sent = (unsigned long long)shape.R * shape.cap[1];
  return most_sent < 0xFFFFFFFFull ? (uint32_t)most_sent : 0xFFFFFFFFu;
}

// a client's buckets from its threshold, the candidates from there on, and what the fullest bin holds
__device__ __forceinline__ ClientRank client_rank(uint32_t thresh_bin, uint32_t top_bin, unsigned long long n_candidates, uint32_t max_bin,
                                                  unsigned long long capacity, uint32_t n) {
  ClientRank r;
  const uint32_t top = top_bin < CVLC_HIST_BINS ? top_bin : CVLC_HIST_BINS - 1;
  const uint32_t nb = thresh_bin <= top ? top - thresh_bin + 1 : 1;
  r.n = (uint32_t)(n_candidates < capacity ? n_candidates : capacity);
  rank_shape(nb, max_bin, (uint64_t)r.n * n, &r);
  r.keytop = sort_keytop(top_bin);
  r.top_bin = top;
  r.thresh_bin = thresh_bin;
  return r;
}

// a client's share of what the encoder's header says of the batch; by one thread, the header starts at zero
__device__ __forceinline__ void add_client(EncHeader* hdr, const ClientRank& r, uint32_t limit) {
  atomicMax(&hdr->most, r.n < limit ? r.n : limit);  // buckets from the limit on are not ranked
  if (r.split) atomicMax(&hdr->most_split, r.n);
}
// Candidates per tile of the final ranking: as many as make the tiles of all clients whole rounds of the blocks, as few rounds as
// tiles of at most `largest` allow.  With powers of two, at least four tiles an SM, some blocks had a tile more than the others:
// one client of 11.2 M coordinates (2048 in 1.4 rounds, now 2800 in one) 18.0 -> 15.6 us between events, 8 of 1.2 M 17.3 -> 14.8, one
// of 52 M, with what is left over, 73 -> 48.
__device__ __forceinline__ uint32_t rank_window(uint32_t most, uint32_t n, uint32_t blocks, uint32_t largest) {
  const uint32_t least = (most + largest - 1) / largest;  // tiles of the largest client
  const uint32_t tiles = (least * n + blocks - 1) / blocks * blocks / n;  // below 2^29: at most 699,051 tiles (of 3072) of at most 512 clients
  const uint32_t window = tiles ? (most + tiles - 1) / tiles : 0u;
  return window > 1024 ? window : 1024;
}

// thread `first` of `stride` writes its share of d zeros
__device__ __forceinline__ void zero_fill(float* __restrict__ out, uint64_t d, uint64_t first, uint64_t stride) {
  const uint64_t nvec = d >> 2;
  float4* ov = reinterpret_cast<float4*>(out);
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  for (uint64_t v = first; v < nvec; v += stride) ov[v] = z;
  if (first < (d & 3)) out[(nvec << 2) + first] = 0.f;
}
// blocks of `threads` for it, `most` at the most
inline unsigned fill_grid(uint64_t coords, uint64_t threads, uint64_t most) {
  const uint64_t want = (coords / 4 + threads - 1) / threads;
  return (unsigned)(want < most ? (want ? want : 1) : most);
}

#endif  // __CUDACC__

}  // namespace cvlc
