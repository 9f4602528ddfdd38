// Exact k+1 nearest-neighbour search (the NN(d, k+1) of Alg. 2) on the sm_103a
// tensor cores.
//
// For a tile of 128 query rows and 256 reference rows the MMA computes, in
// FP32 TMEM accumulators,
//     acc[i][j] = sum_t (-2 q_it) r_jt + (1, 256, 65536, e0, e1, e2)_i . (d0, d1, d2, 1, 256, 65536)_j
//               = ||r_j||^2 + ||q_i||^2 - 2 q_i . r_j = ||q_i - r_j||^2,
// the last term being a 16-wide K-extension that carries both squared norms as
// base-256 digits.  BF16 holds 0..255, -2q and the digits exactly; every
// product and partial sum is an integer below 2^24 in magnitude, so acc is the
// exact squared distance.  Non-negative floats order like their bit patterns,
// so the epilogue tests 32 columns with one compare of their minimum, which
// the TMEM load itself returns (tcgen05.ld.red ... .min.u32), against the
// row's current (k+1)-th distance, and keeps the k+1 smallest (distance, row)
// pairs.  The distance matrix never leaves the SM.
//
// The same scan runs the coarse pass of the FP8 shortlist search: operands
// are the E4M3 roundings of the coordinates shifted by -64 (queries scaled by
// -2, exact in E4M3), one 128-byte K-chunk per tile and four kind::f8f6f4
// MMAs (K = 32 each), and the K-extension carries ||q'||^2 + 2^21 and ||r'||^2
// of the shifted (unrounded) coordinates.  The accumulator then holds
//     coarse = ||q'||^2 + ||r'||^2 - 2 q~ . r~ + 2^21,
// an integer: the bias keeps it positive (E4M3 rounding is within 2^-4 of
// each coordinate, so 2 q~.r~ is within 2 * 0.129 * 128 * 191^2 < 1.21e6 of
// 2 q'.r'), and with the extension issued first every partial sum stays in
// [0, 2^24), so FP32 holds it exactly.
//
// Work: a launch covers T groups of QT query tiles (128 rows each) x S
// reference splits as T x S work items, split-major; a CTA takes one item, or
// (persistent form) items from a queue one after another (see Work below).
//
// Roles (one CTA = QT query tiles x one reference split at a time):
//   warp 0, one thread : TMA producer (the item's query tiles; reference
//                        K-chunks into a ring, the K-extension riding with
//                        the last chunk of each tile)
//   warp 1, one thread : tcgen05.mma issuer (9 MMAs of 128x256x16 per tile);
//                        warp 1 also owns the TMEM allocation; with QT = 2 a
//                        second issuer (warp 2) issues the second query
//                        tile's MMAs
//   warps 4-11         : epilogue: two warps per TMEM lane quarter, each
//                        taking a 128-column half of every tile (QT = 2: its
//                        query tile's 128 x 128 block) with one thread per
//                        query row (TMEM lane); two 256-column FP32
//                        accumulators in flight; each 32-column load also
//                        returns the columns' minimum, and groups whose
//                        minimum is below the row's limit are passed on
//   warps 12-15        : inserters, one per TMEM lane quarter: the rows' lists
//                        of the k+1 nearest (not in the NBNN scan)
// Every wait is bounded; on expiry the CTA records a timeout in the index's
// device error word, drains what it issued and returns.
#include <cudaTypedefs.h>

#include "knn_tc.cuh"
#include "sm103.cuh"
#include "topk.cuh"

namespace lnbnn {
namespace {

using namespace sm103;

constexpr int kBM = kTcQueryTile;         // query rows per query tile (MMA M)
constexpr int kBK = 64;                   // BF16 K elements per 128-byte swizzle row
constexpr int kKChunks = kDim / kBK;      // K-chunks of the BF16 operand (shared memory is laid out for these)
constexpr int kMmaPerChunk = 4;           // 32-byte K-steps per 128-byte chunk (16 BF16 or 32 E4M3)
constexpr uint32_t kAChunkBytes = kBM * kBK * 2;     // 16 KB
constexpr uint32_t kAExtBytes = kBM * kExt * 2;      // 4 KB

// Tile shapes: a CTA computes QT query tiles (128 rows each) against a tile
// of 256 / QT references per step, so every step is 128 x 256 query-reference
// pairs and its FP32 accumulator takes 256 TMEM columns (QT = 2: the two
// query tiles' 128 x 128 blocks side by side).  QT = 2 loads each reference
// tile once for 256 query rows: half the reference bytes per pair.
template <int QT>
struct Shape {
  static_assert(QT == 1 || QT == 2, "one or two query tiles per CTA");
  static constexpr int kTileN = kTcRefTile / QT;                 // references per tile (MMA N)
  static constexpr uint32_t kBChunkBytes = kTileN * kBK * 2;     // 32 or 16 KB
  static constexpr uint32_t kBExtBytes = kTileN * kExt * 2;      // 8 or 4 KB
  static constexpr uint32_t kStageBytes = kBChunkBytes + kBExtBytes;
};

// Warps of a CTA, in warpgroups of four: warp 0 the TMA producer, warp 1 the
// MMA issuer (and the TMEM allocation's owner), warp 2 the second query tile's
// issuer (QT = 2), warp 3 unused; then eight epilogue warps, two per TMEM lane
// quarter; then, for lists kept in registers, four inserter warps.
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 8;
constexpr int kInsWarp0 = kEpiWarp0 + kEpiWarps;
template <class Epilogue>
constexpr int kThreadsOf = 32 * (kInsWarp0 + Epilogue::kInserterWarps);
// Registers a thread of a launch can have (the SM's 65,536 over its threads).
template <class Epilogue>
constexpr int kMaxRegsOf = 65536 / kThreadsOf<Epilogue> / 8 * 8;
// Lists of more than 64 registers a thread: the inserter warps take registers
// that the first warpgroup, whose roles need few, gives up (the epilogue's two
// warpgroups keep theirs).  What counts is that an insertion has no spilled
// operand: k = 50, 20,000 rows x 1.5 million, 184 registers and the spills that
// went with them 7.4 and 9.3 ms, 192 6.4, 200 6.4.
template <class Epilogue, int QT>
constexpr bool kWideLists = Epilogue::KMAX * QT > 32;
constexpr int kRegsFirst = 64, kRegsLaunch = 128, kRegsInserter = 192;
static_assert(kRegsFirst + 2 * kRegsLaunch + kRegsInserter <= 4 * kRegsLaunch, "what is taken has been given up");
constexpr uint32_t kAccCols = kTcRefTile;  // FP32 columns per accumulator (one step)
constexpr uint32_t kTmemCols = 2 * kAccCols;
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s per wait
constexpr uint64_t kItemLimitNs = 60 * kWaitLimitNs;  // a work item, for the warps that wait through all of it

// Shared-memory layout of one CTA: QT query tiles (each AChunks
// 128-byte-swizzle chunks + the 32-byte-swizzle extension), the reference
// ring (Stages stages, each room for one K-chunk of a reference tile and its
// extension), the mbarriers, the TMEM address, abort flag and work-item
// slots, and ListBytes for an epilogue that keeps its lists in shared memory.
template <int AChunks, int Stages, uint32_t ListBytes, int QT>
struct Layout {
  using S = Shape<QT>;
  static constexpr int kStages = Stages;
  static constexpr uint32_t kAQueryBytes = AChunks * kAChunkBytes + 1024 * ((kAExtBytes + 1023) / 1024);
  static constexpr uint32_t kOffA = 0;  // query tile q at kOffA + q * kAQueryBytes; its extension after its chunks
  static constexpr uint32_t kOffB = QT * kAQueryBytes;
  static constexpr uint32_t kOffBar = kOffB + Stages * S::kStageBytes;
  // full, empty per stage; tmem empty per accumulator; A full, A empty,
  // drain; item full, item empty per item slot; lists written; warm-up done,
  // the rows' limits posted, the columns of an item all queued
  static constexpr int kNumBars = 2 * Stages + 2 + 3 + 2 + 2 + 1 + 3;
  // TMEM address, abort flag, "a timeout was reported before" flag, 2 item slots, 2 "an earlier split was not carried" words, work slot
  static constexpr uint32_t kOffMisc = kOffBar + 8 * kNumBars;
  static constexpr uint32_t kOffList = (kOffMisc + 48 + 1023) / 1024 * 1024;
  static constexpr uint32_t kSmemBytes = kOffList + ListBytes + 1024;  // + alignment slack
  static_assert(Stages % AChunks == 0, "a tile's chunks map to fixed stage parities");
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};

// Operand formats.  Either way one K-chunk is one 128-byte (swizzled) row
// per operand row and one MMA consumes 32 bytes of it.
struct FmtBf16 {  // exact search: 128 BF16 coordinates, two chunks
  static constexpr int kChunks = 2;
  static constexpr bool kExtFirst = false;
  template <int N>
  static __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
    mma_bf16(d, a, b, idesc_bf16_f32(kBM, N), acc);
  }
};
struct FmtE4m3 {  // coarse pass: 128 E4M3 coordinates, one chunk
  static constexpr int kChunks = 1;
  static constexpr bool kExtFirst = true;
  template <int N>
  static __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
    mma_f8(d, a, b, idesc_e4m3_f32(kBM, N), acc);
  }
};

template <int kStages>
struct Bars {
  uint32_t base;
  __device__ uint32_t full(int s) const { return base + 8 * s; }
  __device__ uint32_t empty(int s) const { return base + 8 * (kStages + s); }
  __device__ uint32_t tempty(int b) const { return base + 8 * (2 * kStages + b); }
  __device__ uint32_t afull() const { return base + 8 * (2 * kStages + 2); }
  __device__ uint32_t aempty() const { return base + 8 * (2 * kStages + 3); }
  __device__ uint32_t drain() const { return base + 8 * (2 * kStages + 4); }
  __device__ uint32_t ifull(int i) const { return base + 8 * (2 * kStages + 5 + i); }
  __device__ uint32_t iempty(int i) const { return base + 8 * (2 * kStages + 7 + i); }
  __device__ uint32_t lists_done() const { return base + 8 * (2 * kStages + 9); }
  __device__ uint32_t limits() const { return base + 8 * (2 * kStages + 10); }
  __device__ uint32_t queued() const { return base + 8 * (2 * kStages + 11); }
  __device__ uint32_t warmed() const { return base + 8 * (2 * kStages + 12); }
};

// The layout of a kernel instantiation: the format's query chunks; four ring
// stages (two tiles of 256 references in BF16, four in E4M3), for QT = 2 three
// or eight tiles of 128 references (BF16 six stages, E4M3 eight).
template <class Fmt, class Epilogue, int QT>
using LayoutOf = Layout<Fmt::kChunks, QT == 2 ? (Fmt::kChunks == 2 ? 6 : 8) : 4, Epilogue::kListBytes, QT>;

__device__ __forceinline__ void flag_timeout(volatile uint32_t* abort_flag, uint32_t* dev_err) {
  *abort_flag = 1u;
  atomicOr(dev_err, kDevErrTimeout);
}

// Wait until the gate word is nonzero, for at most limit_ns, giving up early
// once another role of the CTA has given up.  Returns false on expiry.
__device__ __forceinline__ bool wait_gate(const uint32_t* gate, uint64_t limit_ns,
                                          const volatile uint32_t* abort_flag) {
  const volatile uint32_t* g = gate;
  if (*g != 0u) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (*g != 0u) return true;
    if ((it & 255u) == 0 && (*abort_flag || globaltimer_ns() - t0 > limit_ns)) return false;
  }
}

// v[j] for a run-time j without dynamic register indexing (no local memory):
// a 5-level select tree on the bits of j.
__device__ __forceinline__ int32_t select32(const uint32_t (&v)[32], int j) {
  uint32_t t[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) t[i] = (j & 1) ? v[2 * i + 1] : v[2 * i];
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = (j & 2) ? t[2 * i + 1] : t[2 * i];
#pragma unroll
  for (int i = 0; i < 4; ++i) t[i] = (j & 4) ? t[2 * i + 1] : t[2 * i];
#pragma unroll
  for (int i = 0; i < 2; ++i) t[i] = (j & 8) ? t[2 * i + 1] : t[2 * i];
  return (int32_t)((j & 16) ? t[1] : t[0]);
}

// What the scan writes (see the epilogues below).
struct ScanOut {
  uint64_t* lists;           // kNN: sorted lists, [splits][stride][K1]
  int64_t stride;
  int K1;
  int32_t* mins;             // NBNN: per (query row, class) minimum distance, [m_pad][C], atomicMin
  int32_t C;
  const int64_t* class_off;  // NBNN: class c owns sorted rows [class_off[c], class_off[c+1])
  const uint32_t* gate;      // null, or a word the producer waits to see nonzero before loading
  int32_t* row_thr;          // kNN: per query row, a shared bound (below), or null
  bool bound_per_tile;       // row_thr read and published every tile, or at a work item's start and end
  uint32_t* done;            // kNN with splits run one after another: per work item, nonzero once its
                             // lists are written, 2 if they also hold every earlier split's keys (zero
                             // before the launch), or null
  int64_t T;                 // query-tile groups of the launch (work item w - T is the same rows' previous split)
  char* work;                // kNN: candidate buffers of the lists in progress, work_slots x tc_work_bytes(entries)
  int64_t work_slots;
  int entries;
  uint32_t* slot_used;       // one word per slot, zero before the launch; null if the grid has no more CTAs than slots
};

// A work slot of the launch for this CTA: its own number where the grid has no
// more CTAs than slots.  Otherwise there is a slot per SM, a CTA fills an SM
// (its shared memory), and so one of the slots is always free.
__device__ __forceinline__ int32_t acquire_slot(const ScanOut& out) {
  if (out.slot_used == nullptr) return (int32_t)blockIdx.x;
  int32_t s = (int32_t)(blockIdx.x % out.work_slots);
  const uint64_t t0 = globaltimer_ns();
  while (atomicExch(out.slot_used + s, 1u) != 0u) {
    s = s + 1 < out.work_slots ? s + 1 : 0;
    if (s == 0 && globaltimer_ns() - t0 > kWaitLimitNs) return -1;
  }
  __threadfence();
  return s;
}
__device__ __forceinline__ void release_slot(const ScanOut& out, int32_t s) {
  if (out.slot_used == nullptr || s < 0) return;
  __threadfence();
  atomicExch(out.slot_used + s, 0u);
}

// kNN (Alg. 2's NN(d, k+1) restricted to the columns one CTA sees): the lists
// are kept by warps of their own.  An epilogue warp that inserted its own
// candidates held up its tile, and with it the other seven and the
// accumulator's return to the MMAs, for as long as the insert took (101-class
// data, k = 50: 3,660 cycles a step against the MMAs' 1,152; k = 100 and
// FP8 shortlist 128 on the 256-class data, heaps: 4,680 and 4,180).
//
// An epilogue warp compares the least value of each 32-column group (which the
// TMEM load returns) with its rows' limits; each of its threads appends the
// octets of columns that hold one below its row's limit to a buffer.  One
// inserter warp per TMEM lane quarter takes the buffers of the quarter's two
// epilogue warps when they are handed over, sorts their columns into the rows'
// lists (registers, or merge_rows) and posts the rows' new limits; the epilogue
// goes on in a second set of buffers meanwhile.  The buffers are in global
// memory (L2): a hit costs the epilogue about 300 cycles of predicated stores
// (copying single columns 1,000), whatever the list length.  The limit may be
// read late: that changes which columns are appended, never which K1 keys the
// list ends with, since keys are compared by (distance, row) and a column at
// the limit passes.  Measured, whole calls before and after (one GB300):
// 101-class data, 200k rows, k = 50 121.6 / 60.5 ms; 256-class data, 15k rows,
// k = 100 95.0 / 32.5 ms, FP8 shortlist 128 84.5 / 26.2 ms, shortlist 24 on
// one image of 632 rows 1.31 / 0.83 ms (all steps together).
//
// The lists of a row in other reference splits share a bound with it:
// row_thr[row] holds the bit pattern of a distance at or below which some list
// already holds K1 entries, so a column farther than it cannot be among the
// row's K1 nearest.  When the lists of a row run at the same time (few query
// tiles, many splits), a merge publishes an improved K1-th distance with an
// atomic minimum, and the inserters read the word every few polls.  When they
// run one after another (many query tiles: the splits of a row are work items
// far apart), a list reads the word once when it starts and publishes once
// when it ends.  Which columns a list drops depends on timing; the K1 nearest
// of the row never are, so the merged result does not.
//
// Warm-up: a list that starts empty would copy every column until its first
// merge.  So the first tiles of an item are run twice, first for a limit alone:
// the columns fall into groups, each group's least value is the distance of
// another column, and so the K1-th smallest of these minima bounds the K1-th
// smallest distance.  A thread keeps the least minima of its column half sorted,
// half of K1 (QT = 2: K1), and the larger of the two halves' last ones is the
// limit.  With 32 columns a group the minimum comes with the load; where that is
// too few groups for a useful limit, eight.  Where a thread cannot keep as many
// minima (lists of more than 128 keys), a group's second-least value stands for
// two columns.  (QT = 2 with the longest lists has no registers for any: the
// largest minimum of exactly as many groups.)
// (row_thr starts at 0x7F7F7F7F, above everything.)  A list's own bound starts
// between the distances (and coarse values) and those of padding rows, so that
// these are never collected: a last split of one tile, mostly padding, held up
// calls of short items by 20 of 45 us.
constexpr int32_t kRealBound = 0x4B7FFFFF;  // bits of 2^24 - 1

struct WarmUp {
  int tiles;    // tiles run twice
  bool octets;  // groups of 8 columns, not 32 (unranked: of 32, not the thread's part of a tile)
  bool pairs;   // a group's second-least value, for two columns
};
// How many minima a thread can keep sorted (0: the limit is the largest).
template <int KMAX, int QT>
constexpr int kRankedMax = KMAX > 0 ? KMAX * QT / 2 : QT == 1 ? 64 : 0;
// rows: of the item's query tile; share: other lists of the rows run meanwhile
// and share their bound.
//
// A tile run twice costs a step; W of an item's n tiles leave about
// K1 (1 + ln(n / W)) columns a row to insert.  The least sum is at W ~ K1 for
// lists in registers (8 K1 for the 64-key ones, whose insertions are dear), a
// few K1 where a merge is paid by the row, whatever n: so a short item runs all
// of its tiles twice.  Whole calls, one GB300, with the tiles limited to a
// quarter or a sixteenth of the item (and none where they had fewer than K1
// groups of 32) against now: 20,000 queries, 2,000 references, k = 10, 24, 100
// and 200 171, 298, 3,351 and 5,552 us / 102, 161, 1,104 and 2,582 us; 20,000
// references, k = 50 and 100 1.88 and 3.76 / 0.57 and 1.45 ms; 500,000, k = 50
// 5.1 / 3.2 ms.  Lists that share a bound get most of it from one another, so
// their items keep that limit, but for a few tiles: 128 queries, 5,000
// references, k = 10 and 100 74 and 1,484 / 56 and 668 us, 11.5 million, k = 40
// all tiles 975, a sixteenth 650 us.
template <int KMAX, int QT, bool Claim>
__device__ __forceinline__ WarmUp warm_up(int ntiles, int K1, int64_t rows, bool share) {
  constexpr int kRanked = kRankedMax<KMAX, QT>;
  if constexpr (kRanked == 0) {
    const int fine = (K1 + 3) / 4;
    return ntiles >= 2 * K1 ? WarmUp{K1, false, false} : WarmUp{ntiles < fine ? 0 : fine, true, false};
  }
  const int need = (K1 * QT + 1) / 2;
  const bool wide = K1 > 32, pairs = need > kRanked;
  const int want = !wide      ? max(K1, 16)
                   : pairs    ? K1 / 2
                   : KMAX > 0 ? 8 * K1
                              : max(16, 3 * K1 * (int)min(rows, int64_t(32)) / 32);
  const int tiles =
      min(want, share ? max(ntiles / (Claim || !wide || pairs ? 4 : 16), min(ntiles, wide ? 16 : 8)) : ntiles);
  const int ranks = pairs ? (need + 1) / 2 : need;
  const bool octets = 4 * tiles < 2 * ranks;
  return {(octets ? 16 : 4) * tiles < ranks ? 0 : tiles, octets, pairs};
}

// The four octets' least (pairs: second-least) values, or the one of all 32.
__device__ __forceinline__ void group_values(const uint32_t (&v)[32], bool octets, bool pairs, int32_t (&y)[4]) {
  int32_t a[4], b[4];
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    a[o] = (int32_t)v[8 * o];
    b[o] = INT32_MAX;
#pragma unroll
    for (int i = 1; i < 8; ++i) {
      const int32_t x = (int32_t)v[8 * o + i];
      b[o] = min(b[o], max(a[o], x));
      a[o] = min(a[o], x);
    }
    y[o] = pairs ? b[o] : a[o];
  }
  if (octets) return;
#pragma unroll
  for (int o = 1; o < 4; ++o) {
    b[0] = min(min(b[0], b[o]), max(a[0], a[o]));
    a[0] = min(a[0], a[o]);
  }
  y[0] = pairs ? b[0] : a[0];
}

// Shared memory of the hand-over between epilogue and inserter warps.
struct HandOver {
  static constexpr uint32_t kGiven = 0;                     // hand-overs made, per epilogue warp (8)
  static constexpr uint32_t kDone = kGiven + 8 * 4;         // hand-overs merged, per epilogue warp
  static constexpr uint32_t kCount = kDone + 8 * 4;         // candidates handed over, per epilogue thread (256)
  static constexpr uint32_t kWarm = kCount + 256 * 4;       // warm-up bound, per epilogue thread
  static constexpr uint32_t kLim = kWarm + 256 * 4;         // limit, per query row (256)
  static constexpr uint32_t kBytes = kLim + 256 * 4;
  uint32_t base;
  __device__ uint32_t given(uint32_t w) const { return base + kGiven + 4 * w; }
  __device__ uint32_t done(uint32_t w) const { return base + kDone + 4 * w; }
  __device__ uint32_t count(uint32_t t) const { return base + kCount + 4 * t; }
  __device__ uint32_t warm(uint32_t t) const { return base + kWarm + 4 * t; }
  __device__ uint32_t lim(uint32_t row) const { return base + kLim + 4 * row; }
};

// The epilogue warps' side: each thread collects its row's candidates, eight
// neighbouring columns at a time: what is in the epilogue's path is then one
// compare and three predicated stores per octet, and the columns are sorted
// out by the inserters, whose 32 lanes each have a row's to sort.
struct Collector {
  HandOver ho;
  uint32_t w, lane;         // epilogue warp, half * 4 + quarter
  uint32_t lim_at;          // its row's limit in shared memory
  const char* mine;         // this thread's two buffers of `cap` entries
  uint32_t cap;
  uint32_t soft;            // entries worth a merge if the inserter is free
  volatile uint32_t* abort_flag;
  uint32_t* dev_err;
  const char* start;        // the buffer being filled
  uint32_t n = 0;           // entries in it
  uint32_t given = 0;       // hand-overs made
  int32_t lim = INT32_MIN;  // a column enters below it (bit pattern)
  __device__ __forceinline__ void read_limit() { lim = (int32_t)ld_shared_u32(lim_at); }
  // Hands the warp's buffers over and goes on with the other ones, once the
  // hand-over before has been merged (without `wait`: only if it has): a vote,
  // since each lane loads the inserter's word for itself and full-mask
  // operations follow.  False when the CTA gives up.
  __device__ __forceinline__ bool hand_over(bool wait) {
    if (!__all_sync(0xffffffffu, ld_shared_acquire(ho.done(w)) == given)) {
      if (!wait) return true;
      const uint64_t t0 = globaltimer_ns();
      for (uint32_t it = 1; !__all_sync(0xffffffffu, ld_shared_acquire(ho.done(w)) == given); ++it) {
        if ((it & 63u) == 0 && __any_sync(0xffffffffu, *abort_flag != 0u || globaltimer_ns() - t0 > kWaitLimitNs)) {
          flag_timeout(abort_flag, dev_err);
          n = 0;  // (the candidates are lost: the call reports the timeout)
          return false;
        }
        __nanosleep(40);  // (the inserters need the issue slots)
      }
    }
    st_shared_u32(ho.count(w * 32 + lane), n);
    __threadfence_block();
    __syncwarp();
    ++given;
    if (lane == 0) st_shared_release(ho.given(w), given);
    start = mine + (given & 1u) * cap * kTcEntryBytes;
    n = 0;
    read_limit();
    return true;
  }
  // 32 columns, some below some row's limit.
  __device__ __forceinline__ void group(const uint32_t (&v)[32], uint32_t col) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const uint32_t* x = v + 8 * o;
      const int32_t a = __vimin3_s32((int32_t)x[0], (int32_t)x[1], (int32_t)x[2]);
      const int32_t b = __vimin3_s32((int32_t)x[3], (int32_t)x[4], (int32_t)x[5]);
      const int32_t c = __vimin3_s32(a, (int32_t)x[6], (int32_t)x[7]);
      push_octet_if_less(start, n, min(b, c), lim, x, col + 8u * o);
    }
  }
  // Two 32-column groups with their minima (mn, from the reducing TMEM load).
  __device__ __forceinline__ void round(const uint32_t (&v0)[32], uint32_t mn0, const uint32_t (&v1)[32], uint32_t mn1,
                                        int64_t col0) {
    if (!__any_sync(0xffffffffu, (int32_t)min(mn0, mn1) < lim)) return;
    // the limit is read again only here, where it matters (a read per tile cost
    // the FP8 pass 4%)
    read_limit();
    if (__any_sync(0xffffffffu, n + 8 > cap)) hand_over(true);
    if (__any_sync(0xffffffffu, (int32_t)mn0 < lim)) group(v0, (uint32_t)col0);
    if (__any_sync(0xffffffffu, (int32_t)mn1 < lim)) group(v1, (uint32_t)col0 + 32u);
    if (__any_sync(0xffffffffu, n >= soft)) hand_over(false);
  }
};

// The inserter warps' side: warp `quarter` has the 32 rows of its TMEM lane
// quarter (QT = 2: of each query tile); lane l holds the state of row l.
template <int KMAX, int QT>
struct Inserter {
  // Lists of up to 64 keys are a thread's registers, and a hand-over's
  // candidates go in one per row and step: a step is a network of 6 KMAX
  // instructions for 32 rows.  Longer ones are in global memory (merge_rows).
  static constexpr bool kRegs = KMAX > 0;
  RegList<kRegs ? KMAX : 0> L[QT];
  HandOver ho;
  uint32_t quarter, lane;
  int K1, cap;
  char* cand;              // this CTA's candidate buffers: [256 epilogue threads][2][cap] entries
  uint32_t done0 = 0, done1 = 0;  // hand-overs merged of the quarter's two epilogue warps
  uint64_t* list[QT];      // the lists of the 32 rows: K1 keys each
  const uint64_t* seed[QT];  // the lists they start from, or null
  uint32_t listed[QT];     // rows whose list has been written
  int32_t kth[QT];         // the list's K1-th distance (INT32_MAX: not full)
  int32_t shared[QT];      // the row's shared bound as last read
  int32_t lim[QT];         // min(kth, shared) + 1; INT32_MIN: no row here
  int32_t* rthr[QT];       // the row's shared bound, or null
  __device__ __forceinline__ void post_limit(int q) {
    if (lim[q] != INT32_MIN) lim[q] = min(kth[q], shared[q]) + 1;  // at the bound a column may still win on its row
    st_shared_u32(ho.lim(q * kBM + quarter * 32 + lane), (uint32_t)lim[q]);
  }
  // Merges what the epilogue warp of half h has handed over; false if nothing.
  __device__ __forceinline__ bool take(int h, bool publish) {
    const uint32_t w = (uint32_t)h * 4 + quarter;
    const int q = QT == 2 ? h : 0;
    const uint32_t done = h == 0 ? done0 : done1;
    // one answer for the warp, whose lanes each load the word the epilogue changes
    if (!__all_sync(0xffffffffu, ld_shared_acquire(ho.given(w)) != done)) return false;
    const int n = (int)ld_shared_u32(ho.count(w * 32 + lane));
    uint32_t* from =
        reinterpret_cast<uint32_t*>(cand) + ((int64_t)w * 64 + (done & 1u)) * cap * kEntryWords;
    const int stride = 2 * cap * kEntryWords;
    if constexpr (kRegs) {
      insert_all(L[q], from + lane * stride, n, lim[q]);
      kth[q] = L[q].worst();
    } else {
      const int keys = pack(from + lane * stride, n, lim[q]);
      const uint32_t rows = __ballot_sync(0xffffffffu, keys > 0);
      const uint64_t* packed = reinterpret_cast<const uint64_t*>(from);
      if (K1 <= 128) {
        kth[q] = merge_rows<4>(packed, stride / 2, keys, list[q], seed[q], rows, listed[q], K1, kth[q]);
      } else {
        kth[q] = merge_rows<8>(packed, stride / 2, keys, list[q], seed[q], rows, listed[q], K1, kth[q]);
      }
      listed[q] |= rows;
    }
    if (publish && rthr[q] && kth[q] < shared[q]) {
      atomicMin(rthr[q], kth[q]);
      shared[q] = kth[q];
    }
    post_limit(q);
    if (h == 0) done0 = done + 1;
    else done1 = done + 1;
    __syncwarp();
    if (lane == 0) st_shared_release(ho.done(w), done + 1);
    return true;
  }
  // Brings a lane's n entries into L1 (about 1,000 cycles for each one alone,
  // from L2 while the operands stream); returns the warp's largest n.
  __device__ __forceinline__ int fetch(const uint32_t* from, int n) const {
    const int most = (int)__reduce_max_sync(0xffffffffu, (uint32_t)n);
#pragma unroll 1
    for (int e = 0; e < most; e += 4) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (e + i < n) {
          prefetch_l1(from + (e + i) * kEntryWords);
          prefetch_l1(from + (e + i) * kEntryWords + 8);
        }
      }
    }
    return most;
  }
  // The columns below `limit` of a lane's n entries into its list: each step
  // takes the least column left of every lane's entry.  The next entry is
  // loaded meanwhile.
  template <class List>
  __device__ __forceinline__ void insert_all(List& list, const uint32_t* from, int n, int32_t limit) const {
    const int most = fetch(from, n);
    uint4 a = make_uint4(0, 0, 0, 0), b = a;
    uint32_t col = 0;
    if (n > 0) {
      a = ld_global_v4(from);
      b = ld_global_v4(from + 4);
      col = ld_global_u32(from + 8);
    }
#pragma unroll 1
    for (int e = 0; e < most; ++e) {
      int32_t v[8] = {(int32_t)a.x, (int32_t)a.y, (int32_t)a.z, (int32_t)a.w,
                      (int32_t)b.x, (int32_t)b.y, (int32_t)b.z, (int32_t)b.w};
      const uint32_t c = col;
      const int32_t bound = e < n ? limit : INT32_MIN;
      if (e + 1 < n) {
        const uint32_t* p = from + (e + 1) * kEntryWords;
        a = ld_global_v4(p);
        b = ld_global_v4(p + 4);
        col = ld_global_u32(p + 8);
      }
#pragma unroll 1
      for (;;) {
        const int32_t m = min(__vimin3_s32(__vimin3_s32(v[0], v[1], v[2]), v[3], v[4]), __vimin3_s32(v[5], v[6], v[7]));
        const bool in = m < bound && m <= list.worst();
        if (!__any_sync(0xffffffffu, in)) break;
        uint32_t j = 0;
#pragma unroll
        for (int i = 7; i >= 0; --i)
          if (v[i] == m) j = (uint32_t)i;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (j == (uint32_t)i) v[i] = INT32_MAX;
        list.insert(in ? m : INT32_MAX, in ? c + j : 0xFFFFFFFFu);
      }
    }
  }
  // The columns below `limit` of a lane's n entries, packed in place (an entry
  // takes as many bytes as eight pairs): (column, distance bits) pairs, as many
  // as returned.
  __device__ __forceinline__ int pack(uint32_t* from, int n, int32_t limit) const {
    const int most = fetch(from, n);
    uint64_t* at = reinterpret_cast<uint64_t*>(from);
    uint64_t* const first = at;
    uint4 a = make_uint4(0, 0, 0, 0), b = a;
    uint32_t col = 0;
    if (n > 0) {
      a = ld_global_v4(from);
      b = ld_global_v4(from + 4);
      col = ld_global_u32(from + 8);
    }
#pragma unroll 1
    for (int e = 0; e < most; ++e) {
      const uint32_t v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
      const uint32_t c = col;
      const int32_t bound = e < n ? limit : INT32_MIN;
      if (e + 1 < n) {
        const uint32_t* p = from + (e + 1) * kEntryWords;
        a = ld_global_v4(p);
        b = ld_global_v4(p + 4);
        col = ld_global_u32(p + 8);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) push_global_if_less(at, (int32_t)v[i], bound, c + (uint32_t)i);
    }
    __syncwarp();
    return (int)(at - first);
  }
  // The rows' shared bounds, read again.
  __device__ __forceinline__ void read_bounds() {
#pragma unroll
    for (int q = 0; q < QT; ++q) {
      const int32_t b = rthr[q] ? min(shared[q], __ldcg(rthr[q])) : shared[q];
      if (b != shared[q]) {
        shared[q] = b;
        post_limit(q);
      }
    }
  }
  // Writes the rows' lists (those in global memory: of the rows that had no
  // candidate).
  __device__ __forceinline__ void finish(int q, uint32_t n_rows) {
    if constexpr (kRegs) {
      if (lane < n_rows) L[q].store(list[q] + lane * K1, K1);
      return;
    }
#pragma unroll 1
    for (uint32_t r = 0; r < n_rows; ++r) {
      if ((listed[q] >> r) & 1u) continue;
      for (int e = (int)lane; e < K1; e += 32)
        list[q][r * K1 + e] = seed[q] ? __ldcg(seed[q] + r * K1 + e) : kEmptyKey;
    }
  }
};

// KMAX: the longest list (16, 24, 32 or 64 keys; 0: up to 256).
template <int KMAX_>
struct KnnEpilogue {
  static constexpr int KMAX = KMAX_;
  static constexpr int kInserterWarps = 4;
  static constexpr bool kClaimsChunks = true;  // can keep its lists across claimed reference chunks
  static constexpr uint32_t kListBytes = HandOver::kBytes;
};

// NBNN epilogue (Alg. 1's NN_C for every class C): the columns are the
// class-sorted references; each thread keeps the minimum over the current
// class and, when the class ends, folds it into mins[row][class] with an
// atomic minimum (other column slices and splits see other parts of the
// class).  All lanes of a warp see the same columns, so the class bookkeeping
// is uniform across the warp.
struct NbnnEpilogue {
  static constexpr int KMAX = 0;
  static constexpr int kInserterWarps = 0;
  static constexpr bool kClaimsChunks = false;
  static constexpr uint32_t kListBytes = 0;
  int32_t* dst;          // mins + row * C
  const int64_t* class_off;
  int64_t n_ref;
  int32_t C;
  int32_t cls;           // class of the current column
  int64_t next;          // first row of the next class
  int32_t run;           // float bits of the running minimum over cls
  bool active;
  __device__ __forceinline__ NbnnEpilogue(const ScanOut& o, int64_t row, bool act, int64_t j_begin)
      : dst(o.mins + (act ? row : 0) * (int64_t)o.C), class_off(o.class_off), n_ref(o.class_off[o.C]), C(o.C),
        run(INT32_MAX), active(act) {
    // class of j_begin: the last c with class_off[c] <= j_begin
    int32_t lo = 0, hi = C;
    while (lo + 1 < hi) {
      const int32_t mid = (lo + hi) >> 1;
      if (class_off[mid] <= j_begin) lo = mid; else hi = mid;
    }
    cls = lo;
    next = class_off[cls + 1];
  }
  __device__ __forceinline__ void flush() {
    if (active && run != INT32_MAX) atomicMin(dst + cls, __float2int_rn(__int_as_float(run)));
    run = INT32_MAX;
  }
  __device__ __forceinline__ void group(const uint32_t (&v)[32], uint32_t mn, int64_t col0) {
    if (col0 + 32 <= next) {  // the whole group lies in class cls
      run = min(run, (int32_t)mn);
      return;
    }
#pragma unroll 1
    for (int j = 0; j < 32; ++j) {
      const int64_t col = col0 + j;
      if (col >= n_ref) return;  // padding rows past the last class
      while (col >= next) {      // class boundaries (empty classes skipped)
        flush();
        ++cls;
        next = class_off[cls + 1];
      }
      run = min(run, select32(v, j));
    }
  }
  __device__ __forceinline__ void round(const uint32_t (&v0)[32], uint32_t mn0, const uint32_t (&v1)[32], uint32_t mn1,
                                        int64_t col0) {
    group(v0, mn0, col0);
    group(v1, mn1, col0 + 32);
  }
  __device__ __forceinline__ void finish() { flush(); }
};

// The work of one launch: T query-tile groups (QT query tiles each) x S
// reference splits = n_items items; item w is group w % T of split w / T
// (split-major, so the CTAs that run at the same time scan the same split and
// L2 serves its tiles to all of them).  queue == null: one CTA per item,
// item = blockIdx.x.  Otherwise a persistent grid: each CTA's producer takes
// the next item from *queue (zero at launch) with an atomic add and hands it
// to the CTA's other roles through a two-slot ring in shared memory; no CTA
// ever waits for another.
struct Work {
  int64_t T;
  int64_t n_items;
  int64_t split_len;
  uint32_t* queue;
  // 0: work items are (query-tile group, reference split) pairs.  > 0 (the
  // claimed-chunk form, persistent): `group` CTAs serve each query-tile
  // group, CTA c the group c / group; each keeps that group's query tiles
  // and its lists for the whole launch and claims reference chunks of
  // split_len rows, in increasing order, from the group's counter
  // queue[c / group]; n_items is then the number of chunks.
  int group;
  // Query rows of each TMEM lane quarter: 32, or for a launch of at most
  // kSpreadRows a quarter of them each, since a quarter's rows have one inserter
  // warp.  Only in the instantiations that such launches have (it cost the others
  // up to 1%: NBNN, the FP8 pass of large batches).  Its 32 lanes
  // hold consecutive operand rows either way, and lanes past the quarter's rows
  // are inactive.  FP8 shortlist 100, 1.5 million references, 16, 32, 64 and 96
  // rows, 32 to a quarter / spread: 602, 922, 956 and 998 / 349, 454, 645 and 841 us;
  // 2,000 references, k = 100, 32 rows 618 / 259 us.
  int quarter;
};
constexpr int64_t kSpreadRows = 96;
template <class Epilogue, bool Claim>
constexpr bool kSpreads = Epilogue::kInserterWarps > 0 && (Claim || Epilogue::KMAX == kTcWideRegListMax);

// Claim: the claimed-chunk form (Work::group > 0), a separate instantiation
// so that the split form's kernels carry none of its code.
template <class Fmt, class Epilogue, int QT, bool Claim>
__global__ void __launch_bounds__(kThreadsOf<Epilogue>, 1)
    tc_scan_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_qe,
                   const __grid_constant__ CUtensorMap tmap_r, const __grid_constant__ CUtensorMap tmap_re, int64_t m,
                   int64_t n_ref, Work work, ScanOut out, uint32_t* __restrict__ dev_err,
                   unsigned long long* __restrict__ stats) {
  using Sh = Shape<QT>;
  constexpr int KC = Fmt::kChunks;
  constexpr int kTileN = Sh::kTileN;
  using L = LayoutOf<Fmt, Epilogue, QT>;
  constexpr int kStages = L::kStages;
  // The epilogue learns that a tile's MMAs are done from the commit that
  // frees the tile's last ring stage: that stage is not reused within
  // two tiles (its next phase then needs this tile's accumulator back, so a
  // parity wait cannot miss a phase); a separate accumulator-full commit per
  // tile cost the MMA thread 2-10% of a step.
  static_assert(kStages >= 2 * KC, "the ring holds two tiles");
  constexpr bool kAsync = Epilogue::kInserterWarps > 0;  // lists kept by inserter warps
  const int quarter_rows = kSpreads<Epilogue, Claim> ? work.quarter : 32;
  constexpr int kListWarps = 4;                        // inserter warps
  constexpr int kEpiPerQuarter = kEpiWarps / 4;
  constexpr int kEpiCols = kAccCols / kEpiPerQuarter;  // accumulator columns per epilogue warp
  constexpr int kRounds = kEpiCols / 64;               // rounds of two 32-column loads per tile
  static_assert(KC <= kKChunks, "the query tile fits the chunks shared memory is laid out for");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const Bars<kStages> bars{sbase + L::kOffBar};
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kOffMisc);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  volatile uint32_t* stale_slot = tmem_slot + 2;
  volatile int64_t* item_slot = reinterpret_cast<volatile int64_t*>(smem + L::kOffMisc + 16);
  volatile uint32_t* chain_broken = reinterpret_cast<volatile uint32_t*>(smem + L::kOffMisc + 32);
  volatile int32_t* work_slot = reinterpret_cast<volatile int32_t*>(smem + L::kOffMisc + 40);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const bool persistent = work.queue != nullptr;
  // MMA issuers: one thread per query tile (warp 1, and for QT = 2 the warp
  // after the epilogue warps), each issuing its tile's MMAs into its half of
  // the accumulator, so that no single thread issues all of a step's MMAs.
  constexpr int kIssuers = QT;
  constexpr int kSecondIssuerWarp = 2;
  const bool issuer = warp == 1 || (kIssuers == 2 && warp == kSecondIssuerWarp);
  if (threadIdx.x == 0) {
    // read by one thread: another CTA may report a timeout meanwhile, and the
    // roles (and lanes) of this one have to agree on what they scan
    const uint32_t reported = *reinterpret_cast<volatile uint32_t*>(dev_err);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bars.full(s), 1);
      mbar_init(bars.empty(s), kIssuers);  // the MMA completions that free the stage
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bars.tempty(b), kEpiWarps);  // one arrival per epilogue warp
      mbar_init(bars.ifull(b), 1);
      // the MMA threads, each epilogue warp and (but for claimed chunks) inserter warp
      mbar_init(bars.iempty(b), kIssuers + kEpiWarps + (kAsync && !Claim ? kListWarps : 0));
    }
    mbar_init(bars.afull(), 1);
    mbar_init(bars.aempty(), kIssuers);
    mbar_init(bars.drain(), kIssuers);
    mbar_init(bars.lists_done(), kListWarps);
    mbar_init(bars.warmed(), kEpiWarps);
    mbar_init(bars.limits(), kListWarps);
    mbar_init(bars.queued(), kEpiWarps);
    *abort_flag = 0u;
    *stale_slot = reported & kDevErrTimeout;
    chain_broken[0] = chain_broken[1] = 0u;
    fence_barrier_init();
  }
  if constexpr (kAsync) {
    if (threadIdx.x < 16) st_shared_u32(sbase + L::kOffList + HandOver::kGiven + 4 * threadIdx.x, 0u);  // given, done
    if (threadIdx.x == 0) {
      *work_slot = acquire_slot(out);
      if (*work_slot < 0) flag_timeout(abort_flag, dev_err);
    }
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // Item i of this CTA for the MMA and epilogue roles (the producer publishes
  // it in the persistent form); n_items means no more work.
  auto consume_item = [&](int i, int64_t* w) -> bool {
    if (!persistent) {
      *w = i == 0 ? (int64_t)blockIdx.x : work.n_items;
      return true;
    }
    const int slot = i & 1;
    if (!mbar_wait(bars.ifull(slot), (uint32_t)((i >> 1) & 1), kWaitLimitNs, abort_flag)) return false;
    *w = item_slot[slot];
    return true;
  };
  static_assert(!Claim || (QT == 1 && Epilogue::kClaimsChunks), "the claimed-chunk form: one query tile per CTA, kNN lists");
  constexpr bool chunked = Claim;
  // (after a timeout reported earlier and not yet collected by lnbnn_sync, no
  // tiles are scanned: every item's lists are still written, empty; the
  // inserters, whose registers are short, need not know)
  auto scanned_tiles = [&](int ntiles) -> int { return *stale_slot != 0u ? 0 : ntiles; };
  auto item_tiles = [&](int64_t w, int64_t* m0, int64_t* j_begin) -> int {
    const int64_t x = chunked ? (int64_t)blockIdx.x / work.group : w % work.T;
    const int64_t y = chunked ? w : w / work.T;
    *m0 = x * (int64_t)(kBM * QT);
    *j_begin = y * work.split_len;
    const int64_t j_end = min(*j_begin + work.split_len, n_ref);
    return (int)((j_end - *j_begin + kTileN - 1) / kTileN);
  };
  // The tiles run twice at the start of this CTA's item i: none where the
  // lists go on from the previous chunk or split.
  auto warm_tiles = [&](int i, int64_t w, int64_t m0, int ntiles) -> WarmUp {
    if (!kAsync || (Claim && i > 0) || (!Claim && out.done != nullptr && w >= work.T)) return WarmUp{0, false, false};
    return warm_up<Epilogue::KMAX, QT, Claim>(ntiles, out.K1, min(m - m0, (int64_t)quarter_rows), out.bound_per_tile && out.row_thr != nullptr);
  };

  if (warp < kEpiWarp0) {
    if constexpr (kWideLists<Epilogue, QT>) reg_dealloc<kRegsFirst>();
    if (warp == 0) {
      if (lane == 0) {
        // ------------------------------------------------------------ producer
        // an optional start gate; with nothing loaded the other roles' waits
        // run out on the abort flag
        bool go = true;
        if (out.gate != nullptr && *stale_slot == 0u && !wait_gate(out.gate, kWaitLimitNs, abort_flag)) {
          flag_timeout(abort_flag, dev_err);
          go = false;
        }
        prefetch_tmap(&tmap_q);
        prefetch_tmap(&tmap_qe);
        prefetch_tmap(&tmap_r);
        prefetch_tmap(&tmap_re);
        int it = 0;       // reference K-chunks issued
        int a_loads = 0;  // query tiles issued
        for (int i = 0; go; ++i) {
          int64_t w;
          if (persistent) {
            const int slot = i & 1;
            if (i >= 2 && !mbar_wait(bars.iempty(slot), (uint32_t)(((i >> 1) - 1) & 1), kWaitLimitNs, abort_flag)) {
              flag_timeout(abort_flag, dev_err);
              break;
            }
            w = *abort_flag ? work.n_items
                            : (int64_t)atomicAdd(work.queue + (chunked ? blockIdx.x / work.group : 0u), 1u);
            if (w > work.n_items) w = work.n_items;
            item_slot[slot] = w;
            mbar_arrive(bars.ifull(slot));
          } else {
            w = i == 0 ? (int64_t)blockIdx.x : work.n_items;
          }
          if (w >= work.n_items) break;
          int64_t m0, j_begin;
          const int ntiles = scanned_tiles(item_tiles(w, &m0, &j_begin));
          // the query tiles: once the previous item's MMAs have read theirs (in
          // the claimed-chunk form, once for the whole launch)
          if (!chunked || a_loads == 0) {
            if (a_loads > 0 && !mbar_wait(bars.aempty(), (uint32_t)((a_loads - 1) & 1), kWaitLimitNs, abort_flag)) {
              flag_timeout(abort_flag, dev_err);
              break;
            }
            mbar_arrive_expect_tx(bars.afull(), QT * (KC * kAChunkBytes + kAExtBytes));
            for (int q = 0; q < QT; ++q) {
              const uint32_t a = sbase + L::kOffA + q * L::kAQueryBytes;
              const int boxes = quarter_rows < 32 ? 4 : 1;  // (of 32 rows each, or one of 128)
              for (int b = 0; b < boxes; ++b) {
                const int32_t qrow = (int32_t)(m0 + q * kBM) + b * quarter_rows;
                for (int kc = 0; kc < KC; ++kc)
                  tma_load_2d(a + kc * kAChunkBytes + b * (kAChunkBytes / 4), &tmap_q, kc * kBK, qrow, bars.afull());
                tma_load_2d(a + KC * kAChunkBytes + b * (kAExtBytes / 4), &tmap_qe, 0, qrow, bars.afull());
              }
            }
            ++a_loads;
          }
          bool ok = true;
          const int warm = warm_tiles(i, w, m0, ntiles).tiles;
          for (int t = -warm; ok && t < ntiles && !*abort_flag; ++t) {
            const int32_t row = (int32_t)(j_begin + (int64_t)(t < 0 ? t + warm : t) * kTileN);
            for (int kc = 0; kc < KC; ++kc, ++it) {
              const int s = it % kStages;
              const uint32_t round = (uint32_t)(it / kStages);
              if (!mbar_wait(bars.empty(s), (round & 1u) ^ 1u, kWaitLimitNs, abort_flag)) {
                flag_timeout(abort_flag, dev_err);
                ok = false;
                break;
              }
              const uint32_t dst = sbase + L::kOffB + s * Sh::kStageBytes;
              const bool last = kc == KC - 1;
              mbar_arrive_expect_tx(bars.full(s), Sh::kBChunkBytes + (last ? Sh::kBExtBytes : 0u));
              tma_load_2d(dst, &tmap_r, kc * kBK, row, bars.full(s));
              if (last) tma_load_2d(dst + Sh::kBChunkBytes, &tmap_re, 0, row, bars.full(s));
            }
          }
          if (!ok || *abort_flag) break;
        }
        // every load issued must land before the CTA may exit
        const uint32_t never = 0;
        if (a_loads > 0) mbar_wait(bars.afull(), (uint32_t)((a_loads - 1) & 1), kWaitLimitNs, &never);
        for (int s = 0; s < kStages; ++s) {
          const int issued = it / kStages + (s < it % kStages ? 1 : 0);
          if (issued > 0) mbar_wait(bars.full(s), (uint32_t)((issued - 1) & 1), kWaitLimitNs, &never);
        }
      }
    } else if (issuer) {
      if (lane == 0) {
        // --------------------------------------------------------- MMA issuers
        const int q_first = kIssuers == QT ? (warp == 1 ? 0 : 1) : 0;  // this thread's query tiles
        const int q_last = kIssuers == QT ? q_first + 1 : QT;
        const long long clk0 = clock64();
        const uint64_t ns0 = globaltimer_ns();
        int it = 0;       // reference K-chunks consumed
        int tg = 0;       // tiles over all items (accumulator use)
        int64_t tiles_done = 0;
        bool ok = true;
        for (int i = 0; ok; ++i) {
          int64_t w;
          if (!consume_item(i, &w)) {
            flag_timeout(abort_flag, dev_err);
            break;
          }
          if (w >= work.n_items) break;
          int64_t m0, j_begin;
          int ntiles = scanned_tiles(item_tiles(w, &m0, &j_begin));
          ntiles += warm_tiles(i, w, m0, ntiles).tiles;
          if ((!chunked || i == 0) && !mbar_wait(bars.afull(), (uint32_t)(i & 1), kWaitLimitNs, abort_flag)) {
            flag_timeout(abort_flag, dev_err);
            break;
          }
          tc_fence_after();
          // no abort-flag read per tile here: shared-memory loads are slow on
          // this thread while the MMAs stream their operands (the per-tile
          // read cost 2% of the FP8 pass), and a role that gives up stops
          // completing barriers, so the next wait below sees the flag
          for (int t = 0; ok && t < ntiles; ++t, ++tg) {
            const int b = tg & 1;
            const uint32_t use = (uint32_t)(tg >> 1);
            if (!mbar_wait(bars.tempty(b), (use & 1u) ^ 1u, kWaitLimitNs, abort_flag)) {
              flag_timeout(abort_flag, dev_err);
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + b * kAccCols;
            for (int kc = 0; kc < KC; ++kc, ++it) {
              const int s = it % kStages;
              const uint32_t round = (uint32_t)(it / kStages);
              if (!mbar_wait(bars.full(s), round & 1u, kWaitLimitNs, abort_flag)) {
                flag_timeout(abort_flag, dev_err);
                ok = false;
                break;
              }
              tc_fence_after();
              // descriptors are built once per stage and advanced by adding the
              // byte offset >> 4 to their start-address field (14 bits of
              // addr >> 4; every shared address is below 256 KB, so the sum
              // never carries out of the field): the MMA thread's issue loop is
              // on the critical path of the N = 128 shape, which issues twice
              // as many MMAs per step
              const uint32_t b_base = sbase + L::kOffB + s * Sh::kStageBytes;
              const uint64_t b_desc = sw128_kmajor_desc(b_base);
              const uint64_t b_ext = sw32_kmajor_desc(b_base + Sh::kBChunkBytes);
              const bool last = kc == KC - 1;  // the norms' K-extension rides with the last chunk
  #pragma unroll
              for (int q = 0; q < QT; ++q) {
                if (q < q_first || q >= q_last) continue;
                const uint32_t a_q = sbase + L::kOffA + q * L::kAQueryBytes;
                const uint64_t a_desc = sw128_kmajor_desc(a_q) + (uint64_t)((kc * kAChunkBytes) >> 4);
                const uint64_t a_ext = sw32_kmajor_desc(a_q + KC * kAChunkBytes);
                const uint32_t d_q = d_tmem + q * kTileN;
                if (Fmt::kExtFirst && last) mma_bf16(d_q, a_ext, b_ext, idesc_bf16_f32(kBM, kTileN), kc != 0 ? 1u : 0u);
  #pragma unroll
                for (int kk = 0; kk < kMmaPerChunk; ++kk)  // K-steps of 32 bytes
                  Fmt::template mma<kTileN>(d_q, a_desc + (uint64_t)(2 * kk), b_desc + (uint64_t)(2 * kk),
                                            (kc | kk) != 0 || (Fmt::kExtFirst && last) ? 1u : 0u);
                if (!Fmt::kExtFirst && last) mma_bf16(d_q, a_ext, b_ext, idesc_bf16_f32(kBM, kTileN), 1u);
              }
              mma_commit(bars.empty(s));  // the producer may refill this stage
            }
          }
          tiles_done += ntiles;
          if (!chunked) mma_commit(bars.aempty());  // the query tiles may be replaced once these MMAs are done
          if (persistent) mbar_arrive(bars.iempty(i & 1));
        }
        // all MMAs issued by this thread must finish before TMEM is released
        const uint32_t never = 0;
        mma_commit(bars.drain());
        mbar_wait(bars.drain(), 0, kWaitLimitNs, &never);
        if (stats && warp == 1) {
          atomicAdd(stats + 0, (unsigned long long)(clock64() - clk0));
          atomicAdd(stats + 1, (unsigned long long)(globaltimer_ns() - ns0));
          atomicAdd(stats + 2, (unsigned long long)tiles_done);
          atomicAdd(stats + 3, 1ull);
        }
      }
    }
  } else if (warp < kInsWarp0) {
    // ------------------------------------------------------------- epilogue
    const int quarter = warp & 3;               // this warp may read TMEM lanes [32*quarter, 32*quarter+32)
    const int half = (warp - kEpiWarp0) >> 2;   // QT = 1: its column half of every tile; QT = 2: its query tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    int tg = 0;
    const uint32_t taddr0 = tmem_base + lane_addr + half * kEpiCols;
    // tile tg's MMAs are done (one answer for the warp: its lanes stay
    // together when a wait runs out)
    auto wait_tile = [&]() -> bool {
      const int itl = tg * KC + KC - 1;  // the tile's last K-chunk
      const bool done = __all_sync(
          0xffffffffu,
          mbar_wait(bars.empty(itl % kStages), (uint32_t)(itl / kStages) & 1u, kWaitLimitNs, abort_flag));
      if (!done) flag_timeout(abort_flag, dev_err);
      tc_fence_after();
      return done;
    };
    // the accumulator goes back: every lane's loads are complete; one arrival
    // per warp after a warp barrier (256 single-thread arrivals on one barrier,
    // while the MMAs read their operands from shared memory, delayed the
    // accumulator's return by ~100 cycles a step)
    auto release_tile = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bars.tempty(tg & 1));
    };
    // the tiles of one work item into the lists of `e`; false if a wait ran out
    auto scan_tiles = [&](auto& e, int ntiles, int64_t col_base) -> bool {
      for (int t = 0; t < ntiles; ++t, ++tg) {
        if (!wait_tile()) return false;
        // rounds of 64 columns; the accumulator goes back as soon as the last
        // round is in registers.  With inserter warps the rounds are one copy of
        // the code (see merge_rows on the instruction cache).
        const uint32_t taddr = taddr0 + (tg & 1) * kAccCols;
        const int64_t col0 = col_base + (int64_t)t * kTileN;
#pragma unroll (kAsync ? 1 : kRounds)
        for (int r = 0; r < kRounds; ++r) {
          uint32_t v0[32], v1[32], mn0, mn1;
          tmem_ld_min_32x32b_x32(taddr + 64 * r, v0, mn0);
          tmem_ld_min_32x32b_x32(taddr + 64 * r + 32, v1, mn1);
          tmem_ld_wait(v0, mn0);
          reg_fence(v1);
          asm volatile("" : "+r"(mn1));
          if (r == kRounds - 1) release_tile();
          e.round(v0, mn0, v1, mn1, col0 + 64 * r);
        }
      }
      return true;
    };
    // one work item after another (or claimed chunk after claimed chunk)
    const int64_t c_off = QT == 2 ? 0 : half * kEpiCols;  // this warp's first column within a tile
    const HandOver ho{sbase + L::kOffList};
    const uint32_t t = (uint32_t)(half * kBM + quarter * 32 + lane);
    Collector e;
    if constexpr (kAsync) {
      e.ho = ho;
      e.w = (uint32_t)(warp - kEpiWarp0);
      e.lane = (uint32_t)lane;
      e.lim_at = ho.lim(QT == 2 ? t : t & 127u);
      e.cap = (uint32_t)out.entries;
      e.mine = out.work + max(*work_slot, 0) * tc_work_bytes(out.entries) + (int64_t)t * 2 * out.entries * kTcEntryBytes;
      e.start = e.mine;
      e.soft = (uint32_t)min(out.K1 < 8 ? 2 : 8, out.entries - 8);
      e.abort_flag = abort_flag;
      e.dev_err = dev_err;
    }
    int i = 0;
    for (;; ++i) {
      int64_t w;
      if (!__all_sync(0xffffffffu, consume_item(i, &w))) {
        flag_timeout(abort_flag, dev_err);
        break;
      }
      if (w >= work.n_items) break;
      int64_t m0, j_begin;
      const int ntiles = scanned_tiles(item_tiles(w, &m0, &j_begin));
      if constexpr (kAsync) {
        if (!Claim || i == 0) {
          const WarmUp wu = warm_tiles(i, w, m0, ntiles);
          // the least minima, sorted, behind slots that nothing displaces
          constexpr int kRanked = kRankedMax<Epilogue::KMAX, QT>;
          const int need = (out.K1 * QT + 1) / 2, ranks = wu.pairs ? (need + 1) / 2 : need;
          int32_t ranked[kRanked > 0 ? kRanked : 1];
#pragma unroll
          for (int j = 0; j < kRanked; ++j) ranked[j] = j < kRanked - ranks ? INT32_MIN : INT32_MAX;
          int32_t most = wu.tiles > 0 ? INT32_MIN : INT32_MAX;
          bool ok = true;
          for (int u = 0; u < wu.tiles; ++u, ++tg) {
            if (!(ok = wait_tile())) break;
            const uint32_t taddr = taddr0 + (tg & 1) * kAccCols;
            int32_t least = INT32_MAX;
#pragma unroll 1
            for (int c = 0; c < kEpiCols; c += 32) {
              uint32_t v[32], mn;
              tmem_ld_min_32x32b_x32(taddr + c, v, mn);
              tmem_ld_wait(v, mn);
              if constexpr (kRanked > 0) {
                int32_t y[4] = {(int32_t)mn, INT32_MAX, INT32_MAX, INT32_MAX};
                if (wu.octets || wu.pairs) group_values(v, wu.octets, wu.pairs, y);
                int left = wu.octets ? 4 : 1;
#pragma unroll 1
                do {
                  const int32_t x = y[0];
                  y[0] = y[1];
                  y[1] = y[2];
                  y[2] = y[3];
#pragma unroll
                  for (int j = kRanked - 1; j > 0; --j) ranked[j] = max(ranked[j - 1], min(ranked[j], x));
                  ranked[0] = min(ranked[0], x);
                } while (--left > 0);
              } else {
                if (wu.octets) most = max(most, (int32_t)mn);
                least = min(least, (int32_t)mn);
              }
            }
            release_tile();
            if (kRanked == 0 && !wu.octets) most = max(most, least);
          }
          if (kRanked > 0 && wu.tiles > 0) most = ranked[kRanked - 1];
          if (!ok) break;
          st_shared_u32(ho.warm(t), (uint32_t)most);
          __syncwarp();
          if (lane == 0) mbar_arrive(bars.warmed());
          if (!__all_sync(0xffffffffu, mbar_wait(bars.limits(), (uint32_t)(i & 1), kWaitLimitNs, abort_flag))) {
            flag_timeout(abort_flag, dev_err);
            break;
          }
          e.read_limit();
        }
        if (!scan_tiles(e, ntiles, j_begin + c_off)) break;
        if (!Claim) {
          if (!e.hand_over(true)) break;
          if (lane == 0) mbar_arrive(bars.queued());
        }
      } else {
        const int64_t row = m0 + (QT == 2 ? half * kBM : 0) + quarter * 32 + lane;
        Epilogue epi(out, row, row < m, j_begin + c_off);
        const bool ok = scan_tiles(epi, ntiles, j_begin + c_off);
        epi.finish();
        if (!ok) break;
      }
      if (persistent) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.iempty(i & 1));
      }
    }
    if constexpr (kAsync && Claim) {
      if (i == 0) {  // no chunk was left for this CTA
        st_shared_u32(ho.warm(t), (uint32_t)INT32_MAX);
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.warmed());
      }
      if (e.hand_over(true) && lane == 0) mbar_arrive(bars.queued());
    }
  } else {
    if constexpr (kAsync) {
      // ----------------------------------------------------------- inserters
      if constexpr (kWideLists<Epilogue, QT>) reg_alloc<kRegsInserter>();
      const uint32_t quarter = (uint32_t)(warp & 3);
      Inserter<Epilogue::KMAX, QT> ins;
      ins.ho = HandOver{sbase + L::kOffList};
      ins.quarter = quarter;
      ins.lane = (uint32_t)lane;
      ins.K1 = out.K1;
      ins.cap = out.entries;
      ins.cand = out.work + max(*work_slot, 0) * tc_work_bytes(out.entries);
      const bool share = out.bound_per_tile && out.row_thr != nullptr;
      // one list per row and split (claimed chunks: per row and CTA of the group)
      for (int i = 0; !Claim || i == 0; ++i) {
        int64_t w = 0;
        if (!Claim) {
          if (!__all_sync(0xffffffffu, consume_item(i, &w))) {
            flag_timeout(abort_flag, dev_err);
            break;
          }
          if (w >= work.n_items) break;
        }
        int64_t m0, j_begin;
        item_tiles(w, &m0, &j_begin);
        const int64_t y = Claim ? (int64_t)(blockIdx.x % (unsigned)work.group) : w / work.T;
        // the previous split of these rows, if it has finished: start from its
        // list.  Its flag says 2 when every earlier split of the rows was
        // carried into it; a warp that cannot say the same of this item marks
        // the item's slot (cleared by the thread that publishes the slot's
        // previous item before that item's slot is released)
        const bool chain = !Claim && out.done != nullptr;
        const uint32_t prev = chain && y > 0 ? ld_acquire_gpu(out.done + (w - out.T)) : 0u;
        const bool carried = __all_sync(0xffffffffu, prev != 0u);
        if (chain && y > 0 && !__all_sync(0xffffffffu, prev == 2u) && lane == 0) chain_broken[i & 1] = 1u;
        bool ok = __all_sync(0xffffffffu, mbar_wait(bars.warmed(), (uint32_t)(i & 1), kWaitLimitNs, abort_flag));
        if (!ok) flag_timeout(abort_flag, dev_err);  // (the lists are written all the same, empty)
#pragma unroll
        for (int q = 0; q < QT; ++q) {
          const int64_t first = m0 + q * kBM + quarter * quarter_rows, row = first + lane;
          const bool active = lane < quarter_rows && row < m;
          ins.list[q] = out.lists + (y * out.stride + first) * out.K1;
          ins.seed[q] = carried ? ins.list[q] - out.stride * out.K1 : nullptr;
          ins.listed[q] = 0u;
          ins.kth[q] = INT32_MAX;
          if constexpr (ins.kRegs) {
            ins.L[q].init(out.K1);
            if (carried && active) ins.L[q].seed(ins.seed[q] + lane * out.K1, out.K1);
            ins.kth[q] = ins.L[q].worst();
          } else if (carried && active) {
            const uint64_t k = __ldcg(ins.seed[q] + lane * out.K1 + out.K1 - 1);
            if (k != kEmptyKey) ins.kth[q] = dist_bits(key_dist(k));
          }
          ins.rthr[q] = active && out.row_thr ? out.row_thr + row : nullptr;
          const uint32_t t = (uint32_t)(q * kBM) + quarter * 32 + (uint32_t)lane;
          int32_t bound = (int32_t)ld_shared_u32(ins.ho.warm(t));
          if (QT == 1) bound = max(bound, (int32_t)ld_shared_u32(ins.ho.warm(t + kBM)));
          ins.shared[q] = ins.rthr[q] ? min(__ldcg(ins.rthr[q]), kRealBound) : kRealBound;
          if (bound < ins.shared[q]) {
            ins.shared[q] = bound;
            if (share && ins.rthr[q]) atomicMin(ins.rthr[q], bound);
          }
          ins.lim[q] = active ? 0 : INT32_MIN;
          ins.post_limit(q);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bars.limits());
        const uint64_t t0 = globaltimer_ns();
        uint32_t nap = 100;  // ns between polls: longer while nothing comes (polls every 100 ns cost the FP8 pass 5%)
        for (uint32_t it = 0; ok; ++it) {
          const bool last = __all_sync(0xffffffffu, mbar_test(bars.queued(), (uint32_t)(i & 1)));
          bool took = false;
          if constexpr (QT == 1) {  // one copy of the code
#pragma unroll 1
            for (int h = 0; h < 2; ++h) took |= ins.take(h, share);
          } else {
            took = ins.take(0, share);
            took |= ins.take(1, share);
          }
          if (share) ins.read_bounds();
          if (took) {
            nap = 100;
            continue;
          }
          if (last) break;
          const bool over = (it & 255u) == 0 && globaltimer_ns() - t0 > kItemLimitNs;
          if (__any_sync(0xffffffffu, *abort_flag != 0u || over)) {
            flag_timeout(abort_flag, dev_err);
            ok = false;
            break;
          }
          __nanosleep(nap);
          nap = min(2 * nap, 1600u);
        }
#pragma unroll
        for (int q = 0; q < QT; ++q) {
          const int64_t left = m - (m0 + q * kBM + quarter * quarter_rows);
          ins.finish(q, (uint32_t)max(int64_t(0), min(left, (int64_t)quarter_rows)));
          if (ins.rthr[q] && !out.bound_per_tile && ins.kth[q] < ins.shared[q]) atomicMin(ins.rthr[q], ins.kth[q]);
        }
        if (chain) {
          // the item's lists are complete once every inserter warp has written
          // its rows' lists; one thread then marks the item done: 2 if its
          // lists hold every earlier split's keys (each split of the rows
          // started from the one before), else 1 (if the wait runs out nothing
          // is marked and a later split simply starts empty)
          __threadfence();
          __syncwarp();
          if (lane == 0) mbar_arrive(bars.lists_done());
          if (warp == kInsWarp0 && lane == 0 && ok &&
              mbar_wait(bars.lists_done(), (uint32_t)(i & 1), kWaitLimitNs, abort_flag)) {
            const uint32_t flag = chain_broken[i & 1] != 0u ? 1u : 2u;
            chain_broken[i & 1] = 0u;
            __threadfence();
            st_release_gpu(out.done + w, flag);
          }
        }
        if (!ok) break;
        if (persistent && !Claim) {
          __syncwarp();
          if (lane == 0) mbar_arrive(bars.iempty(i & 1));
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
  if constexpr (kAsync) {
    if (threadIdx.x == 0) release_slot(out, *work_slot);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// BF16 [rows, cols] row-major, boxes of box_cols x box_rows with the given swizzle.
bool encode_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint32_t cols, uint32_t box_cols,
                 uint32_t box_rows, CUtensorMapSwizzle swizzle) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estride[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// E4M3 bytes [rows, 128] row-major, boxes of 128 x box_rows, 128-byte swizzle.
bool encode_e4m3(CUtensorMap* map, const void* base, uint64_t rows, uint32_t box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t gdim[2] = {(cuuint64_t)kDim, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {(cuuint64_t)kDim};
  cuuint32_t box[2] = {(cuuint32_t)kDim, box_rows};
  cuuint32_t estride[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), gdim, gstride, box, estride,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Main operand (128 K-columns, 64-column boxes, 128-byte swizzle) and its
// 16-column K-extension (32-byte swizzle).
bool encode_operand(CUtensorMap* main, CUtensorMap* ext, const void* bf, const void* ext_base, uint64_t rows,
                    uint32_t box_rows) {
  return encode_bf16(main, bf, rows, kDim, kBK, box_rows, CU_TENSOR_MAP_SWIZZLE_128B) &&
         encode_bf16(ext, ext_base, rows, kExt, kExt, box_rows, CU_TENSOR_MAP_SWIZZLE_32B);
}

}  // namespace

bool make_tc_tensor_maps(const __nv_bfloat16* ref_bf, const __nv_bfloat16* sref_bf, const __nv_bfloat16* ref_ext,
                         const __nv_bfloat16* sref_ext, int64_t n_pad, TcTensorMaps* out) {
  return encode_operand(&out->ref, &out->ref_ext, ref_bf, ref_ext, (uint64_t)n_pad, Shape<1>::kTileN) &&
         encode_operand(&out->sref, &out->sref_ext, sref_bf, sref_ext, (uint64_t)n_pad, Shape<1>::kTileN) &&
         encode_operand(&out->ref_h, &out->ref_ext_h, ref_bf, ref_ext, (uint64_t)n_pad, Shape<2>::kTileN) &&
         encode_operand(&out->sref_h, &out->sref_ext_h, sref_bf, sref_ext, (uint64_t)n_pad, Shape<2>::kTileN);
}

bool make_tc_tensor_maps_e4m3(const uint8_t* ref_f8, const __nv_bfloat16* ref_f8_ext, int64_t n_pad,
                              TcTensorMaps* out) {
  return encode_e4m3(&out->f8, ref_f8, (uint64_t)n_pad, Shape<1>::kTileN) &&
         encode_bf16(&out->f8_ext, ref_f8_ext, (uint64_t)n_pad, kExt, kExt, Shape<1>::kTileN,
                     CU_TENSOR_MAP_SWIZZLE_32B) &&
         encode_e4m3(&out->f8_h, ref_f8, (uint64_t)n_pad, Shape<2>::kTileN) &&
         encode_bf16(&out->f8_ext_h, ref_f8_ext, (uint64_t)n_pad, kExt, kExt, Shape<2>::kTileN,
                     CU_TENSOR_MAP_SWIZZLE_32B);
}

namespace {

template <class Fmt, class Epilogue, int QT>
cudaError_t launch_scan(const CUtensorMap& tr, const CUtensorMap& tre, const void* qop,
                        const __nv_bfloat16* qext, int64_t m, int64_t m_pad, int64_t n_ref, int splits,
                        int64_t split_len, const ScanOut& out, uint32_t* dev_err, unsigned long long* stats,
                        const TcSched& sched, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  if (m_pad % kBM != 0 || split_len % kTcRefTile != 0 || splits < 1) return cudaErrorInvalidValue;
  if (sched.persistent_ctas > 0 && sched.queue == nullptr) return cudaErrorInvalidValue;
  CUtensorMap tq, tqe;
  const bool spread = (sched.group > 0 ? kSpreads<Epilogue, true> : kSpreads<Epilogue, false>) && m <= kSpreadRows;
  const uint32_t box = spread ? 32 : kBM;
  const bool ok = Fmt::kChunks == 1
                      ? encode_e4m3(&tq, qop, (uint64_t)m_pad, box) &&
                            encode_bf16(&tqe, qext, (uint64_t)m_pad, kExt, kExt, box, CU_TENSOR_MAP_SWIZZLE_32B)
                      : encode_operand(&tq, &tqe, qop, qext, (uint64_t)m_pad, box);
  if (!ok) return cudaErrorInvalidValue;
  Work work;
  work.T = (m_pad + kBM * QT - 1) / (kBM * QT);
  work.n_items = work.T * splits;
  work.split_len = split_len;
  work.queue = sched.persistent_ctas > 0 ? sched.queue : nullptr;
  work.group = 0;
  work.quarter = spread ? (int)((m + 3) / 4) : 32;
  ScanOut o = out;
  o.done = splits > 1 ? sched.done : nullptr;
  o.T = work.T;
  int64_t grid = work.queue ? std::min<int64_t>(work.n_items, sched.persistent_ctas) : work.n_items;
  if (sched.group > 0) {
    // the claimed-chunk form: `splits` is the CTAs per query-tile group (the
    // lists' "split" index is the CTA's rank), split_len the chunk length
    if (!Epilogue::kClaimsChunks || sched.queue == nullptr || o.done != nullptr || sched.group != splits)
      return cudaErrorInvalidValue;
    work.group = sched.group;
    work.queue = sched.queue;
    work.n_items = (n_ref + split_len - 1) / split_len;
    grid = work.T * sched.group;
  }
  if (work.n_items > (int64_t)INT32_MAX || grid > (int64_t)INT32_MAX) return cudaErrorInvalidValue;
  if (Epilogue::kInserterWarps > 0) {
    if (sched.work == nullptr || sched.work_slots < 1 || sched.entries < kTcMinEntries || (grid > sched.work_slots && sched.slot_used == nullptr))
      return cudaErrorInvalidValue;
    o.work = sched.work;
    o.work_slots = sched.work_slots;
    o.entries = sched.entries;
    o.slot_used = grid > sched.work_slots ? sched.slot_used : nullptr;
  }
  if constexpr (QT == 1 && Epilogue::kClaimsChunks) {
    if (work.group > 0) {
      tc_scan_kernel<Fmt, Epilogue, QT, true>
          <<<(unsigned)grid, kThreadsOf<Epilogue>, LayoutOf<Fmt, Epilogue, QT>::kSmemBytes,
             s>>>(tq, tqe, tr, tre, m, n_ref, work, o, dev_err, stats);
      return cudaGetLastError();
    }
  }
  if (work.group > 0) return cudaErrorInvalidValue;
  tc_scan_kernel<Fmt, Epilogue, QT, false>
      <<<(unsigned)grid, kThreadsOf<Epilogue>, LayoutOf<Fmt, Epilogue, QT>::kSmemBytes, s>>>(
          tq, tqe, tr, tre, m, n_ref, work, o, dev_err, stats);
  return cudaGetLastError();
}

template <class Fmt, class Epilogue, int QT, bool Claim>
cudaError_t prepare_kernel() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, tc_scan_kernel<Fmt, Epilogue, QT, Claim>);
  if (e != cudaSuccess) return e;
  if (a.numRegs > kMaxRegsOf<Epilogue>) return cudaErrorInvalidKernelImage;
  // the register split counts on what the launch has
  if (kWideLists<Epilogue, QT> && a.numRegs != kRegsLaunch) return cudaErrorInvalidKernelImage;
  return cudaFuncSetAttribute(tc_scan_kernel<Fmt, Epilogue, QT, Claim>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)LayoutOf<Fmt, Epilogue, QT>::kSmemBytes);
}

template <class Fmt, class Epilogue, int QT>
cudaError_t prepare_one() {
  cudaError_t e = prepare_kernel<Fmt, Epilogue, QT, false>();
  if constexpr (QT == 1 && Epilogue::kClaimsChunks) {
    if (e == cudaSuccess) e = prepare_kernel<Fmt, Epilogue, QT, true>();
  }
  return e;
}

// Lists of 33..64 keys run with one query tile per CTA only.
template <class Epilogue>
constexpr bool kTwoQueryTiles = Epilogue::KMAX <= kTcCoarseRegListMax;

// One list kind's kernel for the tile shape the schedule asks for.
template <class Fmt, class Epilogue>
cudaError_t launch_shape(const TcTensorMaps& maps, bool sorted_copy, const void* qop, const __nv_bfloat16* qext,
                         int64_t m, int64_t m_pad, int64_t n_ref, int splits, int64_t split_len, const ScanOut& out,
                         uint32_t* dev_err, unsigned long long* stats, const TcSched& sched, cudaStream_t s) {
  constexpr bool coarse = Fmt::kChunks == 1;
  if constexpr (kTwoQueryTiles<Epilogue>) {
    if (sched.qt == 2) {
      const CUtensorMap& tr = coarse ? maps.f8_h : (sorted_copy ? maps.sref_h : maps.ref_h);
      const CUtensorMap& tre = coarse ? maps.f8_ext_h : (sorted_copy ? maps.sref_ext_h : maps.ref_ext_h);
      return launch_scan<Fmt, Epilogue, 2>(tr, tre, qop, qext, m, m_pad, n_ref, splits, split_len, out, dev_err,
                                           stats, sched, s);
    }
  }
  if (sched.qt != 1) return cudaErrorInvalidValue;
  const CUtensorMap& tr = coarse ? maps.f8 : (sorted_copy ? maps.sref : maps.ref);
  const CUtensorMap& tre = coarse ? maps.f8_ext : (sorted_copy ? maps.sref_ext : maps.ref_ext);
  return launch_scan<Fmt, Epilogue, 1>(tr, tre, qop, qext, m, m_pad, n_ref, splits, split_len, out, dev_err, stats,
                                       sched, s);
}

template <class Fmt, class Epilogue>
cudaError_t prepare_both() {
  cudaError_t e = prepare_one<Fmt, Epilogue, 1>();
  if constexpr (kTwoQueryTiles<Epilogue>) {
    if (e == cudaSuccess) e = prepare_one<Fmt, Epilogue, 2>();
  }
  return e;
}

// The kNN scan with the instantiation for K1.
template <class Fmt>
cudaError_t launch_lists(const TcTensorMaps& maps, bool sorted_copy, const void* qop, const __nv_bfloat16* qext,
                         int64_t m, int64_t m_pad, int64_t n_ref, int splits, int64_t split_len, int K1,
                         const ScanOut& out, uint32_t* dev_err, unsigned long long* stats, const TcSched& sched,
                         cudaStream_t s) {
  switch (tc_list_max(K1, m)) {
    case kTcRegListMax:
      return launch_shape<Fmt, KnnEpilogue<kTcRegListMax>>(maps, sorted_copy, qop, qext, m, m_pad, n_ref, splits,
                                                           split_len, out, dev_err, stats, sched, s);
    case kTcMidRegListMax:
      return launch_shape<Fmt, KnnEpilogue<kTcMidRegListMax>>(maps, sorted_copy, qop, qext, m, m_pad, n_ref, splits,
                                                              split_len, out, dev_err, stats, sched, s);
    case kTcCoarseRegListMax:
      return launch_shape<Fmt, KnnEpilogue<kTcCoarseRegListMax>>(maps, sorted_copy, qop, qext, m, m_pad, n_ref,
                                                                 splits, split_len, out, dev_err, stats, sched, s);
    case kTcWideRegListMax:
      return launch_shape<Fmt, KnnEpilogue<kTcWideRegListMax>>(maps, sorted_copy, qop, qext, m, m_pad, n_ref, splits,
                                                               split_len, out, dev_err, stats, sched, s);
    default:
      return launch_shape<Fmt, KnnEpilogue<0>>(maps, sorted_copy, qop, qext, m, m_pad, n_ref, splits, split_len, out,
                                               dev_err, stats, sched, s);
  }
}

}  // namespace

cudaError_t prepare_tc_kernels() {
  cudaError_t e = prepare_both<FmtBf16, KnnEpilogue<kTcRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtBf16, KnnEpilogue<kTcMidRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtE4m3, KnnEpilogue<kTcMidRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtBf16, KnnEpilogue<kTcCoarseRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtBf16, KnnEpilogue<kTcWideRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtBf16, KnnEpilogue<0>>();
  if (e == cudaSuccess) e = prepare_both<FmtBf16, NbnnEpilogue>();
  if (e == cudaSuccess) e = prepare_both<FmtE4m3, KnnEpilogue<kTcRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtE4m3, KnnEpilogue<kTcCoarseRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtE4m3, KnnEpilogue<kTcWideRegListMax>>();
  if (e == cudaSuccess) e = prepare_both<FmtE4m3, KnnEpilogue<0>>();
  return e;
}

cudaError_t launch_knn_tc(const TcTensorMaps& maps, bool sorted_copy, const __nv_bfloat16* qbf,
                          const __nv_bfloat16* qext, int64_t m, int64_t m_pad, int64_t n_ref, int splits,
                          int64_t split_len, int K1, uint64_t* lists, int64_t stride, int32_t* row_thr,
                          uint32_t* dev_err, unsigned long long* stats, const uint32_t* gate, const TcSched& sched,
                          cudaStream_t s) {
  ScanOut out{};
  out.gate = gate;
  out.row_thr = row_thr;
  out.bound_per_tile = sched.bound_per_tile;
  out.lists = lists;
  out.stride = stride;
  out.K1 = K1;
  return launch_lists<FmtBf16>(maps, sorted_copy, qbf, qext, m, m_pad, n_ref, splits, split_len, K1, out, dev_err,
                               stats, sched, s);
}

cudaError_t launch_coarse_tc(const TcTensorMaps& maps, const uint8_t* qf8, const __nv_bfloat16* qext,
                             int64_t m, int64_t m_pad, int64_t n_ref, int splits, int64_t split_len, int K1,
                             uint64_t* lists, int64_t stride, int32_t* row_thr, uint32_t* dev_err,
                             unsigned long long* stats, const uint32_t* gate, const TcSched& sched, cudaStream_t s) {
  ScanOut out{};
  out.gate = gate;
  out.row_thr = row_thr;
  out.bound_per_tile = sched.bound_per_tile;
  out.lists = lists;
  out.stride = stride;
  out.K1 = K1;
  return launch_lists<FmtE4m3>(maps, false, qf8, qext, m, m_pad, n_ref, splits, split_len, K1, out, dev_err, stats,
                               sched, s);
}

cudaError_t launch_nbnn_tc(const TcTensorMaps& maps, const __nv_bfloat16* qbf, const __nv_bfloat16* qext, int64_t m,
                           int64_t m_pad, int64_t n_ref, int splits, int64_t split_len, int32_t* mins, int32_t C,
                           const int64_t* class_off, uint32_t* dev_err, unsigned long long* stats,
                           const uint32_t* gate, const TcSched& sched, cudaStream_t s) {
  ScanOut out{};
  out.gate = gate;
  out.mins = mins;
  out.C = C;
  out.class_off = class_off;
  return launch_shape<FmtBf16, NbnnEpilogue>(maps, true, qbf, qext, m, m_pad, n_ref, splits, split_len, out, dev_err,
                                             stats, sched, s);
}

}  // namespace lnbnn
