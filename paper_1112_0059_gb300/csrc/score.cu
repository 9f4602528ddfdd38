// Split merge, knn_search output, the Local NBNN class update (Alg. 2) and the
// per-image argmin (Alg. 1 and Alg. 2, last line).
#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "sqdist.cuh"

namespace lnbnn {
namespace {

// Row i's `n_lists` partial lists live at lists[(l * stride + i) * K1]; each is
// sorted ascending.  One warp per row writes the K1 smallest keys of their
// union, ascending: lane j holds the heads of lists j, j + 32, ...; each round
// the warp minimum is written and the list that held it advances.  A key
// names one reference row; it can sit in several lists of a row when a split
// started from the previous split's list, and is written once (a key equal to
// the last one written only advances its lists).
constexpr int kMergeWarps = 4;
// Up to this many lists a thread merges a row on its own (few lists: the
// warp form would leave most lanes idle).
constexpr int kThreadMergeLists = 8;

// The first list of row i to merge: all of them, or only the last split's
// when that split's work item says its list holds every earlier split's keys
// (the scan's done flag 2).  Work item x + y T covers query rows
// [x rows_per_item, (x + 1) rows_per_item) of split y.
__device__ __forceinline__ int first_list(const MergeChain& c, int64_t i, int n_lists) {
  if (c.done == nullptr) return 0;
  const int64_t w = i / c.rows_per_item + (int64_t)(n_lists - 1) * c.T;
  return c.done[w] == 2u ? n_lists - 1 : 0;
}

__global__ void merge_lists_thread_kernel(const uint64_t* __restrict__ lists, int n_lists, int64_t m, int64_t stride,
                                          int K1, MergeChain chain, uint64_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int l0 = first_list(chain, i, n_lists);
  lists += (int64_t)l0 * stride * K1;
  n_lists -= l0;
  int pos[kThreadMergeLists];
  uint64_t head[kThreadMergeLists];
#pragma unroll
  for (int l = 0; l < kThreadMergeLists; ++l) {
    pos[l] = 0;
    head[l] = l < n_lists ? lists[((int64_t)l * stride + i) * K1] : kEmptyKey;
  }
  uint64_t last = kEmptyKey;
  for (int t = 0; t < K1;) {
    uint64_t best = head[0];
    int bl = 0;
#pragma unroll
    for (int l = 1; l < kThreadMergeLists; ++l)
      if (head[l] < best) {
        best = head[l];
        bl = l;
      }
    const bool dup = best != kEmptyKey && best == last;
    if (!dup) {
      out[i * K1 + t] = best;
      ++t;
      last = best;
    }
    if (best == kEmptyKey) continue;
#pragma unroll
    for (int l = 0; l < kThreadMergeLists; ++l)
      if (l == bl) {
        ++pos[l];
        head[l] = pos[l] < K1 ? lists[((int64_t)l * stride + i) * K1 + pos[l]] : kEmptyKey;
      }
  }
}

__global__ void __launch_bounds__(32 * kMergeWarps)
    merge_lists_kernel(const uint64_t* __restrict__ lists, int n_lists, int64_t m, int64_t stride, int K1,
                       MergeChain chain, uint64_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * kMergeWarps + (threadIdx.x >> 5);
  if (i >= m) return;
  const int l0 = first_list(chain, i, n_lists);  // the same for the whole warp (one row)
  lists += (int64_t)l0 * stride * K1;
  n_lists -= l0;
  uint64_t head[kMaxListsPerLane];
  int pos[kMaxListsPerLane];
#pragma unroll
  for (int c = 0; c < kMaxListsPerLane; ++c) {
    const int l = c * 32 + lane;
    pos[c] = 0;
    head[c] = l < n_lists ? lists[((int64_t)l * stride + i) * K1] : kEmptyKey;
  }
  uint64_t last = kEmptyKey;
  for (int t = 0; t < K1;) {
    uint64_t best = kEmptyKey;
    int bc = 0;
#pragma unroll
    for (int c = 0; c < kMaxListsPerLane; ++c)
      if (head[c] < best) {
        best = head[c];
        bc = c;
      }
    uint64_t wmin = best;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wmin = min(wmin, __shfl_xor_sync(0xffffffffu, wmin, off));
    const bool dup = wmin != kEmptyKey && wmin == last;  // warp-uniform
    if (!dup) {
      if (lane == 0) out[i * K1 + t] = wmin;
      ++t;
      last = wmin;
    }
    if (wmin != kEmptyKey && best == wmin) {
#pragma unroll
      for (int c = 0; c < kMaxListsPerLane; ++c)
        if (c == bc) {
          const int l = c * 32 + lane;
          ++pos[c];
          head[c] = pos[c] < K1 ? lists[((int64_t)l * stride + i) * K1 + pos[c]] : kEmptyKey;
        }
    }
  }
}

__global__ void extract_knn_kernel(const uint64_t* __restrict__ lists, int64_t m, int K1, int k,
                                   int32_t* __restrict__ idx, int32_t* __restrict__ dist) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * k) return;
  const int64_t i = e / k;
  const int t = (int)(e - i * k);
  const uint64_t key = lists[i * K1 + t];
  idx[e] = (int32_t)key_row(key);
  dist[e] = (int32_t)key_dist(key);
}

// Image owning descriptor row i, one of [lo, hi): the last whose first row is <= i.
__device__ __forceinline__ int64_t image_of(const int64_t* __restrict__ offsets, int64_t lo, int64_t hi, int64_t i) {
  while (lo + 1 < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (offsets[mid] <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// One warp: the class of the least total, lanes scanning classes lane, lane + 32,
// ...; ties go to the lowest class.
__device__ __forceinline__ void argmin_of(const int64_t* t, int32_t C, int32_t* cls) {
  const int lane = threadIdx.x & 31;
  int64_t best = INT64_MAX;
  int32_t bc = INT32_MAX;
  for (int32_t c = lane; c < C; c += 32) {
    const int64_t v = __ldcg(reinterpret_cast<const long long*>(t + c));
    if (v < best) {  // c increases, so the first minimum seen is the lowest
      best = v;
      bc = c;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const int64_t ov = __shfl_xor_sync(0xffffffffu, best, off);
    const int32_t oc = __shfl_xor_sync(0xffffffffu, bc, off);
    if (ov < best || (ov == best && oc < bc)) {
      best = ov;
      bc = oc;
    }
  }
  if (lane == 0) *cls = bc;
}

// Alg. 2 for one descriptor row i, given its k+1 nearest neighbours sorted by
// (distance, row): dist_B = distance of the (k+1)-th; every class found among
// the first k is updated once with dist_C - dist_B, where dist_C is the
// distance of its first (hence nearest) occurrence in the sorted list.
//
// A warp per row: lane a holds neighbours a, a + 32, ..., so the labels of a
// row are gathered at once, and __match_any_sync finds the first of each class
// (a thread per row gathered and compared k^2 / 2 of them one after another:
// k = 100, 15k rows 1.78 ms).  A block takes consecutive rows; a stretch of at
// least kTableRows of one image is summed in shared memory first (int32: the
// block's rows times the largest distance stay below 2^31), the rest goes
// straight to the totals, with a row per warp whatever its image (the rows of
// one small image at a time left most warps idle: 20,000 images of one row
// against 5,000 references, k = 10, 100 us of a call against 26 for 200 images).
constexpr int kScoreWarps = 8;
constexpr int kScoreMaxRows = 128;    // rows of a block: 128 x 14,565,600 < 2^31
constexpr int kTableRows = 8;
constexpr int kTableClasses = 8192;   // classes up to which the sums fit (32 KB)
constexpr int64_t kMaxDistance = 14565600;
static_assert(kMaxDistance == (int64_t)kDim * 255 * 255 + 2ll * LNBNN_MAX_LOCATION_WEIGHT * 255 * 255 &&
                  kScoreMaxRows * kMaxDistance <= INT32_MAX,
              "a block's sums stay within 32 bits");

// The update of rows [row0, row1) by a block: update(i, add) is called by a warp
// for row i and calls add(class, delta) from any of its lanes.
template <class Update>
__device__ __forceinline__ void sum_rows(const int64_t* offsets, int64_t n_img, int32_t C, int64_t row0, int64_t row1,
                                         bool table, int64_t* totals, uint32_t* dev_err, int32_t* sums, Update update) {
  const int warp = threadIdx.x >> 5;
  unsigned long long* t = reinterpret_cast<unsigned long long*>(totals);
  const int64_t first = image_of(offsets, 0, n_img, row0), last = image_of(offsets, first, n_img, row1 - 1);
  for (int64_t r = row0; r < row1;) {  // stretches of one image (the same for the block), or of small images
    const int64_t img = image_of(offsets, first, last + 1, r);
    const int64_t end = min(offsets[img + 1], row1);
    const bool summed = table && r >= offsets[img] && end - r >= kTableRows;
    const int64_t stop = summed ? end : min(row1, table ? r + 4 * kScoreWarps : row1);
    if (summed) {
      for (int32_t c = threadIdx.x; c < C; c += 32 * kScoreWarps) sums[c] = 0;
      __syncthreads();
    }
    for (int64_t i = r + warp; i < stop; i += kScoreWarps) {
      int64_t own = img;
      if (!summed) {
        own = image_of(offsets, first, last + 1, i);
        if (i < offsets[own] || i >= offsets[own + 1]) {  // only with invalid offsets
          if ((threadIdx.x & 31) == 0) atomicOr(dev_err, kDevErrOffsets);
          continue;
        }
      }
      update(i, [&](int32_t c, int32_t delta) {
        if (summed)
          atomicAdd(sums + c, delta);
        else
          atomicAdd(t + own * C + c, (unsigned long long)(int64_t)delta);
      });
    }
    if (summed) {
      __syncthreads();
      for (int32_t c = threadIdx.x; c < C; c += 32 * kScoreWarps)
        if (sums[c] != 0) atomicAdd(t + img * C + c, (unsigned long long)(int64_t)sums[c]);
      __syncthreads();
    }
    r = stop;
  }
}

template <int G>  // ceil(k / 32) neighbours per lane, or more
__global__ void __launch_bounds__(32 * kScoreWarps)
    lnbnn_score_kernel(const uint64_t* __restrict__ lists, int64_t m, int K1, int k,
                       const int32_t* __restrict__ labels, int64_t n_ref, const int64_t* __restrict__ offsets,
                       int64_t n_img, int32_t C, int rows, bool table, int64_t* __restrict__ totals,
                       uint32_t* __restrict__ dev_err) {
  extern __shared__ int32_t sums[];
  const int lane = threadIdx.x & 31;
  const int64_t row0 = (int64_t)blockIdx.x * rows;
  sum_rows(offsets, n_img, C, row0, min(m, row0 + rows), table, totals, dev_err, sums, [&](int64_t i, auto add) {
    const uint64_t* L = lists + i * K1;
    const uint64_t last = L[k];
    uint64_t key[G];
    int32_t lab[G];
    // A complete list holds k+1 real rows.  Only a search that gave up (a
    // timeout, reported by lnbnn_sync) leaves empty keys: skip such a row
    // rather than gather labels[] at an empty key's row.
    bool ok = (int64_t)key_row(last) < n_ref;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int a = 32 * g + lane;
      key[g] = a < k ? L[a] : last;
      ok = ok && (int64_t)key_row(key[g]) < n_ref;
    }
    if (!__all_sync(0xffffffffu, ok)) return;
#pragma unroll
    for (int g = 0; g < G; ++g) lab[g] = 32 * g + lane < k ? labels[key_row(key[g])] : -1 - lane;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      bool first = __ffs(__match_any_sync(0xffffffffu, lab[g])) - 1 == lane && lab[g] >= 0;
#pragma unroll
      for (int h = 0; h < g; ++h)
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          const int32_t other = __shfl_sync(0xffffffffu, lab[h], j);  // (every lane takes part)
          first = first && other != lab[g];
        }
      const int32_t delta = (int32_t)key_dist(key[g]) - (int32_t)key_dist(last);  // <= 0
      if (first && delta != 0) add(lab[g], delta);
    }
  });
}

// Everything after the scan in one launch, for lists of at most 32 keys: a warp
// per row merges the row's lists, reranks the shortlist by exact distances
// (kRerank), and either adds the row's Alg. 2 update (kScore) or writes its
// neighbours.  The keys stay in the lanes (lane t: the t-th smallest) from the
// merge to the end, and the first kWindow keys of every list are loaded at
// once, the next ones as the list advances.  As kernels of their own (merge,
// rerank, update, argmin) each waited for a launch and for the lists from
// memory again: whole calls took, before and after, 2,000 queries against 5,000
// rows 85 / 76 us, 5 images of 400 to 1,601 from host memory against 1.5 million
// rows 1,414 / 1,388 us, one image of 100 against 11.5 million 508 / 502 us.
//
// kScore: the last block of the launch (a counter zeroed before it) also takes
// the argmin of every image when the totals are few.
struct RowEnd {
  // merge: n_lists sorted lists of K keys, list l of row i at lists + (l * stride + i) * K
  const uint64_t* lists;
  int n_lists, K;
  int64_t stride, m;
  MergeChain chain;
  // rerank: the K1 smallest exact keys of the K shortlisted rows
  const uint8_t* q;
  const uint8_t* ref;
  int K1;
  int64_t n_ref;
  int k;
  // update
  const int32_t* labels;
  const int64_t* offsets;
  int64_t n_img;
  int32_t C;
  int rows;  // rows of a block
  bool table;
  int64_t* totals;
  uint32_t* dev_err;
  int32_t* classes;   // with counter
  uint32_t* counter;  // null: the argmin is a launch of its own
  // neighbours
  int32_t* idx;
  int32_t* dist;
};

__device__ __forceinline__ uint64_t warp_min_key(uint64_t key) {
  const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(key >> 32));
  const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0xFFFFFFFFu);
  return ((uint64_t)hi << 32) | lo;
}

// Lane t's result: the t-th smallest of the row's keys (kEmptyKey past them).
template <int kPerLane, int kWindow>
__device__ __forceinline__ uint64_t merged_key(const RowEnd& p, int64_t i) {
  const int lane = threadIdx.x & 31;
  const int l0 = first_list(p.chain, i, p.n_lists);
  const int n = p.n_lists - l0;
  const uint64_t* lists = p.lists + ((int64_t)l0 * p.stride + i) * p.K;
  if (n == 1) return lane < p.K ? lists[lane] : kEmptyKey;
  uint64_t head[kPerLane][kWindow];
  int next[kPerLane];
#pragma unroll
  for (int c = 0; c < kPerLane; ++c) {
    const int l = c * 32 + lane;
    next[c] = kWindow;
#pragma unroll
    for (int w = 0; w < kWindow; ++w)
      head[c][w] = l < n && w < p.K ? lists[(int64_t)l * p.stride * p.K + w] : kEmptyKey;
  }
  uint64_t mine = kEmptyKey, last = kEmptyKey;
  for (int t = 0; t < p.K;) {
    uint64_t best = head[0][0];
#pragma unroll
    for (int c = 1; c < kPerLane; ++c) best = min(best, head[c][0]);
    const uint64_t least = warp_min_key(best);
    if (least == kEmptyKey) break;
    if (least != last) {  // (a key can sit in several lists of a row: it counts once)
      if (lane == t) mine = least;
      ++t;
      last = least;
    }
#pragma unroll
    for (int c = 0; c < kPerLane; ++c)
      if (head[c][0] == least) {
#pragma unroll
        for (int w = 0; w + 1 < kWindow; ++w) head[c][w] = head[c][w + 1];
        head[c][kWindow - 1] =
            next[c] < p.K ? lists[(int64_t)(c * 32 + lane) * p.stride * p.K + next[c]] : kEmptyKey;
        ++next[c];
      }
  }
  return mine;
}

template <int kPerLane, int kWindow, bool kRerank, bool kScore>
__global__ void __launch_bounds__(32 * kScoreWarps) row_end_kernel(const __grid_constant__ RowEnd p) {
  extern __shared__ int32_t sums[];
  __shared__ bool last_block;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the row's K1 keys, lane by lane
  auto row_key = [&](int64_t i) -> uint64_t {
    uint64_t key = merged_key<kPerLane, kWindow>(p, i);
    if constexpr (kRerank) {
      const uint32_t j = key_row(key);
      const bool real = key != kEmptyKey && (int64_t)j < p.n_ref;
      uint4 qv[8];
      const uint4* qrow = reinterpret_cast<const uint4*>(p.q + i * kDim);
#pragma unroll
      for (int c = 0; c < 8; ++c) qv[c] = __ldg(qrow + c);
      key = real ? make_key(sqdist_u8(qv, p.ref + (int64_t)j * kDim), j) : kEmptyKey;
      uint64_t mine = kEmptyKey;
      for (int r = 0; r < p.K1; ++r) {
        const uint64_t least = warp_min_key(key);
        if (lane == r) mine = least;
        if (key == least) key = kEmptyKey;
      }
      key = mine;
    }
    return key;
  };
  const int64_t row0 = (int64_t)blockIdx.x * p.rows, row1 = min(p.m, row0 + p.rows);
  if constexpr (!kScore) {
    for (int64_t i = row0 + warp; i < row1; i += kScoreWarps) {
      const uint64_t key = row_key(i);
      if (lane < p.k) {
        p.idx[i * p.k + lane] = (int32_t)key_row(key);
        p.dist[i * p.k + lane] = (int32_t)key_dist(key);
      }
    }
  } else {
    sum_rows(p.offsets, p.n_img, p.C, row0, row1, p.table, p.totals, p.dev_err, sums, [&](int64_t i, auto add) {
      const uint64_t key = row_key(i);
      // (an incomplete list, which only a search that gave up leaves, is skipped)
      if (!__all_sync(0xffffffffu, lane > p.k || (int64_t)key_row(key) < p.n_ref)) return;
      const int32_t dist_b = (int32_t)__shfl_sync(0xffffffffu, key_dist(key), p.k);
      const int32_t lab = lane < p.k ? p.labels[key_row(key)] : -1 - lane;
      const bool first = __ffs(__match_any_sync(0xffffffffu, lab)) - 1 == lane && lab >= 0;
      const int32_t delta = (int32_t)key_dist(key) - dist_b;  // <= 0
      if (first && delta != 0) add(lab, delta);
    });
    if (p.counter == nullptr) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_block = atomicAdd(p.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    for (int64_t img = warp; img < p.n_img; img += kScoreWarps) argmin_of(p.totals + img * p.C, p.C, p.classes + img);
  }
}

// Alg. 1's sums: totals[img][c] += the sum over the image's descriptor rows of
// mins[row][c] (= NN_c of that descriptor).  A block takes up to 32 rows and
// 128 classes, whatever the images (a block per image left most SMs idle: 20
// images, 162 us).  Rows of several images are added one after another, so it
// takes no more rows than an image has on average unless there are many blocks
// anyway (20,000 images of one row: 10 classes, 32 rows 45 us, one row 13;
// 4,000 classes, images of 3 rows, whole calls of 6.72 and 6.99 ms); integer
// addition is exact in any order.
constexpr int kSumRows = 32;
constexpr int64_t kSumBlocks = 16 * 152;
__global__ void nbnn_sum_kernel(const int32_t* __restrict__ mins, int64_t m, int32_t C,
                                const int64_t* __restrict__ offsets, int64_t n_img, int rows,
                                int64_t* __restrict__ totals) {
  const int32_t c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const int64_t row0 = (int64_t)blockIdx.x * rows, row1 = min(m, row0 + rows);
  for (int64_t r = row0; r < row1;) {
    const int64_t img = image_of(offsets, 0, n_img, r);
    const int64_t end = min(offsets[img + 1], row1);
    if (r < offsets[img] || r >= end) {  // only with invalid offsets, flagged elsewhere
      ++r;
      continue;
    }
    int64_t acc = 0;
#pragma unroll 8
    for (int64_t i = r; i < end; ++i) acc += mins[i * C + c];
    atomicAdd(reinterpret_cast<unsigned long long*>(totals) + img * C + c, (unsigned long long)acc);
    r = end;
  }
}

__global__ void argmin_kernel(const int64_t* __restrict__ totals, int64_t n_img, int32_t C,
                              int32_t* __restrict__ classes) {
  const int64_t img = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (img < n_img) argmin_of(totals + img * C, C, classes + img);
}

}  // namespace

cudaError_t launch_merge_lists(const uint64_t* lists, int splits, int64_t m, int64_t stride, int K1, uint64_t* out,
                               cudaStream_t s, const MergeChain& chain) {
  if (m == 0) return cudaSuccess;
  if (splits < 1 || splits > 32 * kMaxListsPerLane) return cudaErrorInvalidValue;
  if (chain.done != nullptr && (chain.T < 1 || chain.rows_per_item < 1)) return cudaErrorInvalidValue;
  if (splits <= kThreadMergeLists) {
    merge_lists_thread_kernel<<<(unsigned)((m + 127) / 128), 128, 0, s>>>(lists, splits, m, stride, K1, chain, out);
    return cudaGetLastError();
  }
  merge_lists_kernel<<<(unsigned)((m + kMergeWarps - 1) / kMergeWarps), 32 * kMergeWarps, 0, s>>>(
      lists, splits, m, stride, K1, chain, out);
  return cudaGetLastError();
}

cudaError_t launch_extract_knn(const uint64_t* lists, int64_t m, int K1, int k, int32_t* idx, int32_t* dist,
                               cudaStream_t s) {
  const int64_t n = m * k;
  if (n == 0) return cudaSuccess;
  extract_knn_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(lists, m, K1, k, idx, dist);
  return cudaGetLastError();
}

// A row per warp while the rows do not fill the chip that way, then more (the
// sums are written to the totals once per block).
static int score_rows(int64_t m) {
  return (int)std::min<int64_t>(kScoreMaxRows, kScoreWarps * std::max<int64_t>(1, m / 8192));
}

cudaError_t launch_row_end(const RowLists& in, const RowRerank* rerank, const RowScore* score, int32_t k, int32_t* idx,
                           int32_t* dist, cudaStream_t s, bool* argmin_done) {
  if (in.m == 0) return cudaSuccess;
  if (in.K < 1 || in.K > 32 || in.n_lists < 1 || in.n_lists > 32 * kMaxListsPerLane) return cudaErrorInvalidValue;
  RowEnd p{};
  p.lists = in.lists;
  p.n_lists = in.n_lists;
  p.K = in.K;
  p.stride = in.stride;
  p.m = in.m;
  p.chain = in.chain;
  p.k = k;
  p.n_ref = in.n_ref;
  p.rows = score_rows(in.m);
  if (rerank) {
    p.q = rerank->q;
    p.ref = rerank->ref;
    p.K1 = rerank->K1;
  }
  size_t smem = 0;
  if (score) {
    p.labels = score->labels;
    p.offsets = score->offsets;
    p.n_img = score->n_img;
    p.C = score->C;
    p.table = score->C <= kTableClasses;
    p.totals = score->totals;
    p.dev_err = score->dev_err;
    p.classes = score->classes;
    // one block takes the argmin of up to 64 images x 256 classes in a few us
    // (an image's is one round trip to memory for a warp, whatever its classes:
    // 400 images x 10 classes took 20 us that way, 3 as a launch of their own)
    p.counter = score->n_img <= 64 && score->n_img * score->C <= 16384 ? score->counter : nullptr;
    if (argmin_done) *argmin_done = p.counter != nullptr;
    smem = p.table ? sizeof(int32_t) * (size_t)score->C : 0;
  } else {
    p.idx = idx;
    p.dist = dist;
  }
  const unsigned blocks = (unsigned)((in.m + p.rows - 1) / p.rows);
  auto launch = [&](auto kernel) { kernel<<<blocks, 32 * kScoreWarps, smem, s>>>(p); };
  auto pick = [&](auto per_lane, auto window) {
    constexpr int L = decltype(per_lane)::value, W = decltype(window)::value;
    if (rerank && score) launch(row_end_kernel<L, W, true, true>);
    if (rerank && !score) launch(row_end_kernel<L, W, true, false>);
    if (!rerank && score) launch(row_end_kernel<L, W, false, true>);
    if (!rerank && !score) launch(row_end_kernel<L, W, false, false>);
  };
  using std::integral_constant;
  if (in.n_lists <= 32)
    pick(integral_constant<int, 1>{}, integral_constant<int, 6>{});
  else if (in.n_lists <= 160)
    pick(integral_constant<int, 5>{}, integral_constant<int, 2>{});
  else
    pick(integral_constant<int, kMaxListsPerLane>{}, integral_constant<int, 2>{});
  return cudaGetLastError();
}

cudaError_t launch_lnbnn_score(const uint64_t* lists, int64_t m, int K1, int k, const int32_t* labels, int64_t n_ref,
                               const int64_t* offsets, int64_t n_img, int32_t C, int64_t* totals, uint32_t* dev_err,
                               cudaStream_t s) {
  if (m == 0 || n_img == 0) return cudaSuccess;
  const int rows = score_rows(m);
  const bool table = C <= kTableClasses;
  const unsigned blocks = (unsigned)((m + rows - 1) / rows);
  const size_t smem = table ? sizeof(int32_t) * (size_t)C : 0;
  auto launch = [&](auto kernel) {
    kernel<<<blocks, 32 * kScoreWarps, smem, s>>>(lists, m, K1, k, labels, n_ref, offsets, n_img, C, rows, table, totals,
                                                  dev_err);
  };
  if (k <= 32)
    launch(lnbnn_score_kernel<1>);
  else if (k <= 64)
    launch(lnbnn_score_kernel<2>);
  else if (k <= 128)
    launch(lnbnn_score_kernel<4>);
  else
    launch(lnbnn_score_kernel<8>);
  return cudaGetLastError();
}

cudaError_t launch_nbnn_sum(const int32_t* mins, int64_t m, int32_t C, const int64_t* offsets, int64_t n_img,
                            int64_t* totals, cudaStream_t s) {
  if (n_img == 0 || m == 0) return cudaSuccess;
  const int64_t ranges = (C + 127) / 128;
  const int rows =
      (int)std::min<int64_t>(kSumRows, std::max<int64_t>(1, std::max<int64_t>(m / n_img, m * ranges / kSumBlocks)));
  dim3 grid((unsigned)((m + rows - 1) / rows), (unsigned)ranges);
  nbnn_sum_kernel<<<grid, 128, 0, s>>>(mins, m, C, offsets, n_img, rows, totals);
  return cudaGetLastError();
}

cudaError_t launch_argmin(const int64_t* totals, int64_t n_img, int32_t C, int32_t* classes, cudaStream_t s) {
  if (n_img == 0) return cudaSuccess;
  argmin_kernel<<<(unsigned)((n_img * 32 + 255) / 256), 256, 0, s>>>(totals, n_img, C, classes);
  return cudaGetLastError();
}

}  // namespace lnbnn
