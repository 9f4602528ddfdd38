// Split merge, knn_search output, the Local NBNN class update (Alg. 2) and the
// per-image argmin (Alg. 1 and Alg. 2, last line).
#include <algorithm>

#include "internal.cuh"

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

// Image owning descriptor row i: the last image whose first row is <= i.
__device__ __forceinline__ int64_t image_of(const int64_t* __restrict__ offsets, int64_t n_img, int64_t i) {
  int64_t lo = 0, hi = n_img;  // answer in [0, n_img)
  while (lo + 1 < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (offsets[mid] <= i) lo = mid; else hi = mid;
  }
  return lo;
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
// straight to the totals.
constexpr int kScoreWarps = 8;
constexpr int kScoreMaxRows = 128;    // rows of a block: 128 x 14,565,600 < 2^31
constexpr int kTableRows = 8;
constexpr int kTableClasses = 8192;   // classes up to which the sums fit (32 KB)
template <int G>  // ceil(k / 32) neighbours per lane, or more
__global__ void __launch_bounds__(32 * kScoreWarps)
    lnbnn_score_kernel(const uint64_t* __restrict__ lists, int64_t m, int K1, int k,
                       const int32_t* __restrict__ labels, int64_t n_ref, const int64_t* __restrict__ offsets,
                       int64_t n_img, int32_t C, int rows, bool table, int64_t* __restrict__ totals,
                       uint32_t* __restrict__ dev_err) {
  extern __shared__ int32_t sums[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long* t = reinterpret_cast<unsigned long long*>(totals);
  const int64_t row1 = min(m, ((int64_t)blockIdx.x + 1) * rows);
  for (int64_t r = (int64_t)blockIdx.x * rows; r < row1;) {  // stretches of one image (the same for the block)
    const int64_t img = image_of(offsets, n_img, r);
    const int64_t end = min(offsets[img + 1], row1);
    if (r < offsets[img] || r >= end) {  // only with invalid offsets
      if (threadIdx.x == 0) atomicOr(dev_err, kDevErrOffsets);
      ++r;
      continue;
    }
    const bool summed = table && end - r >= kTableRows;
    if (summed) {
      for (int32_t c = threadIdx.x; c < C; c += 32 * kScoreWarps) sums[c] = 0;
      __syncthreads();
    }
    for (int64_t i = r + warp; i < end; i += kScoreWarps) {
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
      if (!__all_sync(0xffffffffu, ok)) continue;
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
        if (first && delta != 0) {
          if (summed)
            atomicAdd(sums + lab[g], delta);
          else
            atomicAdd(t + img * C + lab[g], (unsigned long long)(int64_t)delta);
        }
      }
    }
    if (summed) {
      __syncthreads();
      for (int32_t c = threadIdx.x; c < C; c += 32 * kScoreWarps)
        if (sums[c] != 0) atomicAdd(t + img * C + c, (unsigned long long)(int64_t)sums[c]);
      __syncthreads();
    }
    r = end;
  }
}

// Alg. 1's sums: totals[img][c] += the sum over the image's descriptor rows of
// mins[row][c] (= NN_c of that descriptor).  A block takes 32 rows and 128
// classes, whatever the images (a block per image left most SMs idle: 20
// images, 162 us); integer addition is exact in any order.
constexpr int kSumRows = 32;
__global__ void nbnn_sum_kernel(const int32_t* __restrict__ mins, int64_t m, int32_t C,
                                const int64_t* __restrict__ offsets, int64_t n_img, int64_t* __restrict__ totals) {
  const int32_t c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const int64_t row1 = min(m, ((int64_t)blockIdx.x + 1) * kSumRows);
  for (int64_t r = (int64_t)blockIdx.x * kSumRows; r < row1;) {
    const int64_t img = image_of(offsets, n_img, r);
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

// One warp per image; lanes scan classes lane, lane+32, ...; ties -> lowest class.
__global__ void argmin_kernel(const int64_t* __restrict__ totals, int64_t n_img, int32_t C,
                              int32_t* __restrict__ classes) {
  const int64_t img = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (img >= n_img) return;
  const int64_t* t = totals + img * C;
  int64_t best = INT64_MAX;
  int32_t bc = INT32_MAX;
  for (int32_t c = lane; c < C; c += 32) {
    const int64_t v = t[c];
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
  if (lane == 0) classes[img] = bc;
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

cudaError_t launch_lnbnn_score(const uint64_t* lists, int64_t m, int K1, int k, const int32_t* labels, int64_t n_ref,
                               const int64_t* offsets, int64_t n_img, int32_t C, int64_t* totals, uint32_t* dev_err,
                               cudaStream_t s) {
  if (m == 0 || n_img == 0) return cudaSuccess;
  // a row per warp while the rows do not fill the chip that way, then more (the
  // table is written to the totals once per block)
  const int rows = (int)std::min<int64_t>(kScoreMaxRows, kScoreWarps * std::max<int64_t>(1, m / 8192));
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
  dim3 grid((unsigned)((m + kSumRows - 1) / kSumRows), (unsigned)((C + 127) / 128));
  nbnn_sum_kernel<<<grid, 128, 0, s>>>(mins, m, C, offsets, n_img, totals);
  return cudaGetLastError();
}

cudaError_t launch_argmin(const int64_t* totals, int64_t n_img, int32_t C, int32_t* classes, cudaStream_t s) {
  if (n_img == 0) return cudaSuccess;
  argmin_kernel<<<(unsigned)((n_img * 32 + 255) / 256), 256, 0, s>>>(totals, n_img, C, classes);
  return cudaGetLastError();
}

}  // namespace lnbnn
