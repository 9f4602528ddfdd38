// NBNN as a sum of log-odds increments (Section 3.1): each query descriptor d
// changes the log-odds of every class C by
//
//   inc(d, C) = log [P(C|d) P(Cbar)] / [P(Cbar|d) P(C)]            Eq. (eqn:log-odds)
//
// with equal priors P(C) = 1/|classes| and the posterior of the NBNN Gaussian
// kernel on each class's nearest neighbour, P(C|d) ~ exp(-beta D_C),
// D_C = ||d - NN_C(d)||^2, beta = 1/(2 sigma^2).  The image goes to the class
// with the largest sum (Eq. (eqn:log-increments)); the "positive increments
// only" variant (Table 1) adds only increments > 0.
//
// Written without the normalisation, which cancels:
//   inc(d, C) = -beta D_C - log sum_{C' != C} exp(-beta D_C') + log(|classes| - 1).
// Shifting by the row minimum Dmin keeps every exponential <= 1 and the sums
// >= 1, so nothing underflows into a log(0):
//   * C not the unique nearest class: with x = beta (D_C - Dmin) and
//     S = sum_C' exp(-beta (D_C' - Dmin)) >= 1 + exp(-x),
//       inc = -x - log(S - exp(-x)) + log(|classes| - 1);
//   * C the unique nearest class, D2 the second smallest distance and
//     S2 = sum_{C' != C} exp(-beta (D_C' - D2)) >= 1,
//       inc = beta (D2 - Dmin) - log S2 + log(|classes| - 1).
// All of it is float64.  The input is the [m, C] table of NN_C distances that
// the tensor-core scan of the class-sorted references fills for Alg. 1.
//
// Blocks take chunks of rows, not whole images: one block per image and 128
// classes left most SMs idle (8 images of the 101-class data: 8 blocks, 4.1 ms
// of a 6.2 ms call; float64 runs at about two multiply-adds a cycle and SM).  A
// chunk is 8 rows from the image's first, so the sums do not depend on what
// else is in the batch.  Up to kTableClasses classes a block finds its rows'
// statistics, keeps exp(-x) of every class in shared memory for the sums (one
// exponential and one logarithm per row and class in all), and adds its rows'
// increments in row order.  With more classes a chunk is too much for a block
// and its table too large: the statistics are a launch of a warp per row, and a
// block takes a chunk and 256 classes (one block for a whole image, as long as
// the chunks' sums had to be in shared memory, took 88 ms for 1,000 rows and
// 4,097 classes).
#include <math.h>

#include <algorithm>

#include "internal.cuh"

namespace lnbnn {
namespace {

constexpr int kChunk = 8;            // rows of a chunk; an image's last one takes its remainder too
constexpr int kThreads = 256;        // of a block, at most
constexpr int kWarps = kThreads / 32;
constexpr int kTableClasses = 1024;  // classes up to which exp(-x) of 8 rows is kept (64 KB)

struct RowStat {
  double s;       // sum over classes of exp(-beta (D_C - Dmin)), in [1, |classes|]
  double inc;     // the increment of the unique nearest class
  int32_t dmin;   // smallest class distance of the row
  int32_t cstar;  // the unique nearest class, or -1 when two or more classes tie at Dmin
};
static_assert(sizeof(RowStat) == kLogoddsRowStatBytes, "room per row in the call's scratch");

__device__ __forceinline__ double warp_sum(double v) {
  // xor butterfly: both partners add the same two values, so every lane ends
  // with the same bits and the order is fixed
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// One warp: the statistics of a row of class minima, and exp(-x) per class
// into `table` unless null.
__device__ __forceinline__ RowStat row_stat(const int32_t* __restrict__ d, int32_t C, double beta, double log_c1,
                                            double* table) {
  const int lane = threadIdx.x & 31;
  int32_t best = INT32_MAX, bc = INT32_MAX, ties = 0, sec = INT32_MAX;  // sec: the second smallest value
  for (int32_t c = lane; c < C; c += 32) {
    const int32_t v = d[c];
    if (v < best) {
      sec = best;
      best = v;
      bc = c;
      ties = 1;
    } else if (v == best) {
      ++ties;
    } else {
      sec = min(sec, v);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const int32_t ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int32_t oc = __shfl_xor_sync(0xffffffffu, bc, off);
    const int32_t ot = __shfl_xor_sync(0xffffffffu, ties, off);
    const int32_t os = __shfl_xor_sync(0xffffffffu, sec, off);
    sec = min(min(sec, os), ob == best ? INT32_MAX : max(ob, best));
    if (ob < best) {
      best = ob;
      bc = oc;
      ties = ot;
    } else if (ob == best) {
      bc = min(bc, oc);
      ties += ot;
    }
  }
  double t = 0.0;  // all classes but bc
  for (int32_t c = lane; c < C; c += 32) {
    const double e = exp(-beta * (double)(d[c] - best));
    if (table) table[c] = e;
    if (c != bc) t += e;
  }
  t = warp_sum(t);
  RowStat r;
  r.s = 1.0 + t;
  r.dmin = best;
  r.cstar = ties == 1 ? bc : -1;
  r.inc = 0.0;
  if (ties == 1) {
    const double gap = beta * (double)(sec - best);
    if (gap < 600.0) {
      r.inc = log_c1 - log(t);
    } else {  // t underflows: relative to the second smallest distance instead
      double s2 = 0.0;
      for (int32_t c = lane; c < C; c += 32)
        if (c != bc) s2 += exp(-beta * (double)(d[c] - sec));
      r.inc = gap - log(warp_sum(s2)) + log_c1;
    }
  }
  return r;
}

// Image owning descriptor row i: the last image whose first row is <= i.
__device__ __forceinline__ int64_t image_of(const int64_t* __restrict__ offsets, int64_t n_img, int64_t i) {
  int64_t lo = 0, hi = n_img;
  while (lo + 1 < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (offsets[mid] <= i) lo = mid; else hi = mid;
  }
  return lo;
}

// Partial sums of a chunk, [C] doubles over its own rows of the table of class
// minima (8 rows take 32 C bytes), once every thread has read them.
__device__ __forceinline__ double* partials(int32_t* mins, int64_t row, int32_t C) {
  return reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(mins + row * C) + 7) & ~uintptr_t(7));
}
// Where several blocks have the classes of a chunk, the partial sum of class c
// takes the place of the class's minima in the chunk's first two rows (32 bits
// each), which only the thread that adds up class c reads.
__device__ __forceinline__ void put_partial(int32_t* mins, int64_t row, int32_t C, int32_t c, double v) {
  mins[row * C + c] = __double2loint(v);
  mins[(row + 1) * C + c] = __double2hiint(v);
}
__device__ __forceinline__ double partial(const int32_t* mins, int64_t row, int32_t C, int32_t c) {
  return __hiloint2double(mins[(row + 1) * C + c], mins[row * C + c]);
}

// The rows [r0, r1) of block b, of image img; false if it has none.  Block b <
// n_slots owns the chunk [off + 8 j, off + 8 j + 8) of the image at off that
// holds row 8 b (every chunk of 8 rows holds one such row; an image's last
// chunk, of 8 to 15 rows, belongs to the first of its two); block n_slots + i
// owns image i if it has fewer rows.  split: the image has other chunks.
__device__ __forceinline__ bool chunk_of(const int64_t* __restrict__ offsets, int64_t n_img, int64_t m, int64_t n_slots,
                                         int64_t b, int64_t* img, int64_t* r0, int64_t* r1, bool* split) {
  *split = false;
  if (b >= n_slots) {
    *img = b - n_slots;
    *r0 = max(offsets[*img], (int64_t)0);
    *r1 = min(offsets[*img + 1], m);
    return *r0 < *r1 && *r1 - *r0 < kChunk;
  }
  const int64_t p = b * kChunk;
  *img = image_of(offsets, n_img, p);
  const int64_t o0 = max(offsets[*img], (int64_t)0), o1 = min(offsets[*img + 1], m);
  if (p < o0 || p >= o1 || o1 - o0 < kChunk) return false;
  const int64_t chunks = (o1 - o0) / kChunk, j = (p - o0) / kChunk;
  if (j >= chunks) return false;  // in the remainder, which the chunk before has
  *split = chunks > 1;
  *r0 = o0 + j * kChunk;
  *r1 = j == chunks - 1 ? o1 : *r0 + kChunk;
  return true;
}

// The increment of a row with statistics t to class c, x = beta (D_c - Dmin), e = exp(-x).
__device__ __forceinline__ double increment(const RowStat& t, int32_t c, double x, double e, double log_c1) {
  return c == t.cstar ? t.inc : -x - log(t.s - e) + log_c1;
}

__device__ __forceinline__ void add_count(unsigned long long* counts, int64_t img, unsigned long long n) {
  if (!counts) return;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(counts + img, n);
}

// Up to kTableClasses classes: statistics and sums of a chunk.  kFull: kThreads
// threads (a stride known to the compiler).
template <bool kFull>
__global__ void __launch_bounds__(kThreads)
    logodds_chunk_kernel(int32_t* __restrict__ mins, int64_t m, int32_t C, double beta, double log_c1, int positive_only,
                         const int64_t* __restrict__ offsets, int64_t n_img, int64_t n_slots,
                         double* __restrict__ totals, unsigned long long* __restrict__ counts) {
  extern __shared__ double table[];           // [8][C]
  double* part = table + (int64_t)kChunk * C;  // [C], with split only
  __shared__ RowStat st[kChunk];
  int64_t img, r0, r1;
  bool split;
  if (!chunk_of(offsets, n_img, m, n_slots, blockIdx.x, &img, &r0, &r1, &split)) return;
  const int threads = kFull ? kThreads : (int)blockDim.x;
  unsigned long long n = 0;
  for (int64_t r = r0; r < r1; r += kChunk) {
    const int rows = (int)min(r1 - r, (int64_t)kChunk);
    __syncthreads();
    for (int i = threadIdx.x >> 5; i < rows; i += threads >> 5) {
      const RowStat t = row_stat(mins + (r + i) * C, C, beta, log_c1, table + (int64_t)i * C);
      if ((threadIdx.x & 31) == 0) st[i] = t;
    }
    __syncthreads();
    for (int32_t c = threadIdx.x; c < C; c += threads) {
      double* sum = split ? part + c : totals + img * C + c;
      double acc = r == r0 ? 0.0 : *sum;
#pragma unroll 4
      for (int i = 0; i < rows; ++i) {
        const double x = beta * (double)(mins[(r + i) * C + c] - st[i].dmin);
        const double inc = increment(st[i], c, x, table[(int64_t)i * C + c], log_c1);
        if (!positive_only || inc > 0.0) {
          acc += inc;
          ++n;
        }
      }
      *sum = acc;
    }
  }
  add_count(counts, img, n);
  if (split) {
    __syncthreads();  // the rows have been read
    double* out = partials(mins, r0, C);
    for (int32_t c = threadIdx.x; c < C; c += threads) out[c] = part[c];
  }
}

// More classes.  The statistics of a row by a warp:
__global__ void __launch_bounds__(kThreads)
    logodds_rowstat_kernel(const int32_t* __restrict__ mins, int64_t m, int32_t C, double beta, double log_c1,
                           RowStat* __restrict__ stat) {
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (row >= m) return;
  const RowStat t = row_stat(mins + row * C, C, beta, log_c1, nullptr);
  if ((threadIdx.x & 31) == 0) stat[row] = t;
}

// the sums of a chunk over kThreads classes:
__global__ void __launch_bounds__(kThreads)
    logodds_range_kernel(int32_t* __restrict__ mins, int64_t m, int32_t C, double beta, double log_c1, int positive_only,
                         const int64_t* __restrict__ offsets, int64_t n_img, int64_t n_slots,
                         const RowStat* __restrict__ stat, double* __restrict__ totals,
                         unsigned long long* __restrict__ counts) {
  int64_t img, r0, r1;
  bool split;
  if (!chunk_of(offsets, n_img, m, n_slots, blockIdx.x, &img, &r0, &r1, &split)) return;
  unsigned long long n = 0;
  const int32_t c = (int32_t)blockIdx.y * kThreads + threadIdx.x;
  if (c < C) {
    double acc = 0.0;
#pragma unroll 4
    for (int64_t r = r0; r < r1; ++r) {
      const double x = beta * (double)(mins[r * C + c] - stat[r].dmin);
      const double inc = increment(stat[r], c, x, exp(-x), log_c1);
      if (!positive_only || inc > 0.0) {
        acc += inc;
        ++n;
      }
    }
    if (split)
      put_partial(mins, r0, C, c, acc);
    else
      totals[img * C + c] = acc;
  }
  add_count(counts, img, n);
}

// and these sums in the chunks' order, an image and kThreads classes a block.
__global__ void __launch_bounds__(kThreads)
    logodds_total_kernel(const int32_t* __restrict__ mins, int64_t m, int32_t C, const int64_t* __restrict__ offsets,
                         double* __restrict__ totals) {
  const int64_t img = blockIdx.x;
  const int32_t c = (int32_t)blockIdx.y * kThreads + threadIdx.x;
  const int64_t o0 = max(offsets[img], (int64_t)0), o1 = min(offsets[img + 1], m);
  const int64_t chunks = o1 <= o0 ? 0 : (o1 - o0) / kChunk;
  if (c >= C || chunks < 2) return;
  double v = 0.0;
#pragma unroll 8
  for (int64_t j = 0; j < chunks; ++j) v += partial(mins, o0 + j * kChunk, C, c);
  totals[img * C + c] = v;
}

// One block per image: the chunks' sums (unless summed), then the argmax over
// classes, the lowest class on ties.  kFull: kThreads threads.
template <bool kFull>
__global__ void __launch_bounds__(kThreads)
    logodds_finish_kernel(int32_t* __restrict__ mins, int64_t m, int32_t C, const int64_t* __restrict__ offsets,
                          bool summed, double* __restrict__ totals, int32_t* __restrict__ classes) {
  __shared__ double best_s[kWarps];
  __shared__ int32_t class_s[kWarps];
  const int threads = kFull ? kThreads : (int)blockDim.x;
  const int64_t img = blockIdx.x;
  const int64_t o0 = max(offsets[img], (int64_t)0), o1 = min(offsets[img + 1], m);
  const int64_t chunks = summed || o1 <= o0 ? 0 : (o1 - o0) / kChunk;
  double best = -INFINITY;
  int32_t bc = INT32_MAX;
  for (int32_t c = threadIdx.x; c < C; c += threads) {
    double v;
    if (chunks > 1) {
      v = 0.0;
#pragma unroll 8
      for (int64_t j = 0; j < chunks; ++j) v += partials(mins, o0 + j * kChunk, C)[c];
      totals[img * C + c] = v;
    } else {
      v = totals[img * C + c];
    }
    if (v > best || bc == INT32_MAX) {  // c increases: the first maximum seen is the lowest
      best = v;
      bc = c;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, best, off);
    const int32_t oc = __shfl_xor_sync(0xffffffffu, bc, off);
    if (oc != INT32_MAX && (bc == INT32_MAX || ov > best || (ov == best && oc < bc))) {
      best = ov;
      bc = oc;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    best_s[threadIdx.x >> 5] = best;
    class_s[threadIdx.x >> 5] = bc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (threads >> 5); ++w)
      if (class_s[w] != INT32_MAX && (bc == INT32_MAX || best_s[w] > best || (best_s[w] == best && class_s[w] < bc))) {
        best = best_s[w];
        bc = class_s[w];
      }
    classes[img] = bc;
  }
}

}  // namespace

cudaError_t prepare_logodds() {
  const int bytes = (int)sizeof(double) * (kChunk + 1) * kTableClasses;
  cudaError_t e =
      cudaFuncSetAttribute(logodds_chunk_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(logodds_chunk_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

int64_t logodds_rowstat_bytes(int64_t m, int32_t C) { return C > kTableClasses ? m * kLogoddsRowStatBytes : 0; }

cudaError_t launch_logodds(int32_t* mins, void* rowstat, int64_t m, int32_t C, double beta, bool positive_only,
                           const int64_t* offsets, int64_t n_img, double* totals, int64_t* counts, int32_t* classes,
                           cudaStream_t s, int* launches) {
  *launches = 0;
  if (n_img == 0) return cudaSuccess;
  auto launched = [&]() {
    ++*launches;
    return cudaGetLastError();
  };
  const bool tabled = C <= kTableClasses;
  const double log_c1 = log((double)(C - 1));
  unsigned long long* counts_u = reinterpret_cast<unsigned long long*>(counts);
  // a thread per class and a warp per row of a chunk, of an image with fewer rows as many
  const int64_t class_warps = std::min<int64_t>((C + 31) / 32, kWarps);
  if (m > 0) {
    const int64_t n_slots = (m + kChunk - 1) / kChunk, blocks = n_slots + n_img;
    cudaError_t e;
    if (tabled) {
      const int64_t warps = std::max<int64_t>(class_warps, std::min<int64_t>((m + n_img - 1) / n_img, kWarps));
      (warps == kWarps ? logodds_chunk_kernel<true> : logodds_chunk_kernel<false>)<<<
          (unsigned)blocks, (unsigned)(32 * warps), sizeof(double) * (kChunk + 1) * (size_t)C, s>>>(
          mins, m, C, beta, log_c1, positive_only ? 1 : 0, offsets, n_img, n_slots, totals, counts_u);
      e = launched();
    } else {
      RowStat* stat = static_cast<RowStat*>(rowstat);
      // a row per block while the rows do not fill the chip that way
      const int64_t rows = std::min<int64_t>(kWarps, std::max<int64_t>(1, m / 1024));
      logodds_rowstat_kernel<<<(unsigned)((m + rows - 1) / rows), (unsigned)(32 * rows), 0, s>>>(mins, m, C, beta,
                                                                                                log_c1, stat);
      e = launched();
      if (e != cudaSuccess) return e;
      const dim3 grid((unsigned)blocks, (unsigned)((C + kThreads - 1) / kThreads));
      logodds_range_kernel<<<grid, kThreads, 0, s>>>(mins, m, C, beta, log_c1, positive_only ? 1 : 0, offsets, n_img,
                                                     n_slots, stat, totals, counts_u);
      e = launched();
      if (e != cudaSuccess) return e;
      logodds_total_kernel<<<dim3((unsigned)n_img, grid.y), kThreads, 0, s>>>(mins, m, C, offsets, totals);
      e = launched();
    }
    if (e != cudaSuccess) return e;
  }
  // (blocks of fewer threads only where there are many: see the chunks)
  const unsigned finish = n_img > 1024 ? (unsigned)(32 * class_warps) : kThreads;
  (finish == kThreads ? logodds_finish_kernel<true> : logodds_finish_kernel<false>)<<<(unsigned)n_img, finish, 0, s>>>(
      mins, m, C, offsets, !tabled || m == 0, totals, classes);
  return launched();
}

}  // namespace lnbnn
