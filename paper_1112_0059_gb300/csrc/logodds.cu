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
// block finds its rows' statistics, keeps exp(-x) of every class in shared
// memory for the sums (one exponential and one logarithm per row and class in
// all), and adds its rows' increments in row order; a chunk is 8 rows from the
// image's first, so the sums do not depend on what else is in the batch.
#include <math.h>

#include "internal.cuh"

namespace lnbnn {
namespace {

constexpr int kChunk = 8;            // rows of a chunk; an image's last one takes its remainder too
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTableClasses = 1024;  // classes up to which exp(-x) of 8 rows is kept (64 KB)
constexpr int kPartClasses = 4096;   // classes up to which images are split into chunks

struct RowStat {
  double s;       // sum over classes of exp(-beta (D_C - Dmin)), in [1, |classes|]
  double inc;     // the increment of the unique nearest class
  int32_t dmin;   // smallest class distance of the row
  int32_t cstar;  // the unique nearest class, or -1 when two or more classes tie at Dmin
};

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
__device__ __forceinline__ double* partial(int32_t* mins, int64_t row, int32_t C) {
  return reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(mins + row * C) + 7) & ~uintptr_t(7));
}

// Block b < n_slots owns the chunk [off + 8 j, off + 8 j + 8) of the image at
// off that holds row 8 b (every chunk of 8 rows holds one such row; an image's
// last chunk, of 8 to 15 rows, belongs to the first of its two); block
// n_slots + i owns image i if it has fewer rows.  `whole`: block i owns image i.
__global__ void __launch_bounds__(kThreads)
    logodds_chunk_kernel(int32_t* __restrict__ mins, int64_t m, int32_t C, double beta, double log_c1, int positive_only,
                         const int64_t* __restrict__ offsets, int64_t n_img, int64_t n_slots, bool whole, bool tabled,
                         double* __restrict__ totals, unsigned long long* __restrict__ counts) {
  extern __shared__ double smem[];
  __shared__ RowStat st[kChunk];
  const int64_t b = blockIdx.x;
  int64_t img, r0, r1;
  bool split = false;  // the image has other chunks
  if (whole || b >= n_slots) {
    img = whole ? b : b - n_slots;
    r0 = max(offsets[img], (int64_t)0);
    r1 = min(offsets[img + 1], m);
    if (r0 >= r1 || (!whole && r1 - r0 >= kChunk)) return;
  } else {
    const int64_t p = b * kChunk;
    img = image_of(offsets, n_img, p);
    const int64_t o0 = max(offsets[img], (int64_t)0), o1 = min(offsets[img + 1], m);
    if (p < o0 || p >= o1 || o1 - o0 < kChunk) return;
    const int64_t chunks = (o1 - o0) / kChunk, j = (p - o0) / kChunk;
    if (j >= chunks) return;  // in the remainder, which the chunk before has
    split = chunks > 1;
    r0 = o0 + j * kChunk;
    r1 = j == chunks - 1 ? o1 : r0 + kChunk;
  }
  double* table = tabled ? smem : nullptr;                     // [8][C]
  double* part = smem + (tabled ? (int64_t)kChunk * C : 0);    // [C], with split only
  const int warp = threadIdx.x >> 5;
  unsigned long long n = 0;
  for (int64_t r = r0; r < r1; r += kChunk) {
    const int rows = (int)min(r1 - r, (int64_t)kChunk);
    __syncthreads();
    for (int i = warp; i < rows; i += kWarps) {
      const RowStat t = row_stat(mins + (r + i) * C, C, beta, log_c1, table ? table + (int64_t)i * C : nullptr);
      if ((threadIdx.x & 31) == 0) st[i] = t;
    }
    __syncthreads();
    for (int32_t c = threadIdx.x; c < C; c += kThreads) {
      double* sum = split ? part + c : totals + img * C + c;
      double acc = r == r0 ? 0.0 : *sum;
#pragma unroll 4
      for (int i = 0; i < rows; ++i) {
        const double x = beta * (double)(mins[(r + i) * C + c] - st[i].dmin);
        const double e = table ? table[(int64_t)i * C + c] : exp(-x);
        const double inc = c == st[i].cstar ? st[i].inc : -x - log(st[i].s - e) + log_c1;
        if (!positive_only || inc > 0.0) {
          acc += inc;
          ++n;
        }
      }
      *sum = acc;
    }
  }
  if (counts) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(counts + img, n);
  }
  if (split) {
    __syncthreads();  // the rows have been read
    double* out = partial(mins, r0, C);
    for (int32_t c = threadIdx.x; c < C; c += kThreads) out[c] = part[c];
  }
}

// One block per image: the chunks' sums in their order, then the argmax over
// classes, the lowest class on ties.
__global__ void __launch_bounds__(kThreads)
    logodds_finish_kernel(int32_t* __restrict__ mins, int64_t m, int32_t C, const int64_t* __restrict__ offsets,
                          bool whole, double* __restrict__ totals, int32_t* __restrict__ classes) {
  __shared__ double best_s[kWarps];
  __shared__ int32_t class_s[kWarps];
  const int64_t img = blockIdx.x;
  const int64_t o0 = max(offsets[img], (int64_t)0), o1 = min(offsets[img + 1], m);
  const int64_t chunks = whole || o1 <= o0 ? 0 : (o1 - o0) / kChunk;
  double best = -INFINITY;
  int32_t bc = INT32_MAX;
  for (int32_t c = threadIdx.x; c < C; c += kThreads) {
    double v;
    if (chunks > 1) {
      v = 0.0;
#pragma unroll 8
      for (int64_t j = 0; j < chunks; ++j) v += partial(mins, o0 + j * kChunk, C)[c];
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
    for (int w = 1; w < kWarps; ++w)
      if (class_s[w] != INT32_MAX && (bc == INT32_MAX || best_s[w] > best || (best_s[w] == best && class_s[w] < bc))) {
        best = best_s[w];
        bc = class_s[w];
      }
    classes[img] = bc;
  }
}

}  // namespace

cudaError_t prepare_logodds() {
  return cudaFuncSetAttribute(logodds_chunk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(double) * (kChunk + 1) * kTableClasses);
}

cudaError_t launch_logodds(int32_t* mins, int64_t m, int32_t C, double beta, bool positive_only, const int64_t* offsets,
                           int64_t n_img, double* totals, int64_t* counts, int32_t* classes, cudaStream_t s) {
  if (n_img == 0) return cudaSuccess;
  const bool whole = C > kPartClasses, tabled = C <= kTableClasses;
  if (m > 0) {
    const int64_t n_slots = whole ? 0 : (m + kChunk - 1) / kChunk;
    const size_t smem = sizeof(double) * (size_t)C * ((tabled ? kChunk : 0) + (whole ? 0 : 1));
    logodds_chunk_kernel<<<(unsigned)(n_slots + n_img), kThreads, smem, s>>>(
        mins, m, C, beta, log((double)(C - 1)), positive_only ? 1 : 0, offsets, n_img, n_slots, whole, tabled, totals,
        reinterpret_cast<unsigned long long*>(counts));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  logodds_finish_kernel<<<(unsigned)n_img, kThreads, 0, s>>>(mins, m, C, offsets, whole || m == 0, totals, classes);
  return cudaGetLastError();
}

}  // namespace lnbnn
