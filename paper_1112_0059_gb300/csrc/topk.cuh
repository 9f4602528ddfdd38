// The k+1 nearest of Alg. 2: sorted lists, and merging them with candidates
// collected since.
#pragma once

#include "internal.cuh"

namespace lnbnn {

// Above every distance and coarse value, below those of padding rows.
constexpr uint32_t kDistLimit = (1u << 24) - 1;

// Bits of a non-negative float as int32, ordered like the float, for a whole
// distance (exact below 2^24), and back.
__device__ __forceinline__ int32_t dist_bits(uint32_t dist) { return __float_as_int((float)dist); }
__device__ __forceinline__ uint32_t bits_dist(uint32_t bits) { return (uint32_t)__float2int_rn(__uint_as_float(bits)); }

__device__ __forceinline__ void prefetch_l1(const uint32_t* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p) : "memory");
}
__device__ __forceinline__ uint32_t ld_global_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_global_v4(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_global_u64(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Sorted list of the K1 smallest (distance, row) pairs seen so far, held in one
// thread's registers, the distances as the bit patterns of their floats:
// ascending in slots [KMAX-K1, KMAX); the slots below hold -1, which no
// distance displaces, so the list always has K1 live entries and its largest
// is slot KMAX-1 (INT32_MAX while the list is not full).
template <int KMAX>
struct RegList {
  int32_t d[KMAX];
  uint32_t r[KMAX];

  __device__ __forceinline__ void init(int K1) {
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      d[i] = i < KMAX - K1 ? -1 : INT32_MAX;
      r[i] = 0xFFFFFFFFu;
    }
  }
  __device__ __forceinline__ int32_t worst() const { return d[KMAX - 1]; }
  // Start from a finished list of K1 ascending keys (kEmptyKey: no entry).
  __device__ __forceinline__ void seed(const uint64_t* src, int K1) {
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i >= KMAX - K1) {
        const uint64_t k = __ldcg(src + (i - (KMAX - K1)));
        d[i] = k == kEmptyKey ? INT32_MAX : dist_bits(key_dist(k));
        r[i] = key_row(k);
      }
      // at most four keys in flight: the list itself holds the registers
      if ((i & 3) == 3) asm volatile("" ::: "memory");
    }
  }
  // new[i] = old[i-1] if (x, row) sorts before it, else min((x, row), old[i]);
  // a pair that sorts after the largest changes nothing.
  __device__ __forceinline__ void insert(int32_t x, uint32_t row) {
    const int64_t key = ((int64_t)x << 32) | row;
    bool before = key < (((int64_t)d[KMAX - 1] << 32) | r[KMAX - 1]);
#pragma unroll
    for (int i = KMAX - 1; i > 0; --i) {
      const bool shift = key < (((int64_t)d[i - 1] << 32) | r[i - 1]);
      d[i] = shift ? d[i - 1] : (before ? x : d[i]);
      r[i] = shift ? r[i - 1] : (before ? row : r[i]);
      before = shift;
    }
    if (before) {
      d[0] = x;
      r[0] = row;
    }
  }
  // Writes the K1 live entries ascending (unfilled slots as kEmptyKey).
  __device__ __forceinline__ void store(uint64_t* out, int K1) const {
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
      if (i >= KMAX - K1)
        out[i - (KMAX - K1)] = d[i] == INT32_MAX ? kEmptyKey : make_key(bits_dist((uint32_t)d[i]), r[i]);
  }
};

template <>
struct RegList<0> {};

// A bitonic stage between elements `stride` >= 32 apart: registers of one lane.
template <int S, int R, typename Key>
__device__ __forceinline__ void between_registers(Key (&k)[R][S], int size, int stride) {
#pragma unroll
  for (int d = S / 2; d > 0; d >>= 1) {
    if (stride == 32 * d) {
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int s = 0; s < S; ++s)
          if ((s & d) == 0) {
            const bool up = ((32 * s) & size) == 0;
            const Key a = k[i][s], b = k[i][s | d];
            const bool keep = (a < b) == up;
            k[i][s] = keep ? a : b;
            k[i][s | d] = keep ? b : a;
          }
    }
  }
}

// Candidate entries: eight neighbouring columns' distance bits, then the first
// one's column (row of the references).
constexpr int kEntryWords = 16;

// Merges the rows of the mask `rows` (row r < 32; its counters and result are
// lane r's): n candidates at cand + r * cand_stride, (row, distance bits)
// pairs in increasing row order, into the K1 smallest (distance, row) keys, ascending,
// at list + r * K1.  The list holds keys already where `listed` has the row;
// otherwise it starts from seed + r * K1 if there is a seed, or empty.
// Returns the bits of the lane's row's K1-th distance (INT32_MAX: not full),
// `kth` for rows not merged.
//
// R rows at a time: the candidates are sorted bitonically, N = 32 S at a time,
// and the smaller half of list and candidates merged; lane l holds elements l,
// l + 32, ...  The sort runs on 32-bit keys (a distance is below 2^24, so it
// has room for the candidate's place), a shuffle and a minimum or maximum per
// key and stage; candidates must therefore come in increasing row order among
// equal distances.  Only the merge compares 64-bit (distance, row) keys: the
// list may hold rows from other columns.  A stage waits on its shuffle, so R
// rows share it.  The stages run in rolled loops and the function is not
// inlined: straight-line code past what the instruction cache holds (about
// 10 KB for all roles of the scan kernel) runs at a third of the speed (6
// cycles an instruction against 2 measured on one warp).
template <int S, int R>
__device__ __noinline__ int32_t merge_rows(const uint64_t* cand, int cand_stride, int n_cand, uint64_t* list,
                                           const uint64_t* seed, uint32_t rows, uint32_t listed, int K1, int32_t kth) {
  constexpr int N = 32 * S;
  const int lane = threadIdx.x & 31;
  while (rows != 0u) {
    int row[R], n[R], most = 0;
    uint64_t l[R][S];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      row[i] = __ffs(rows) - 1;  // -1: fewer than R rows are left
      rows &= rows - 1;
      n[i] = row[i] < 0 ? 0 : __shfl_sync(0xffffffffu, n_cand, row[i] & 31);
      most = max(most, n[i]);
      const uint64_t* src = row[i] < 0                       ? nullptr
                            : ((listed >> row[i]) & 1u) != 0 ? list + row[i] * K1
                            : seed != nullptr                ? seed + row[i] * K1
                                                             : nullptr;
#pragma unroll
      for (int s = 0; s < S; ++s)
        l[i][s] = src != nullptr && lane + 32 * s < K1 ? ld_global_u64(src + lane + 32 * s) : kEmptyKey;
    }
#pragma unroll 1
    for (int off = 0; off < most; off += N) {
      uint32_t c[R][S];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const int e = lane + 32 * s;
          c[i][s] = 0xFFFFFFFFu;
          if (off + e < n[i]) {
            const uint32_t d = bits_dist((uint32_t)(ld_global_u64(cand + (int64_t)row[i] * cand_stride + off + e) >> 32));
            if (d < kDistLimit) c[i][s] = (d << 8) | (uint32_t)e;  // (a padding row's distance is above it)
          }
        }
      // the first power of two that holds them all is sorted; the rest of c is
      // empty, above all, and stays where it is
      int span = 32;
      while (span < N && span < most - off) span <<= 1;
#pragma unroll 1
      for (int size = 2; size <= span; size <<= 1) {
#pragma unroll 1
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
          if (S > 1 && stride >= 32) {
            between_registers<S, R>(c, size, stride);
          } else {
#pragma unroll
            for (int s = 0; s < S; ++s) {
              if (s > 0 && 32 * s >= span) break;
              const bool low = ((lane & stride) == 0) == (((lane + 32 * s) & size) == 0);
#pragma unroll
              for (int i = 0; i < R; ++i) {
                const uint32_t o = __shfl_xor_sync(0xffffffffu, c[i][s], stride);
                c[i][s] = low ? min(c[i][s], o) : max(c[i][s], o);
              }
            }
          }
        }
      }
      // both ascending: element e of the list against element N - 1 - e of the
      // candidates leaves the N smallest, as a bitonic sequence
#pragma unroll
      for (int i = 0; i < R; ++i) {
        uint64_t k[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, c[i][S - 1 - s], 31);
          k[s] = kEmptyKey;
          if (o != 0xFFFFFFFFu)
            k[s] = make_key(o >> 8, (uint32_t)ld_global_u64(cand + (int64_t)row[i] * cand_stride + off + (o & 255u)));
        }
#pragma unroll
        for (int s = 0; s < S; ++s) l[i][s] = min(l[i][s], k[s]);
      }
#pragma unroll 1
      for (int stride = N >> 1; stride > 0; stride >>= 1) {
        if (S > 1 && stride >= 32) {
          between_registers<S, R>(l, 2 * N, stride);
        } else {
          const bool low = (lane & stride) == 0;
#pragma unroll
          for (int s = 0; s < S; ++s)
#pragma unroll
            for (int i = 0; i < R; ++i) {
              const uint64_t o = __shfl_xor_sync(0xffffffffu, l[i][s], stride);
              l[i][s] = (l[i][s] < o) == low ? l[i][s] : o;
            }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (row[i] < 0) continue;
      uint64_t last = kEmptyKey;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (lane + 32 * s < K1) list[row[i] * K1 + lane + 32 * s] = l[i][s];
        if ((K1 - 1) >> 5 == s) last = l[i][s];
      }
      const uint32_t d = __shfl_sync(0xffffffffu, (uint32_t)(last >> 32), (K1 - 1) & 31);
      if (lane == row[i]) kth = d == 0xFFFFFFFFu ? INT32_MAX : dist_bits(d);
    }
  }
  __syncwarp();
  return kth;
}

}  // namespace lnbnn
