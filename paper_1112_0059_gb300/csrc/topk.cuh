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

// Candidate entries: eight neighbouring columns' distance bits, then the first
// one's column (row of the references).
constexpr int kEntryWords = 16;

// Merges the rows of the mask `rows` (row r < 32; its counters and result are
// lane r's): n candidates at cand + r * cand_stride, (row, distance bits)
// pairs, into the K1 <= 32 S smallest (distance, row) keys, ascending, at
// list + r * K1.  The list holds keys already where `listed` has the row;
// otherwise it starts from seed + r * K1 if there is a seed, or empty.
// Returns the bits of the lane's row's K1-th distance (INT32_MAX: not full),
// `kth` for rows not merged.
//
// One row after another, by counting: lane l holds the list's keys l, l + 32,
// ... and candidate l of (up to) 32.  Each candidate in turn is shown to every
// lane, which counts it for those of its keys that it sorts before; a key's new
// place is its old one plus its count, a candidate's the number of list keys
// (summed over the lanes by one reduction) and candidates before it.  A row has
// ten or so candidates when its warp's buffers come, so this is less than a
// bitonic sort and merge of 32 S keys, which took 3,900 cycles a row whatever
// their number: 256-class data, 15k rows, k = 100 35.7 / 32.9 ms, FP8 shortlist
// 128 28.4 / 27.2 ms.  Of about 2,600 cycles a row, 900 wait for the row's keys
// (from L2; the next row's are loaded meanwhile, but the operands stream at the
// same time and shared memory leaves L1 28 KB), 1,300 show the candidates (a
// shuffle waits its turn behind the MMAs' operand reads, so four are shown at a
// time: one at a time 34.9 ms, eight 33.3) and 440 store.  Straight-line code
// past what the instruction cache holds (about 10 KB for all roles of the scan
// kernel) runs at a third of the speed (6 cycles an instruction against 2
// measured on one warp), so the function is rolled and not inlined.
template <int S>
__device__ __noinline__ int32_t merge_rows(const uint64_t* cand, int cand_stride, int n_cand, uint64_t* list,
                                           const uint64_t* seed, uint32_t rows, uint32_t listed, int K1, int32_t kth) {
  constexpr int W = (S + 3) / 4;  // words of four 8-bit counts
  constexpr int U = 4;            // candidates shown at a time
  const int lane = threadIdx.x & 31;
  uint64_t l[S], next_l[S], c = 0, next_c = 0;
  int row = -1, n = 0, next_n = 0;
#pragma unroll
  for (int s = 0; s < S; ++s) l[s] = next_l[s] = kEmptyKey;
#pragma unroll 1
  do {
    const int next = __ffs(rows) - 1;  // -1: no row is left
    if (next >= 0) {
      rows &= rows - 1;
      next_n = __shfl_sync(0xffffffffu, n_cand, next);
      const uint64_t* src = ((listed >> next) & 1u) != 0 ? list + next * K1 : seed != nullptr ? seed + next * K1 : nullptr;
#pragma unroll
      for (int s = 0; s < S; ++s)
        next_l[s] = src != nullptr && lane + 32 * s < K1 ? ld_global_u64(src + lane + 32 * s) : kEmptyKey;
      next_c = lane < next_n ? ld_global_u64(cand + (int64_t)next * cand_stride + lane) : 0;
    }
    if (row >= 0) {
      uint64_t* to = list + row * K1;
      bool all = ((listed >> row) & 1u) == 0;  // nothing is written yet
#pragma unroll 1
      for (int off = 0;;) {
        uint64_t key = kEmptyKey;
        if (off + lane < n) {
          const uint32_t d = bits_dist((uint32_t)(c >> 32));
          if (d < kDistLimit) key = make_key(d, (uint32_t)c);  // (a padding row's distance is above it)
        }
        const int shown = min(n - off, 32);
        uint32_t count[W], above = 0;
        int rank = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) count[w] = 0;
#pragma unroll 1
        for (int j = 0; j < shown; j += U) {
          uint64_t x[U];
          uint32_t one[U][W], g[U];
#pragma unroll
          for (int u = 0; u < U; ++u) x[u] = __shfl_sync(0xffffffffu, key, j + u);
#pragma unroll
          for (int u = 0; u < U; ++u) {
            rank += x[u] < key;
#pragma unroll
            for (int w = 0; w < W; ++w) {
              one[u][w] = 0;
#pragma unroll
              for (int s = 4 * w; s < min(S, 4 * w + 4); ++s)
                if (x[u] < l[s]) one[u][w] += 1u << (8 * (s & 3));
              count[w] += one[u][w];
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            g[u] = 0;  // list keys that x sorts before
#pragma unroll
            for (int w = 0; w < W; ++w) g[u] = __dp4a(__reduce_add_sync(0xffffffffu, one[u][w]), 0x01010101u, g[u]);
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (lane == j + u) above = g[u];
        }
        // a place for every key: nothing moves before the first candidate's
        uint32_t last = 0;
        bool at_end = false;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const int by = (int)((count[s / 4] >> (8 * (s & 3))) & 255u), at = lane + 32 * s + by;
          if (at < K1 && (all || by > 0)) to[at] = l[s];
          if (at == K1 - 1) {
            at_end = true;
            last = (uint32_t)(l[s] >> 32);
          }
        }
        const int at = 32 * S - (int)above + rank;
        if (key != kEmptyKey && at < K1) {
          to[at] = key;
          if (at == K1 - 1) {
            at_end = true;
            last = (uint32_t)(key >> 32);
          }
        }
        const uint32_t holder = __ballot_sync(0xffffffffu, at_end);
        const uint32_t d = __shfl_sync(0xffffffffu, last, __ffs(holder) - 1);
        if (lane == row) kth = d == 0xFFFFFFFFu ? INT32_MAX : dist_bits(d);
        off += 32;
        if (off >= n) break;
        __syncwarp();
        all = false;
#pragma unroll
        for (int s = 0; s < S; ++s) l[s] = lane + 32 * s < K1 ? ld_global_u64(to + lane + 32 * s) : kEmptyKey;
        if (off + lane < n) c = ld_global_u64(cand + (int64_t)row * cand_stride + off + lane);
      }
    }
    row = next;
    n = next_n;
    c = next_c;
#pragma unroll
    for (int s = 0; s < S; ++s) l[s] = next_l[s];
  } while (row >= 0);
  __syncwarp();
  return kth;
}

}  // namespace lnbnn
