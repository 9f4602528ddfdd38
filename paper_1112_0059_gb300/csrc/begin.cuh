// The part of a call's first kernel beside the query preparation (Begin).
#pragma once

#include <algorithm>

#include "internal.cuh"

namespace lnbnn {

constexpr int kBeginThreads = 256;

// Blocks for the fills and the check, 0 if there is nothing to do: a few
// thousand words each, at most four per SM's worth.
inline unsigned begin_blocks(const Begin& b) {
  int64_t words = b.offsets ? b.n_img + 1 : 0;
  for (int i = 0; i < b.n; ++i) words += b.f[i].words;
  return (unsigned)std::min<int64_t>((words + 4095) / 4096, 608);
}

// Block `block` of `blocks` (kBeginThreads threads each).
__device__ __forceinline__ void begin_part(const Begin& b, int64_t block, int64_t blocks) {
  const int64_t at = block * kBeginThreads + threadIdx.x, step = blocks * kBeginThreads;
#pragma unroll 1
  for (int k = 0; k < b.n; ++k) {
    uint32_t* p = b.f[k].p;
    const int64_t words = b.f[k].words;
    const uint32_t v = b.f[k].v;
    int64_t done = 0;
    if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
      done = words & ~int64_t(3);
      for (int64_t i = at; i < words / 4; i += step) reinterpret_cast<uint4*>(p)[i] = make_uint4(v, v, v, v);
    }
    for (int64_t i = done + at; i < words; i += step) p[i] = v;
  }
  if (b.offsets == nullptr) return;
  for (int64_t i = at; i <= b.n_img; i += step) {
    bool bad = false;
    if (i == 0) bad = b.offsets[0] != 0;
    if (i == b.n_img) bad = bad || b.offsets[b.n_img] != b.m;
    if (i < b.n_img) bad = bad || b.offsets[i + 1] < b.offsets[i];
    if (bad) atomicOr(b.dev_err, kDevErrOffsets);
  }
}

}  // namespace lnbnn
