// Exact squared distance of two 128-byte rows.
#pragma once

#include "internal.cuh"

namespace lnbnn {

// ||q - r||^2 over one 128-byte row, 16 bytes at a time.
__device__ __forceinline__ uint32_t sqdist_u8(const uint4 (&q)[8], const uint8_t* __restrict__ r) {
  uint32_t acc = 0;
  const uint4* rv = reinterpret_cast<const uint4*>(r);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 b = __ldg(rv + i);
    uint32_t d;
    d = __vabsdiffu4(q[i].x, b.x);
    acc = __dp4a(d, d, acc);
    d = __vabsdiffu4(q[i].y, b.y);
    acc = __dp4a(d, d, acc);
    d = __vabsdiffu4(q[i].z, b.z);
    acc = __dp4a(d, d, acc);
    d = __vabsdiffu4(q[i].w, b.w);
    acc = __dp4a(d, d, acc);
  }
  return acc;
}

}  // namespace lnbnn
