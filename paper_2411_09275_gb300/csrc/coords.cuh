// Every coordinate in [0, 2^30): a value is out of range exactly when one of
// its two top bits is set.
#pragma once

#include <algorithm>

#include "common.cuh"

namespace pkd {

static_assert(PKD_COORD_LIMIT == (1 << 30), "range test by the top two bits");

// The grid's threads' share of the OR of cnt values: a scalar head up to the
// first 16-byte boundary, then 16-byte loads, four in flight per thread, then
// a scalar tail.
__device__ __forceinline__ unsigned coord_bits(const int32_t* c, uint64_t cnt) {
  const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t head = min(cnt, (uint64_t)(((16u - ((uintptr_t)c & 15u)) & 15u) >> 2));
  unsigned b = 0;
  if (tid < head) b |= (unsigned)c[tid];
  const int4* v4 = reinterpret_cast<const int4*>(c + head);
  const uint64_t n4 = (cnt - head) >> 2;
  uint64_t i = tid;
  for (; i + 3 * nth < n4; i += 4 * nth) {
    const int4 a0 = v4[i], a1 = v4[i + nth], a2 = v4[i + 2 * nth], a3 = v4[i + 3 * nth];
    b |= (unsigned)(a0.x | a0.y | a0.z | a0.w | a1.x | a1.y | a1.z | a1.w);
    b |= (unsigned)(a2.x | a2.y | a2.z | a2.w | a3.x | a3.y | a3.z | a3.w);
  }
  for (; i < n4; i += nth) {
    const int4 a = v4[i];
    b |= (unsigned)(a.x | a.y | a.z | a.w);
  }
  const uint64_t t0 = head + 4 * n4;
  if (tid < cnt - t0) b |= (unsigned)c[t0 + tid];
  return b;
}

// Blocks of 256 threads for coord_bits: four 16-byte loads a thread, at most
// eight blocks per SM.
inline unsigned coord_blocks(uint64_t cnt) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((cnt + 4095) / 4096, 152 * 8));
}

}  // namespace pkd
