// copy16.cuh -- 16-byte streaming copies shared by the move kernels
// (pack_kernels.cu) and the segment kernel (segment_kernels.cu); device code.
#pragma once

#include <stdint.h>

#include "kvx_internal.h"

namespace kvx {
namespace {

constexpr int kInflight = 8;  // 16-byte vectors per lane between loads and stores

// Streaming (evict-first) accesses: every byte is touched exactly once.
__device__ __forceinline__ uint4 ld16(const uint8_t* p) {
  return __ldcs(reinterpret_cast<const uint4*>(p));
}
__device__ __forceinline__ void st16(uint8_t* p, const uint4& v) {
  __stcs(reinterpret_cast<uint4*>(p), v);
}

// One warp's copy of nbytes (a multiple of 16).
__device__ __forceinline__ void copy_flat(uint8_t* dst, const uint8_t* src, int64_t nbytes, int lane) {
  int64_t off = (int64_t)lane * 16;
  constexpr int64_t kStep = 32 * 16;
  for (; off + (kInflight - 1) * kStep < nbytes; off += kInflight * kStep) {
    uint4 v[kInflight];
#pragma unroll
    for (int i = 0; i < kInflight; ++i) v[i] = ld16(src + off + i * kStep);
#pragma unroll
    for (int i = 0; i < kInflight; ++i) st16(dst + off + i * kStep, v[i]);
  }
  for (; off < nbytes; off += kStep) st16(dst + off, ld16(src + off));
}

}  // namespace
}  // namespace kvx
