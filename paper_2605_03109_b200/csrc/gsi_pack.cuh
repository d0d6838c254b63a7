// Layouts of the copies that the persistent kernel streams (see PersistGroup::P).
#pragma once

#include <cuda_fp8.h>

#include "gsi_common.cuh"
#include "gsi_persistent.cuh"

namespace gsi {
namespace pack {

// 16-bit slot of element (row, col) of a [rows][k] matrix in 16 x 16 tiles: within a tile four
// 8 x 8 blocks of 64 elements, each row-major.
__device__ __forceinline__ size_t t16_slot(int row, int col, int k) {
  const size_t tile = (size_t)(row >> 4) * (k >> 4) + (col >> 4);
  return tile * 256 + ((row >> 3) & 1) * 64 + ((col >> 3) & 1) * 128 + (row & 7) * 8 + (col & 7);
}

// Sixteen rows (block R) of the image in FP8 (Section 7.4), by one thread block of at least 256
// threads.  Row scale = max|row| / 448 (1 for a zero row), code = nearest E4M3 of element / scale
// (ties to even, saturating); both divisions are single IEEE fp32 operations, so the codes follow
// from the bf16 image alone.  s_scale: sixteen floats of shared memory, free again after the next
// barrier.
__device__ __forceinline__ void fp8_rows16(const uint16_t* src, int rows, int k, unsigned char* dst, int R,
                                           float* s_scale) {
  const int kt = k >> 4, tid = threadIdx.x;
  if (tid < 256) {
    const int r = tid >> 4, sub = tid & 15;
    float amax = 0.f;
    if (R * 16 + r < rows)
      for (int j = sub; j < k; j += 16)
        amax = fmaxf(amax, fabsf(__uint_as_float((uint32_t)src[(size_t)(R * 16 + r) * k + j] << 16)));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (sub == 0) s_scale[r] = amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f;
  }
  __syncthreads();
  unsigned char* out = dst + (size_t)R * persist_image_row_bytes(k, true);
  for (int wi = tid; wi < kt * 128; wi += blockDim.x) {   // one pair of codes per step
    const int reg = wi & 3, lane = (wi >> 2) & 31, K = wi >> 7;
    const int r16 = (lane >> 2) + (reg & 1) * 8, row = R * 16 + r16;
    const int col = K * 16 + 2 * (lane & 3) + (reg >> 1) * 8;
    unsigned short pair = 0;
    if (row < rows) {
      const float sc = s_scale[r16];
      const float a = __uint_as_float((uint32_t)src[(size_t)row * k + col] << 16);
      const float b = __uint_as_float((uint32_t)src[(size_t)row * k + col + 1] << 16);
      const unsigned lo = __nv_cvt_float_to_fp8(__fdiv_rn(a, sc), __NV_SATFINITE, __NV_E4M3);
      const unsigned hi = __nv_cvt_float_to_fp8(__fdiv_rn(b, sc), __NV_SATFINITE, __NV_E4M3);
      pair = (unsigned short)(lo | (hi << 8));
    }
    reinterpret_cast<unsigned short*>(out)[wi] = pair;
  }
  if (tid < 16) reinterpret_cast<float*>(out + (size_t)kt * 256)[tid] = s_scale[tid];
}

}  // namespace pack
}  // namespace gsi
