// Epilogue pieces shared by the product kernels (symgemm.cu, symgemm_f32.cu).
#pragma once

#include <cuda_fp16.h>

#include "internal.h"

namespace psd {

__device__ __forceinline__ void raise_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// Two values as FP16, a in the low half: rounded to nearest, to +-65504 beyond
// FP16's range (a NaN stays a NaN).
__device__ __forceinline__ uint32_t pack_h2_sat(float a, float b) {
  uint32_t r;
  asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
// x as an FP16 pair hi + lo (bits), both saturating.
__device__ __forceinline__ void split_h2_sat(float x, uint16_t& hi, uint16_t& lo) {
  hi = static_cast<uint16_t>(pack_h2_sat(x, 0.f));
  lo = static_cast<uint16_t>(pack_h2_sat(x - __half2float(__ushort_as_half(hi)), 0.f));
}

// Row stride (words) of a warp's 32 x 32 FP32 staging square.
constexpr int kStgWords = 33;

// One 32 x 32 chunk of the final output out = (X + lam~ acc) / 2 in FP32,
// reading only the upper triangle of the caller's X (column-major).
__device__ __forceinline__ void epilogue_chunk_final(const BlockRec& br, int r0, int c0,
                                                     const uint32_t (&v)[32], uint8_t* wbuf,
                                                     int lane, float lam, ComplAcc* ca) {
  uint32_t* stg = reinterpret_cast<uint32_t*>(wbuf);
  const int n = br.n;
  const float* X = br.X;
  const int64_t ld = br.ld;
  float* out = br.out;
  const int64_t ldo = br.ld_out;
  const int r = r0 + lane;
  const bool diag = (r0 == c0);
  const bool row_ok = r < n;
  float o[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int c = c0 + j;
    float x = 0.f;
    const bool upper = !diag || j >= lane;
    if (row_ok && c < n && upper) x = X[static_cast<int64_t>(c) * ld + r];
    o[j] = 0.5f * fmaf(lam, __uint_as_float(v[j]), x);
    if (ca && row_ok && c < n && upper) compl_add(*ca, o[j], x, c == r ? 1.f : 2.f);
  }
  float* sf = reinterpret_cast<float*>(stg);
  if (diag) {
#pragma unroll
    for (int j = 0; j < 32; ++j) sf[lane * kStgWords + j] = o[j];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < lane) o[j] = sf[j * kStgWords + lane];
    __syncwarp();
  }
  if (row_ok) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (c0 + j < n) out[static_cast<int64_t>(c0 + j) * ldo + r] = o[j];
  }
  if (!diag) {
#pragma unroll
    for (int j = 0; j < 32; ++j) sf[lane * kStgWords + j] = o[j];
    __syncwarp();
    const int c = c0 + lane;
    if (c < n) {
#pragma unroll 4
      for (int rr = 0; rr < 32; ++rr)
        if (r0 + rr < n) out[static_cast<int64_t>(r0 + rr) * ldo + c] = sf[rr * kStgWords + lane];
    }
    __syncwarp();
  }
}

}  // namespace psd
