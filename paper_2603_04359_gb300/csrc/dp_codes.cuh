// b-bit codes and their digit planes: the parts that the SIMT and the tensor-core activation kernels share
// (grids, exact decisions and the plane format are described in quant_dp.cu).
#pragma once
#include "common.cuh"

namespace cat {

struct DpMode {
  int bits;      // 2..8
  int asym;      // 0: symmetric, 1: asymmetric
  int planes;    // digit planes D
  float qmax;    // symmetric: 2^(b-1) - 1; asymmetric: N = 2^b - 1
};

// Order-preserving key of a float (max of keys = key of the max), for signed min / max atomics.
__device__ __forceinline__ uint32_t fkey(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ uint32_t e4m3_digit(int d) { return (d < 0 ? 0x80u : 0u) | (uint32_t)(d < 0 ? -d : d); }

// The digits' E4M3 bytes of one code.
__device__ __forceinline__ void code_digits(int q, const DpMode& m, uint32_t* b0, uint32_t* b1) {
  if (m.planes == 1) {
    *b0 = e4m3_digit(q);
    *b1 = 0u;
  } else if (m.asym) {
    *b0 = (uint32_t)(q & 15);
    *b1 = (uint32_t)(q >> 4);
  } else {
    const int lo = ((q + 8) & 15) - 8;
    *b0 = e4m3_digit(lo);
    *b1 = e4m3_digit((q - lo) / 16);
  }
}

// Per-row asymmetric grid: float32 estimate inputs and the float64 operands of the exact route.
struct AsymRow {
  float inv;      // fl(N / fl(hi - lo)); 0 for a zero or non-finite row
  double lo, r;   // lo and hi - lo in float64
  int z;
};

__device__ __forceinline__ AsymRow asym_row(float hi, float lo, float N) {
  AsymRow a;
  a.lo = lo;
  a.r = (double)hi - (double)lo;
  a.inv = 0.f;
  a.z = 0;
  if (!(isfinite(hi) && isfinite(lo)) || !(a.r > 0.0)) return a;
  a.inv = __fdiv_rn(N, __fsub_rn(hi, lo));
  a.z = (int)rint(((double)N * -a.lo) / a.r);
  return a;
}

__device__ __forceinline__ int asym_code(float v, const AsymRow& a, float N) {
  if (a.inv == 0.f || !isfinite(v)) return a.inv == 0.f ? 0 : a.z;
  const float p = __fmul_rn(v, a.inv);
  float rq = rintf(p);
  // exact route; also where 1 / step overflowed (hi - lo below N / FLT_MAX): p - rq is then NaN
  if (!(fabsf(p - rq) <= 0.5f - 0x1p-12f)) rq = (float)rint(((double)N * (double)v) / a.r);
  int q = (int)rq + a.z;
  const int top = (int)N;
  return q < 0 ? 0 : (q > top ? top : q);
}

}  // namespace cat
