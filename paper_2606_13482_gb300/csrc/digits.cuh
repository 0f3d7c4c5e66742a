// 10-bit digits of FP64 values and their FP16 products on the tensor cores
// (error-free fixed-point splitting, Ozaki et al. 2012); see near_mma.cu.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace efie {

constexpr int NM_PIECE = 512;        // columns after which the 32-bit sums are drained
constexpr int NM_ENAN = 30000;       // exponent of a row or vector with an Inf or NaN: outputs NaN

// ---------------------------------------------------------------- digits
// E with |x| < 2^E for every x whose high word, sign cleared, is at most mx
__device__ __forceinline__ int nm_exponent(int mx) {
  const int f = mx >> 20;
  return f == 2047 ? NM_ENAN : max(f, 1) - 1022;  // (zeros and subnormal numbers as 2^-1022)
}
// of a matrix row: not below -850, where an entry is nothing beside its row's largest
__device__ __forceinline__ int nm_row_exponent(int mx) { return max(nm_exponent(mx), -850); }
// A digit sum T of a row with exponent er and a vector with exponent ex counts units of
// 2^(er + ex - off), off about 50, which may be below 2^-1022 while the value is a normal
// number.  So ex is cut to +-100, which with er makes one FP64 factor, and the rest, zero but
// for vectors below 2^-100 or above 2^100, goes into the exponent of the double T by integer
// arithmetic: the value rounds, underflows and overflows as FP64 does.  (48,000
// unknowns, 64 vectors: 1.5% of the near field; a multiplication by the rest took 3%, for the
// drains are bound by the FP64 pipe.)
struct NmCol {
  int e, rest;  // rest shifted to the exponent field
  bool bad;
};
__device__ __forceinline__ NmCol nm_col(int ex) {
  const int e = min(max(ex, -100), 100);
  return {e, (int)((uint32_t)(ex - e) << 20), ex == NM_ENAN};
}
__device__ __forceinline__ double nm_scale(int er, const NmCol& x, int off) {
  return __hiloint2double(er == NM_ENAN || x.bad ? 0x7ff80000 : (er + x.e - off + 1023) << 20, 0);
}
// t 2^rest for an integer t below 2^63
__device__ __forceinline__ double nm_raise(double t, const NmCol& x) {
  const int hi = __double2hiint(t);
  return __hiloint2double(hi == 0 ? 0 : hi + x.rest, __double2loint(t));
}
// q = round-toward-zero(v 2^59), v = x 2^-(E + 1), |v| < 1/2, from the bits of x
__device__ __forceinline__ int64_t nm_fixed(double x, int E) {
  const int hi = __double2hiint(x);
  const int f = (hi >> 20) & 0x7ff;
  uint64_t m = ((uint64_t)(uint32_t)((hi & 0xfffff) | (f ? 0x100000 : 0)) << 32) | (uint32_t)__double2loint(x);
  const int k = E - (max(f, 1) - 1023) - 1;  // >= 0
  m = k > 63 ? 0 : (m << 5) >> k;
  return hi < 0 ? -(int64_t)m : (int64_t)m;
}
// NS digits of q, d[0] the leading one, each in [-512, 511]
template <int NS>
__device__ __forceinline__ void nm_digits(int64_t q, int* d) {
  if (NS == 5) q = (q + 512) >> 10;
  uint64_t u = (uint64_t)(q + (NS == 5 ? 0x0002008020080200LL : 0x0802008020080200LL));  // + 512 at every digit
#pragma unroll
  for (int k = NS - 1; k >= 0; --k) {
    d[k] = (int)((uint32_t)u & 1023u);
    u >>= 10;
  }
}
// two unsigned digits u0, u1 in [0, 1023] -> half2 (u0 - 512, u1 - 512): 0x6400 | u is 1024 + u
__device__ __forceinline__ uint32_t nm_pack(int u0, int u1) {
  const uint32_t w = 0x64006400u | (uint32_t)u0 | ((uint32_t)u1 << 16);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __floats2half2_rn(1536.f, 1536.f));
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void nm_mma(float* d, const uint32_t* a, uint32_t b0, uint32_t b1, const float* c) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

}  // namespace efie
