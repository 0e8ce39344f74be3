// exp() in double precision for sums of many terms, table-driven (P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15(2), 1989):
//   x = (32 m + j) * ln2/32 + r,  |r| <= ln2/64,   exp(x) = 2^m * 2^(j/32) * P(r),
// P = the Taylor polynomial of degree 6 (truncation 3.5e-18 relative), ln2/32 split in two for the reduction.
// Cost per term: 9 fp64 instructions with the addition to the sum, two conversions, two shuffles, six others; measured 3.5 terms
// per SM and clock from registers (a general exp() with its subtraction: 2.9); the row scan around it reaches 2.6.  The table has one entry per lane of a warp and
// is read with two shuffles: no shared memory, no bank conflicts.  Error: about one unit in the last place per term.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace jet {

// 2^(j/32), j = 0 .. 31, correctly rounded.
static __device__ const double kExp2Over32[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0, 0x1.172b83c7d517bp+0,
    0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0, 0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0,
    0x1.3dea64c123422p+0, 0x1.44e086061892dp+0, 0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0,
    0x1.6247eb03a5585p+0, 0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0, 0x1.ae89f995ad3adp+0,
    0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0, 0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0,
    0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0};

// The calling lane's table entry, fetched once per kernel; scale_down(m) makes every later result 2^-m times exp(x).
struct Exp64Table {
  int lo, hi;
  __device__ __forceinline__ void scale_down(int m) { hi -= static_cast<int>(static_cast<uint32_t>(m) << 20); }
  __device__ __forceinline__ explicit Exp64Table(int lane) {
    const double t = __ldg(kExp2Over32 + lane);
    lo = __double2loint(t);
    hi = __double2hiint(t);
  }
};

// Largest |x| the table form covers (the interval number must fit the rounding trick below).
constexpr float kExp64Range = 5e4f;

struct Exp64 { double s, p; };

// (s, p) with s * p = exp(x) * 2^-shift, xd = x.  Called by whole warps; the result must be in the normal range.
__device__ __forceinline__ Exp64 exp64(float x, double xd, const Exp64Table& tab) {
  constexpr float kMagic = 12582912.0f;                      // 1.5 * 2^23: rounds to an integer in the low mantissa bits
  const float t = fmaf(x, 46.16624130844683f, kMagic);       // 32 / ln2
  const uint32_t k = __float_as_uint(t);
  const double kd = static_cast<double>(t - kMagic);
  double r = fma(kd, -0x1.62e42fee00000p-6, xd);
  r = fma(kd, -0x1.a39ef35793c76p-38, r);
  double p = fma(1.0 / 720.0, r, 1.0 / 120.0);
  p = fma(p, r, 1.0 / 24.0);
  p = fma(p, r, 1.0 / 6.0);
  p = fma(p, r, 0.5);
  p = fma(p, r, 1.0);
  p = fma(p, r, 1.0);
  const int lo = __shfl_sync(0xffffffffu, tab.lo, static_cast<int>(k));        // (lane = k mod 32: the magic constant is a multiple of 32)
  const int hi = __shfl_sync(0xffffffffu, tab.hi, static_cast<int>(k));
  // 2^m: the bits of k above the table index, moved to the exponent field (the magic constant's own bits fall off the top)
  return {__hiloint2double(hi + static_cast<int>((k & 0xFFFFFFE0u) << 15), lo), p};
}

}  // namespace jet
