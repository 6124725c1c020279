// Exact base-256 digits of FP64 numbers for products on the tensor cores
// (ozgemm.cu: complex matrix products; ozgrid.cu: the FP64 grid passes).
//
// A set of numbers shares a power of two: x is held as 64-bit fixed point,
// X = round(x 2^(1084 - bmax)) with bmax the largest exponent field of the
// set (|x| < 2^(bmax - 1022), |X| <= 2^62), and X = sum_t d_t 256^(7 - t) with
// eight balanced digits |d_t| <= 128, each exact in BF16.  The products of
// digits of order o = t + u have the unit 256^(14 - o); orders 0 .. 7 are kept
// in one FP32 tensor-memory accumulator each (kOzOrders of them, `cw` columns
// apart), exact for orders 0 .. 5 over kOzChunk K steps of 16 (6 x 160 x 2^14 <
// 2^24), and summed exactly in 64-bit integers.
#pragma once

#include <math.h>
#include <stdint.h>

#include "tc.cuh"

namespace etdm {

constexpr int kOzS = 8;       // base-256 digits per operand (and product orders kept)
constexpr int kOzChunk = 10;  // K steps between read-outs
constexpr int kOzBad = 0x7ff; // exponent field of a set with an infinity or NaN

static_assert(6LL * kOzChunk * 16 * 128 * 128 <= (1LL << 24), "orders 0-5 of a chunk are exact in FP32");

__device__ __forceinline__ int exp_field(double x) { return (int)((__double2hiint(x) >> 20) & 0x7ff); }

// round(x 2^(1084 - bmax)) for |x| < 2^(bmax - 1022) (larger x saturate at +-2^62)
__device__ __forceinline__ long long to_fixed(double x, int bmax) {
  const long long b = __double_as_longlong(x);
  const int f = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffLL;
  m |= f ? (1LL << 52) : 0;
  const int sh = 9 - (bmax - max(f, 1));
  if (sh > 9) {
    m = 1LL << 62;
  } else if (sh >= 0) {
    m <<= sh;
  } else {
    const int r = min(-sh, 63);
    m = (m + (1LL << (r - 1))) >> r;
  }
  return b < 0 ? -m : m;
}

// 128 added to every byte: byte 7 - t is digit t + 128
__device__ __forceinline__ unsigned long long biased(long long x) {
  return (unsigned long long)x + 0x8080808080808080ULL;
}

// digit t as a float (exact)
template <int T>
__device__ __forceinline__ float digit(unsigned long long y) {
  const uint32_t w = T < 4 ? (uint32_t)(y >> 32) : (uint32_t)y;
  return __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 + (3 - (T & 3)))), 8388736.f);
}

__device__ __forceinline__ int oz_int(uint32_t bits) { return __float2int_rn(__uint_as_float(bits)); }

// 4 columns of the eight accumulators, cw columns apart, of a lane quarter
__device__ __forceinline__ void oz_ld_issue(uint32_t t, uint32_t (&r)[32], uint32_t cw) {
#pragma unroll
  for (int o = 0; o < 8; ++o)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[4 * o]), "=r"(r[4 * o + 1]), "=r"(r[4 * o + 2]), "=r"(r[4 * o + 3])
                 : "r"(t + o * cw));
}

// column j of oz_ld_issue's registers into (hi, lo): orders 0-3 and 4-7.
// |i0 256 + i1|, |i2 256 + i3| < 2^31 by the chunk bound.
__device__ __forceinline__ void oz_add(const uint32_t (&r)[32], int j, long long &hi, long long &lo) {
  const int j01 = oz_int(r[j]) * 256 + oz_int(r[4 + j]);
  const int j23 = oz_int(r[8 + j]) * 256 + oz_int(r[12 + j]);
  hi += (long long)j01 * 65536 + j23;
  lo += (long long)oz_int(r[16 + j]) * 16777216 + (long long)oz_int(r[20 + j]) * 65536 +
        (long long)oz_int(r[24 + j]) * 256 + oz_int(r[28 + j]);
}

// v 2^e without intermediate overflow or double rounding in the normal range
__device__ __forceinline__ double oz_scale(double v, int e) {
  const int f = exp_field(v) + e;
  if (f > 0 && f < 0x7ff && exp_field(v) > 0)
    return __hiloint2double(__double2hiint(v) + e * (1 << 20), __double2loint(v));
  return v == 0.0 ? 0.0 : scalbn(v, e);
}

}  // namespace etdm
