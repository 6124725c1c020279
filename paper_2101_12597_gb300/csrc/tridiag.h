// Sturm counts and interval sections of a real symmetric tridiagonal matrix:
// the eigenvalues of kpoint.cu's bisection.  Plain arithmetic, compiled for the
// device and, in the tests, for the host.
//
// A block's eigenvalues are found to their own last bit, not to a fraction of
// its norm: inverse iteration takes them as shifts, and the eigenvalues of a
// null space (rounding noise of 1e-17 of the norm) that share one shift give
// vectors that are nearly parallel, of which Gram-Schmidt keeps no basis (to
// 2^-54 of the norm, exp(A) of an A(k) whose occupied-occupied and
// virtual-virtual blocks are zero was wrong by 5e-9 at n = 144, 3e-8 at 512;
// now 5e-16).  For the same reason every block is scaled by its own norm.
#pragma once

#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define ETDM_HD __host__ __device__ __forceinline__
#else
#define ETDM_HD inline
#endif

namespace etdm {

constexpr int kTriBits = 200;  // sections end at 2^-kTriBits of the block's norm

// the smallest e^2 of a scaled block (|T| < 1): a smaller off-diagonal counts as
// 2^-210, below what the sections resolve
constexpr double kTriE2Min = 0x1p-420;

ETDM_HD long long tri_bits(double v) {
  long long b;
  memcpy(&b, &v, 8);
  return b;
}
ETDM_HD double tri_double(long long b) {
  double v;
  memcpy(&v, &b, 8);
  return v;
}
ETDM_HD int tri_exp(double v) { return (int)((tri_bits(v) >> 52) & 0x7ff); }

// v 2^k by the exponent field, k such that it stays below 2^1000; a zero of its
// sign where it leaves the normal range
ETDM_HD double tri_shift(double v, int k) {
  const int f = tri_exp(v);
  const long long b = tri_bits(v);
  return tri_double(f > 0 && f + k > 0 ? b + ((long long)k << 52) : b & (1LL << 63));
}

// Eigenvalues of rows [p, q) below x (block scaled to |T| < 1, |x| < 1.1;
// kTriE2Min <= e2 <= 1): the signs of the leading principal minors p_j =
// (d_j - x) p_(j-1) - e_(j-1)^2 p_(j-2), a change of sign per eigenvalue below
// x (a zero's sign does not matter: its neighbours have opposite ones, and
// either way one change falls on the two rows).  Three FP64 operations per row
// (the quotient form divides).  Every second row, minors that have left
// 2^+-100 are shifted by their exponents to bring the larger of the last two to
// 1: a row grows them by at most 4 and shrinks the larger by no less than
// 2^-422, so they stay in range wherever x lies, also far below the norm
// (every eighth row was not enough there), and two in a row never vanish.
ETDM_HD int tri_count(const double *d, const double *e2, int p, int q, double x) {
  auto changes = [](double v, double w) {  // of sign, 0 or 1
    return (int)((unsigned long long)(tri_bits(v) ^ tri_bits(w)) >> 63);
  };
  double pm = 1.0, pc = d[p] - x;
  int c = changes(pm, pc), j = p + 1;
  for (; j + 1 < q; j += 2) {
    const double p1 = fma(d[j] - x, pc, -(e2[j - 1] * pm));
    const double p2 = fma(d[j + 1] - x, p1, -(e2[j] * pc));
    c += changes(pc, p1) + changes(p1, p2);
    pm = p1;
    pc = p2;
    const int em = tri_exp(pm), ec = tri_exp(pc), top = ec > em ? ec : em;
    if ((unsigned)(top - 923) > 200u) {
      pc = tri_shift(pc, 1023 - top);
      pm = tri_shift(pm, 1023 - top);
    }
  }
  if (j < q) c += changes(pc, fma(d[j] - x, pc, -(e2[j - 1] * pm)));
  return c;
}

// the interval is not yet one eigenvalue to its last bit
ETDM_HD bool tri_open(double lo, double hi) {
  return hi - lo > 2.2204460492503131e-16 * (fabs(lo) + fabs(hi));
}

// section point m (1 .. P) of [lo, hi], w = (hi - lo) / (P + 1)
ETDM_HD double tri_point(double lo, double w, int m) { return fma(w, (double)m, lo); }

// rounds of P points that reach 2^-kTriBits of the norm
inline int tri_rounds(int P) { return (int)ceil((kTriBits + 1) / log2(P + 1.0)); }

}  // namespace etdm
