// FP64 grid passes on the 5th-generation tensor cores: basis -> grid density
// (Eq. 2, 12) and grid -> basis potential matrix (Eq. 11) of the FP64 path and
// of the full-A path, in exact base-256 digits (ozdigits.cuh).
//
// FP64 FMA bounds these passes on this part (1.05 TFLOP/s): the 4 x 4 x 4-tile
// kernels of grid.cu take 11.2 ms (density) and 9.4 ms (V) for 96 atoms on a
// 96^3 grid.  Here a 4 x 4 x 8 tile of 128 points with n <= 128 list entries is
//   density:  Y = X D_loc (128 x n x n),  rho_p = sum_b Y_pb X_pb ,
//   V:        V_loc = X^T (v X)           (n x n x 128),
// with X, D and v in 64-bit fixed point and the products' digits on tcgen05;
// sums stay exact in 64- and 128-bit integers up to rho (one rounding to FP64)
// and to V's 64-bit fixed point, so no FP64 arithmetic is left in either pass
// and V is independent of the order of its additions.
//
//   X: one entry per function and tile, periodic images of a function that
//      reach the tile summed (the phase between images is 1 at the Gamma point;
//      a box of 6.4 A has some 150 images of 16 functions per tile); with
//      k-points one entry per image, the pair's lattice offset looked up.
//      Evaluated once in FP64 at set-up and kept twice, with all of its 53 bits:
//      for the density, whose rows are points, as a left-justified mantissa and
//      its distance from the point's largest exponent, [entry][128]; for V, whose
//      rows are entries, in fixed point with the power of two of the entry's
//      largest value in the tile.  (One power of two for the whole system left
//      the density around a molecule, where X is 1e-16 of the largest, with
//      relative errors of 2e-2; now 2e-14.)
//   D: positive semidefinite, so |D_ab| <= sqrt(D_aa D_bb): D_ab 2^-(e_a + e_b)
//      with D_aa < 2^2e_a in fixed point, and X_pa 2^e_a in the density pass,
//      in fixed point with the power of two of the point's largest of these.
//      Where the density is faint it keeps its relative accuracy, which
//      rho^(1/3) passes on to v (one power of two for all of D left 1e-9 of v,
//      and 6e-11 of H, on an atom whose orbitals are empty; one per tile 1e-12
//      and 3e-13).
//   v: fixed point with the power of two of its largest element in the tile.
//   V: 64-bit fixed point with a factor 2 in reserve over the Cauchy-Schwarz
//      bound of |V_ab|, max |v dV| (sum X_a^2 sum X_b^2)^(1/2) (sums wrap
//      harmlessly in between): the unit is 2^-62 of that bound, where an FP64
//      sum rounds at 2^-53 of the terms it adds.
//
// One persistent block per SM: 8 or 16 warps read the accumulators (lane quarter
// w % 4, column part w / 4), two or one sets of eight warps cut the digits of
// the K steps of 16 in turn into a four-stage ring, warp 24 issues the MMAs.  The
// columns of a tile go in passes of 64 (eight orders of 64 columns fill tensor
// memory), the last one 64, 32 or 16 wide.  A tile's K is at most 128, one exact
// chunk.
//
// What bounds it: a K step's MMAs take 1152 tensor cycles, its digits some 3500
// instructions and a column's read-out 50 per warp, and the three do not overlap
// fully (the accumulators fill tensor memory).  The inputs of a step are loaded
// a step of the set ahead, by lanes along consecutive elements: X is kept twice,
// [entry][point] for the density and [pair of points][entry] for V, and D is
// read by its columns.  With one set of builders and V's rows 1 KB apart, D's
// 2 KB, a step waited for its loads: 32 waters 1.23 and 1.21 ms, now 1.07 and
// 1.03 ms (11.2 and 9.4 ms on the FP64 pipe), of which the exponents of single
// values and of entries and tiles take 0.04 each; the points' shifts take another
// 0.02 with the conversion of D.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "device.cuh"
#include "host.h"
#include "kpoint.h"
#include "ozdigits.cuh"

namespace etdm {

constexpr int kOxP = 128;                       // points per tile (4 x 4 x 8)
constexpr int kOxN = 128;                       // list entries per tile, at most
constexpr int kOxCols = 64;                     // columns of a pass, at most
constexpr int kOxA = kOzS * 128 * 32, kOxB = kOzS * kOxCols * 32;
constexpr int kOxStage = kOxA + kOxB;           // 48 KB
constexpr int kOxStages = 4;
constexpr int kOxBldW = 8;                      // warps of a builder set
constexpr int kOxThreads = 25 * 32;
// Warps of a pass: the density's builders wait for gathered elements of D, V's
// read-out has the atomics (16 + 1 x 8 and 8 + 2 x 8 warps, 32 waters, with one
// power of two for X: density 1.16 and 1.03 ms, V 1.00 and 1.08 ms)
template <bool RHO>
struct OxRoles {
  static constexpr int epi = RHO ? 8 : 16, sets = RHO ? 2 : 1;
  static constexpr int parts = epi / 4;               // column parts of the read-out
  static constexpr int mma = epi + sets * kOxBldW;    // the MMA warp
  static_assert((mma + 1) * 32 == kOxThreads, "every role has its warps");
};
constexpr int kOxParts = 256;                   // partial maxima of a fixed-point conversion

struct OxArgs {
  GridGeom g;               // 4 x 4 x 8 tiles
  KGeom G;                  // lattice offsets (k-points)
  int n_tiles;
  const int *ptr, *id;      // entries of a tile; mu, or the image key (k-points)
  const long long *x;       // density: [entry][128] words of ox_word
  const long long *xt;      // V: per tile [64 pairs of points][entry][2], fixed point
  const short *pexp;        // density: [tile][128] exponent field of a point's largest |X|
  const uint8_t *pmin;      // density: [tile][128] bits from max |X_pa| max 2^e_a to max |X_pa 2^e_a|
  const short *q;           // V: [entry] bits from the entry's unit to the function's
  const long long *dfix;    // density: scaled D, or DR per offset
  const int *ee, *ct;       // density: exponents e_a of the functions; -max e_a of a tile
  const int *bexp;          // exponent field of v dV
  double *rho;
  const long long *vt;      // V: v dV in tile order
  const int *vq;            // V: [tile] bits from the tile's unit of v to the largest
  unsigned long long *V;    // V: sums, [M][M] (upper triangle), or [offset][M][M]
  int full;                 // V: both triangles
  int *flags;
};

__device__ __forceinline__ int ox_point(const GridGeom &g, int t, int p) {
  const int bz = t % g.nbz, by = (t / g.nbz) % g.nby, bx = t / (g.nbz * g.nby);
  const int i = bx * 4 + (p >> 5), j = by * 4 + ((p >> 3) & 3), k = bz * 8 + (p & 7);
  return (i < g.nx && j < g.ny && k < g.nz) ? (i * g.ny + j) * g.nz + k : -1;
}

// index of the lattice offset n_a - n_b of two image keys, -1 beyond the table
__device__ __forceinline__ int ox_ridx(const KGeom &G, int ka, int kb) {
  const int rx = ((ka >> 6) & 7) - ((kb >> 6) & 7), ry = ((ka >> 3) & 7) - ((kb >> 3) & 7),
            rz = (ka & 7) - (kb & 7);
  if (abs(rx) > G.Rm[0] || abs(ry) > G.Rm[1] || abs(rz) > G.Rm[2]) return -1;
  return ((rx + G.Rm[0]) * (2 * G.Rm[1] + 1) + ry + G.Rm[1]) * (2 * G.Rm[2] + 1) + rz + G.Rm[2];
}

// ---- set-up -------------------------------------------------------------------
// X of a tile's entries in FP64 (into the tables' memory): entry e sums the
// images keys[ek[e]] .. keys[ek[e + 1] - 1]; the exponent fields of a point's
// and of an entry's largest |X| in the tile, and sum X^2 per function
__global__ void __launch_bounds__(kOxP) ox_basis_kernel(GridGeom g, Tables tb, const int *ptr, const int *id,
                                                        int shift, const int *ek, const int *keys, double *x,
                                                        short *pexp, short *xe, double *s2) {
  __shared__ int big[kOxN];
  const int t = blockIdx.x, p = threadIdx.x, e0 = ptr[t], n = ptr[t + 1] - e0;
  const int bz = t % g.nbz, by = (t / g.nbz) % g.nby, bx = t / (g.nbz * g.nby);
  const int i = bx * 4 + (p >> 5), j = by * 4 + ((p >> 3) & 3), k = bz * 8 + (p & 7);
  const bool in = i < g.nx && j < g.ny && k < g.nz;
  big[p] = 1;
  __syncthreads();
  int top = 1;
  for (int e = 0; e < n; ++e) {
    double s = 0.0;
    for (int q = ek[e0 + e]; in && q < ek[e0 + e + 1]; ++q) {
      const int key = keys[q], mu = key >> 9;
      const int ix = ((key >> 6) & 7) - 4 + kImgMax, iy = ((key >> 3) & 7) - 4 + kImgMax,
                iz = (key & 7) - 4 + kImgMax;
      const long ax = ((long)mu * kImgN + ix) * g.nx + i, ay = ((long)mu * kImgN + iy) * g.ny + j,
                 az = ((long)mu * kImgN + iz) * g.nz + k;
      const double r2 = __dadd_rn(__dadd_rn(tb.sq[0][ax], tb.sq[1][ay]), tb.sq[2][az]);
      if (r2 < tb.rc2[mu]) s += tb.norm[mu] * tb.ex[0][ax] * tb.ex[1][ay] * tb.ex[2][az];
    }
    x[(long)(e0 + e) * kOxP + p] = s;
    const int f = exp_field(s), m = __reduce_max_sync(0xffffffffu, f);
    top = max(top, f);
    double q = s * s;
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if ((p & 31) == 0) {
      atomicMax(&big[e], m);
      atomicAdd(s2 + (id[e0 + e] >> shift), q);
    }
  }
  pexp[(long)t * kOxP + p] = (short)top;
  __syncthreads();
  if (p < n) xe[e0 + p] = (short)big[p];
}

// X as a left-justified mantissa (53 bits, 2^61 <= |m| < 2^62) and, in its lowest
// seven bits, the distance k of its exponent field from the point's largest,
// top: X = m 2^(top - 1084 - k).  Zero 128 bits below the largest, and for
// subnormal numbers (their squares are no FP64 numbers).
__device__ __forceinline__ long long ox_word(double v, int top) {
  const long long b = __double_as_longlong(v);
  const int f = exp_field(v), k = top - f;
  if (f == 0 || k > 127) return 0;
  const long long m = ((b & 0xfffffffffffffLL) | (1LL << 52)) << 9;
  return (b < 0 ? -m : m) | k;
}
// its fixed-point value in the unit 2^(top - 1084 + s), s + k >= 0 unless it is zero
__device__ __forceinline__ long long ox_value(long long w, int s) {
  const int r = min(max(s + ((int)w & 127), 0), 63);
  return ((w & ~511LL) + (long long)((1ULL << r) >> 1)) >> r;
}

// h with sum X^2 < 2^2h for a function's sum of squares
__device__ __forceinline__ int ox_hexp(double s2) { return (max(exp_field(s2), 1) - 1021) >> 1; }

// the tables of X (x holds it in FP64 on entry), and the entries' exponent
// fields q as the bits from their units to those of their functions
__global__ void __launch_bounds__(kOxP) ox_xfix_kernel(const int *ptr, const int *id, int shift, int M,
                                                       const short *pexp, const double *s2, long long *x,
                                                       long long *xt, uint8_t *kx, short *q, int *hx) {
  __shared__ short xe[kOxN];
  const int t = blockIdx.x, p = threadIdx.x, e0 = ptr[t], n = ptr[t + 1] - e0;
  if (p < n) xe[p] = q[e0 + p];
  __syncthreads();
  if (p < n)  // at least 0: X^2 <= sum X^2; a unit 100 bits away adds nothing
    q[e0 + p] = (short)min(ox_hexp(s2[id[e0 + p] >> shift]) - xe[p] + 1022, 100);
  const int top = pexp[(long)t * kOxP + p];
  long long *const xp = xt + (long)e0 * kOxP + (long)(p >> 1) * n * 2 + (p & 1);
  for (int e = 0; e < n; ++e) {
    const double v = __longlong_as_double(x[(long)(e0 + e) * kOxP + p]);
    xp[2 * e] = to_fixed(v, xe[e]);
    const long long w = ox_word(v, top);
    x[(long)(e0 + e) * kOxP + p] = w;
    kx[(long)(e0 + e) * kOxP + p] = w ? (uint8_t)(w & 127) : 255;
  }
  for (int m = blockIdx.x * kOxP + p; m < M; m += gridDim.x * kOxP) hx[m] = ox_hexp(s2[m]);
}

// ---- per evaluation: D and v in fixed point --------------------------------------
// e with d < 2^2e
__device__ __forceinline__ int ox_dexp(double d) { return (exp_field(d) - 1021) >> 1; }
// that of an infinity or NaN: a tile with such a function has no density (where
// an element of D is not finite, those of its row and column on the diagonal
// are neither)
constexpr int kOxBad = (kOzBad - 1021) >> 1;

// D_ab 2^-(e_a + e_b) (one bit in reserve for rounding), the exponents and the
// tiles' largest ones (kOxBad: no number), the points' shifts pmin; diag: the
// offset 0 of DR (its diagonal bounds every offset)
__global__ void __launch_bounds__(256) ox_dfix_kernel(const double *D, long n, const double *diag, int M,
                                                      int shift, int n_tiles, const int *ptr, const int *id,
                                                      const uint32_t *kx, long long *dst, int *ee, int *ct,
                                                      uint32_t *pmin) {
  const long MM = (long)M * M, gtid = (long)blockIdx.x * 256 + threadIdx.x, gs = (long)gridDim.x * 256;
  for (long q = gtid; q < n; q += gs) {
    const long r = q % MM;
    const int a = (int)(r / M), b = (int)(r % M);
    dst[q] = to_fixed(D[q], 1023 + ox_dexp(diag[(long)a * (M + 1)]) + ox_dexp(diag[(long)b * (M + 1)]));
  }
  for (long a = gtid; a < M; a += gs) ee[a] = ox_dexp(diag[a * (M + 1)]);
  const int lane = threadIdx.x & 31;
  for (long t = gtid >> 5; t < n_tiles; t += gs >> 5) {
    const int e0 = ptr[t], n = ptr[t + 1] - e0;
    int ex[4], m = -2000;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = lane + 32 * q;
      ex[q] = e < n ? ox_dexp(diag[(long)(id[e0 + e] >> shift) * (M + 1)]) : -2000;
      m = max(m, ex[q]);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) ct[t] = -m;
    // four points a lane, in 16-bit pairs: the least k + (max e - e_a) over the
    // entries, 255 at most (32 entries' loads in flight)
    uint32_t least[2] = {0x00ff00ffu, 0x00ff00ffu};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (32 * q >= n) break;
      uint32_t k4[32];
#pragma unroll
      for (int l = 0; l < 32; ++l)
        k4[l] = 32 * q + l < n ? __ldg(kx + (long)(e0 + 32 * q + l) * 32 + lane) : 0xffffffffu;
      const uint32_t d = min(m - ex[q], 255) * 0x00010001u;
#pragma unroll
      for (int l = 0; l < 32; ++l) {
        const uint32_t dl = __shfl_sync(0xffffffffu, d, l);
        least[0] = __viaddmin_u16x2(__byte_perm(k4[l], 0, 0x4140), dl, least[0]);
        least[1] = __viaddmin_u16x2(__byte_perm(k4[l], 0, 0x4342), dl, least[1]);
      }
    }
    pmin[t * 32 + lane] = __byte_perm(least[0], least[1], 0x6420);
  }
}

// partial maxima of the exponent fields of src
__global__ void __launch_bounds__(256) ox_max_kernel(const double *src, long n, double scale, int *part) {
  __shared__ int sm[8];
  int m = 1;
  for (long e = (long)blockIdx.x * 256 + threadIdx.x; e < n; e += (long)gridDim.x * 256)
    m = max(m, exp_field(src[e] * scale));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) m = max(m, sm[q]);
    part[blockIdx.x] = m;
  }
}
__device__ __forceinline__ int ox_total_max(const int *part, int np) {
  __shared__ int sm[8];
  int m = (int)threadIdx.x < np ? part[threadIdx.x] : 1;
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  m = sm[0];
  for (int q = 1; q < 8; ++q) m = max(m, sm[q]);
  return m;
}
// v dV in tile order (0 outside the grid), a warp per tile, in the unit of the
// tile's largest; vq: the bits from there to the largest of all
__global__ void __launch_bounds__(256) ox_vfix_kernel(GridGeom g, int n_tiles, const double *v, const int *part,
                                                      int np, long long *dst, int *vq, int *bexp) {
  const int b = ox_total_max(part, np), lane = threadIdx.x & 31;
  if (blockIdx.x == 0 && threadIdx.x == 0) *bexp = b;
  for (long t = ((long)blockIdx.x * 256 + threadIdx.x) >> 5; t < n_tiles; t += gridDim.x * 8L) {
    double x[4];
    int m = 1;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int gp = ox_point(g, (int)t, lane + 32 * u);
      x[u] = gp < 0 ? 0.0 : v[gp] * g.dV;
      m = max(m, exp_field(x[u]));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) vq[t] = min(b - m, 100);
#pragma unroll
    for (int u = 0; u < 4; ++u) dst[t * kOxP + lane + 32 * u] = b == kOzBad ? 0 : to_fixed(x[u], m);
  }
}

// ---- the passes -----------------------------------------------------------------
struct OxBars {
  uint64_t full[kOxStages], empty[kOxStages], acc_full, acc_empty, fin;
  uint64_t part_full[2], part_empty[2];
  uint32_t tbase;
  int stop;
  __int128 part[2][OxRoles<true>::parts - 1][kOxP];  // column parts of rho, two tiles in flight
  int id[OxRoles<true>::sets * kOxBldW][kOxN], ee[OxRoles<true>::sets * kOxBldW][kOxN];  // entries of a builder warp's tile
};

// columns of pass h of a tile of n entries: 64, and the last 64, 32 or 16
__device__ __forceinline__ int ox_cols(int n, int h) {
  const int rem = n - h * kOxCols;
  return rem > 32 ? 64 : rem > 16 ? 32 : 16;
}

// digit T of the eight values y (row r of a block of `rows` rows, columns h * 8 ..)
template <int T, int N>
__device__ __forceinline__ void ox_put(const unsigned long long (&y)[N], uint8_t *dst) {
  uint32_t w[N / 2];
#pragma unroll
  for (int u = 0; u < N / 2; ++u) w[u] = pack_bf16(digit<T>(y[2 * u]), digit<T>(y[2 * u + 1]));
  if constexpr (N == 8) *(uint4 *)dst = make_uint4(w[0], w[1], w[2], w[3]);
  else *(uint2 *)dst = make_uint2(w[0], w[1]);
}
template <int N>
__device__ __forceinline__ void ox_put_all(const unsigned long long (&y)[N], uint8_t *dst, int stride) {
  ox_put<0, N>(y, dst);
  ox_put<1, N>(y, dst + stride);
  ox_put<2, N>(y, dst + 2 * stride);
  ox_put<3, N>(y, dst + 3 * stride);
  ox_put<4, N>(y, dst + 4 * stride);
  ox_put<5, N>(y, dst + 5 * stride);
  ox_put<6, N>(y, dst + 6 * stride);
  ox_put<7, N>(y, dst + 7 * stride);
}

// floor(x y / 2^62) of two fixed-point numbers of at most 2^62
__device__ __forceinline__ long long ox_mul62(long long x, long long y) {
  return (long long)(((unsigned long long)__mul64hi(x, y) << 2) | ((unsigned long long)(x * y) >> 62));
}

// MMAs of one K step: digit q of A times digits 0 .. 7 - q of B, CW columns each,
// into the orders q .. 7 (at most 256 columns per MMA)
template <int CW, bool FRESH>
__device__ __forceinline__ void ox_mma(uint32_t tmem, uint32_t a0, uint32_t b0) {
  constexpr int per = 256 / CW;  // digits of B in one MMA
#pragma unroll
  for (int q = 0; q < kOzS; ++q) {
    const uint64_t A = smem_desc(a0 + q * 128 * 32);
#pragma unroll
    for (int u = 0; u < kOzS - q; u += per) {
      const int nd = per < kOzS - q - u ? per : kOzS - q - u;
      if (FRESH && q == 0) mma_bf16<false>(tmem + (q + u) * CW, A, smem_desc(b0 + u * CW * 32), idesc_bf16(nd * CW));
      else mma_bf16<true>(tmem + (q + u) * CW, A, smem_desc(b0 + u * CW * 32), idesc_bf16(nd * CW));
    }
  }
}
template <int CW>
__device__ __forceinline__ void ox_mma_step(uint32_t tmem, uint32_t a0, bool fresh) {
  if (fresh) ox_mma<CW, true>(tmem, a0, a0 + kOxA);
  else ox_mma<CW, false>(tmem, a0, a0 + kOxA);
}

// RHO: density, else V; KP: entries are images, matrices per lattice offset
template <bool RHO, bool KP>
__global__ void __launch_bounds__(kOxThreads, 1) ox_pass_kernel(OxArgs g) {
  using W = OxRoles<RHO>;
  extern __shared__ __align__(1024) uint8_t dsm[];
  __shared__ OxBars S;
  const int tid = threadIdx.x, w = uniform(tid >> 5), lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kOxStages; ++s) {
      mbar_init(&S.full[s], kOxBldW);
      mbar_init(&S.empty[s], 1);
    }
    mbar_init(&S.acc_full, 1);
    mbar_init(&S.acc_empty, W::epi);
    for (int q = 0; q < 2; ++q) {
      mbar_init(&S.part_full[q], W::epi - 4);  // the warps of the parts from 1 up
      mbar_init(&S.part_empty[q], 4);           // the warps of part 0
    }
    mbar_init(&S.fin, 1);
    S.stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 0) tmem_alloc(&S.tbase);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = uniform(S.tbase);
  volatile int *stop = &S.stop;
  const int M = g.g.M;
  const long MM = (long)M * M;

  if (w == W::mma) {
    // --------------------------------- MMA issue ---------------------------------
    int fill = 0, ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x) {
      const int n = uniform(g.ptr[t + 1] - g.ptr[t]), nks = RHO ? (n + 15) / 16 : kOxP / 16;
      for (int h = 0; h * kOxCols < n && ok; ++h, ++ch) {
        const int cw = ox_cols(n, h);
        if (ch > 0 && !mbar_wait_warp(&S.acc_empty, (ch - 1) & 1, stop)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int ks = 0; ks < nks; ++ks, ++fill) {
          const int s = fill % kOxStages, use = fill / kOxStages;
          if (!mbar_wait_warp(&S.full[s], use & 1, stop)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = su32(dsm + s * kOxStage);
          if (cw == 64) ox_mma_step<64>(tmem, a0, ks == 0);
          else if (cw == 32) ox_mma_step<32>(tmem, a0, ks == 0);
          else ox_mma_step<16>(tmem, a0, ks == 0);
          mma_commit(&S.empty[s]);
        }
        if (ok) mma_commit(&S.acc_full);
      }
    }
    if (!ok && lane == 0) atomicExch((int *)stop, 1);
    mma_commit(&S.fin);  // every MMA issued has completed before the TMEM is released
    mbar_wait_warp(&S.fin, 0);
  } else if (w >= W::epi) {
    // ----------------------------- digits of each K step -----------------------------
    // The inputs of a step are loaded while the previous one's digits are cut
    // (one step's chain of L2 loads is about as long as its MMAs).
    // The sets take the steps in turn.
    const int bw = w - W::epi, set = bw / kOxBldW, bt = tid - (W::epi + set * kOxBldW) * 32;
    const int r = bt & 127, hh = bt >> 7;  // A: row, half of the K step
    int first = 0;                         // steps of the tiles before
    bool ok = true;
    for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x) {
      const int e0 = g.ptr[t], n = g.ptr[t + 1] - e0, nks = RHO ? (n + 15) / 16 : kOxP / 16;
      const int steps = (n + kOxCols - 1) / kOxCols * nks;
      int rm = 0;
      if (RHO) {
        const int top = -g.ct[t];  // ids and exponents of the tile's entries, a copy per warp
        rm = g.pmin[(long)t * kOxP + r];
        __syncwarp();
        for (int e = lane; e < n; e += 32) {
          const int id = __ldg(g.id + e0 + e);
          S.id[bw][e] = id;
          S.ee[bw][e] = min(top - __ldg(g.ee + (KP ? id >> 9 : id)), 512);
        }
        __syncwarp();
      }
      // inputs of step st: pass h = st / nks, K step ks = st % nks.  A: 8 values
      // of row r; B: row bi of the pass, 4 consecutive K per item, cw * 4 items
      auto load = [&](int st, long long (&xa)[8], long long (&xb)[4], longlong2 (&xv)[2]) {
        const int h = st / nks, ks = st - h * nks, cw = ox_cols(n, h);
        const int bi = bt & (cw - 1), bq = bt / cw, be = h * kOxCols + bi;
        const bool in = bt < cw * 4 && be < n;
        if (RHO) {  // rows: points, K: entries
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int e = ks * 16 + hh * 8 + u;
            xa[u] = e < n ? __ldg(g.x + (long)(e0 + e) * kOxP + r) : 0;
          }
          const int idb = in ? S.id[bw][be] : 0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {  // D[k][b] = D[b][k]: the lanes along b read consecutive elements
            const int e = ks * 16 + bq * 4 + u;
            xb[u] = 0;
            if (in && e < n) {
              const int ide = S.id[bw][e];
              if (KP) {
                const int ri = ox_ridx(g.G, ide, idb);
                if (ri >= 0) xb[u] = __ldg(g.dfix + ri * MM + (long)(ide >> 9) * M + (idb >> 9));
              } else {
                xb[u] = __ldg(g.dfix + (long)ide * M + idb);
              }
            }
          }
        } else {  // rows: entries, K: points
          const longlong2 *px = (const longlong2 *)(g.xt + (long)e0 * kOxP) + (long)ks * 8 * n;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const longlong2 z = r < n ? __ldg(px + (hh * 4 + u) * n + r) : make_longlong2(0, 0);
            xa[2 * u] = z.x;
            xa[2 * u + 1] = z.y;
          }
          const longlong2 *pv = (const longlong2 *)(g.vt + (long)t * kOxP + ks * 16 + min(bq, 3) * 4);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const longlong2 z = in ? __ldg(px + (bq * 2 + u) * n + be) : make_longlong2(0, 0);
            xb[2 * u] = z.x;
            xb[2 * u + 1] = z.y;
            xv[u] = __ldg(pv + u);
          }
        }
      };
      long long xa[8], xb[4];
      longlong2 xv[2];
      const int st0 = (set + W::sets - first % W::sets) % W::sets;
      if (st0 < steps) load(st0, xa, xb, xv);
      for (int st = st0; st < steps; st += W::sets) {
        const int fill = first + st;
        const int h = st / nks, ks = st - h * nks, cw = ox_cols(n, h);
        const int bi = bt & (cw - 1), bq = bt / cw;
        const int s = fill % kOxStages, use = fill / kOxStages;
        // (voted: a lane that gave up alone would leave the others at a __syncwarp)
        if (use > 0 && !mbar_wait_warp(&S.empty[s], (use - 1) & 1, stop)) { ok = false; break; }
        uint8_t *stg = dsm + s * kOxStage;
        unsigned long long ya[8], yb[4];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int e = ks * 16 + hh * 8 + u;
          ya[u] = biased(RHO ? (e < n ? ox_value(xa[u], S.ee[bw][e] - rm) : 0) : xa[u]);
        }
        if (RHO) {
#pragma unroll
          for (int u = 0; u < 4; ++u) yb[u] = biased(xb[u]);
        } else {  // W = v X
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            yb[2 * u] = biased(ox_mul62(xb[2 * u], xv[u].x));
            yb[2 * u + 1] = biased(ox_mul62(xb[2 * u + 1], xv[u].y));
          }
        }
        if (st + W::sets < steps) load(st + W::sets, xa, xb, xv);
        ox_put_all<8>(ya, stg + kstep_off(r, hh * 8), 128 * 32);
        if (bt < cw * 4) ox_put_all<4>(yb, stg + kOxA + kstep_off(bi, bq * 4), cw * 32);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.full[s]);
      }
      first += steps;
    }
    if (!ok) atomicExch((int *)stop, 1);
  } else {
    // ------------------------------- read-out -------------------------------
    const int quad = w & 3, part = w >> 2, row = quad * 32 + lane;
    const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16);
    int ch = 0, nt = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < g.n_tiles && ok; t += gridDim.x, ++nt) {
      const int e0 = g.ptr[t], n = g.ptr[t + 1] - e0;
      const int gp = RHO ? ox_point(g.g, t, row) : 0;
      const int rm = RHO ? (int)g.pmin[(long)t * kOxP + row] : 0;
      const int rexp = RHO ? (int)g.pexp[(long)t * kOxP + row] - g.ct[t] - rm : 0;
      const bool bad = RHO && g.ct[t] == -kOxBad;
      // ids and, from bit 24, units (V) or shifts (density) of the tile's entries,
      // entry lane + 32 q
      int ent[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = lane + 32 * q;
        ent[q] = e < n ? __ldg(g.id + e0 + e) : 0;
        if (RHO && e < n) ent[q] = min(-g.ct[t] - __ldg(g.ee + (KP ? ent[q] >> 9 : ent[q])), 512);
        if (!RHO && e < n) ent[q] |= (int)__ldg(g.q + e0 + e) << 24;
      }
      auto entry = [&](int b) {  // (b: the same in every lane)
        const int lo = b & 32 ? ent[1] : ent[0], hi = b & 32 ? ent[3] : ent[2];
        return __shfl_sync(0xffffffffu, b & 64 ? hi : lo, b & 31);
      };
      const int ida = RHO ? 0 : ent[quad] & 0xffffff;  // entry `row`
      // bits from the unit of the tile's sums to V's, without the column's; at
      // least 6 (2^-1084 x 2^-1084 x 2^56 against 2^(-1084 - 1022))
      const int ra = RHO ? 0 : 6 + (ent[quad] >> 24) + __ldg(g.vq + t);
      // density: X of the next four columns, loaded a group ahead
      long long xn[4];
      auto ahead = [&](int b0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) xn[j] = b0 + j < n ? __ldg(g.x + (long)(e0 + b0 + j) * kOxP + row) : 0;
      };
      if (RHO) ahead(part * (ox_cols(n, 0) / W::parts));
      __int128 acc = 0;
      for (int h = 0; h * kOxCols < n; ++h, ++ch) {
        const int cw = ox_cols(n, h), cp = cw / W::parts;  // columns of this part
        ok = __all_sync(0xffffffffu, mbar_wait(&S.acc_full, ch & 1, stop));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int c0 = 0; c0 < cp; c0 += 4) {
          const int b0 = h * kOxCols + part * cp + c0;
          long long x4[4];
          if (RHO) {
#pragma unroll
            for (int j = 0; j < 4; ++j) x4[j] = ox_value(xn[j], entry(b0 + j) - rm);
            const int b1 = c0 + 4 < cp ? b0 + 4 : (h + 1) * kOxCols + part * (ox_cols(n, h + 1) / W::parts);
            if (c0 + 4 < cp || (h + 1) * kOxCols < n) ahead(b1);
          }
          uint32_t r[32];
          oz_ld_issue(tbase + part * cp + c0, r, cw);
          tmem_ld_wait(r);
          if (c0 + 4 >= cp) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int b = b0 + j;
            const int eb = RHO ? 0 : entry(b), idb = eb & 0xffffff;
            long long hi = 0, lo = 0;
            oz_add(r, j, hi, lo);
            const __int128 T = ((__int128)hi << 32) + lo;  // |T| <= 2^75
            if (RHO) {
              // (a column beyond n has X = 0)
              acc += ((__int128)(long long)(T >> 13) * x4[j]) >> 8;
            } else if (b < n && b <= row && row < n) {
              const int r = min(ra + (eb >> 24), 100);
              const long long v = (long long)((T + ((__int128)1 << (r - 1))) >> r);
              if (v != 0) {
                if (KP) {  // VR[n_a - n_b][mu_a][mu_b], and the transposed pair
                  const int ri = ox_ridx(g.G, ida, idb);
                  if (ri >= 0) {
                    const int ma = ida >> 9, mb = idb >> 9;
                    atomicAdd(g.V + ri * MM + (long)ma * M + mb, (unsigned long long)v);
                    if (b != row)
                      atomicAdd(g.V + ox_ridx(g.G, idb, ida) * MM + (long)mb * M + ma, (unsigned long long)v);
                  }
                } else {  // entries ascend: mu_b <= mu_a
                  atomicAdd(g.V + (long)idb * M + ida, (unsigned long long)v);
                  if (g.full && b != row) atomicAdd(g.V + (long)ida * M + idb, (unsigned long long)v);
                }
              }
            }
          }
        }
      }
      if (!ok) break;
      if (RHO) {
        // the column parts of each point, summed exactly
        const int q = nt & 1;
        if (part > 0) {
          if (nt >= 2) ok = __all_sync(0xffffffffu, mbar_wait(&S.part_empty[q], ((nt >> 1) - 1) & 1, stop));
          S.part[q][part - 1][row] = acc;
          __syncwarp();
          if (lane == 0) mbar_arrive(&S.part_full[q]);
          continue;
        }
        ok = __all_sync(0xffffffffu, mbar_wait(&S.part_full[q], (nt >> 1) & 1, stop));
#pragma unroll
        for (int c = 0; c < W::parts - 1; ++c) acc += S.part[q][c][row];
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.part_empty[q]);
        if (ok && gp >= 0) {
          const bool neg = acc < 0;
          unsigned __int128 u = neg ? -(unsigned __int128)acc : (unsigned __int128)acc;
          // the leading 63 bits as FP64
          const unsigned long long top = (unsigned long long)(u >> 64);
          const int lz = top ? __clzll((long long)top) : 64 + __clzll((long long)(unsigned long long)u);
          const int drop = max(0, 65 - lz);
          const double m = (double)(long long)(unsigned long long)(u >> drop);
          const double v = oz_scale(m, drop + 2 * rexp - 2152);
          g.rho[gp] = bad ? nan("") : neg ? -v : v;
        }
      }
    }
    if (!ok) atomicExch((int *)stop, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (w == 0) tmem_dealloc(tmem);
  if (tid == 0 && S.stop) atomicExch(g.flags + FLAG_ERR, ETDM_ERR_TIMEOUT);
}

// H += the fixed-point sums (upper triangle), unit 2^(bV + h_a + h_b - 1084)
__global__ void __launch_bounds__(256) ox_vadd_kernel(const unsigned long long *V, int M, const int *hx,
                                                      const int *bexp, double *H) {
  const int b = *bexp;
  const long MM = (long)M * M;
  for (long e = (long)blockIdx.x * 256 + threadIdx.x; e < MM; e += (long)gridDim.x * 256) {
    const int i = (int)(e / M), j = (int)(e % M);
    if (i > j) continue;
    H[e] += b == kOzBad ? nan("") : oz_scale((double)(long long)V[e], b + hx[i] + hx[j] - 1084);
  }
}
// the sums as FP64, in place (a matrix per blockIdx.y)
__global__ void __launch_bounds__(256) ox_vcvt_kernel(double *V, int M, const int *hx, const int *bexp) {
  const int b = *bexp;
  const unsigned e = blockIdx.x * 256 + threadIdx.x, MM = (unsigned)M * M;
  if (e >= MM) return;
  const int h = hx[e / (unsigned)M] + hx[e % (unsigned)M];
  double *const v = V + (size_t)blockIdx.y * MM + e;
  *v = b == kOzBad ? nan("") : oz_scale((double)__double_as_longlong(*v), b + h - 1084);
}

// ---- host side -------------------------------------------------------------------
namespace {

OxArgs ox_args(etdm_handle *h) {
  const OxGrid &o = h->ox;
  OxArgs a{};
  a.g = o.geom;
  a.G = h->kg;
  a.n_tiles = o.n_tiles;
  a.ptr = o.ptr; a.id = o.id; a.x = o.x; a.xt = o.xt; a.pexp = o.pexp; a.pmin = o.pmin;
  a.q = o.q;
  a.dfix = o.dfix; a.ee = o.ee; a.ct = o.ct; a.bexp = o.bexp; a.vt = o.vt; a.vq = o.vq;
  a.flags = h->d_flags;
  return a;
}

template <bool RHO, bool KP>
cudaError_t ox_launch(const OxArgs &a, int sms, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(ox_pass_kernel<RHO, KP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kOxStages * kOxStage);
  if (e != cudaSuccess) return e;
  ox_pass_kernel<RHO, KP><<<std::min(a.n_tiles, sms), kOxThreads, kOxStages * kOxStage, s>>>(a);
  return cudaGetLastError();
}

int ox_parts(long n) { return (int)std::max<long>(1, std::min<long>(kOxParts, (n + 2047) / 2048)); }

}  // namespace

// Tables of the passes from the 4 x 4 x 8 tiles' image lists (ptr, keys on the
// host and on the device).  `images`: one entry per image, else per function.
// Leaves h->ox.n_tiles = 0 (the passes of grid.cu run) when a tile has more
// than 128 entries, the tables (2.1 KB per entry) would take more than half of
// the free memory, or a function has no finite sum of squares.
void ox_setup(etdm_handle *h, const GridGeom &geom, int n_tiles, const std::vector<int> &kptr,
              const std::vector<int> &keys, const int *d_keys, bool images, cudaStream_t s) {
  OxGrid &o = h->ox;
  std::vector<int> ptr(n_tiles + 1, 0), id, ek;
  for (int t = 0; t < n_tiles; ++t) {
    for (int e = kptr[t]; e < kptr[t + 1]; ++e)
      if (images || e == kptr[t] || (keys[e] >> 9) != (keys[e - 1] >> 9)) {
        id.push_back(images ? keys[e] : keys[e] >> 9);
        ek.push_back(e);
      }
    ptr[t + 1] = (int)id.size();
    if (ptr[t + 1] - ptr[t] > kOxN) return;
  }
  const long ne = (long)id.size();
  if (ne == 0 || h->M >= (images ? 1 << 15 : 1 << 24)) return;  // (ids share a word with 8 bits)
  ek.push_back((int)keys.size());
  const long mats = images ? h->kg.nR : 1, MM = (long)h->M * h->M;
  const size_t nptr = ptr.size(), nV = h->kpath ? 0 : (size_t)MM, nint = nptr + id.size() + ek.size();
  const size_t bytes = (size_t)ne * (kOxP * 17 + 2) + (size_t)n_tiles * kOxP * 11 +
                       ((size_t)mats * MM + nV) * 8 + (nint + kOxParts + 1 + 2 * h->M + 2 * n_tiles) * sizeof(int) +
                       (size_t)h->M * 8 + 20 * 256;
  if (bytes > (size_t)256 << 20) {  // leave what the rest of the set-up may need
    size_t avail = 0, total = 0;
    CUDA_TRY(cudaMemGetInfo(&avail, &total));
    if (bytes > avail / 2) return;
  }
  unsigned char *p = nullptr;  // one allocation: each costs a small system's set-up some 15 us
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  h->allocs.push_back(p);
  auto take = [&p](size_t n) {
    unsigned char *q = p;
    p += (n + 255) & ~(size_t)255;
    return q;
  };
  o.x = (long long *)take((size_t)ne * kOxP * 8);  // (the allocation's address)
  o.xt = (long long *)take((size_t)ne * kOxP * 8);
  o.vt = (long long *)take((size_t)n_tiles * kOxP * 8);
  o.dfix = (long long *)take((size_t)mats * MM * 8);
  if (nV) o.V = (unsigned long long *)take(nV * 8);
  o.pexp = (short *)take((size_t)n_tiles * kOxP * sizeof(short));
  o.q = (short *)take((size_t)ne * sizeof(short));
  o.kx = take((size_t)ne * kOxP);
  o.pmin = take((size_t)n_tiles * kOxP);
  o.ptr = (int *)take(nint * sizeof(int));
  o.id = o.ptr + nptr;
  const int *d_ek = o.id + id.size();
  o.part = (int *)take(kOxParts * sizeof(int));
  o.bexp = (int *)take(sizeof(int));
  o.ee = (int *)take(h->M * sizeof(int));
  o.hx = (int *)take(h->M * sizeof(int));
  o.ct = (int *)take(n_tiles * sizeof(int));
  o.vq = (int *)take(n_tiles * sizeof(int));
  double *d_s2 = (double *)take(h->M * 8);
  CUDA_TRY(cudaMemsetAsync(d_s2, 0, h->M * 8, s));
  std::vector<int> up(ptr);
  up.insert(up.end(), id.begin(), id.end());
  up.insert(up.end(), ek.begin(), ek.end());
  CUDA_TRY(cudaMemcpyAsync(o.ptr, up.data(), nint * sizeof(int), cudaMemcpyHostToDevice, s));
  Tables tb;
  for (int a = 0; a < 3; ++a) {
    tb.sq[a] = h->d_sq + h->tab_off[a];
    tb.ex[a] = h->d_ex + h->tab_off[a];
  }
  tb.norm = h->d_norm;
  tb.rc2 = h->d_rc2;
  const int shift = images ? 9 : 0;
  ox_basis_kernel<<<n_tiles, kOxP, 0, s>>>(geom, tb, o.ptr, o.id, shift, d_ek, d_keys, (double *)o.x, o.pexp,
                                           o.q, d_s2);
  CUDA_TRY(cudaGetLastError());
  ox_xfix_kernel<<<n_tiles, kOxP, 0, s>>>(o.ptr, o.id, shift, h->M, o.pexp, d_s2, o.x, o.xt, o.kx, o.q,
                                          o.hx);
  CUDA_TRY(cudaGetLastError());
  std::vector<double> s2(h->M);
  CUDA_TRY(cudaMemcpyAsync(s2.data(), d_s2, h->M * 8, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  for (double v : s2)
    if (!std::isfinite(v)) return;
  o.geom = geom;
  o.images = images;
  o.n_tiles = n_tiles;
}

// rho on the grid from D [M][M] (Gamma point) or DR [offset][M][M]
cudaError_t launch_ox_rho(etdm_handle *h, const double *D, double *rho, cudaStream_t s) {
  const OxGrid &o = h->ox;
  const long n = (o.images ? (long)h->kg.nR : 1L) * h->M * h->M;
  const long work = std::max(n, (long)o.n_tiles * 32);
  ox_dfix_kernel<<<(int)std::min<long>(8 * h->num_sms, (work + 255) / 256), 256, 0, s>>>(
      D, n, D + (o.images ? (h->kg.nR - 1) / 2 : 0) * (long)h->M * h->M, h->M, o.images ? 9 : 0, o.n_tiles,
      o.ptr, o.id, (const uint32_t *)o.kx, o.dfix, o.ee, o.ct, (uint32_t *)o.pmin);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  OxArgs a = ox_args(h);
  a.rho = rho;
  return o.images ? ox_launch<true, true>(a, h->num_sms, s) : ox_launch<true, false>(a, h->num_sms, s);
}

namespace {
// V of the potential v into the zeroed sums V
cudaError_t ox_vmat(etdm_handle *h, const double *v, unsigned long long *V, bool full, cudaStream_t s) {
  const OxGrid &o = h->ox;
  const int np = ox_parts(h->G);
  ox_max_kernel<<<np, 256, 0, s>>>(v, h->G, o.geom.dV, o.part);
  ox_vfix_kernel<<<(int)std::min<long>(8 * h->num_sms, ((long)o.n_tiles + 7) / 8), 256, 0, s>>>(
      o.geom, o.n_tiles, v, o.part, np, o.vt, o.vq, o.bexp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  OxArgs a = ox_args(h);
  a.V = V;
  a.full = full;
  return o.images ? ox_launch<false, true>(a, h->num_sms, s) : ox_launch<false, false>(a, h->num_sms, s);
}
}  // namespace

// H (upper triangle) += V
cudaError_t launch_ox_vmat(etdm_handle *h, const double *v, double *H, cudaStream_t s) {
  const OxGrid &o = h->ox;
  const long MM = (long)h->M * h->M;
  cudaError_t e = cudaMemsetAsync(o.V, 0, MM * 8, s);
  if (e != cudaSuccess) return e;
  if ((e = ox_vmat(h, v, o.V, false, s)) != cudaSuccess) return e;
  ox_vadd_kernel<<<(int)std::min<long>(4 * h->num_sms, (MM + 255) / 256), 256, 0, s>>>(o.V, h->M, o.hx, o.bexp, H);
  return cudaGetLastError();
}

// VR [offset][M][M] = V (overwritten)
cudaError_t launch_ox_vmat_k(etdm_handle *h, const double *v, double *VR, cudaStream_t s) {
  const OxGrid &o = h->ox;
  const long n = (long)h->kg.nR * h->M * h->M;
  cudaError_t e = cudaMemsetAsync(VR, 0, n * 8, s);
  if (e != cudaSuccess) return e;
  if ((e = ox_vmat(h, v, (unsigned long long *)VR, true, s)) != cudaSuccess) return e;
  const unsigned bx = (unsigned)(((long)h->M * h->M + 255) / 256);
  ox_vcvt_kernel<<<dim3(bx, h->kg.nR), 256, 0, s>>>(VR, h->M, o.hx, o.bexp);
  return cudaGetLastError();
}

}  // namespace etdm
