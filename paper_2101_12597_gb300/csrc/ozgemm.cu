// FP64 complex products of the full-A path on the 5th-generation tensor cores.
//
// FP64 runs at 1/64 of the FP32 rate on this part (1.05 TFLOP/s measured), so
// the batched products of the full-A path were bound by the FP64 pipe: 8.2 ms
// for 8 x 512^3 complex multiply-adds.  Here a product is evaluated in exact
// integer arithmetic on BF16 operands:
//   - a row of A (a column of B) is taken as 64-bit fixed point with the power
//     of two of its largest component, X = round(x 2^(62 - E)), |X| <= 2^62,
//     and X is written in eight balanced base-256 digits, |d_t| <= 128, each
//     exact in BF16 (d_0 the leading digit).  A component down to 2^-9 of the
//     row's largest keeps all of its 53 bits; every component is within 2^-63
//     of the largest.
//   - digit products of order o = t + u <= 7 are accumulated in one FP32
//     tensor-memory accumulator per order.  A product is an integer of at most
//     2^14, o + 1 of them fall on order o, and a chunk is 160 elements of K:
//     the orders up to 5 stay below 2^24 (6 x 160 x 2^14), exact whatever the
//     accumulator rounds; orders 6 and 7 can pass 2^24 only when nearly all
//     digits are extreme with one sign, and then lose units of 2^-62 of
//     |A_i| |B_j|.  The orders above 7 are dropped: below 2^-61 |A_i| |B_j| per
//     element of K.  FP64 accumulation rounds every addition at 2^-53.
//   - the read-out adds the eight exact integers of a chunk into two 64-bit
//     integers per output (orders 0-3 and 4-7), and one FP64 multiply-add at
//     the end gives the result, rounded once.
// The error is relative to the largest elements of the row and the column, not to
// the terms of the sum as in FP64: K 2^-61 |A_i| |B_j| at most.  Factors that are
// products themselves carry 2^-53 of those norms already; where elements far
// below them matter and may be exact (rho^(1/3) of orbitals' tails) the caller
// makes the factors of like size: O = C0 + C0 (U - I), and O f O^dagger in two
// factors O f^(1/2).
// A complex matrix product is one real product with K' = 2k: A' rows are the
// (re, im) pairs as stored, B' has two rows per column j of B, (re, -im) for
// the real and (im, re) for the imaginary part of C_ij, which come out
// interleaved as C is stored.
//
// What bounds it: 36 digit products per multiply-add; per K step of 16 the
// MMAs of a 128 x 64 tile take 1152 tensor cycles and about 1310 cycles of
// shared-memory traffic (12 MMAs re-read A and B slices; 48 KB of copies in).
// 128 x 64 outputs x 8 orders fill tensor memory (512 columns), so the
// read-out of a chunk is not overlapped with MMAs; a 128 x 32 tile would
// overlap it but reads the A slices from L2 twice as often.  Measured, 8
// products of 512^3: 0.37 ms with both digit passes (0.30 ms without), 8.2 ms
// on the FP64 pipe; largest error over |A||B| 5e-18 (FP64: 1.2e-16).
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "device.cuh"
#include "host.h"
#include "kpoint.h"
#include "ozdigits.cuh"
#include "tc.cuh"

namespace etdm {

constexpr int kOzRows = 128, kOzCols = 64;     // real output tile
constexpr int kOzA = kOzS * kOzRows * 32;      // A digits of a K step of 16 (32 KB)
constexpr int kOzB = kOzS * kOzCols * 32;      // B digits of a K step (16 KB)
constexpr int kOzStage = kOzA + kOzB;
constexpr int kOzStages = 4;
constexpr int kOzEpiW = 16;                    // read-out warps (lane quarter w % 4, columns 16 (w / 4))
constexpr int kOzThreads = (kOzEpiW + 2) * 32;

struct OzArgs {
  const uint8_t *asl, *bsl;   // [batch][row block][K step][digit][4 KB], [batch][column block]...[2 KB]
  const int *rexp, *cexp;     // exponent fields, [batch][nrb * 128], [batch][ncb * 32]
  double2 *C;
  long sC;
  int m, n, ldc, nks, nrb, ncb, batch;
  double alpha, beta;
  int *flags;
};

// Digits of one operand.  ROWC: the elements of a row are contiguous in memory
// (a block takes 8 rows, a warp per row for the maxima), else the rows are
// (16 rows per block).  B operands (ISB) write two real rows per row.  The
// digits go out as whole 128-byte core matrices (8 rows x 16 bytes).
template <int T, bool ISB>
__device__ __forceinline__ void put_digits(const unsigned long long (&yr)[4],
                                           const unsigned long long (&yi)[4], uint8_t *blk,
                                           int off0, int off1) {
  uint32_t w0[4], w1[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float r = digit<T>(yr[q]), i = digit<T>(yi[q]);
    w0[q] = pack_bf16(r, ISB ? -i : i);
    if (ISB) w1[q] = pack_bf16(i, r);
  }
  uint8_t *d = blk + T * (ISB ? kOzCols : kOzRows) * 32;
  *(uint4 *)(d + off0) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
  if (ISB) *(uint4 *)(d + off1) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
}

template <bool ROWC, bool ISB>
__global__ void __launch_bounds__(256) oz_slice_kernel(const double2 *Xb, long sX, int ld, int rows,
                                                       int K, int conj, uint8_t *dst, int *exps,
                                                       int nblk, int nks) {
  constexpr int R = ROWC ? 8 : 16;
  constexpr int BR = ISB ? kOzCols / 2 : kOzRows;  // rows of the operand per block of digits
  __shared__ int mx[R];
  const int b = blockIdx.y, r0 = blockIdx.x * R, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const double2 *X = Xb + (long)b * sX;
  if (tid < R) mx[tid] = 1;
  __syncthreads();
  {
    int m = 1;
    if (ROWC) {
      const int r = r0 + w;
      if (r < rows) {
        const double2 *x = X + (long)r * ld;
#pragma unroll 4
        for (int k = lane; k < K; k += 32) {
          const double2 z = x[k];
          m = max(m, max(exp_field(z.x), exp_field(z.y)));
        }
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) mx[w] = m;
    } else {
      const int r = r0 + (tid & 15);
      if (r < rows) {
#pragma unroll 4
        for (int k = tid >> 4; k < K; k += 16) {
          const double2 z = X[(long)k * ld + r];
          m = max(m, max(exp_field(z.x), exp_field(z.y)));
        }
        atomicMax(&mx[tid & 15], m);
      }
    }
  }
  __syncthreads();
  if (tid < R) exps[(long)b * nblk * BR + r0 + tid] = mx[tid];
  const int lr = ROWC ? (lane & 7) : (lane & 15);
  const int r = r0 + lr, bm = mx[lr];
  const bool in = r < rows && bm != kOzBad;
  const int rr = r % BR;
  uint8_t *base = dst + ((long)b * nblk + r / BR) * nks * (kOzS * (ISB ? kOzCols : kOzRows) * 32);
  const int gs = ROWC ? 32 : 16;
  for (int g = ROWC ? w * 4 + (lane >> 3) : w * 2 + (lane >> 4); g < nks * 2; g += gs) {
    unsigned long long yr[4], yi[4];
    double2 z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = g * 4 + q;
      z[q] = make_double2(0.0, 0.0);
      if (in && k < K) z[q] = ROWC ? X[(long)r * ld + k] : X[(long)k * ld + r];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      yr[q] = biased(to_fixed(z[q].x, bm));
      yi[q] = biased(to_fixed(conj ? -z[q].y : z[q].y, bm));
    }
    uint8_t *blk = base + (long)(g >> 1) * (kOzS * (ISB ? kOzCols : kOzRows) * 32);
    const int h = (g & 1) * 8;
    const int off0 = kstep_off(ISB ? 2 * rr : rr, h), off1 = kstep_off(ISB ? 2 * rr + 1 : rr, h);
    put_digits<0, ISB>(yr, yi, blk, off0, off1);
    put_digits<1, ISB>(yr, yi, blk, off0, off1);
    put_digits<2, ISB>(yr, yi, blk, off0, off1);
    put_digits<3, ISB>(yr, yi, blk, off0, off1);
    put_digits<4, ISB>(yr, yi, blk, off0, off1);
    put_digits<5, ISB>(yr, yi, blk, off0, off1);
    put_digits<6, ISB>(yr, yi, blk, off0, off1);
    put_digits<7, ISB>(yr, yi, blk, off0, off1);
  }
}

// ---- the product ----------------------------------------------------------------
struct OzBars {
  uint64_t full[kOzStages], empty[kOzStages], acc_full, acc_empty, fin;
  uint32_t tbase;
  int stop;
};

__global__ void __launch_bounds__(kOzThreads, 1) oz_product_kernel(OzArgs g) {
  extern __shared__ __align__(1024) uint8_t dsm[];
  __shared__ OzBars S;
  const int tid = threadIdx.x, w = uniform(tid >> 5), lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < kOzStages; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    mbar_init(&S.acc_full, 1);
    mbar_init(&S.acc_empty, kOzEpiW);
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
  const int per = g.nrb * g.ncb, ntiles = per * g.batch, nks = g.nks;

  if (w == kOzEpiW) {
    // --------------------------- digits of each K step ---------------------------
    if (lane == 0) {
      asm volatile("fence.proxy.async.global;" ::: "memory");
      int fill = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int b = t / per, rb = (t % per) / g.ncb, cb = t % g.ncb;
        const uint8_t *as = g.asl + ((size_t)b * g.nrb + rb) * nks * kOzA;
        const uint8_t *bs = g.bsl + ((size_t)b * g.ncb + cb) * nks * kOzB;
        for (int ks = 0; ks < nks; ++ks, ++fill) {
          const int s = fill % kOzStages, use = fill / kOzStages;
          if (use > 0 && !mbar_wait(&S.empty[s], (use - 1) & 1, stop)) { ok = false; break; }
          mbar_expect_tx(&S.full[s], kOzStage);
          bulk_g2s(dsm + s * kOzStage, as + (size_t)ks * kOzA, kOzA, &S.full[s]);
          bulk_g2s(dsm + s * kOzStage + kOzA, bs + (size_t)ks * kOzB, kOzB, &S.full[s]);
        }
      }
      if (!ok) atomicExch((int *)stop, 1);
      // the copies still in flight land before the block exits
      for (int q = 0; q < kOzStages && q < fill; ++q)
        mbar_wait(&S.full[(fill - 1 - q) % kOzStages], ((fill - 1 - q) / kOzStages) & 1);
    }
  } else if (w == kOzEpiW + 1) {
    // --------------------------------- MMA issue ---------------------------------
    const uint32_t id256 = idesc_bf16(256), id192 = idesc_bf16(192), id128 = idesc_bf16(128),
                   id64 = idesc_bf16(64);
    int fill = 0, ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      for (int ks = 0; ks < nks; ++ks, ++fill) {
        const bool fresh = ks % kOzChunk == 0;
        if (fresh && ch > 0 && !mbar_wait_warp(&S.acc_empty, (ch - 1) & 1, stop)) { ok = false; break; }
        const int s = fill % kOzStages, use = fill / kOzStages;
        if (!mbar_wait_warp(&S.full[s], use & 1, stop)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a0 = su32(dsm + s * kOzStage), b0 = a0 + kOzA;
        // digit q of A times digits 0 .. 7 - q of B (consecutive rows in
        // shared memory) adds into the orders q .. 7 (consecutive columns)
        const uint64_t B0 = smem_desc(b0), B4 = smem_desc(b0 + 4 * kOzCols * 32);
        if (fresh) {
          mma_bf16<false>(tmem, smem_desc(a0), B0, id256);
          mma_bf16<false>(tmem + 256, smem_desc(a0), B4, id256);
        } else {
          mma_bf16<true>(tmem, smem_desc(a0), B0, id256);
          mma_bf16<true>(tmem + 256, smem_desc(a0), B4, id256);
        }
#pragma unroll
        for (int q = 1; q < kOzS; ++q) {
          const uint64_t A = smem_desc(a0 + q * kOzRows * 32);
          const uint32_t d = tmem + q * kOzCols;
          const int nc = kOzS - q;  // digits of B
          mma_bf16<true>(d, A, B0, nc >= 4 ? id256 : nc == 3 ? id192 : nc == 2 ? id128 : id64);
          if (nc > 4) mma_bf16<true>(d + 256, A, B4, nc == 7 ? id192 : nc == 6 ? id128 : id64);
        }
        mma_commit(&S.empty[s]);
        if (ks % kOzChunk == kOzChunk - 1 || ks == nks - 1) {
          mma_commit(&S.acc_full);
          ++ch;
        }
      }
    }
    if (!ok && lane == 0) atomicExch((int *)stop, 1);
    mma_commit(&S.fin);  // every MMA issued has completed before the TMEM is released
    mbar_wait_warp(&S.fin, 0);
  } else {
    // ------------------------- read-out and outputs -------------------------
    const int quad = w & 3, part = w >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + part * 16;
    const int nch = (nks + kOzChunk - 1) / kOzChunk;
    int ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int b = t / per, rb = (t % per) / g.ncb, cb = t % g.ncb;
      long long hi[16], lo[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0;
      for (int c = 0; c < nch; ++c, ++ch) {
        ok = __all_sync(0xffffffffu, mbar_wait(&S.acc_full, ch & 1, stop));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int cg = 0; cg < 4; ++cg) {
          uint32_t r[32];
          oz_ld_issue(tbase + cg * 4, r, kOzCols);
          tmem_ld_wait(r);
          if (cg == 3) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) oz_add(r, j, hi[cg * 4 + j], lo[cg * 4 + j]);
        }
      }
      if (!ok) break;
      const int i = rb * kOzRows + quad * 32 + lane;
      if (i >= g.m) continue;
      const int ea = g.rexp[(long)b * g.nrb * kOzRows + i];
      const int j0 = cb * (kOzCols / 2) + part * 8;  // complex columns j0 .. j0 + 7
      double2 *out = g.C + (long)b * g.sC + (long)i * g.ldc + j0;
      const int *ce = g.cexp + (long)b * g.ncb * (kOzCols / 2) + j0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (j0 + c >= g.n) break;
        const int eb = ce[c];
        double2 v;
        if (ea == kOzBad || eb == kOzBad) {
          v = make_double2(nan(""), nan(""));
        } else {
          const int e = ea + eb - 2112;
          v.x = oz_scale(fma((double)hi[2 * c], 4294967296.0, (double)lo[2 * c]), e);
          v.y = oz_scale(fma((double)hi[2 * c + 1], 4294967296.0, (double)lo[2 * c + 1]), e);
        }
        if (g.alpha != 1.0) { v.x *= g.alpha; v.y *= g.alpha; }
        if (g.beta != 0.0) {
          const double2 o = out[c];
          v.x = fma(g.beta, o.x, v.x);
          v.y = fma(g.beta, o.y, v.y);
        }
        out[c] = v;
      }
    }
    if (!ok) atomicExch((int *)stop, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (w == 0) tmem_dealloc(tmem);
  if (tid == 0 && S.stop) atomicExch(g.flags + FLAG_ERR, ETDM_ERR_TIMEOUT);
}

// ---- host side -------------------------------------------------------------------
namespace {
int oz_ksteps(int k) { return (k + 7) / 8; }
size_t oz_a_bytes(int n) { return (size_t)((n + kOzRows - 1) / kOzRows) * oz_ksteps(n) * kOzA; }
size_t oz_b_bytes(int n) { return (size_t)((2 * n + kOzCols - 1) / kOzCols) * oz_ksteps(n) * kOzB; }
int oz_rows_pad(int n, int q) { return (n + q - 1) / q * q; }

template <bool ISB>
cudaError_t oz_slice(const OzMat &X, int b0, int rows, int k, int batch, uint8_t *dst, int *exps,
                     cudaStream_t s) {
  constexpr int BR = ISB ? kOzCols / 2 : kOzRows;
  const int nblk = (rows + BR - 1) / BR, nks = oz_ksteps(k);
  const double2 *p = X.p + b0 * X.stride;
  if (X.rows_contiguous)
    oz_slice_kernel<true, ISB><<<dim3(nblk * BR / 8, batch), 256, 0, s>>>(p, X.stride, X.ld, rows, k, X.conj,
                                                                          dst, exps, nblk, nks);
  else
    oz_slice_kernel<false, ISB><<<dim3(nblk * BR / 16, batch), 256, 0, s>>>(p, X.stride, X.ld, rows, k, X.conj,
                                                                            dst, exps, nblk, nks);
  return cudaGetLastError();
}
}  // namespace

// Workspace for n x n products over a batch: as many matrices at a time as 512
// MB holds.  Without memory for it the products stay on the FP64 kernel.
void oz_alloc(etdm_handle *h, int n, int batch) {
  OzWork &W = h->oz;
  const size_t per = oz_a_bytes(n) + oz_b_bytes(n);
  W.group = (int)std::min<size_t>(batch, std::max<size_t>(1, ((size_t)512 << 20) / per));
  const size_t ex = (size_t)W.group * (oz_rows_pad(n, kOzRows) + oz_rows_pad(n, kOzCols / 2));
  unsigned char *p = nullptr;
  if (cudaMalloc(&p, per * W.group + ex * sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    W = OzWork{};
    return;
  }
  h->allocs.push_back(p);
  W.n = n;
  W.sms = h->num_sms;
  W.a = p;
  W.b = p + oz_a_bytes(n) * W.group;
  W.rexp = (int *)(p + per * W.group);
  W.cexp = W.rexp + (size_t)W.group * oz_rows_pad(n, kOzRows);
}

// C = alpha A B + beta C over a batch, A m x k by rows, B n x k by the columns of
// the product's second factor (m, n, k <= W.n)
cudaError_t oz_gemm(const OzWork &W, const OzMat &A, const OzMat &B, double2 *C, long sC, int ldc, int m,
                    int n, int k, int batch, double alpha, double beta, int *flags, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(oz_product_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kOzStages * kOzStage);
  if (e != cudaSuccess) return e;
  for (int b0 = 0; b0 < batch; b0 += W.group) {
    const int nb = std::min(W.group, batch - b0);
    if ((e = oz_slice<false>(A, b0, m, k, nb, W.a, W.rexp, s)) != cudaSuccess) return e;
    if ((e = oz_slice<true>(B, b0, n, k, nb, W.b, W.cexp, s)) != cudaSuccess) return e;
    OzArgs g{};
    g.asl = W.a; g.bsl = W.b; g.rexp = W.rexp; g.cexp = W.cexp;
    g.C = C + b0 * sC; g.sC = sC;
    g.m = m; g.n = n; g.ldc = ldc;
    g.nks = oz_ksteps(k);
    g.nrb = (m + kOzRows - 1) / kOzRows;
    g.ncb = (2 * n + kOzCols - 1) / kOzCols;
    g.batch = nb;
    g.alpha = alpha; g.beta = beta;
    g.flags = flags;
    const int tiles = g.nrb * g.ncb * nb;
    oz_product_kernel<<<std::min(tiles, W.sms), kOzThreads, kOzStages * kOzStage, s>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// C = alpha op(A) op(B) + beta C for a batch of n x n matrices (n = W.n)
cudaError_t launch_oz_zgemm(const OzWork &W, const double2 *A, int opa, const double2 *B, int opb,
                            double2 *C, int batch, double alpha, double beta, int *flags,
                            cudaStream_t s) {
  const int n = W.n;
  const long nn = (long)n * n;
  // rows of op(A): contiguous for A, columns of A for A^dagger; columns of op(B)
  return oz_gemm(W, OzMat{A, nn, n, opa == 0, opa}, OzMat{B, nn, n, opb != 0, opb}, C, nn, n, n, n, n, batch,
                 alpha, beta, flags, s);
}

}  // namespace etdm
