// Potential and energy terms on the grid (Eq. 1): the spectral Poisson solve
// v_H(G) = 4 pi rho(G) / G^2 (G != 0), the external potential of Gaussian ion
// charges, Slater exchange, and the grid sums of the energy, in FP64.
//
// The 1-D transforms are mixed-radix Stockham (radices 2..13) on lines held in
// shared memory.  An evaluation runs five passes on half a spectrum (rho is
// real): z forward (two real lines as one complex line), y forward, x forward
// with the Poisson kernel and x inverse, y inverse, z inverse with the
// potential and the energy sums.  The set-up's v_ext takes the plain complex
// 3-D transform (fft3d).
//
// A warp-wide FP64 operation holds its scheduler for about 75 cycles here, so
// the passes count FP64 operations per warp: half the spectrum, the Poisson
// kernel from a table (it cost two divisions per point), an FP32-seeded cube
// root, one thread per output in the radices from 5 up (a thread per radix-13
// butterfly ran 676 of them in a row), and few lines per block so that every
// SM has work.
#include <math.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace etdm {

constexpr int kFftLines = 16;
constexpr int kFftThreads = 256;

struct FftPlan {
  int n;
  int nst;
  int radix[12];
};

static FftPlan make_plan(int n) {
  FftPlan p{};
  p.n = n;
  int m = n;
  const int order[] = {4, 2, 3, 5, 7, 11, 13};
  for (int r : order) {
    while (m % r == 0) { p.radix[p.nst++] = r; m /= r; }
  }
  return p;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// w(k) = exp(sign * 2 pi i k / n) from the forward table exp(-2 pi i k / n)
__device__ __forceinline__ double2 tw_at(const double2 *tw, int k, int sign) {
  double2 w = tw[k];
  if (sign > 0) w.y = -w.y;
  return w;
}

template <int R>
__device__ __forceinline__ void dft_small(double2 *v, const double2 *tw, int n, int sign) {
  double2 out[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    double2 acc = v[0];
#pragma unroll
    for (int r = 1; r < R; ++r) {
      int idx = (int)(((long)r * q % R) * (n / R));
      double2 w = tw_at(tw, idx, sign);
      double2 t = cmul(v[r], w);
      acc.x += t.x; acc.y += t.y;
    }
    out[q] = acc;
  }
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = out[q];
}

__device__ __forceinline__ void dft4(double2 *v, int sign) {
  double2 a = make_double2(v[0].x + v[2].x, v[0].y + v[2].y);
  double2 b = make_double2(v[0].x - v[2].x, v[0].y - v[2].y);
  double2 c = make_double2(v[1].x + v[3].x, v[1].y + v[3].y);
  double2 d = make_double2(v[1].x - v[3].x, v[1].y - v[3].y);
  // forward: multiply d by -i; inverse: by +i
  double2 dr = sign < 0 ? make_double2(d.y, -d.x) : make_double2(-d.y, d.x);
  v[0] = make_double2(a.x + c.x, a.y + c.y);
  v[2] = make_double2(a.x - c.x, a.y - c.y);
  v[1] = make_double2(b.x + dr.x, b.y + dr.y);
  v[3] = make_double2(b.x - dr.x, b.y - dr.y);
}

template <int R>
__device__ void stockham_stage(const double2 *in, double2 *out, int n, int Ns, int lines,
                               const double2 *tw, int sign) {
  const int nb = n / R;
  for (int q = threadIdx.x; q < lines * nb; q += blockDim.x) {
    int l = q / nb, j = q % nb;
    const double2 *src = in + (long)l * n;
    double2 v[R];
    int k = j % Ns;
    int step = n / (Ns * R);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      double2 x = src[j + r * nb];
      if (r > 0 && k > 0) x = cmul(x, tw_at(tw, (r * k * step) % n, sign));
      v[r] = x;
    }
    if (R == 4) dft4(v, sign);
    else if (R == 2) {
      double2 a = v[0], b = v[1];
      v[0] = make_double2(a.x + b.x, a.y + b.y);
      v[1] = make_double2(a.x - b.x, a.y - b.y);
    } else dft_small<R>(v, tw, n, sign);
    double2 *dst = out + (long)l * n;
    int base = (j / Ns) * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[base + r * Ns] = v[r];
  }
}

// Layout [A][n][Bdim]; transform along n.  Each block takes kFftLines lines.
__global__ void __launch_bounds__(kFftThreads) fft_axis_kernel(double2 *data, long A, long Bdim,
                                                               const double2 *tw, FftPlan plan,
                                                               int sign) {
  extern __shared__ double2 fsm[];
  const int n = plan.n;
  double2 *b0 = fsm, *b1 = fsm + kFftLines * n;
  long a0, bb0;
  int lines;
  if (Bdim == 1) {
    a0 = (long)blockIdx.x * kFftLines;
    bb0 = 0;
    lines = (int)min((long)kFftLines, A - a0);
  } else {
    long chunks = (Bdim + kFftLines - 1) / kFftLines;
    a0 = blockIdx.x / chunks;
    bb0 = (blockIdx.x % chunks) * kFftLines;
    lines = (int)min((long)kFftLines, Bdim - bb0);
  }
  // load
  if (Bdim == 1) {
    const double2 *src = data + a0 * n;
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) b0[q] = src[q];
  } else {
    for (int q = threadIdx.x; q < kFftLines * n; q += blockDim.x) {
      int i = q / kFftLines, l = q % kFftLines;
      if (l < lines) b0[l * n + i] = data[(a0 * n + i) * Bdim + bb0 + l];
    }
  }
  __syncthreads();
  int Ns = 1;
  double2 *in = b0, *out = b1;
  for (int s = 0; s < plan.nst; ++s) {
    int R = plan.radix[s];
    switch (R) {
      case 2: stockham_stage<2>(in, out, n, Ns, lines, tw, sign); break;
      case 3: stockham_stage<3>(in, out, n, Ns, lines, tw, sign); break;
      case 4: stockham_stage<4>(in, out, n, Ns, lines, tw, sign); break;
      case 5: stockham_stage<5>(in, out, n, Ns, lines, tw, sign); break;
      case 7: stockham_stage<7>(in, out, n, Ns, lines, tw, sign); break;
      case 11: stockham_stage<11>(in, out, n, Ns, lines, tw, sign); break;
      default: stockham_stage<13>(in, out, n, Ns, lines, tw, sign); break;
    }
    __syncthreads();
    Ns *= R;
    double2 *t = in; in = out; out = t;
  }
  if (Bdim == 1) {
    double2 *dst = data + a0 * n;
    for (int q = threadIdx.x; q < lines * n; q += blockDim.x) dst[q] = in[q];
  } else {
    for (int q = threadIdx.x; q < kFftLines * n; q += blockDim.x) {
      int i = q / kFftLines, l = q % kFftLines;
      if (l < lines) data[(a0 * n + i) * Bdim + bb0 + l] = in[l * n + i];
    }
  }
}

__global__ void twiddle_kernel(double2 *tw, int n) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    double s, c;
    sincospi(2.0 * (double)k / (double)n, &s, &c);
    tw[k] = make_double2(c, -s);
  }
}

cudaError_t launch_twiddles(etdm_handle *h, cudaStream_t s) {
  long off = 0;
  for (int a = 0; a < 3; ++a) {
    twiddle_kernel<<<(h->n[a] + 127) / 128, 128, 0, s>>>(h->d_tw + off, h->n[a]);
    off += h->n[a];
  }
  return cudaGetLastError();
}

// sign -1: F(k) = sum_j f(j) e^{-2 pi i jk/n}; sign +1: unnormalized inverse.
cudaError_t fft3d(etdm_handle *h, double2 *data, int sign, cudaStream_t s) {
  const int nx = h->n[0], ny = h->n[1], nz = h->n[2];
  const long dims_A[3] = {1, nx, (long)nx * ny};
  const long dims_B[3] = {(long)ny * nz, nz, 1};
  const long tw_off[3] = {0, nx, (long)nx + ny};
  for (int ax = 2; ax >= 0; --ax) {
    int n = h->n[ax];
    FftPlan plan = make_plan(n);
    long A = dims_A[ax], Bd = dims_B[ax];
    long blocks = (Bd == 1) ? (A + kFftLines - 1) / kFftLines
                            : A * ((Bd + kFftLines - 1) / kFftLines);
    size_t sm = (size_t)2 * kFftLines * n * sizeof(double2);
    cudaError_t e = allow_smem(fft_axis_kernel, 2 * kFftLines * kMaxFFT * (int)sizeof(double2));
    if (e != cudaSuccess) return e;
    fft_axis_kernel<<<(unsigned)blocks, kFftThreads, sm, s>>>(data, A, Bd, h->d_tw + tw_off[ax],
                                                              plan, sign);
  }
  return cudaGetLastError();
}

__device__ __forceinline__ double gcomp(int k, int n, double h) {
  int sk = (k < (n + 1) / 2) ? k : k - n;
  double val = 1.0 / ((double)n * h);
  return (2.0 * M_PI) * ((double)sk * val);
}

// v_ext(G) = -(4 pi / (Omega G^2)) exp(-G^2 sigma^2 / 2) sum_I Z_I exp(-i G.R_I)
__global__ void vext_recip_kernel(double2 *out, int nx, int ny, int nz, double hx, double hy,
                                  double hz, const double *pos, const double *Z, int n_atoms,
                                  double omega, double sigma) {
  long G = (long)nx * ny * nz;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < G;
       e += (long)gridDim.x * blockDim.x) {
    int k = (int)(e % nz), j = (int)((e / nz) % ny), i = (int)(e / ((long)ny * nz));
    double gx = gcomp(i, nx, hx), gy = gcomp(j, ny, hy), gz = gcomp(k, nz, hz);
    double g2 = gx * gx + gy * gy + gz * gz;
    double2 acc = make_double2(0.0, 0.0);
    if (e != 0) {
      for (int I = 0; I < n_atoms; ++I) {
        double ph = -(gx * pos[3 * I] + gy * pos[3 * I + 1] + gz * pos[3 * I + 2]);
        double sn, cs;
        sincos(ph, &sn, &cs);
        acc.x += Z[I] * cs;
        acc.y += Z[I] * sn;
      }
      double f = -4.0 * M_PI / (omega * g2) * exp(-g2 * sigma * sigma / 2.0);
      acc.x *= f;
      acc.y *= f;
    }
    out[e] = acc;
  }
}

cudaError_t launch_vext_recip(etdm_handle *h, cudaStream_t s) {
  vext_recip_kernel<<<2048, 256, 0, s>>>(h->d_fft, h->n[0], h->n[1], h->n[2], h->h[0], h->h[1],
                                         h->h[2], h->d_pos, h->d_Z, h->n_atoms, h->omega,
                                         h->sigma);
  return cudaGetLastError();
}

__global__ void real_part_kernel(const double2 *src, double *dst, long n) {
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long)gridDim.x * blockDim.x)
    dst[e] = src[e].x;
}

cudaError_t launch_real_part(etdm_handle *h, const double2 *src, double *dst, cudaStream_t s) {
  real_part_kernel<<<2048, 256, 0, s>>>(src, dst, h->G);
  return cudaGetLastError();
}

// ---- the evaluation's passes -----------------------------------------------------
constexpr int kPotThreads = 128;
constexpr int kPotLinesMax = 8;  // lines (z: pairs of real lines) per block, at most

struct PotArgs {
  int nx, ny, nz, nzh;
  FftPlan px, py, pz;
  const double2 *twx, *twy, *twz;  // forward twiddles
  double2 *H;                      // [nx][ny][nzh] half spectrum
  const double *kp;                // [nx][ny][nzh] 4 pi / (|G|^2 Ng), 0 at G = 0
  const double *rho, *vext;        // vext: null for a self-interaction potential
  double *v, *part;
  double dV, fk;
  int lines;                       // per block
};

// One output element of a radix-R stage: sum_r x_r w^(r idx), idx = (j mod Ns)
// n / (Ns R) + q n / R for output q of butterfly j.
template <int R>
__device__ void stage_outputs(const double2 *in, double2 *out, int n, int Ns, int lines,
                              const double2 *tw, int sign) {
  const int nb = n / R, step = n / (Ns * R);
  for (int e = threadIdx.x; e < lines * n; e += blockDim.x) {
    const int l = e / n, o = e % n;
    const int blk = o / (Ns * R), w = o % (Ns * R), q = w / Ns, k = w % Ns;
    const double2 *src = in + (long)l * n + blk * Ns + k;
    int idx = k * step + q * nb;
    if (idx >= n) idx -= n;
    double2 acc = src[0];
    int m = 0;
#pragma unroll
    for (int r = 1; r < R; ++r) {
      m += idx;
      if (m >= n) m -= n;
      const double2 x = src[r * nb], t = tw_at(tw, m, sign);
      acc.x = fma(x.x, t.x, fma(-x.y, t.y, acc.x));
      acc.y = fma(x.x, t.y, fma(x.y, t.x, acc.y));
    }
    out[(long)l * n + o] = acc;
  }
}

// Radix 3: a + (b + c), a - (b + c) / 2 +- i s (b - c) sin(2 pi / 3)
__device__ void stage3(const double2 *in, double2 *out, int n, int Ns, int lines, const double2 *tw,
                       int sign) {
  const int nb = n / 3, step = n / (Ns * 3);
  const double h = sign < 0 ? -0.86602540378443864676 : 0.86602540378443864676;
  for (int e = threadIdx.x; e < lines * nb; e += blockDim.x) {
    const int l = e / nb, j = e % nb, k = j % Ns;
    const double2 *src = in + (long)l * n;
    const double2 a = src[j];
    double2 b = src[j + nb], c = src[j + 2 * nb];
    if (k > 0) {
      b = cmul(b, tw_at(tw, k * step, sign));
      c = cmul(c, tw_at(tw, 2 * k * step, sign));
    }
    const double2 t = make_double2(b.x + c.x, b.y + c.y), d = make_double2(b.x - c.x, b.y - c.y);
    const double2 u = make_double2(fma(-0.5, t.x, a.x), fma(-0.5, t.y, a.y));
    double2 *dst = out + (long)l * n + (j / Ns) * Ns * 3 + k;
    dst[0] = make_double2(a.x + t.x, a.y + t.y);
    dst[Ns] = make_double2(fma(-h, d.y, u.x), fma(h, d.x, u.y));
    dst[2 * Ns] = make_double2(fma(h, d.y, u.x), fma(-h, d.x, u.y));
  }
}

// transform of `lines` lines held in b0; the result's buffer; ends with a block barrier
__device__ double2 *fft_lines(double2 *b0, double2 *b1, const FftPlan &pl, int lines, const double2 *tw,
                              int sign) {
  int Ns = 1;
  for (int s = 0; s < pl.nst; ++s) {
    const int R = pl.radix[s];
    switch (R) {
      case 2: stockham_stage<2>(b0, b1, pl.n, Ns, lines, tw, sign); break;
      case 3: stage3(b0, b1, pl.n, Ns, lines, tw, sign); break;
      case 4: stockham_stage<4>(b0, b1, pl.n, Ns, lines, tw, sign); break;
      case 5: stage_outputs<5>(b0, b1, pl.n, Ns, lines, tw, sign); break;
      case 7: stage_outputs<7>(b0, b1, pl.n, Ns, lines, tw, sign); break;
      case 11: stage_outputs<11>(b0, b1, pl.n, Ns, lines, tw, sign); break;
      default: stage_outputs<13>(b0, b1, pl.n, Ns, lines, tw, sign); break;
    }
    __syncthreads();
    Ns *= R;
    double2 *t = b0;
    b0 = b1;
    b1 = t;
  }
  return b0;
}

__global__ void __launch_bounds__(kPotThreads) pot_zfwd_kernel(PotArgs a) {
  extern __shared__ double2 psm[];
  const int n = a.nz, nzh = a.nzh, lb = a.lines;
  const long NL = (long)a.nx * a.ny, L0 = (long)blockIdx.x * lb * 2;
  double2 *tw = psm, *b0 = psm + n, *b1 = b0 + lb * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = a.twz[i];
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int p = q / n, z = q % n;
    const long La = L0 + 2 * p;
    b0[q] = make_double2(La < NL ? a.rho[La * n + z] : 0.0, La + 1 < NL ? a.rho[(La + 1) * n + z] : 0.0);
  }
  __syncthreads();
  const double2 *X = fft_lines(b0, b1, a.pz, lb, tw, -1);
  // F_a(k) = (X(k) + conj X(-k)) / 2,  F_b(k) = (X(k) - conj X(-k)) / (2i)
  for (int q = threadIdx.x; q < lb * nzh; q += blockDim.x) {
    const int p = q / nzh, k = q % nzh;
    const long La = L0 + 2 * p;
    const double2 F = X[p * n + k], G = X[p * n + (k ? n - k : 0)];
    if (La < NL) a.H[La * nzh + k] = make_double2(0.5 * (F.x + G.x), 0.5 * (F.y - G.y));
    if (La + 1 < NL) a.H[(La + 1) * nzh + k] = make_double2(0.5 * (F.y + G.y), 0.5 * (G.x - F.x));
  }
}

// y lines (fixed x, kz), in place
__global__ void __launch_bounds__(kPotThreads) pot_y_kernel(PotArgs a, int sign) {
  extern __shared__ double2 psm[];
  const int n = a.ny, nzh = a.nzh, lb = a.lines;
  const long nl = (long)a.nx * nzh, q0 = (long)blockIdx.x * lb;
  const int lines = (int)min((long)lb, nl - q0);
  double2 *tw = psm, *b0 = psm + n, *b1 = b0 + lb * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = a.twy[i];
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int y = q / lb, l = q % lb;
    if (l < lines) b0[l * n + y] = a.H[((q0 + l) / nzh * n + y) * nzh + (q0 + l) % nzh];
  }
  __syncthreads();
  const double2 *Y = fft_lines(b0, b1, a.py, lines, tw, sign);
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int y = q / lb, l = q % lb;
    if (l < lines) a.H[((q0 + l) / nzh * n + y) * nzh + (q0 + l) % nzh] = Y[l * n + y];
  }
}

// x lines: forward, Poisson kernel, inverse, in place
__global__ void __launch_bounds__(kPotThreads) pot_x_kernel(PotArgs a) {
  extern __shared__ double2 psm[];
  const int n = a.nx, lb = a.lines;
  const long stride = (long)a.ny * a.nzh, q0 = (long)blockIdx.x * lb;
  const int lines = (int)min((long)lb, stride - q0);
  double2 *tw = psm, *b0 = psm + n, *b1 = b0 + lb * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = a.twx[i];
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int x = q / lb, l = q % lb;
    if (l < lines) b0[l * n + x] = a.H[x * stride + q0 + l];
  }
  __syncthreads();
  double2 *X = fft_lines(b0, b1, a.px, lines, tw, -1);
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int x = q / lb, l = q % lb;
    if (l < lines) {
      const double f = a.kp[x * stride + q0 + l];
      const double2 v = X[l * n + x];
      X[l * n + x] = make_double2(v.x * f, v.y * f);
    }
  }
  __syncthreads();
  const double2 *Y = fft_lines(X, X == b0 ? b1 : b0, a.px, lines, tw, +1);
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int x = q / lb, l = q % lb;
    if (l < lines) a.H[x * stride + q0 + l] = Y[l * n + x];
  }
}

// r^(1/3), r >= 0: FP32 seed and two Newton steps with the FP32 slope's
// reciprocal (the error shrinks by 2^-22 in each, so the second one ends at
// FP64 rounding), nine FP64 operations; cbrt() outside FP32's comfortable range
__device__ __forceinline__ double root3(double r) {
  if (!(r > 1e-30 && r < 1e30)) return cbrt(r);
  const float yf = cbrtf((float)r);
  const double s = (double)(1.f / (3.f * yf * yf));
  double y = (double)yf;
  y = fma(-fma(y * y, y, -r), s, y);
  return fma(-fma(y * y, y, -r), s, y);
}

// z lines, inverse: two half spectra rebuilt into one complex line; then, per
// point, v = v_ext + v_H + v_x and the energy sums.  SIC: v_H[n] + v_x^pol[n]
// of an orbital density and part[b] = -f_k dV sum (n v_H / 2 + 3/4 n v_x^pol).
template <bool SIC>
__global__ void __launch_bounds__(kPotThreads) pot_zinv_kernel(PotArgs a) {
  extern __shared__ double2 psm[];
  const int n = a.nz, nzh = a.nzh, lb = a.lines;
  const long NL = (long)a.nx * a.ny, L0 = (long)blockIdx.x * lb * 2;
  double2 *tw = psm, *b0 = psm + n, *b1 = b0 + lb * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = a.twz[i];
  for (int q = threadIdx.x; q < lb * n; q += blockDim.x) {
    const int p = q / n, k = q % n;
    const long La = L0 + 2 * p;
    const bool up = k >= nzh;
    const int kk = up ? n - k : k;
    double2 va = La < NL ? a.H[La * nzh + kk] : make_double2(0.0, 0.0);
    double2 vb = La + 1 < NL ? a.H[(La + 1) * nzh + kk] : make_double2(0.0, 0.0);
    if (up) { va.y = -va.y; vb.y = -vb.y; }
    b0[q] = make_double2(va.x - vb.y, va.y + vb.x);
  }
  __syncthreads();
  const double2 *Z = fft_lines(b0, b1, a.pz, lb, tw, +1);
  const double cx = SIC ? 1.2407009817988000333 : 0.98474502184269655;  // (6 / pi)^(1/3), (3 / pi)^(1/3)
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  for (int q = threadIdx.x; q < lb * 2 * n; q += blockDim.x) {
    const int pl = q / n, z = q % n;  // line L0 + pl, pl = 2 p + (0 | 1)
    const long L = L0 + pl;
    if (L >= NL) continue;
    const double2 zz = Z[(pl >> 1) * n + z];
    const double h = (pl & 1) ? zz.y : zz.x;
    const long gp = L * n + z;
    const double r = a.rho[gp], rp = r > 0.0 ? r : 0.0;
    const double vx = -cx * root3(rp);
    s1 = fma(r, h, s1);
    s2 = fma(rp, vx, s2);  // eps_x = (3/4) rho v_x
    if (SIC) {
      a.v[gp] = h + vx;
    } else {
      const double ve = a.vext[gp];
      a.v[gp] = ve + h + vx;
      s0 = fma(r, ve, s0);
    }
  }
  if (!SIC) s0 = block_sum(s0);
  s1 = block_sum(s1);
  s2 = block_sum(s2);
  if (threadIdx.x == 0) {
    if (SIC) {
      a.part[blockIdx.x] = -a.fk * a.dV * (0.5 * s1 + 0.75 * s2);
    } else {
      a.part[3 * blockIdx.x] = a.dV * s0;
      a.part[3 * blockIdx.x + 1] = 0.5 * a.dV * s1;
      a.part[3 * blockIdx.x + 2] = 0.75 * a.dV * s2;
    }
  }
}

__global__ void pot_kernel_kernel(double *kp, int nx, int ny, int nz, int nzh, double hx, double hy,
                                  double hz) {
  const long total = (long)nx * ny * nzh;
  const double Ng = (double)nx * ny * nz;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long)gridDim.x * blockDim.x) {
    const int k = (int)(e % nzh), j = (int)((e / nzh) % ny), i = (int)(e / ((long)ny * nzh));
    const double gx = gcomp(i, nx, hx), gy = gcomp(j, ny, hy), gz = gcomp(k, nz, hz);
    kp[e] = e == 0 ? 0.0 : 4.0 * M_PI / ((gx * gx + gy * gy + gz * gz) * Ng);
  }
}

// lines per block: about two blocks per SM, up to kPotLinesMax
static int pot_lines(long lines, int sms) {
  return (int)std::max<long>(1, std::min<long>(kPotLinesMax, (lines + 2L * sms - 1) / (2L * sms)));
}

int pot_blocks(const etdm_handle *h) {
  const long pairs = ((long)h->n[0] * h->n[1] + 1) / 2;
  const int lb = pot_lines(pairs, h->num_sms);
  return (int)((pairs + lb - 1) / lb);
}

cudaError_t launch_potential_setup(etdm_handle *h, cudaStream_t s) {
  pot_kernel_kernel<<<1024, 256, 0, s>>>(h->d_kpois64, h->n[0], h->n[1], h->n[2], h->n[2] / 2 + 1,
                                         h->h[0], h->h[1], h->h[2]);
  return cudaGetLastError();
}

// The five passes: v and the energy partials (3 per block of pot_blocks) of
// rho, or (sic) the orbital potential and one partial per block.
cudaError_t launch_potential(etdm_handle *h, const double *rho, double *v, double *part, bool sic,
                             double fk, cudaStream_t s) {
  PotArgs a{};
  a.nx = h->n[0]; a.ny = h->n[1]; a.nz = h->n[2];
  a.nzh = a.nz / 2 + 1;
  a.px = make_plan(a.nx); a.py = make_plan(a.ny); a.pz = make_plan(a.nz);
  a.twx = h->d_tw; a.twy = h->d_tw + a.nx; a.twz = h->d_tw + a.nx + a.ny;
  a.H = h->d_fft;
  a.kp = h->d_kpois64;
  a.rho = rho; a.vext = h->d_vext; a.v = v; a.part = part;
  a.dV = h->dV; a.fk = fk;
  const long pairs = ((long)a.nx * a.ny + 1) / 2, ly = (long)a.nx * a.nzh, lx = (long)a.ny * a.nzh;
  const int bz = pot_lines(pairs, h->num_sms), by = pot_lines(ly, h->num_sms), bx = pot_lines(lx, h->num_sms);
  auto smem = [](int n, int lb) { return (size_t)(n + 2 * lb * n) * sizeof(double2); };
  const size_t sz = smem(a.nz, bz), sy = smem(a.ny, by), sx = smem(a.nx, bx);
  const int most = (int)smem(kMaxFFT, kPotLinesMax);
  for (auto k : {pot_zfwd_kernel, pot_x_kernel, pot_zinv_kernel<false>, pot_zinv_kernel<true>})
    if (const cudaError_t e = allow_smem(k, most)) return e;
  if (const cudaError_t e = allow_smem(pot_y_kernel, most)) return e;
  const unsigned gz = (unsigned)((pairs + bz - 1) / bz), gy = (unsigned)((ly + by - 1) / by),
                 gx = (unsigned)((lx + bx - 1) / bx);
  a.lines = bz;
  pot_zfwd_kernel<<<gz, kPotThreads, sz, s>>>(a);
  a.lines = by;
  pot_y_kernel<<<gy, kPotThreads, sy, s>>>(a, -1);
  a.lines = bx;
  pot_x_kernel<<<gx, kPotThreads, sx, s>>>(a);
  a.lines = by;
  pot_y_kernel<<<gy, kPotThreads, sy, s>>>(a, +1);
  a.lines = bz;
  if (sic) pot_zinv_kernel<true><<<gz, kPotThreads, sz, s>>>(a);
  else pot_zinv_kernel<false><<<gz, kPotThreads, sz, s>>>(a);
  return cudaGetLastError();
}

}  // namespace etdm
