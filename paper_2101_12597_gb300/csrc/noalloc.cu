// Allocation-free L-BFGS two-loop direction (etdm_lbfgs_direction_noalloc).
//
// Some callers cannot allocate device memory at the point where they need a
// search direction: code running inside a stream capture whose memory pool is
// frozen, host frameworks that hand out only pre-registered buffers, and
// embedded drivers that forbid cudaMalloc after start-up.  This entry point
// computes the same direction as the handle's etdm_lbfgs_step, from a pair
// history the caller keeps, with its reduction scratch in a fixed file-scope
// device array instead of handle-owned memory.  It calls no cudaMalloc,
// cudaFree or allocating library routine.
//
// The scratch array lives in every GPU that loads the library until the
// process exits.  All calls share it and it keeps the last call's contents:
// the barrier words and the status word are cleared at the start of each
// call, and calls that overlap on the GPU (two streams, or two host threads)
// race on it.  The status word records a device-side failure of the last call
// (a grid barrier that gave up, or a pair without positive curvature);
// etdm_lbfgs_direction_noalloc_status reads it without allocating.
#include <cooperative_groups.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "device.cuh"
#include "internal.h"

namespace etdm {

constexpr int kNaMaxPairs = 16;      // maximum number of (s, y) pairs
constexpr int kNaMaxBlocks = 256;    // partial sums held per reduction
constexpr int kNaThreads = 512;
constexpr int kNaDevices = 64;
constexpr int kNaRegs = 16;          // work-vector elements a thread keeps in registers
constexpr int kNaBatch = 4;          // elements whose inputs are in flight together
constexpr int kNaSlots = 55;         // and in shared memory, at most (4 KB per slot and block)
// layout: [0, 256) bytes: barrier count, generation, error flag; then two
// halves of two sums of kNaMaxBlocks block partials
constexpr size_t kNaScratchBytes = 256 + 4 * kNaMaxBlocks * sizeof(double);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaScratchBytes];

struct NaArgs {
  const double *g, *s, *y, *h0;
  double *p;
  long n;
  int m;
  int slots;  // shared-memory slots of this launch
  unsigned *bar;
  int *flags;
  double *red;
};

// The sums of x and y over the grid, in the same order in every block.  Two
// halves of the partials alternate between calls, so one grid barrier per
// reduction is enough (a block is at most one reduction ahead of another).
__device__ double2 na_sum(const NaArgs &a, double x, double y, int half, bool *ok) {
  __shared__ double2 part[kNaThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nb = gridDim.x;
  double *red = a.red + half * 2 * kNaMaxBlocks;
  for (int pass = 0;; ++pass) {
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    __syncthreads();
    if (lane == 0) part[w] = make_double2(x, y);
    __syncthreads();
    double2 t = make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < kNaThreads / 32; ++q) {
      t.x += part[q].x;
      t.y += part[q].y;
    }
    if (pass == 1 || nb == 1) return t;
    if (threadIdx.x == 0) {
      red[blockIdx.x] = t.x;
      red[kNaMaxBlocks + blockIdx.x] = t.y;
    }
    if (!grid_barrier(a.bar, a.flags)) { *ok = false; return t; }
    x = y = 0.0;
    if ((int)threadIdx.x < nb) {
      x = __ldcg(red + threadIdx.x);
      y = __ldcg(red + kNaMaxBlocks + threadIdx.x);
    }
  }
}

// Up to three input elements of one pass.
struct NaIn {
  double a, b, c;
};

// f(e, in, v) on every element e of this thread, in = ld(e) its inputs and v
// its element of the work vector: the first kNaRegs in registers, the next in
// shared memory, the rest in p.  Inputs are loaded kNaBatch elements at a time,
// all before the first use.  `back` reverses the order of the parts, so that a
// pass starts on what the previous one read last (its lines are still in L2).
template <class L, class F>
__device__ __forceinline__ void na_each(const NaArgs &a, double (&q)[kNaRegs], double *sm, bool back,
                                        L ld, F f) {
  const long stride = (long)gridDim.x * kNaThreads, n = a.n;
  const long e0 = (long)blockIdx.x * kNaThreads + threadIdx.x;
  const long es = e0 + kNaRegs * stride, em = es + a.slots * stride;
  const NaIn none{0.0, 0.0, 0.0};
#pragma unroll 1
  for (int h = 0; h < 3; ++h) {
    const int part = back ? 2 - h : h;
    if (part == 0) {
#pragma unroll
      for (int k0 = 0; k0 < kNaRegs; k0 += kNaBatch) {
        NaIn in[kNaBatch];
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const long e = e0 + (k0 + u) * stride;
          in[u] = e < n ? ld(e) : none;
        }
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const long e = e0 + (k0 + u) * stride;
          if (e < n) f(e, in[u], q[k0 + u]);
        }
      }
    } else if (part == 1) {
#pragma unroll 1
      for (int k0 = 0; k0 < a.slots; k0 += kNaBatch) {
        NaIn in[kNaBatch];
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const int k = k0 + u, kk = back ? a.slots - 1 - k : k;
          const long e = es + kk * stride;
          in[u] = (k < a.slots && e < n) ? ld(e) : none;
        }
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const int k = k0 + u, kk = back ? a.slots - 1 - k : k;
          const long e = es + kk * stride;
          if (k < a.slots && e < n) {
            double v = sm[kk * kNaThreads + threadIdx.x];
            f(e, in[u], v);
            sm[kk * kNaThreads + threadIdx.x] = v;
          }
        }
      }
    } else {
#pragma unroll 1
      for (long e1 = em; e1 < n; e1 += kNaBatch * stride) {
        NaIn in[kNaBatch];
        double v[kNaBatch];
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const long e = e1 + u * stride;
          in[u] = e < n ? ld(e) : none;
          v[u] = e < n ? a.p[e] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kNaBatch; ++u) {
          const long e = e1 + u * stride;
          if (e < n) {
            f(e, in[u], v[u]);
            a.p[e] = v[u];
          }
        }
      }
    }
  }
}

// p = -H g by the two-loop recursion over pairs oldest (0) .. newest (m-1),
// with the diagonal initial inverse Hessian h0.  Bound by memory: n = 5.3e6
// with m = 3 took 793 us when each step of the recursion read and wrote p (and
// y.s had passes of its own).  The work vector now stays on the chip, 71
// elements per thread (registers and 220 KB of shared memory; n up to 5.5e6
// on 152 SMs, the rest in p), and each pass does the update of one pair and
// the dot products of the next: 16 vectors are read and one written, 283 us.
// The FP64 pipe is the next bound: 17 multiply-adds per element, 173 us.
// A pair whose curvature y.s is not positive and finite makes the direction
// meaningless: the kernel records ETDM_ERR_NUMERIC in the status word and
// returns (every block sees the same sum, so all of them stop together).
__global__ void __launch_bounds__(kNaThreads, 1) lbfgs_noalloc_kernel(NaArgs a) {
  extern __shared__ double na_sm[];
  __shared__ double rho[kNaMaxPairs], alph[kNaMaxPairs];
  const long n = a.n;
  const int m = a.m;
  double q[kNaRegs];
  bool ok = true, back = false;
  int half = 0;
  double c = 0.0;              // pending update v -= c x
  const double *x = nullptr;
  for (int i = m - 1; i >= 0; --i) {
    const double *si = a.s + (long)i * n, *yi = a.y + (long)i * n;
    double ps = 0.0, pq = 0.0;
    if (i == m - 1) {
      na_each(a, q, na_sm, back,
              [&](long e) { return NaIn{__ldg(si + e), __ldg(yi + e), __ldg(a.g + e)}; },
              [&](long, const NaIn &in, double &v) {
                v = in.c;
                ps = fma(in.b, in.a, ps);
                pq = fma(in.a, v, pq);
              });
    } else {
      na_each(a, q, na_sm, back,
              [&](long e) { return NaIn{__ldg(si + e), __ldg(yi + e), __ldg(x + e)}; },
              [&](long, const NaIn &in, double &v) {
                v = fma(-c, in.c, v);
                ps = fma(in.b, in.a, ps);
                pq = fma(in.a, v, pq);
              });
    }
    back = !back;
    const double2 t = na_sum(a, ps, pq, half, &ok);
    half ^= 1;
    if (!ok) return;
    if (!(t.x > 0.0) || isinf(t.x)) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(a.flags + FLAG_ERR, ETDM_ERR_NUMERIC);
      return;
    }
    const double r = 1.0 / t.x;
    c = r * t.y;
    x = yi;
    if (threadIdx.x == 0) { rho[i] = r; alph[i] = c; }
  }
  if (m == 0) {
    for (long e = (long)blockIdx.x * kNaThreads + threadIdx.x; e < n; e += (long)gridDim.x * kNaThreads)
      a.p[e] = -(a.g[e] * a.h0[e]);
    return;
  }
  for (int i = 0; i < m; ++i) {
    const double *yi = a.y + (long)i * n;
    double pq = 0.0;
    if (i == 0) {  // the pending update is of pair 0
      na_each(a, q, na_sm, back, [&](long e) { return NaIn{__ldg(yi + e), __ldg(a.h0 + e), 0.0}; },
              [&](long, const NaIn &in, double &v) {
                v = fma(-c, in.a, v) * in.b;
                pq = fma(in.a, v, pq);
              });
    } else {
      na_each(a, q, na_sm, back, [&](long e) { return NaIn{__ldg(yi + e), __ldg(x + e), 0.0}; },
              [&](long, const NaIn &in, double &v) {
                v = fma(c, in.b, v);
                pq = fma(in.a, v, pq);
              });
    }
    back = !back;
    const double2 t = na_sum(a, pq, 0.0, half, &ok);
    half ^= 1;
    if (!ok) return;
    c = alph[i] - rho[i] * t.x;
    x = a.s + (long)i * n;
  }
  na_each(a, q, na_sm, back, [&](long e) { return NaIn{__ldg(x + e), 0.0, 0.0}; },
          [&](long e, const NaIn &in, double &v) {
            v = -fma(c, in.a, v);
            a.p[e] = v;
          });
}

namespace {

struct NaDevice {
  bool ready = false;
  unsigned char *scratch = nullptr;  // device address of g_noalloc_scratch
  int blocks_max = 0;
};

std::mutex g_na_mutex;
NaDevice g_na[kNaDevices];

int na_fail(int code, const std::string &msg) {
  set_unbound_error(msg);
  return code;
}

}  // namespace

}  // namespace etdm

using namespace etdm;

namespace etdm {
namespace {

// The device's scratch address and launch size, looked up once per device with
// that device current (the array's host-side name is not a device address).
int na_device(NaDevice **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaDevices)
    return na_fail(ETDM_ERR_CUDA, "no current CUDA device");
  NaDevice *d = &g_na[dev];
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!d->ready) {
    void *ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess)
      return na_fail(ETDM_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    int sms = 0, bps = 0, coop = 0;
    if (cudaFuncSetAttribute(lbfgs_noalloc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kNaSlots * kNaThreads * 8) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, lbfgs_noalloc_kernel, kNaThreads,
                                                      kNaSlots * kNaThreads * 8) != cudaSuccess ||
        !coop || bps < 1)
      return na_fail(ETDM_ERR_CUDA, "cannot size the cooperative two-loop kernel");
    d->scratch = (unsigned char *)ptr;
    d->blocks_max = std::min(kNaMaxBlocks, sms * bps);
    d->ready = true;
  }
  *out = d;
  return ETDM_OK;
}

}  // namespace
}  // namespace etdm

extern "C" int etdm_lbfgs_direction_noalloc(const double *g_dev, const double *s_dev,
                                            const double *y_dev, int32_t m, int64_t n,
                                            const double *h0_dev, double *p_dev,
                                            void *stream) {
  if (m < 0 || m > kNaMaxPairs)
    return na_fail(ETDM_ERR_INVALID_ARG,
                   "m must be in [0, " + std::to_string(kNaMaxPairs) + "] (scratch limit)");
  if (n < 0 || n > (int64_t)1 << 40) return na_fail(ETDM_ERR_INVALID_ARG, "n out of range");
  if (n == 0) return ETDM_OK;
  if (!g_dev || !h0_dev || !p_dev || (m > 0 && (!s_dev || !y_dev)))
    return na_fail(ETDM_ERR_INVALID_ARG, "g, h0, p (and s, y when m > 0) are required");
  NaDevice *d = nullptr;
  int rc = na_device(&d);
  if (rc != ETDM_OK) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  // barrier words and the status word must start at zero
  cudaError_t e = cudaMemsetAsync(d->scratch, 0, 256, s);
  if (e != cudaSuccess)
    return na_fail(ETDM_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
  NaArgs a;
  a.g = g_dev; a.s = s_dev; a.y = y_dev; a.h0 = h0_dev; a.p = p_dev;
  a.n = (long)n; a.m = m;
  a.bar = (unsigned *)d->scratch;
  a.flags = (int *)(d->scratch + 64);
  a.red = (double *)(d->scratch + 256);
  // four elements per thread, then every SM; shared memory for the elements
  // beyond the registers
  const long want = (n + 4L * kNaThreads - 1) / (4L * kNaThreads);
  const int blocks = (int)std::max(1L, std::min((long)d->blocks_max, want));
  const long per = (n + (long)blocks * kNaThreads - 1) / ((long)blocks * kNaThreads);
  a.slots = (int)std::max(0L, std::min<long>(kNaSlots, per - kNaRegs));
  void *args[] = {&a};
  e = cudaLaunchCooperativeKernel((void *)lbfgs_noalloc_kernel, dim3(blocks), dim3(kNaThreads),
                                  args, (size_t)a.slots * kNaThreads * 8, s);
  if (e != cudaSuccess)
    return na_fail(ETDM_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
  return ETDM_OK;
}

extern "C" int etdm_lbfgs_direction_noalloc_status(void *stream) {
  NaDevice *d = nullptr;
  int rc = na_device(&d);
  if (rc != ETDM_OK) return rc;
  // wait for the calls queued on `stream`, then copy the status word into a
  // local (a pageable copy: no pinned staging buffer, nothing allocated)
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  int word = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&word, d->scratch + 64, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess)
    return na_fail(ETDM_ERR_CUDA, std::string("status read: ") + cudaGetErrorString(e));
  if (word == ETDM_ERR_TIMEOUT)
    return na_fail(ETDM_ERR_TIMEOUT,
                   "the last allocation-free direction gave up at a grid barrier "
                   "(blocks not co-resident?); its output is incomplete");
  if (word == ETDM_ERR_NUMERIC)
    return na_fail(ETDM_ERR_NUMERIC,
                   "the last allocation-free direction met a pair with y.s <= 0 (or not "
                   "finite); its output is incomplete");
  if (word != 0) return na_fail(word, "the last allocation-free direction failed on the device");
  return ETDM_OK;
}
