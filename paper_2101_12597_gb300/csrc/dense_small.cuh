// The dense chains of small systems (M <= 32) on one block with every matrix in
// shared memory (included by dense.cu, which defines the element types, the
// argument block and the workspace slots).
//
// A chain is some ten to thirty dependent products of a few hundred outputs, so
// latency bounds it: in the general chains a phase is described in a stack
// frame, copied to shared memory, and reads its operands back from L2, 2 to 3
// us each.  Here a phase is a call of one resident function on offsets into
// shared memory: operands are read there, results go there and, for the kernels
// and chains that read them later, to their places in global memory.  FP64
// products split K over up to eight lanes, one multiply-add chain each, because
// a warp-wide FP64 operation holds its scheduler for some 70 cycles; float
// pairs keep the order of phase_direct (the same bits), since their rounding
// decides the O slices.  Measured, forward / reverse: 8 atoms (M = 16, N = 4,
// FP64) 33 / 54 -> 17 / 24 us; two water-like units (M = 16, N = 8, float pairs)
// 46 / 74 -> 21 / 29 us; what is left is some 1 us a product of loads, FP64 or
// pair chains and the block barrier.
// The arithmetic and the outputs are those of dense_forward and dense_reverse.
#pragma once

namespace etdm {

constexpr int kSmallM = 32;                    // functions, at most
constexpr int kSmallBytes = 200 * 1024;        // shared memory, at most

// offsets (elements) of the matrices; the first five are loaded
struct SmallFwd {
  int A, C0, T, q, K, S, U, O, total;
  __host__ __device__ SmallFwd(int M, int N, int V) {
    const int NN = N * N;
    A = 0; C0 = A + N * V; T = C0 + M * M; q = T + M * M;
    K = q + kQslots * NN; S = K + 2 * NN; U = S + 2 * NN; O = U + M * N;
    total = O + M * N;
  }
};
struct SmallRev {
  int A, C0, H, O, TO, q, SJ, G, Ub, kb, sb, Kt, St, Ab, w, total;
  __host__ __device__ SmallRev(int M, int N, int V) {
    const int NN = N * N, MN = M * N;
    A = 0; C0 = A + N * V; H = C0 + M * M; O = H + M * M; TO = O + MN; q = TO + MN;
    SJ = q + kQslots * NN; G = SJ + NN; Ub = G + MN; kb = Ub + MN; sb = kb + 2 * NN;
    Kt = sb + 2 * NN; St = Kt + NN; Ab = St + NN; w = Ab + N * V;
    total = w + kWslots * NN;
  }
};
inline bool small_fits(int M, int N, int V) {
  return M <= kSmallM && std::max(SmallFwd(M, N, V).total, SmallRev(M, N, V).total) * 8 <= kSmallBytes;
}

extern __shared__ __align__(16) unsigned char small_sm[];

// out[m n] = alpha op(A) op(B) (+ alpha2 A2 B2) + sum b_q C_q + diag I, with
// A(i, k) at A + i iA + k kA and B(k, j) at B + k kB + j jB; also to gout
// (nullptr: not; out64: as FP64)
template <class R>
__device__ __noinline__ void small_prod(int out, void *gout, int m, int n, int K, int A, int iA, int kA,
                                        int B, int kB, int jB, double alpha, int c0 = -1, double b0 = 0.0,
                                        int c1 = -1, double b1 = 0.0, int c2 = -1, double b2 = 0.0,
                                        double diag = 0.0, int A2 = -1, int B2 = -1, double alpha2 = 0.0,
                                        bool out64 = false) {
  using X = Num<R>;
  R *sm = reinterpret_cast<R *>(small_sm);
  const int mn = m * n;
  int ls = 0;  // log2 of the lanes of an output
  if constexpr (!X::kPair)
    while (ls < 3 && (mn << (ls + 1)) <= NT && (2 << ls) <= K) ++ls;
  for (int base = 0; base < (mn << ls); base += NT) {
    const int idx = base + threadIdx.x, e = idx >> ls;
    const bool in = e < mn;
    const int i = e / n, j = e - i * n;
    R v = X::zero();
    if constexpr (X::kPair) {
      if (in) {
        R acc[2] = {X::zero(), X::zero()};
        for (int q = 0; q < 2; ++q) {
          const int Aq = q ? A2 : A, Bq = q ? B2 : B;
          if (Aq < 0) break;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int k0 = c * BK, k1 = min(K, k0 + BK);
            if (k0 >= K) break;
            Mac<R> mac;
            for (int k = k0; k < k1; k += 4) {
#pragma unroll
              for (int u = 0; u < 4; ++u)
                mac.step(u, k + u < k1 ? sm[Aq + i * iA + (k + u) * kA] : X::zero(),
                         k + u < k1 ? sm[Bq + (k + u) * kB + j * jB] : X::zero());
            }
            acc[c] = X::fma(q ? alpha2 : alpha, mac.total(), acc[c]);
          }
        }
        v = K > BK ? X::add(acc[0], acc[1]) : acc[0];
      }
    } else {
      const int sub = idx & ((1 << ls) - 1);
      if (in) {
        double s = 0.0;
#pragma unroll 4
        for (int k = sub; k < K; k += 1 << ls) s = fma(sm[A + i * iA + k * kA], sm[B + k * kB + j * jB], s);
        v = alpha == 1.0 ? s : alpha * s;
        if (A2 >= 0) {
          s = 0.0;
#pragma unroll 4
          for (int k = sub; k < K; k += 1 << ls) s = fma(sm[A2 + i * iA + k * kA], sm[B2 + k * kB + j * jB], s);
          v = fma(alpha2, s, v);
        }
      }
      for (int o = 1; o < 1 << ls; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (sub) continue;
    }
    if (!in) continue;
    if (c0 >= 0) v = X::fma(b0, sm[c0 + e], v);
    if (c1 >= 0) v = X::fma(b1, sm[c1 + e], v);
    if (c2 >= 0) v = X::fma(b2, sm[c2 + e], v);
    if (i == j && diag != 0.0) v = X::add(v, X::from(diag));
    sm[out + e] = v;
    if (gout) {
      if (out64) static_cast<double *>(gout)[e] = X::dbl(v);
      else X::st(gout, e, v);
    }
  }
  __syncthreads();
}

// X <- s (X + X^T) for n consecutive N x N matrices
template <class R>
__device__ __noinline__ void small_sym(int x, int n, int N, double s) {
  using X = Num<R>;
  R *sm = reinterpret_cast<R *>(small_sm);
  const int NN = N * N;
  for (int e = threadIdx.x; e < n * NN; e += NT) {
    const int q = e / NN, r = e - q * NN, i = r / N, j = r - i * N;
    if (i > j) continue;
    R *p = sm + x + q * NN;
    const R a = p[i * N + j], b = p[j * N + i];
    p[i * N + j] = X::scale2(X::add(a, b), s);
    if (i != j) p[j * N + i] = X::scale2(X::add(b, a), s);
  }
  __syncthreads();
}

// sum over a warp of a(e) b(e), e = lane, lane + 32, .. < n, in every lane
template <class F>
__device__ __forceinline__ double small_dot(int first, int step, int n, F f) {
  double s = 0.0;
  for (int e = first; e < n; e += step) s += f(e);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <class R>
__device__ __forceinline__ void small_load(int dst, const void *src, int n) {
  R *sm = reinterpret_cast<R *>(small_sm);
  for (int e = threadIdx.x; e < n; e += NT) sm[dst + e] = Num<R>::ld(src, e);
}

template <class R>
__global__ void __launch_bounds__(NT) dense_forward_small_kernel(DenseArgs a) {
  using X = Num<R>;
  R *sm = reinterpret_cast<R *>(small_sm);
  __shared__ double t[3];
  __shared__ int sh_j;
  const int M = a.M, N = a.N, V = a.V, NN = N * N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SmallFwd f(M, N, V);
  auto qs = [&](int k) { return f.q + k * NN; };
  auto gq = [&](int k) { return a.Qk + (long)k * NN; };
  for (int e = tid; e < N * V; e += NT) {
    const R x = X::ld_f64(a.A, e);
    sm[f.A + e] = x;
    if (X::kPair) X::st(a.Af, e, x);
  }
  small_load<R>(f.C0, a.C0, M * M);
  small_load<R>(f.T, a.T, M * M);
  __syncthreads();
  // P = A A^T (in the place of Q), P^2, P^3, P^4
  small_prod<R>(qs(kQ1), a.P, N, N, V, f.A, V, 1, f.A, 1, V, 1.0);
  small_prod<R>(qs(kQ2), nullptr, N, N, N, qs(kQ1), N, 1, qs(kQ1), N, 1, 1.0);
  small_prod<R>(qs(kQ3), nullptr, N, N, N, qs(kQ1), N, 1, qs(kQ2), N, 1, 1.0);
  small_prod<R>(qs(kQ4), nullptr, N, N, N, qs(kQ2), N, 1, qs(kQ2), N, 1, 1.0);
  if (warp < 3) {
    const int x = qs(warp == 0 ? kQ1 : warp == 1 ? kQ2 : kQ4);
    const double s = small_dot(lane, 32, NN, [&](int e) {
      const double d = X::dbl(sm[x + e]);
      return d * d;
    });
    if (lane == 0) t[warp] = s;
  }
  __syncthreads();
  if (tid == 0) {  // the doublings, as dense_forward takes them
    const double t1 = t[0], t2 = t[1], t4 = t[2];
    int jf = 0, j = 0;
    for (double lim = 1.0; t1 > lim && jf <= kJmax; lim *= 16.0) ++jf;
    if (!(t1 == t1) || isinf(t1)) jf = kJmax + 1;
    double l1 = 1.0, l2 = 1.0, l4 = 1.0;
    while (j < jf && !(t1 <= l1) && !(t2 <= l2) && !(t4 <= l4)) {
      l1 *= 16.0; l2 *= 256.0; l4 *= 65536.0;
      ++j;
    }
    if (jf > kJmax) {
      atomicExch(a.flags + FLAG_ERR, ETDM_ERR_NUMERIC);
      j = -1;
    } else {
      a.flags[FLAG_J] = j;
      a.scal[0] = ldexp(1.0, -2 * j);
    }
    sh_j = j;
  }
  __syncthreads();
  const int J = sh_j;
  if (J < 0) return;
  const double sc = ldexp(1.0, -2 * J), sc2 = sc * sc, sc3 = sc2 * sc, sc4 = sc2 * sc2;
  auto cf = [&](const double *c, int k) { return k <= kTaylor ? c[k] : 0.0; };
  for (int e = tid; e < NN; e += NT) {
    const R q1 = X::scale2(sm[qs(kQ1) + e], sc), q2 = X::scale2(sm[qs(kQ2) + e], sc2),
            q3 = X::scale2(sm[qs(kQ3) + e], sc3), q4 = X::scale2(sm[qs(kQ4) + e], sc4);
    const R q[4] = {X::from(e / N == e % N ? 1.0 : 0.0), q1, q2, q3};
    R bc = X::zero(), bs = X::zero();
    for (int r = 0; r < 4; ++r) {
      bc = X::fma(cf(a.ck, 8 + r), q[r], bc);
      bs = X::fma(cf(a.sk, 8 + r), q[r], bs);
    }
    const R o[6] = {q1, q2, q3, q4, bc, bs};
    const int s[6] = {kQ1, kQ2, kQ3, kQ4, kBc2, kBs2};
#pragma unroll
    for (int w = 0; w < 6; ++w) {
      sm[qs(s[w]) + e] = o[w];
      X::st(gq(s[w]), e, o[w]);
    }
  }
  __syncthreads();
  for (int w = 0; w < 2; ++w) {  // T = B_1 + Q^4 B_2
    const double *c = w ? a.sk : a.ck;
    small_prod<R>(qs(w ? kTs : kTc), gq(w ? kTs : kTc), N, N, N, qs(kQ4), N, 1, qs(w ? kBs2 : kBc2), N, 1,
                  1.0, qs(kQ1), cf(c, 5), qs(kQ2), cf(c, 6), qs(kQ3), cf(c, 7), cf(c, 4));
  }
  for (int w = 0; w < 2; ++w) {  // k = cos sqrt(Q) - 1, s = sin sqrt(Q) / sqrt(Q)
    const double *c = w ? a.sk : a.ck;
    small_prod<R>(w ? f.S : f.K, w ? a.St : a.Kt, N, N, N, qs(kQ4), N, 1, qs(w ? kTs : kTc), N, 1, 1.0,
                  qs(kQ1), cf(c, 1), qs(kQ2), cf(c, 2), qs(kQ3), cf(c, 3), cf(c, 0));
  }
  for (int u = 0; u < J; ++u) {  // doubling: k' = 4k + 2k^2, s' = s + s k
    const int k0 = f.K + (u & 1) * NN, k1 = f.K + (1 - (u & 1)) * NN;
    const int s0 = f.S + (u & 1) * NN, s1 = f.S + (1 - (u & 1)) * NN;
    small_prod<R>(k1, a.Kt + (long)(u + 1) * NN, N, N, N, k0, N, 1, k0, N, 1, 2.0, k0, 4.0);
    small_prod<R>(s1, a.St + (long)(u + 1) * NN, N, N, N, s0, N, 1, k0, N, 1, 1.0, s0, 1.0);
  }
  const int kJ = f.K + (J & 1) * NN, sJ = f.S + (J & 1) * NN;
  for (int e = tid; e < NN; e += NT) {
    const R x = X::add(sm[kJ + e], X::from(e / N == e % N ? 1.0 : 0.0));
    sm[f.U + e] = x;
    X::st(a.Uocc, e, x);
  }
  small_prod<R>(f.U + NN, a.Uocc + NN, V, N, N, f.A, 1, V, sJ, N, 1, -1.0);  // -A^T s(P)
  small_prod<R>(f.O, a.O, M, N, M, f.C0, M, 1, f.U, N, 1, 1.0);              // O = C0 U_occ
  // (the results below are read from global memory only; they take C0's place)
  if (a.Vacc) {
    small_prod<R>(f.C0, a.TO, M, N, M, f.T, M, 1, f.O, N, 1, 1.0);
  } else {
    small_prod<R>(f.C0, a.D, M, M, N, f.O, N, 1, f.O, 1, N, 2.0);  // D = 2 O O^T
    for (int e = tid; e < M * M; e += NT) X::st(a.H, e, sm[f.T + e]);
  }
}

template <class R>
__global__ void __launch_bounds__(NT) dense_reverse_small_kernel(DenseArgs a, int want_grad) {
  using X = Num<R>;
  R *sm = reinterpret_cast<R *>(small_sm);
  __shared__ double rs[20];  // kin: 8 warps, external, Hartree, exchange, correction: 4 + 4 warps
  const int M = a.M, N = a.N, V = a.V, NN = N * N, MM = M * M, MN = M * N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SmallRev f(M, N, V);
  const bool mixed = a.Vacc != nullptr;
  const int J = a.flags[FLAG_J];
  const double sc = a.scal[0];
  const void *const Hg = mixed ? a.Vacc : (const void *)a.H;  // upper triangle
  auto qs = [&](int k) { return f.q + k * NN; };
  auto w = [&](int k) { return f.w + k * NN; };
  if (want_grad || mixed) {
    for (int e = tid; e < MM; e += NT) {
      const int i = e / M, c = e - i * M;
      const R x = X::ld(Hg, i > c ? (long)c * M + i : e);
      sm[f.H + e] = x;
      if (!mixed && i > c) X::st(a.H, e, x);
    }
    small_load<R>(f.O, a.O, MN);
    if (mixed) small_load<R>(f.TO, a.TO, MN);
  }
  if (want_grad) {
    small_load<R>(f.A, X::kPair ? (const void *)a.Af : (const void *)a.A, N * V);
    small_load<R>(f.C0, a.C0, MM);
    small_load<R>(f.q, a.Qk, kQslots * NN);
    small_load<R>(f.SJ, a.St + (long)J * NN, NN);
  }
  // energy terms, straight from global memory
  if (warp < 8) {
    const double s = small_dot(tid, 256, mixed ? MN : MM, [&](int e) {
      if (mixed) return 2.0 * X::dbl(X::ld(a.O, e)) * X::dbl(X::ld(a.TO, e));
      return X::dbl(X::ld(a.D, e)) * X::dbl(X::ld(a.T, e));
    });
    if (lane == 0) rs[warp] = s;
  } else if (warp < 11) {
    const double s = small_dot(lane, 32, a.n_gridpart, [&](int b) { return a.gridpart[3 * b + warp - 8]; });
    if (lane == 0) rs[warp] = s;
  } else if (warp < 15) {
    const double s = mixed ? small_dot(tid - 352, 128, MN, [&](int e) { return X::dbl(X::ld(a.TO, e)) * a.dO[e]; })
                           : 0.0;
    if (lane == 0) rs[warp] = -4.0 * s;
  }
  __syncthreads();
  if (want_grad || mixed) {  // Gbar = dE/dO = 4 H O (4 V O + 4 T O), Ubar = C0^T Gbar
    small_prod<R>(f.G, a.Gbar, M, N, M, f.H, M, 1, f.O, N, 1, 4.0, mixed ? f.TO : -1, 4.0);
    if (warp >= 12) {
      const double s = mixed ? small_dot(tid - 384, 128, MN, [&](int e) { return X::dbl(sm[f.G + e]) * a.dO[e]; })
                             : 0.0;
      if (lane == 0) rs[warp + 3] = s;
    }
    if (want_grad) small_prod<R>(f.Ub, a.Ubar, M, N, M, f.C0, 1, M, f.G, N, 1, 1.0);
    else __syncthreads();
  }
  if (tid == 0) {
    double kin = 0.0, corr = 0.0;
    for (int b = 0; b < 8; ++b) kin += rs[b];
    if (mixed)
      for (int b = 11; b < 19; ++b) corr += rs[b];
    const double E = kin + rs[8] + rs[9] + rs[10] + corr;
    a.eterms[0] = kin; a.eterms[1] = rs[8]; a.eterms[2] = rs[9]; a.eterms[3] = rs[10] + corr;
    if (a.E) *a.E = E;
    if (!(E == E) || isinf(E)) atomicExch(a.flags + FLAG_ERR, ETDM_ERR_NUMERIC);
  }
  if (!want_grad) return;
  const int Ubv = f.Ub + NN;
  // Sbar_J = -A Ubar_v, Abar = -S_J Ubar_v^T; symmetric cotangents of k_J and s_J
  int kb = f.kb, sb = f.sb;
  for (int e = tid; e < NN; e += NT) sm[kb + e] = sm[f.Ub + e];
  small_prod<R>(sb, nullptr, N, N, V, f.A, V, 1, Ubv, N, 1, -1.0);
  small_prod<R>(f.Ab, nullptr, N, V, N, f.SJ, N, 1, Ubv, 1, N, -1.0);
  small_sym<R>(kb, 1, N, 0.5);
  small_sym<R>(sb, 1, N, 0.5);
  for (int u = J - 1; u >= 0; --u) {  // the doublings, as in dense_reverse
    const int ko = f.kb + f.kb + NN - kb, so = f.sb + f.sb + NN - sb;  // the other halves
    small_load<R>(f.Kt, a.Kt + (long)u * NN, NN);
    small_load<R>(f.St, a.St + (long)u * NN, NN);
    __syncthreads();
    small_prod<R>(so, nullptr, N, N, N, sb, N, 1, f.Kt, N, 1, 0.5, sb, 0.5);
    small_prod<R>(ko, nullptr, N, N, N, kb, N, 1, f.Kt, N, 1, 2.0, kb, 2.0, -1, 0.0, -1, 0.0, 0.0, f.St, sb, 0.5);
    small_sym<R>(ko, 1, N, 1.0);
    small_sym<R>(so, 1, N, 1.0);
    kb = ko;
    sb = so;
  }
  // back through k = B_0 + Q^4 T_c, s = B_0 + Q^4 T_s and T = B_1 + Q^4 B_2
  small_prod<R>(w(kQ4b), nullptr, N, N, N, kb, N, 1, qs(kTc), N, 1, 1.0, -1, 0.0, -1, 0.0, -1, 0.0, 0.0, sb, qs(kTs), 1.0);
  small_prod<R>(w(kTcb), nullptr, N, N, N, qs(kQ4), N, 1, kb, N, 1, 1.0);
  small_prod<R>(w(kTsb), nullptr, N, N, N, qs(kQ4), N, 1, sb, N, 1, 1.0);
  small_prod<R>(w(kQ4b), nullptr, N, N, N, w(kTcb), N, 1, qs(kBc2), N, 1, 1.0, w(kQ4b), 1.0, -1, 0.0, -1, 0.0, 0.0,
                w(kTsb), qs(kBs2), 1.0);
  small_prod<R>(w(kBc2b), nullptr, N, N, N, qs(kQ4), N, 1, w(kTcb), N, 1, 1.0);
  small_prod<R>(w(kBs2b), nullptr, N, N, N, qs(kQ4), N, 1, w(kTsb), N, 1, 1.0);
  for (int e = tid; e < NN; e += NT) {
    const R bcb[3] = {sm[kb + e], sm[w(kTcb) + e], sm[w(kBc2b) + e]};
    const R bsb[3] = {sm[sb + e], sm[w(kTsb) + e], sm[w(kBs2b) + e]};
    R qb[4] = {X::zero(), X::zero(), X::zero(), X::zero()};
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int r = 1; r < 4; ++r) {
        const int k = 4 * b + r;
        if (k <= kTaylor) qb[r] = X::fma(a.ck[k], bcb[b], X::fma(a.sk[k], bsb[b], qb[r]));
      }
    sm[w(kQ1bB) + e] = qb[1];
    sm[w(kQ2bB) + e] = qb[2];
    sm[w(kQ3b) + e] = qb[3];
  }
  __syncthreads();
  static_assert(kQ2bB == kQ1bB + 1 && kQ3b == kQ2bB + 1, "three consecutive slots");
  small_sym<R>(w(kQ4b), 1, N, 0.5);
  small_sym<R>(w(kQ1bB), 3, N, 0.5);
  // Q^4 = Q^2 Q^2, Q^3 = Q Q^2, Q^2 = Q Q
  small_prod<R>(w(kQ2b), nullptr, N, N, N, w(kQ4b), N, 1, qs(kQ2), N, 1, 1.0, w(kQ2bB), 0.5, -1, 0.0, -1, 0.0, 0.0,
                qs(kQ1), w(kQ3b), 0.5);
  small_prod<R>(w(kQ1bt), nullptr, N, N, N, w(kQ3b), N, 1, qs(kQ2), N, 1, 0.5, w(kQ1bB), 0.5);
  static_assert(kQ1bt == kQ2b + 1, "two consecutive slots");
  small_sym<R>(w(kQ2b), 2, N, 1.0);
  small_prod<R>(w(kQ1b), nullptr, N, N, N, w(kQ2b), N, 1, qs(kQ1), N, 1, 1.0, w(kQ1bt), 0.5);
  small_sym<R>(w(kQ1b), 1, N, 1.0);
  // g = Abar + 2 sc Qbar A, as FP64 (into Gbar's place)
  small_prod<R>(f.Ab, a.g, N, V, N, w(kQ1b), N, 1, f.A, V, 1, 2.0 * sc, f.Ab, 1.0, -1, 0.0, -1, 0.0, 0.0, -1, -1, 0.0,
                true);
  if (!a.resid) return;
  // Eq. 45 from R = Ubar - U_occ (U_occ^T Ubar), as in dense_reverse
  small_load<R>(f.O, a.Uocc, MN);
  __syncthreads();
  small_prod<R>(w(kQ4b), nullptr, N, N, M, f.O, 1, N, f.Ub, N, 1, 1.0);
  small_prod<R>(f.G, nullptr, M, N, N, f.O, N, 1, w(kQ4b), N, 1, -1.0, f.Ub, 1.0);
  if (warp == 0) {
    const double s = small_dot(lane, 32, MN, [&](int e) {
      const double d = X::dbl(sm[f.G + e]);
      return d * d;
    });
    if (lane == 0) *a.resid = s / (16.0 * N);
  }
}

}  // namespace etdm
