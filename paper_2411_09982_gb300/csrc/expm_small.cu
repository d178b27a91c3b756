// FP64 exponentials of small matrices (d <= 32), one CTA per matrix, everything in shared
// memory:  U_b = e^{-i tau_b} exp(-i W_b)  by scaling and squaring of the Taylor polynomial
// of degree m (App. A.5), W_b = Hbar_b - tau_b I.
//
// The step-by-step form launches one batched product per Taylor and squaring step, each
// reading and writing whole matrices, and forms complex products of matrices whose real or
// imaginary part is zero.  At these sizes GB300's FP64 pipe (about two FMAs per cycle and SM)
// bounds both forms; this one saves
//   * the launches and passes between the steps (d = 2, 50 intervals: 11 launches of 3-5 us);
//   * for real symmetric W (real operators, which the plan detects) all complex arithmetic:
//     exp(-i A) = cos A - i sin A, and the degree-m Taylor polynomial splits exactly into
//     C = sum (-1)^k Y^k / (2k)! and S = A sum (-1)^k Y^k / (2k+1)! in Y = A^2.  With powers
//     up to Y^p, 2 p >= m / 2, each series needs one further product (degree 16: seven real
//     products), and a squaring two: C' = (C + S)(C - S), S' = 2 S C.  All factors are
//     polynomials in A, so every product is symmetric and its lower triangle suffices:
//     d^2 (d + 1) flops a product against 8 d^3, 15 of them against 10 (degree 16, four
//     squarings).
// Measured (GB300): d = 30, 1000 real intervals of four squarings 2.45 -> 0.46 ms; the
// strongly driven qubit (d = 2, 50 intervals) nine launches of 40 us -> one of 9.
#include "common.cuh"

#include <algorithm>

namespace mg {

constexpr int ES_MAXD = 32;
constexpr int ES_PITCH = 33;                        // odd: rows start in different banks
constexpr int ES_MAT = ES_MAXD * ES_PITCH;
// One output of a symmetric product per thread (at most 528), two of a complex one: an even
// share of warps for the four FP64 quarters of an SM (288 threads with up to two outputs each
// left one quarter a third more than the others).
constexpr int ES_THREADS_REAL = 544;
constexpr int ES_THREADS = 512;

struct SmallSeries {
  double c[9], s[9];   // (-1)^k / (2k)!, (-1)^k / (2k+1)!
  int kc, ks, p;       // degrees in Y, largest power formed
};

// Row and column of entry e of the lower triangle, row by row.
__device__ __forceinline__ void tri_index(int e, int& i, int& j) {
  i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= e) ++i;   // the square root may be off by one
  while (i * (i + 1) / 2 > e) --i;
  j = e - i * (i + 1) / 2;
}

__global__ void __launch_bounds__(ES_THREADS_REAL)
expm_small_real_kernel(int d, const double2* __restrict__ W, const double* __restrict__ tau, int sq,
                       const int* __restrict__ sq_dev, const __grid_constant__ SmallSeries ser, double2* __restrict__ U) {
  extern __shared__ double sm[];
  double* A = sm;
  double* Y[5] = {nullptr, sm + ES_MAT, sm + 2 * ES_MAT, sm + 3 * ES_MAT, sm + 4 * ES_MAT};
  double *C = sm + 5 * ES_MAT, *S = sm + 6 * ES_MAT, *T1 = sm + 7 * ES_MAT, *T2 = sm + 8 * ES_MAT;
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x;
  const int n = d * (d + 1) / 2;
  const int s = sq_dev ? sq_dev[b] : sq;
  const double2* Wb = W + (long long)b * d * d;
  const double scale = ldexp(1.0, -s);
  for (int e = tid; e < d * d; e += nth) A[(e / d) * ES_PITCH + e % d] = scale * Wb[e].x;
  __shared__ double phase[2];
  if (tid == 0) {
    phase[0] = 1.0;
    phase[1] = 0.0;
    if (tau) sincos(tau[b], &phase[1], &phase[0]);
  }
  __syncthreads();
  // dst = f(P Q) on the lower triangle and its mirror, P and Q symmetric and commuting
  auto product = [&](double* dst, const double* P, const double* Q, auto f) {
    for (int e = tid; e < n; e += nth) {
      int i, j;
      tri_index(e, i, j);
      const double *pr = P + i * ES_PITCH, *qr = Q + j * ES_PITCH;
      double x0 = 0.0, x1 = 0.0;
      int k = 0;
      for (; k + 1 < d; k += 2) {
        x0 = fma(pr[k], qr[k], x0);
        x1 = fma(pr[k + 1], qr[k + 1], x1);
      }
      if (k < d) x0 = fma(pr[k], qr[k], x0);
      const double v = f(i, j, x0 + x1);
      dst[i * ES_PITCH + j] = v;
      dst[j * ES_PITCH + i] = v;
    }
  };
  auto same = [](int, int, double x) { return x; };
  // sum_{j <= top} co[first + j] Y^j at (i, j), Y^0 = I
  auto poly = [&](const double* co, int first, int top, int i, int j) {
    double v = i == j ? co[first] : 0.0;
#pragma unroll
    for (int q = 1; q <= 4; ++q)
      if (q <= top) v = fma(co[first + q], Y[q][i * ES_PITCH + j], v);
    return v;
  };
  product(Y[1], A, A, same);
  __syncthreads();
  if (ser.p >= 2) product(Y[2], Y[1], Y[1], same);
  if (ser.p >= 2) __syncthreads();
  if (ser.p >= 3) product(Y[3], Y[2], Y[1], same);
  if (ser.p >= 4) product(Y[4], Y[2], Y[2], same);
  if (ser.p >= 3) __syncthreads();
  const int p = ser.p;
  const bool hc = ser.kc > p, hs = ser.ks > p;   // a second block: high part times Y^p
  for (int e = tid; e < d * d; e += nth) {
    const int i = e / d, j = e % d;
    if (hc) T1[i * ES_PITCH + j] = poly(ser.c, p, ser.kc - p, i, j);
    else C[i * ES_PITCH + j] = poly(ser.c, 0, ser.kc, i, j);
    if (hs) T2[i * ES_PITCH + j] = poly(ser.s, p, ser.ks - p, i, j);
    else S[i * ES_PITCH + j] = poly(ser.s, 0, ser.ks, i, j);
  }
  __syncthreads();
  if (hc) product(C, T1, sm + p * ES_MAT, [&](int i, int j, double x) { return x + poly(ser.c, 0, p - 1, i, j); });
  if (hs) product(S, T2, sm + p * ES_MAT, [&](int i, int j, double x) { return x + poly(ser.s, 0, p - 1, i, j); });
  __syncthreads();
  product(T2, A, S, same);   // sin = A S
  __syncthreads();
  double* Sn = T2;
  double *P = T1, *M = S, *Cn = Y[1], *Sf = Y[2];   // free from here on
  for (int q = 0; q < s; ++q) {
    for (int e = tid; e < d * d; e += nth) {
      const int o = (e / d) * ES_PITCH + e % d;
      P[o] = C[o] + Sn[o];
      M[o] = C[o] - Sn[o];
    }
    __syncthreads();
    product(Cn, P, M, same);
    product(Sf, Sn, C, [](int, int, double x) { return 2.0 * x; });
    __syncthreads();
    double* t = C; C = Cn; Cn = t;
    t = Sn; Sn = Sf; Sf = t;
  }
  const double cs = phase[0], sn = phase[1];
  double2* Ub = U + (long long)b * d * d;
  for (int e = tid; e < d * d; e += nth) {
    const int o = (e / d) * ES_PITCH + e % d;
    Ub[e] = make_double2(cs * C[o] - sn * Sn[o], -(sn * C[o] + cs * Sn[o]));
  }
}

// General complex W: Paterson-Stockmeyer with blocks of p, then squarings, as the batched
// products form them (the same coefficients, operands and order of terms).
struct SmallPs {
  double a[17];   // 1 / j!, zero beyond degree m
  int m, p;
};

__global__ void __launch_bounds__(ES_THREADS)
expm_small_kernel(int d, const double2* __restrict__ W, const double* __restrict__ tau, int sq,
                  const int* __restrict__ sq_dev, const __grid_constant__ SmallPs ps, double2* __restrict__ U) {
  extern __shared__ double sm[];
  double2* base = reinterpret_cast<double2*>(sm);
  double2* P[5] = {nullptr, base, base + ES_MAT, base + 2 * ES_MAT, base + 3 * ES_MAT};
  double2 *R = base + 4 * ES_MAT, *Rn = base + 5 * ES_MAT;
  const int b = blockIdx.x, tid = threadIdx.x, nth = blockDim.x, n = d * d;
  const int s = sq_dev ? sq_dev[b] : sq;
  const double scale = ldexp(1.0, -s);
  const double2* Wb = W + (long long)b * n;
  for (int e = tid; e < n; e += nth) {
    const double2 w = Wb[e];
    P[1][(e / d) * ES_PITCH + e % d] = make_double2(scale * w.y, -(scale * w.x));   // -i W
  }
  __shared__ double phase[2];
  if (tid == 0) {
    phase[0] = 1.0;
    phase[1] = 0.0;
    if (tau) sincos(tau[b], &phase[1], &phase[0]);
  }
  __syncthreads();
  auto product = [&](double2* dst, const double2* L, const double2* Q, auto f) {
    for (int e = tid; e < n; e += nth) {
      const int i = e / d, j = e % d;
      const double2* lr = L + i * ES_PITCH;
      double re = 0.0, im = 0.0;
      for (int k = 0; k < d; ++k) {
        const double2 x = lr[k], y = Q[k * ES_PITCH + j];
        re = fma(x.x, y.x, re);
        re = fma(-x.y, y.y, re);
        im = fma(x.x, y.y, im);
        im = fma(x.y, y.x, im);
      }
      dst[i * ES_PITCH + j] = f(i, j, make_double2(re, im));
    }
    __syncthreads();
  };
  auto same = [](int, int, double2 x) { return x; };
  const int p = ps.p, m = ps.m;
#pragma unroll
  for (int q = 2; q <= 4; ++q)
    if (q <= p) product(P[q], P[q - 1], P[1], same);
  // v + sum_{1 <= j <= top} a_{first + j} X^j + a_first I
  auto terms = [&](double2 v, int first, int top, int i, int j) {
#pragma unroll
    for (int q = 1; q <= 4; ++q)
      if (q <= top) {
        const double2 x = P[q][i * ES_PITCH + j];
        v.x = fma(ps.a[first + q], x.x, v.x);
        v.y = fma(ps.a[first + q], x.y, v.y);
      }
    if (i == j) v.x += ps.a[first];
    return v;
  };
  const int q = m / p, r = m - q * p;
  const int top = r == 0 ? q - 1 : q;
  for (int e = tid; e < n; e += nth)
    R[(e / d) * ES_PITCH + e % d] = terms(make_double2(0.0, 0.0), top * p, r == 0 ? p : p - 1, e / d, e % d);
  __syncthreads();
  const double2* Yp = base + (p - 1) * ES_MAT;
  for (int i0 = top - 1; i0 >= 0; --i0) {
    product(Rn, R, Yp, [&](int i, int j, double2 x) { return terms(x, i0 * p, p - 1, i, j); });
    double2* t = R; R = Rn; Rn = t;
  }
  for (int k = 0; k < s; ++k) {
    product(Rn, R, R, same);
    double2* t = R; R = Rn; Rn = t;
  }
  const double cs = phase[0], sn = phase[1];
  double2* Ub = U + (long long)b * n;
  for (int e = tid; e < n; e += nth) {
    const double2 v = R[(e / d) * ES_PITCH + e % d];
    Ub[e] = make_double2(cs * v.x + sn * v.y, cs * v.y - sn * v.x);
  }
}

int expm_small_max_dim() { return ES_MAXD; }

int launch_expm_small(int batch, int d, const double* W, const double* tau, int m, int p, int sq, const int* sq_dev,
                      int real_sym, double* U, cudaStream_t s) {
  if (batch <= 0) return MG_OK;
  const double2* W2 = reinterpret_cast<const double2*>(W);
  double2* U2 = reinterpret_cast<double2*>(U);
  double f[18];
  f[0] = 1.0;
  for (int j = 1; j < 18; ++j) f[j] = f[j - 1] / j;
  if (real_sym) {
    SmallSeries ser{};
    ser.kc = m / 2;
    ser.ks = (m - 1) / 2;
    ser.p = (ser.kc + 1) / 2;
    for (int k = 0; k <= ser.kc; ++k) ser.c[k] = (k & 1) ? -f[2 * k] : f[2 * k];
    for (int k = 0; k <= ser.ks; ++k) ser.s[k] = (k & 1) ? -f[2 * k + 1] : f[2 * k + 1];
    const int threads = std::min(ES_THREADS_REAL, (d * (d + 1) / 2 + 31) / 32 * 32);
    const int smem = 9 * ES_MAT * (int)sizeof(double);
    MG_TRY(ensure_smem_limit(reinterpret_cast<const void*>(expm_small_real_kernel), smem));
    expm_small_real_kernel<<<batch, threads, smem, s>>>(d, W2, tau, sq, sq_dev, ser, U2);
    return check_launch("expm_small_real_kernel");
  }
  SmallPs ps{};
  ps.m = m;
  ps.p = p;
  for (int j = 0; j <= m; ++j) ps.a[j] = f[j];
  const int threads = std::min(ES_THREADS, ((d * d + 1) / 2 + 31) / 32 * 32);
  const int smem = 6 * ES_MAT * (int)sizeof(double2);
  MG_TRY(ensure_smem_limit(reinterpret_cast<const void*>(expm_small_kernel), smem));
  expm_small_kernel<<<batch, threads, smem, s>>>(d, W2, tau, sq, sq_dev, ps, U2);
  return check_launch("expm_small_kernel");
}

}  // namespace mg
