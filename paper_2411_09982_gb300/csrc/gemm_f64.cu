// Native-FP64 batched complex matrix product (the MG_PREC_FP64 path and the
// FP64 re-orthonormalisation).
//
//   C[b] = scale * opA(A[b]) * B[b] + sum_m coef_m P_m[b] + diag * I
//
// with opA = identity or conjugate transpose.  GB300's FP64 throughput is a
// small fraction of its tensor-core throughput, so this kernel is bound by the
// FP64 pipe: a warp's FMA takes about 68 cycles of its quarter of the SM, next to
// which shared-memory loads cost nothing.  So a tile needs no reuse in registers,
// only little padding and many CTAs: 16 x 16 complex outputs, one per thread,
// operands staged in K-slabs of 16.  (64 x 64 tiles, four by four outputs per thread,
// took 266 us for one product of d = 64 against 25, 662 against 336 for 64 of d = 81,
// and 8.0 ms against 6.8 for one of d = 1000; 32 x 32 tiles lie between.)
#include "common.cuh"

namespace mg {

constexpr int FTM = 16;   // tile edge
constexpr int FBK = 16;   // K per slab

struct AddDev {
  const double* src[3];
  double coef[3];
  long long stride;
  int n;
  double diag;
  double scale;
  const int* item_sq;   // null, or per-item squaring counts: item b is skipped when item_sq[b] <= sq_step
  int sq_step;
};

__global__ void __launch_bounds__(256)
cgemm_f64_kernel(int d, const double* __restrict__ A, long long sA, int opA,
                 const double* __restrict__ B, long long sB, double* __restrict__ C, long long sC,
                 AddDev add) {
  __shared__ double2 As[FBK][FTM + 1];   // As[k][i] = opA(A)[i][k]
  __shared__ double2 Bs[FBK][FTM];       // Bs[k][j] = B[k][j]

  const int b = blockIdx.z;
  if (add.item_sq && add.item_sq[b] <= add.sq_step) return;   // uniform over the CTA
  const double2* Ab = reinterpret_cast<const double2*>(A + b * sA);
  const double2* Bb = reinterpret_cast<const double2*>(B + b * sB);
  const int i0 = blockIdx.y * FTM, j0 = blockIdx.x * FTM;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double accr = 0.0, acci = 0.0;
  for (int k0 = 0; k0 < d; k0 += FBK) {
    double2 v = make_double2(0.0, 0.0), w = v;
    if (opA == 0) {   // A[i0 + ty][k0 + tx]
      if (i0 + ty < d && k0 + tx < d) v = Ab[(long long)(i0 + ty) * d + (k0 + tx)];
      As[tx][ty] = v;
    } else {          // conj(A[k0 + ty][i0 + tx])
      if (i0 + tx < d && k0 + ty < d) v = Ab[(long long)(k0 + ty) * d + (i0 + tx)];
      As[ty][tx] = make_double2(v.x, -v.y);
    }
    if (k0 + ty < d && j0 + tx < d) w = Bb[(long long)(k0 + ty) * d + (j0 + tx)];
    Bs[ty][tx] = w;
    __syncthreads();
    const int kmax = min(FBK, d - k0);   // zero padding beyond d adds nothing
#pragma unroll
    for (int k = 0; k < FBK; ++k) {
      if (k >= kmax) break;
      const double2 x = As[k][ty], y = Bs[k][tx];
      accr = fma(x.x, y.x, accr);
      accr = fma(-x.y, y.y, accr);
      acci = fma(x.x, y.y, acci);
      acci = fma(x.y, y.x, acci);
    }
    __syncthreads();
  }
  const int i = i0 + ty, j = j0 + tx;
  if (i >= d || j >= d) return;
  const long long off = (long long)i * d + j;
  double re = add.scale * accr, im = add.scale * acci;
  for (int m = 0; m < add.n; ++m) {
    const double2 p = reinterpret_cast<const double2*>(add.src[m] + b * add.stride)[off];
    re = fma(add.coef[m], p.x, re);
    im = fma(add.coef[m], p.y, im);
  }
  if (i == j) re += add.diag;
  reinterpret_cast<double2*>(C + b * sC)[off] = make_double2(re, im);
}

int launch_cgemm_f64(int batch, int d, const double* A, long long strideA, int opA, const double* B,
                     long long strideB, double* C, long long strideC, const AddTerms& add,
                     cudaStream_t s) {
  if (batch <= 0) return MG_OK;
  if (batch > 65535) return MG_EUNSUPPORTED;
  AddDev a{};
  a.n = add.n;
  for (int m = 0; m < 3; ++m) { a.src[m] = add.src[m]; a.coef[m] = add.coef[m]; }
  a.stride = add.stride;
  a.diag = add.diag;
  a.scale = add.scale;
  a.item_sq = add.item_sq;
  a.sq_step = add.sq_step;
  const dim3 grid(ceil_div(d, FTM), ceil_div(d, FTM), batch);
  cgemm_f64_kernel<<<grid, 256, 0, s>>>(d, A, strideA, opA, B, strideB, C, strideC, a);
  return check_launch("cgemm_f64_kernel");
}

}  // namespace mg
