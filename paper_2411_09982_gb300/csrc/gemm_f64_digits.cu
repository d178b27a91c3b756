// FP64 complex matrix products on the tcgen05 tensor cores, to FP64 accuracy.
//
//   C[b] = opA(A[b]) B[b] + sum_m coef_m P_m[b] + diag I        (FP64 in, FP64 out)
//
// GB300's FP64 pipe gives 1.1 TFLOP/s, its BF16 tensor cores 1900.  A product of the
// exponential or of the propagators (MG_PREC_FP64) is therefore formed from integer digits
// whose products the tensor cores accumulate exactly (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump, Numerical Algorithms 59, 2012):
//   * Every row of A (column of B) is scaled by the power of two 2^E that bounds it and
//     rounded to 63-bit fixed point: an entry a becomes F = rint(a 2^{62 - E}), |F| < 2^62,
//     and F = sum_{s<8} q_s 2^{8 (7 - s)} with balanced base-256 digits |q_s| <= 128 (the
//     first at most 64), each exact in BF16 (stored as q_s 2^{-8 s}).  Entries down to 2^-9
//     of the row's largest keep all 53 bits of their mantissa.
//   * Digit products q_s q_t with s + t <= 7 (36 of 64) are summed by level l = s + t in FP32
//     TMEM accumulators.  Their levels up to 5 have to stay exact integers below 2^24 (the
//     rounding of level 6 and 7 weighs 2^-62 of the leading digit product and less), so the
//     accumulators are drained into 64-bit integer registers every n K steps of 32: by
//     Cauchy-Schwarz a level's sum over n steps is at most n sqrt(ea eb), ea and eb the
//     largest digit energies (sums of q_s^2) of one K step in A's rows and B's columns, which
//     the slicers record per item.  Full random digits give n = 12 and 18 (levels 0..3),
//     whatever the operands 6 and 10 steps are exact, and most matrices of the exponential
//     take one drain per sweep.
//   * The two 64-bit sums (levels 0..3 and 4..7) are joined and rounded to FP64 on the integer
//     pipe, the product's only rounding beside that of F.
// The error is about 2^-58 of (largest entry of the row of A) x (largest entry of the column
// of B) beside the rounding of the result: below FP64 arithmetic's, whose K roundings
// accumulate.  Whole evolutions against quad precision (relative 2-norm, here / FP64 pipe):
// spin chain d = 64, six squarings per interval 2.1e-14 / 5.6e-14, four 4.4e-15 / 3.2e-14;
// transmon chain d = 81 2.7e-14 / 1.1e-13; transmon-resonator d = 80 1.1e-12 / 1.6e-12.
// (Base-128 digits, 56 bits, need fewer drains but gave 2.3e-14, 1.3e-14, 1.0e-13, 1.1e-12.)
// Operands that the scheme does not cover -- a NaN, an infinity, a row or column whose largest
// entry lies outside 2^-400 .. 2^400 -- are marked by the slicers; such an item is computed in
// FP64 arithmetic once a CTA's digit tiles are done (f8_pipe_tiles).  So are, where a caller's own
// operands are multiplied, tiles with entries too weak for the digits (f64d_weak_kernel).
//
// Structure of the product kernel (persistent, one CTA of 640 threads per SM, 128 x 64
// complex output tiles; every tile makes two sweeps over K, levels 4..7 first):
//   warp 0      TMA producer: 32 KiB slots (4 digits of the A or B tile, K = 32, SWIZZLE_64B)
//               in a ring of six.  Levels 0..3 need the digits 0..3 of A and B (two slots per
//               K step), levels 4..7 all eight (four slots).
//   warp 1      MMA issuer: M = 128, N = 128 (64 real, 64 imaginary columns), K = 16; four
//               levels fill the 512 TMEM columns.  In the sweep of levels 4..7 the order
//               (A 0..3, B 0..3), (A 0..3, B 4..7), (A 4..7, B 0..3) frees two slots while
//               ten digit pairs are still to be multiplied, so a ring of 1.5 K steps keeps
//               loads in flight.
//   warps 4..19 drains: tcgen05.ld, float -> int, 64-bit accumulation in registers (32 sums
//               per thread).  The low words of levels 4..7 wait in a per-CTA scratch (L2)
//               while levels 0..3 are swept onto the high ones.  Rounding to FP64, addends
//               and stores run while the next tile's MMAs are issued.  These warps take
//               registers over from the first four (setmaxnreg).
// Measured (GB300, one product of a batch, slicing included, against the FP64-pipe kernel of
// gemm_f64.cu): d = 729, batch 16 2531 -> 103 us (30 TFLOP/s of the product's 8 d^3); d = 256,
// batch 128 108 -> 5.4 us; d = 81, batch 256 5.0 -> 0.86 us.  The tensor pipe is 55% busy at
// d = 256 and 729, 29% at d = 81.  Small K is bound by the epilogue's latency, which is why it has 16 warps (eight
// warps of 64 sums: d = 84 exponentials 2.93 -> 2.42 ms, d = 256 12.1 -> 10.7, d = 729 the
// same); at d = 729 the slicers take 12% (HBM-bound), the drains 11%, and the operands arrive
// at 43 bytes per cycle and SM, near what L2 delivers.
// Every wait is bounded (SplitCtl::wait_ns, at most 4 s): a wait that gives up records
// MG_DEV_TIMEOUT, the CTA's unfinished tiles become NaN, and it leaves once its own copies
// and MMAs have completed.
#include "common.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

namespace mg {

constexpr int F8_L = 8;                 // digits
constexpr int F8_BM = 128;              // output rows per tile
constexpr int F8_BN = 64;               // complex output columns per tile
constexpr int F8_BK = 32;               // K per slot
constexpr int F8_SLOTS = 6;
constexpr int F8_SLOT_BYTES = 4 * F8_BM * F8_BK * 2;
constexpr int F8_THREADS = 640;         // warps 0..3: loads, MMAs (two idle); warps 4..19: drains and epilogue
constexpr int F8_EPI_WARPS = 16;
constexpr int F8_SEG_LO = 6;            // K steps per drain of levels 4..7 that are exact whatever the digits
constexpr int F8_SEG_HI = 10;           // and of levels 0..3
constexpr int F8_VALS = 32;             // sums per epilogue thread
constexpr int F8_EPI = F8_EPI_WARPS * 32;
constexpr int F8_STAGE_BYTES = F8_EPI_WARPS * 2048;   // epilogue staging: 32 rows x 4 complex (8 real) columns per warp
// Register split (setmaxnreg): the launch holds 640 x 96 = 128 x 64 + 512 x 104
constexpr int F8_REGS_LAUNCH = 96;
constexpr int F8_REGS_IO = 64;
constexpr int F8_REGS_EPI = 104;
static_assert(128 * F8_REGS_IO + F8_EPI * F8_REGS_EPI <= F8_THREADS * F8_REGS_LAUNCH, "a larger split would wait forever");
constexpr int F8_EXP_MAX = 400;

struct F8Geom {
  int d, Kh, Kp;
  long long a_elems, b_elems;   // BF16 elements per item
};
static F8Geom f8_geom(int d) {
  F8Geom g;
  g.d = d;
  g.Kh = ceil_div(d, F8_BK) * F8_BK;
  g.Kp = 2 * g.Kh;
  g.a_elems = (long long)F8_L * d * g.Kp;        // rows [Re | 0 | Im | 0]
  g.b_elems = (long long)F8_L * 3 * d * g.Kh;    // planes -Im, Re, Im of the columns
  return g;
}

// The product's kernels have to be compiled to the register count their split starts from
// (asked for once per kernel).
static int f8_check_registers(const void* kern, std::atomic<bool>& checked) {
  if (checked.load(std::memory_order_relaxed)) return MG_OK;
  cudaFuncAttributes at;
  MG_CUDA_TRY(cudaFuncGetAttributes(&at, kern));
  if (at.numRegs < F8_REGS_LAUNCH) {
    set_last_message("the FP64 digit product is compiled to %d registers, its split needs %d", at.numRegs, F8_REGS_LAUNCH);
    return MG_EUNSUPPORTED;
  }
  checked.store(true, std::memory_order_relaxed);
  return MG_OK;
}
static std::atomic<bool> f8_checked[2];

// operand buffer: digits of all items, then row (column) exponents, then the items' marks and
// digit energies
size_t f64d_a_bytes(int d, int batch) {
  return ((size_t)f8_geom(d).a_elems * 2 + (size_t)d * 4 + 12) * batch;
}
size_t f64d_b_bytes(int d, int batch) {
  return ((size_t)f8_geom(d).b_elems * 2 + (size_t)d * 4 + 12) * batch;
}

// ---------------------------------------------------------------------------
// slicers
// ---------------------------------------------------------------------------
// E with |a| < 2^E; zero -> -2^29; subnormals -> -1022; NaN and infinities -> 1025
__device__ __forceinline__ int f8_exp(double a) {
  const int hi = __double2hiint(a), bexp = (hi >> 20) & 0x7FF;
  return bexp == 0 ? ((((uint32_t)hi << 1) | (uint32_t)__double2loint(a)) ? -1022 : -(1 << 29)) : bexp - 1022;
}
// exponents are stored as E + 4096; 0 is a row or column without a nonzero entry
constexpr int F8_EBIAS = 4096;
__device__ __forceinline__ int f8_exponent(int stored) { return stored ? stored - F8_EBIAS : 0; }
__device__ __forceinline__ bool f8_marked(int E) { return E > F8_EXP_MAX || (E < -F8_EXP_MAX && E > -(1 << 28)); }

constexpr unsigned long long F8_BIAS = 0x8080808080808080ull;   // 128 in every base-256 position
// F + bias for F = rint(a 2^{62 - E}), |F| < 2^62: digit s is byte 7 - s of the sum, less 128.
// The fixed-point value is formed on the integer pipe.
__device__ __forceinline__ unsigned long long f8_fixed(double a, int E) {
  const long long bits = __double_as_longlong(a);
  const int bexp = (int)((bits >> 52) & 0x7FF);
  const int sh = max(bexp, 1) - 1075 + 62 - E;               // <= 9, 10 for subnormals
  unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | ((unsigned long long)(bexp != 0) << 52);
  if (sh >= 0) m <<= min(sh, 10);
  else if (sh > -56) m = (m + (1ull << (-sh - 1))) >> -sh;
  else m = 0;
  return (bits < 0 ? 0ull - m : m) + F8_BIAS;
}
// q_s 2^{-8 s} of a biased value as FP32 (exact): the byte in the low mantissa bits of
// 2^{23 - 8 s}, less (2^23 + 128) 2^{-8 s}
__device__ __forceinline__ float f8_digit(unsigned long long f, int s) {
  const uint32_t q = (uint32_t)(f >> (8 * (7 - s))) & 0xFFu;
  const uint32_t magic = 0x4B000000u - ((uint32_t)(8 * s) << 23);
  return __uint_as_float(magic | q) - __uint_as_float(magic | 128u);
}
// BF16 pair (lo in the low half); the digits are exact in the high 16 bits of their FP32 form
__device__ __forceinline__ uint32_t f8_pack(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// Digit energies, the bound on the level sums: sum of q_s^2 over s <= 5 (high half) and s <= 3
// (low half) in units of 64, rounded up, so that the sum over one row's (column's) 32
// positions of a K step fits 16 bits each.
__device__ __forceinline__ uint32_t f8_energy(const unsigned long long (&f)[4]) {
  int e3 = 0, e5 = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int hi = (int)((uint32_t)(f[q] >> 32) ^ 0x80808080u);             // digits 0..3 as signed bytes
    const int lo = (int)(((uint32_t)f[q] ^ 0x80808080u) & 0xFFFF0000u);     // digits 4, 5
    e3 = __dp4a(hi, hi, e3);
    e5 = __dp4a(lo, lo, e5);
  }
  return ((uint32_t)(e3 + e5 + 63) >> 6 << 16) | ((uint32_t)(e3 + 63) >> 6);
}
// over the 8 lanes that share a row's K step, then the larger of both halves of two values
__device__ __forceinline__ uint32_t f8_energy_step(uint32_t e) {
  for (int o = 1; o < 8; o <<= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  return e;
}
__device__ __forceinline__ uint32_t f8_energy_max(uint32_t a, uint32_t b) { return __vmaxu2(a, b); }
// the warp's largest into the item's two words (s <= 5, s <= 3)
__device__ __forceinline__ void f8_energy_store(uint32_t e, uint32_t* item, int lane) {
  for (int o = 16; o >= 8; o >>= 1) e = f8_energy_max(e, __shfl_xor_sync(0xffffffffu, e, o));
  if (lane == 0) {
    if (item[0] < (e >> 16)) atomicMax(item, e >> 16);
    if (item[1] < (e & 0xFFFFu)) atomicMax(item + 1, e & 0xFFFFu);
  }
}
// K steps that keep every level sum of a segment below 2^24 by Cauchy-Schwarz, given the
// largest energies of both operands' K steps: n sqrt(ea eb) <= 2^24 (0.1% below, for the
// rounding of this expression)
__device__ __forceinline__ int f8_seg(uint32_t ea, uint32_t eb, int least, int steps) {
  const float e = (float)ea * (float)eb;   // in units of 64^2
  const int n = e > 0.f ? (int)(fminf(261881.0f * rsqrtf(e), 4096.0f)) : steps;
  return min(max(n, least), steps);
}

// A digits, one warp per row: row exponent, then 4 consecutive elements per lane and step.
// grid (ceil(d / 8), batch), block 256.  Bound by the digit stores (32 bytes per complex
// entry written, 16 read).
__global__ void __launch_bounds__(256)
f64d_slice_a_kernel(int d, int Kp, const double2* __restrict__ A, long long sA2, __nv_bfloat16* __restrict__ out,
                    long long item_elems, int* __restrict__ ea, int* __restrict__ bad, uint32_t* __restrict__ energy,
                    const int* __restrict__ item_sq, int sq_step) {
  const int lane = threadIdx.x & 31, row = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y;
  if (row >= d) return;
  if (item_sq && item_sq[b] <= sq_step) return;
  const int Kh = Kp / 2;
  const double2* a = A + b * sA2 + (long long)row * d;
  int E = -(1 << 29);
  for (int k = lane; k < d; k += 32) {
    const double2 v = a[k];
    E = max(E, max(f8_exp(v.x), f8_exp(v.y)));
  }
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  const bool mark = f8_marked(E);
  if (E < -(1 << 28)) E = 0;   // all-zero row
  if (lane == 0) {
    ea[(long long)b * d + row] = E + F8_EBIAS;
    if (mark) atomicOr(bad + b, 1);
  }
  __nv_bfloat16* o = out + b * item_elems + (long long)row * Kp;
  const long long ds = (long long)d * Kp;
  uint32_t en = 0;
  for (int k0 = 0; k0 < Kh; k0 += 128) {
    const int k = k0 + 4 * lane;
    unsigned long long re[4], im[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 v = k + q < d ? a[k + q] : make_double2(0.0, 0.0);
      re[q] = f8_fixed(v.x, E);
      im[q] = f8_fixed(v.y, E);
    }
    en = f8_energy_max(en, f8_energy_max(f8_energy_step(f8_energy(re)), f8_energy_step(f8_energy(im))));
    if (k >= Kh) continue;
#pragma unroll
    for (int s = 0; s < F8_L; ++s) {
      *reinterpret_cast<uint2*>(o + s * ds + k) =
          make_uint2(f8_pack(f8_digit(re[0], s), f8_digit(re[1], s)), f8_pack(f8_digit(re[2], s), f8_digit(re[3], s)));
      *reinterpret_cast<uint2*>(o + s * ds + Kh + k) =
          make_uint2(f8_pack(f8_digit(im[0], s), f8_digit(im[1], s)), f8_pack(f8_digit(im[2], s), f8_digit(im[3], s)));
    }
  }
  f8_energy_store(en, energy + 2 * b, lane);
}

// Column exponents (preset to 0): grid (ceil(d/64), ceil(d/64), batch), block 256.
__global__ void __launch_bounds__(256)
f64d_col_exponent_kernel(int d, const double2* __restrict__ B, long long sB2, int* __restrict__ eb,
                         const int* __restrict__ item_sq, int sq_step) {
  __shared__ int red[4][64];
  const int j0 = blockIdx.x * 64, k0 = blockIdx.y * 64, b = blockIdx.z;
  if (item_sq && item_sq[b] <= sq_step) return;
  const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
  const double2* Bb = B + b * sB2;
  int E = -(1 << 29);
  if (j0 + c < d)
    for (int k = k0 + g; k < min(d, k0 + 64); k += 4) {
      const double2 v = Bb[(long long)k * d + j0 + c];
      E = max(E, max(f8_exp(v.x), f8_exp(v.y)));
    }
  red[g][c] = E;
  __syncthreads();
  if (g == 0 && j0 + c < d) {
    E = max(max(red[0][c], red[1][c]), max(red[2][c], red[3][c]));
    if (E > -(1 << 28)) atomicMax(eb + (long long)b * d + j0 + c, E + F8_EBIAS);
  }
}

// Column digits of a 32 (k) x 64 (j) block, staged in shared memory.  ADJ = false: B planes
// (-Im, Re, Im; row j of a plane is column j along k).  ADJ = true: the same columns written
// as A rows of the adjoint, [Re | -Im].  grid (ceil(d/64), Kh/32, batch), block 256.
template <bool ADJ>
__global__ void __launch_bounds__(256)
f64d_slice_col_kernel(int d, int Kp, const double2* __restrict__ B, long long sB2, __nv_bfloat16* __restrict__ out,
                      long long item_elems, int* __restrict__ eb, int* __restrict__ bad, uint32_t* __restrict__ energy,
                      const int* __restrict__ item_sq, int sq_step) {
  __shared__ double2 tile[32][65];
  __shared__ int ex[64];
  const int b = blockIdx.z;
  if (item_sq && item_sq[b] <= sq_step) return;
  const int j0 = blockIdx.x * 64, k0 = blockIdx.y * 32, tid = threadIdx.x, Kh = Kp / 2;
  const double2* Bb = B + b * sB2;
  if (tid < 64) {
    const int E = j0 + tid < d ? f8_exponent(eb[(long long)b * d + j0 + tid]) : 0;
    if (f8_marked(E)) atomicOr(bad + b, 1);
    ex[tid] = E;
  }
  for (int e = tid; e < 32 * 64; e += 256) {
    const int kk = e >> 6, c = e & 63;
    tile[kk][c] = (k0 + kk < d && j0 + c < d) ? Bb[(long long)(k0 + kk) * d + j0 + c] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  uint32_t en = 0;
  for (int e = tid; e < 8 * 64; e += 256) {   // 8 lanes per column
    const int g = e & 7, r = e >> 3, j = j0 + r, k = k0 + 4 * g;
    const int E = ex[r];
    unsigned long long re[4], im[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 v = tile[4 * g + q][r];
      re[q] = f8_fixed(v.x, E);
      im[q] = f8_fixed(ADJ ? -v.y : v.y, E);
    }
    en = f8_energy_max(en, f8_energy_max(f8_energy_step(f8_energy(re)), f8_energy_step(f8_energy(im))));
    if (j >= d) continue;
    if constexpr (ADJ) {
      __nv_bfloat16* o = out + b * item_elems + (long long)j * Kp + k;
      const long long ds = (long long)d * Kp;
#pragma unroll
      for (int s = 0; s < F8_L; ++s) {
        *reinterpret_cast<uint2*>(o + s * ds) = make_uint2(f8_pack(f8_digit(re[0], s), f8_digit(re[1], s)),
                                                           f8_pack(f8_digit(re[2], s), f8_digit(re[3], s)));
        *reinterpret_cast<uint2*>(o + s * ds + Kh) = make_uint2(f8_pack(f8_digit(im[0], s), f8_digit(im[1], s)),
                                                                f8_pack(f8_digit(im[2], s), f8_digit(im[3], s)));
      }
    } else {
      const long long plane = (long long)d * Kh;
      __nv_bfloat16* o = out + b * item_elems + (long long)j * Kh + k;
#pragma unroll
      for (int s = 0; s < F8_L; ++s) {
        const uint2 wi = make_uint2(f8_pack(f8_digit(im[0], s), f8_digit(im[1], s)),
                                    f8_pack(f8_digit(im[2], s), f8_digit(im[3], s)));
        __nv_bfloat16* os = o + s * 3 * plane;
        *reinterpret_cast<uint2*>(os) = make_uint2(wi.x ^ 0x80008000u, wi.y ^ 0x80008000u);
        *reinterpret_cast<uint2*>(os + plane) = make_uint2(f8_pack(f8_digit(re[0], s), f8_digit(re[1], s)),
                                                           f8_pack(f8_digit(re[2], s), f8_digit(re[3], s)));
        *reinterpret_cast<uint2*>(os + 2 * plane) = wi;
      }
    }
  }
  f8_energy_store(en, energy + 2 * b, tid & 31);
}

// Row digits of a real symmetric matrix (both operands of its products are such rows), one
// warp per row: entry k is X[k] + sz Z[k] (Z null: X[k]), or with CW the real part of a complex
// matrix W times 2^{-sq} (an exact change of the row's exponent).  grid (ceil(d / 8), batch).
// Entries are bounded above (the exponential scales them to norm about 1) and finite, so no
// row is marked; the product takes scales down to the smallest subnormal (f8_value).
template <bool CW>
__global__ void __launch_bounds__(256)
f64r_slice_kernel(int d, int Kh, const double* __restrict__ X, const double* __restrict__ Z, double sz, long long sX,
                  int sq, const int* __restrict__ sq_dev, __nv_bfloat16* __restrict__ out, long long item_elems,
                  int* __restrict__ ex, uint32_t* __restrict__ energy, const int* __restrict__ item_sq, int sq_step) {
  const int lane = threadIdx.x & 31, row = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y;
  if (row >= d) return;
  if (item_sq && item_sq[b] <= sq_step) return;
  const double* x = X + b * sX + (long long)row * d * (CW ? 2 : 1);
  const double* z = Z ? Z + b * sX + (long long)row * d : nullptr;
  auto load = [&](int k) {
    if constexpr (CW) return x[2 * k];
    else return z ? fma(sz, z[k], x[k]) : x[k];
  };
  int E = -(1 << 29);
  for (int k = lane; k < d; k += 32) E = max(E, f8_exp(load(k)));
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  const int s = CW ? (sq_dev ? sq_dev[b] : sq) : 0;
  if (E < -(1 << 28)) E = s;                 // all-zero row
  if (lane == 0) ex[(long long)b * d + row] = E - s + F8_EBIAS;
  __nv_bfloat16* o = out + b * item_elems + (long long)row * Kh;
  const long long ds = (long long)d * Kh;
  uint32_t en = 0;
  for (int k0 = 0; k0 < Kh; k0 += 128) {
    const int k = k0 + 4 * lane;
    unsigned long long f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) f[q] = f8_fixed(k + q < d ? load(k + q) : 0.0, E);
    en = f8_energy_max(en, f8_energy_step(f8_energy(f)));
    if (k >= Kh) continue;
#pragma unroll
    for (int g = 0; g < F8_L; ++g)
      *reinterpret_cast<uint2*>(o + g * ds + k) =
          make_uint2(f8_pack(f8_digit(f[0], g), f8_digit(f[1], g)), f8_pack(f8_digit(f[2], g), f8_digit(f[3], g)));
  }
  f8_energy_store(en, energy + 2 * b, lane);
}

// Real symmetric matrices: two linear combinations of up to four matrices in one pass,
// dst_o = sum_m coef[o][m] src_m + diag[o] I (dst_1 may be null).
struct RealComb {
  const double* src[4];
  double coef[2][4], diag[2];
  double* dst[2];
  int n;
};
__global__ void __launch_bounds__(256) f64r_lincomb_kernel(int d, long long total, const __grid_constant__ RealComb a) {
  const long long per = (long long)d * d;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    const long long r = e % per;
    const bool dg = r / d == r % d;
    double v0 = dg ? a.diag[0] : 0.0, v1 = dg ? a.diag[1] : 0.0;
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (m < a.n) {
        const double x = a.src[m][e];
        v0 = fma(a.coef[0][m], x, v0);
        v1 = fma(a.coef[1][m], x, v1);
      }
    if (a.dst[0]) a.dst[0][e] = v0;
    if (a.dst[1]) a.dst[1][e] = v1;
  }
}

// U_b = e^{-i tau_b} (C_b - i S_b); grid (x, batch)
__global__ void __launch_bounds__(256)
f64r_phase_kernel(long long per, const double* __restrict__ tau, const double* __restrict__ C,
                  const double* __restrict__ S, double2* __restrict__ U) {
  __shared__ double ph[2];
  const long long o = blockIdx.y * per;
  if (threadIdx.x == 0) {
    ph[0] = 1.0;
    ph[1] = 0.0;
    if (tau) sincos(tau[blockIdx.y], &ph[1], &ph[0]);
  }
  __syncthreads();
  const double cs = ph[0], sn = ph[1];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < per; e += (long long)gridDim.x * blockDim.x) {
    const double c = C[o + e], s = S[o + e];
    U[o + e] = make_double2(cs * c - sn * s, -(sn * c + cs * s));
  }
}

// ---------------------------------------------------------------------------
// product
// ---------------------------------------------------------------------------
struct F8Args {
  const double* A;            // the operands themselves, for marked items (complex products)
  const double* B;
  long long sA, sB;           // doubles
  int opA;
  int d, Kp, batch, ntn, ntm;   // Kp: length of the K axis; per item ntm x ntn tiles
  const int* ea;
  const int* eb;
  const int* bad_a;
  const int* bad_b;
  const unsigned char* weak;  // per tile: the digits do not hold its weakest entries (null: not asked)
  const uint32_t* en_a;       // per item: largest digit energies of a K step (f8_energy)
  const uint32_t* en_b;
  double* C;
  long long sC;               // doubles
  const double* add_src[3];
  double add_coef[3];
  long long add_stride;       // doubles
  int add_n;
  double diag;
  int scale2;                 // real products only: the product times 2^scale2
  uint32_t* scratch;          // per CTA: the low words of F8_VALS x F8_EPI sums of levels 4..7
  int* status;
  const int* item_sq;
  int sq_step;
  unsigned long long wait_ns;
  int stall;                  // test only: the MMA issuer waits on a barrier nothing completes
};

__device__ __forceinline__ bool f8_done(const F8Args& p, int b) { return p.item_sq && p.item_sq[b] <= p.sq_step; }
// tile t (of item b) runs in FP64 arithmetic
__device__ __forceinline__ bool f8_pipe_tile(const F8Args& p, int b, long long t) {
  return ((p.bad_a && (p.bad_a[b] | p.bad_b[b]) != 0) || (p.weak && p.weak[t])) && !f8_done(p, b);
}
__device__ __forceinline__ bool f8_skip(const F8Args& p, int b, long long t) {
  return (p.bad_a && (p.bad_a[b] | p.bad_b[b]) != 0) || (p.weak && p.weak[t]) || f8_done(p, b);
}

// Where the operands are a caller's own (any range of magnitudes in a row), FP64 arithmetic
// bounds the error of an entry by about d u M_ij + u |P_ij|, M = |A| |B| and P the addends; the
// digits' is sqrt(d) 2^-61 2^{Ea_i + Eb_j} whatever the entry's own terms are (the standard
// deviation of rounding each entry at 2^-63 of its row's or column's scale and of leaving out
// the digit pairs s + t >= 8).  This kernel forms M in FP32 (the larger component's magnitude,
// rounded down, scaled by 2^{57 - Ea}, 2^{57 - Eb}) and sends a tile to FP64 arithmetic where
// an entry has M + |P| / d < 2^{114 - 8} / sqrt(d).  M = 0 is a zero of the operands'
// structure, which the digits give exactly, unless some entry in reach is below 2^-110 of its
// row or column.  128 x 64 outputs per CTA (the product's tiles), 4 x 4 per thread, K in slabs of
// 16 until every output of the tile holds: the terms only add up.  Bound by latency.  Exponentials
// of dense matrices, in us without the check / with every K / as it is: 64 of d = 64 1012 / 1218 /
// 1149, 37 of d = 100 1294 / 1582 / 1438, 10 of d = 200 1632 / 2080 / 1767, 5 of d = 400 2268 /
// 3029 / 2424.  (256 threads of 8 x 4 outputs took 42 us a launch at d = 81, batch 64, against 16.)
constexpr int F8_NK = 16;              // K per slab
constexpr int F8_WEAK_THREADS = 512;
// the larger component's magnitude times 2^k, rounded down (0 below FP32's normal range,
// infinity above it); without FP64 instructions
__device__ __forceinline__ float f8_magnitude(double2 v, int k) {
  const int hi = max(__double2hiint(v.x) & 0x7FFFFFFF, __double2hiint(v.y) & 0x7FFFFFFF);
  const int fe = (hi >> 20) - 1023 + 127 + k;
  if (hi < 0x00100000 || fe <= 0) return 0.f;
  return fe >= 255 ? __int_as_float(0x7F800000) : __int_as_float((fe << 23) | ((hi & 0xFFFFF) << 3));
}
__device__ __forceinline__ bool f8_nonzero(double2 v) {
  return (((unsigned long long)__double_as_longlong(v.x) | (unsigned long long)__double_as_longlong(v.y)) << 1) != 0;
}
__global__ void __launch_bounds__(F8_WEAK_THREADS)
f64d_weak_kernel(const __grid_constant__ F8Args p, float least, unsigned char* __restrict__ weak) {
  __shared__ __align__(16) float As[F8_NK][F8_BM + 4], Bs[F8_NK][F8_BN];
  const int b = blockIdx.y, tid = threadIdx.x, d = p.d;
  const long long t = (long long)b * gridDim.x + blockIdx.x;
  if (f8_done(p, b) || (p.bad_a[b] | p.bad_b[b]) != 0) {   // not multiplied, or in FP64 arithmetic anyway
    if (tid == 0) weak[t] = 0;
    return;
  }
  const int i0 = blockIdx.x / p.ntn * F8_BM, j0 = blockIdx.x % p.ntn * F8_BN;
  const double2* A = reinterpret_cast<const double2*>(p.A + b * p.sA);
  const double2* B = reinterpret_cast<const double2*>(p.B + b * p.sB);
  const int* ea = p.ea + (long long)b * d;
  const int* eb = p.eb + (long long)b * d;
  // loads: four entries of A and two of B per thread and slab of K, one slab ahead
  auto row = [&](int q) { return p.opA ? tid & 127 : (tid >> 4) + 32 * q; };
  auto ka = [&](int q) { return p.opA ? (tid >> 7) + 4 * q : tid & 15; };
  const int jb = tid & 63;
  double2 av[4], bv[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + row(q), k = k0 + ka(q);
      av[q] = make_double2(0.0, 0.0);
      if (i < d && k < d) av[q] = A[p.opA ? (long long)k * d + i : (long long)i * d + k];
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = k0 + (tid >> 6) + 8 * q;
      bv[q] = make_double2(0.0, 0.0);
      if (j0 + jb < d && k < d) bv[q] = B[(long long)k * d + j0 + jb];
    }
  };
  load(0);
  const int Eb = j0 + jb < d ? f8_exponent(eb[j0 + jb]) : 0;
  int Ea[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) Ea[q] = i0 + row(q) < d ? f8_exponent(ea[i0 + row(q)]) : 0;
  const int c0 = (tid & 15) * 4, r0 = (tid >> 4) * 4;   // outputs: 4 x 4
  constexpr float kTiny = 1.1102230246251565e-16f;      // 2^{57 - 110}
  const float per_d = 1.0f / (float)d;
  float m[4][4] = {}, add[4][4] = {};                   // M so far, |P| / d
  bool tiny = false;
  // an output of this thread does not hold the bound with the terms so far (zero: M = 0 counts)
  auto short_of = [&](bool zero) {
    bool low = false;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        low |= i0 + r0 + r < d && j0 + c0 + c < d && m[r][c] + add[r][c] < least && (m[r][c] > 0.f || zero);
    return low;
  };
  for (int k0 = 0; k0 < d; k0 += F8_NK) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = f8_magnitude(av[q], 57 - Ea[q]);
      tiny |= v < kTiny && f8_nonzero(av[q]);
      As[ka(q)][row(q)] = v;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float v = f8_magnitude(bv[q], 57 - Eb);
      tiny |= v < kTiny && f8_nonzero(bv[q]);
      Bs[(tid >> 6) + 8 * q][jb] = v;
    }
    __syncthreads();
    if (k0 + F8_NK < d) load(k0 + F8_NK);
    if (i0 + r0 < d && j0 + c0 < d) {
#pragma unroll
      for (int k = 0; k < F8_NK; ++k) {
        const float4 x = *reinterpret_cast<const float4*>(&As[k][r0]), y = *reinterpret_cast<const float4*>(&Bs[k][c0]);
        const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) m[r][c] = fmaf(xs[r], ys[c], m[r][c]);
      }
    }
    // M only grows: a tile of dense operands is done after one slab, with addends after two
    if (!__syncthreads_or(short_of(true))) {
      if (tid == 0) weak[t] = 0;
      return;
    }
    if (k0 == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int i = i0 + r0 + r, j = j0 + c0 + c;
          if (i >= d || j >= d) continue;
          const int k = 114 - f8_exponent(ea[i]) - f8_exponent(eb[j]);
          float v = i == j ? f8_magnitude(make_double2(p.diag, 0.0), k) : 0.f;
#pragma unroll
          for (int q = 0; q < 3; ++q)
            if (q < p.add_n) {
              const float x = f8_magnitude(reinterpret_cast<const double2*>(p.add_src[q] + b * p.add_stride)[(long long)i * d + j], k);
              if (x > 0.f) v = fmaf(fabsf((float)p.add_coef[q]), x, v);
            }
          add[r][c] = v * per_d;
        }
    }
  }
  const bool any_tiny = __syncthreads_or(tiny);
  const bool low = __syncthreads_or(short_of(any_tiny));
  if (tid == 0) weak[t] = low;
}

// The tiles of marked items, and weak ones, in FP64 arithmetic, once a CTA's digit tiles are
// done: no wait of theirs is open then, however long this takes.  16 x 16 outputs per group of
// 256 threads (two groups: the epilogue warps), dealt over all groups of the grid; operands
// through shared memory, sums in the order of cgemm_f64_kernel (the same bits).
__device__ __noinline__ void f8_pipe_tiles(const F8Args& p, double2* stage, int et) {
  const int g = et >> 8, tx = et & 15, ty = (et >> 4) & 15, d = p.d;
  double2* As = stage + g * (16 * 17 + 16 * 16);   // [k][i], pitch 17
  double2* Bs = As + 16 * 17;                      // [k][j]
  const int per_item = p.ntm * p.ntn;
  const long long tiles = (long long)per_item * p.batch;
  const int all = 2 * (int)gridDim.x;
  int turn = 2 * (int)blockIdx.x + g;              // 16 x 16 outputs until this group's next ones
  auto sync = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + g) : "memory"); };
  for (long long t0 = 0; t0 < tiles; t0 += 32) {
    const long long tl = t0 + (et & 31);
    unsigned todo = __ballot_sync(0xffffffffu, tl < tiles && f8_pipe_tile(p, (int)(tl / per_item), tl));
    for (; todo; todo &= todo - 1) {
      const long long t = t0 + __ffs(todo) - 1;
      const int b = (int)(t / per_item), rem = (int)(t % per_item);
      const double2* A = reinterpret_cast<const double2*>(p.A + b * p.sA);
      const double2* B = reinterpret_cast<const double2*>(p.B + b * p.sB);
      constexpr int PER = F8_BM * F8_BN / 256;
      int u = turn;
      for (; u < PER; u += all) {
        const int i0 = rem / p.ntn * F8_BM + u / (F8_BN / 16) * 16, j0 = rem % p.ntn * F8_BN + u % (F8_BN / 16) * 16;
        if (i0 >= d || j0 >= d) continue;
        double re = 0.0, im = 0.0;
        for (int k0 = 0; k0 < d; k0 += 16) {
          double2 v = make_double2(0.0, 0.0), w = v;
          if (p.opA == 0) {   // A[i0 + ty][k0 + tx]
            if (i0 + ty < d && k0 + tx < d) v = A[(long long)(i0 + ty) * d + k0 + tx];
            As[tx * 17 + ty] = v;
          } else {            // conj(A[k0 + ty][i0 + tx])
            if (i0 + tx < d && k0 + ty < d) v = A[(long long)(k0 + ty) * d + i0 + tx];
            As[ty * 17 + tx] = make_double2(v.x, -v.y);
          }
          if (k0 + ty < d && j0 + tx < d) w = B[(long long)(k0 + ty) * d + j0 + tx];
          Bs[ty * 16 + tx] = w;
          sync();
          const int kmax = min(16, d - k0);
          for (int k = 0; k < kmax; ++k) {
            const double2 x = As[k * 17 + ty], y = Bs[k * 16 + tx];
            re = fma(x.x, y.x, re);
            re = fma(-x.y, y.y, re);
            im = fma(x.x, y.y, im);
            im = fma(x.y, y.x, im);
          }
          sync();
        }
        const int i = i0 + ty, j = j0 + tx;
        if (i < d && j < d) {
          const long long off = (long long)i * d + j;
          for (int m = 0; m < p.add_n; ++m) {
            const double2 v = reinterpret_cast<const double2*>(p.add_src[m] + b * p.add_stride)[off];
            re = fma(p.add_coef[m], v.x, re);
            im = fma(p.add_coef[m], v.y, im);
          }
          if (i == j) re += p.diag;
          reinterpret_cast<double2*>(p.C + b * p.sC)[off] = make_double2(re, im);
        }
      }
      turn = u - PER;
    }
  }
}

// polls until the phase completes, the CTA aborts or the limit runs out
__device__ __forceinline__ bool f8_wait(uint64_t* bar, uint32_t parity, unsigned long long limit, volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort || global_ns() - t0 > limit) return false;
  }
  return true;
}

// (t 2^32 + w) 2^k rounded to FP64, |t| < 2^63; k keeps the result below 2^1024, and with
// TINY = false above FP64's smallest normal number (otherwise what lies below that becomes 0).
template <bool TINY>
__device__ __forceinline__ double f8_value(long long t, uint32_t w, int k) {
  const uint32_t neg = (uint32_t)((unsigned long long)t >> 63);
  const unsigned long long s = 0ull - neg;
  w = (w ^ (uint32_t)s) + neg;                                   // |T|, 96 bits
  unsigned long long u = ((unsigned long long)t ^ s) + (neg & (w == 0u));
  uint32_t t1 = (uint32_t)(u >> 32), t0 = (uint32_t)u;
  int e = k + 95 + 1022;                                         // biased exponent less one if t1's top bit is set
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const bool z = t1 == 0u;
    t1 = z ? t0 : t1;
    t0 = z ? w : t0;
    w = z ? 0u : w;
    e -= z ? 32 : 0;
  }
  const int lz = __clz((int)t1);
  const uint32_t m1 = __funnelshift_l(t0, t1, lz), m0 = __funnelshift_l(w, t0, lz);   // 64 bits, the top one set
  // 53 bits and the rounding bit; a carry runs into the exponent as it should
  const unsigned long long m = ((unsigned long long)m1 << 32 | m0) >> 11;
  const unsigned long long bits = ((unsigned long long)(uint32_t)(e - lz) << 52) + m + ((m0 >> 10) & 1u);
  return t1 == 0u || (TINY && e <= lz) ? 0.0 : __longlong_as_double((long long)(bits | (unsigned long long)neg << 63));
}

// The same on the FP64 pipe, |t| < 2^51.  A warp's FP64 instruction takes about 68 cycles of
// its quarter of the SM, the integer form some 50 dependent instructions: the epilogues send
// every fourth value here, which is where the two balance.
__device__ __forceinline__ double f8_value_fp64(long long t, uint32_t w, int k) {
  // t 2^-64 and w 2^-96, exact: (1.5 2^52 + t) 2^-64 - 1.5 2^-12, (2^52 + w) 2^-96 - 2^-44
  const double h = __longlong_as_double(t + 0x3F38000000000000ll) - 0.0003662109375;
  const double l = __hiloint2double(0x3D300000, (int)w) - 5.684341886080802e-14;
  return (h + l) * __hiloint2double(max(k + 96 + 1023, 0) << 20, 0);   // 2^{k + 96}; 0 from k = -1119 down
}

// Drain of one accumulator set (levels l0 .. l0 + 3) into the thread's sums, in units of
// 2^{-8 (l0 + 3)}, from the integers G_l = 2^{8 l} g_l.
template <bool CPLX>
__device__ __forceinline__ void f8_drain(uint32_t tbase, int l0, long long (&acc)[F8_VALS]) {
  const float m0 = l0 ? 4294967296.0f : 1.0f;   // 2^{8 l0}
  const float m1 = m0 * 256.0f, m2 = m0 * 65536.0f, m3 = m0 * 16777216.0f;
#pragma unroll
  for (int c = 0; c < F8_VALS; c += 4) {
    // complex: values 0..15 are the real parts of the thread's 16 columns, 16..31 the imaginary
    // parts; real: 32 columns
    const uint32_t col = tbase + (CPLX && c >= F8_VALS / 2 ? F8_BN + c - F8_VALS / 2 : c);
    uint32_t g[4][4];
#pragma unroll
    for (int l = 0; l < 4; ++l) tmem_ld4(col + l * 128, g[l]);
    tmem_wait_ld();
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      acc[c + v] += (long long)__float2int_rn(__uint_as_float(g[0][v]) * m0) * 16777216 +
                    (long long)__float2int_rn(__uint_as_float(g[1][v]) * m1) * 65536;
      acc[c + v] += (long long)__float2int_rn(__uint_as_float(g[2][v]) * m2) * 256 +
                    __float2int_rn(__uint_as_float(g[3][v]) * m3);
    }
  }
}

constexpr uint32_t kF8Idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

// tile `rem` of an item: row by row, or (SYM: real symmetric products) the lower triangle
template <bool CPLX>
__device__ __forceinline__ void f8_tile(const F8Args& p, int rem, int& mt, int& nt) {
  if constexpr (CPLX) {
    mt = rem / p.ntn;
    nt = rem % p.ntn;
  } else {
    mt = 0;
    while ((mt + 1) * (mt + 2) / 2 <= rem) ++mt;   // at most 32 row tiles
    nt = rem - mt * (mt + 1) / 2;
  }
}

// CPLX: 128 x 64 complex tiles as described above.  Otherwise products of commuting real
// symmetric matrices (polynomials in one matrix): both operands are row digits, tiles are
// 128 x 128 real entries on and below the diagonal, and every entry is written on both sides
// of it; addends are symmetric too.
template <bool CPLX>
__global__ void __launch_bounds__(F8_THREADS, 1)
f64d_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ F8Args p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  double2* staging = reinterpret_cast<double2*>(smem + F8_SLOTS * F8_SLOT_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + F8_SLOTS * F8_SLOT_BYTES + F8_STAGE_BYTES);
  uint64_t* empty = full + F8_SLOTS;
  uint64_t* accfull = empty + F8_SLOTS;    // an accumulator set is complete
  uint64_t* accempty = accfull + 1;        // ... and drained
  uint64_t* mmadone = accempty + 1;        // closing commit
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mmadone + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* pipe_flag = abort_flag + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < F8_SLOTS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accfull, 1);
    mbar_init(accempty, F8_EPI_WARPS);
    mbar_init(mmadone, 1);
    *abort_flag = 0;
    *pipe_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int steps = p.Kp / F8_BK, half = steps / 2;
  const int per_item = CPLX ? p.ntn * p.ntm : p.ntm * (p.ntm + 1) / 2;
  const long long tiles = (long long)per_item * p.batch;
  // drains of an item's sweep (0: levels 4..7, 1: levels 0..3)
  auto segments = [&](int b, int sweep) {
    const int n = f8_seg(p.en_a[2 * b + sweep], p.en_b[2 * b + sweep], sweep == 0 ? F8_SEG_LO : F8_SEG_HI, steps);
    return (steps + n - 1) / n;
  };

  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(F8_REGS_IO));
  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      long long n = 0;   // slots filled
      bool ok = true;
      for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int b = (int)(t / per_item);
        int mt, nt;
        f8_tile<CPLX>(p, (int)(t % per_item), mt, nt);
        if (f8_skip(p, b, t)) continue;
        for (int sweep = 0; sweep < 2 && ok; ++sweep) {
          const int per_step = sweep == 0 ? 4 : 2;
          for (int st = 0; st < steps && ok; ++st) {
            const bool imag = st >= half;
            for (int q = 0; q < per_step; ++q) {
              // slot order: A digits 0..3, B 0..3, B 4..7, A 4..7
              const int s = (int)(n % F8_SLOTS);
              if (!f8_wait(&empty[s], (uint32_t)((n / F8_SLOTS) & 1) ^ 1u, p.wait_ns, abort_flag)) {
                ok = false;
                break;
              }
              mbar_expect_tx(&full[s], F8_SLOT_BYTES);
              unsigned char* dst = smem + s * F8_SLOT_BYTES;
              if (q == 0 || q == 3)
                tma_load_4d(dst, &tmA, &full[s], st * F8_BK, mt * F8_BM, q == 0 ? 0 : 4, b);
              else if constexpr (!CPLX)
                tma_load_4d(dst, &tmB, &full[s], st * F8_BK, nt * F8_BM, q == 1 ? 0 : 4, b);
              else
                tma_load_5d(dst, &tmB, &full[s], (imag ? st - half : st) * F8_BK, nt * F8_BN, imag ? 0 : 1,
                            q == 1 ? 0 : 4, b);
              ++n;
            }
          }
        }
      }
      if (!ok) {
        if (!*abort_flag) atomicExch(p.status, MG_DEV_TIMEOUT);
        *abort_flag = 1;
      }
      // no copy into this CTA's shared memory stays in flight
      const long long from = n > F8_SLOTS ? n - F8_SLOTS : 0;
      for (long long i = from; i < n; ++i) {
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(&full[i % F8_SLOTS], (uint32_t)((i / F8_SLOTS) & 1)) && global_ns() - t0 < 4000000000ull) {
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      long long n = 0;
      uint32_t set = 0;   // accumulator sets begun
      bool ok = !p.stall || f8_wait(mmadone, 0, p.wait_ns, abort_flag);
      for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int b = (int)(t / per_item);
        if (f8_skip(p, b, t)) continue;
        for (int sweep = 0; sweep < 2 && ok; ++sweep) {
          const int ns = segments(b, sweep);
          for (int sg = 0; sg < ns && ok; ++sg) {
            const int st0 = (int)((long long)steps * sg / ns), st1 = (int)((long long)steps * (sg + 1) / ns);
            if (!f8_wait(accempty, (set & 1) ^ 1u, p.wait_ns, abort_flag)) { ok = false; break; }
            tc_fence_after();
            for (int st = st0; st < st1; ++st) {
              uint32_t sa[4];   // shared-memory address of the step's slots
#pragma unroll
              for (int q = 0; q < 4; ++q) sa[q] = smem_u32(smem + (int)((n + q) % F8_SLOTS) * F8_SLOT_BYTES);
              auto ready = [&](int q) {
                const long long i = n + q;
                return f8_wait(&full[i % F8_SLOTS], (uint32_t)((i / F8_SLOTS) & 1), p.wait_ns, abort_flag);
              };
              const bool fst = st == st0;
              // the digit pairs (s0 + s, t0 + u), s, u < 4, of levels lmin .. lmax
              auto group = [&](uint32_t abase, uint32_t bbase, int s0, int t0, int lmin, int lmax, bool (&first)[4]) {
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)
#pragma unroll
                  for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                      const int l = s0 + s + t0 + u;
                      if (l < lmin || l > lmax) continue;
                      const uint64_t ad = sw64_kmajor_desc(abase + s * 8192 + kk * 32);
                      const uint64_t bd = sw64_kmajor_desc(bbase + u * 8192 + kk * 32);
                      tc_mma_bf16(tmem + (l & 3) * 128, ad, bd, kF8Idesc, first[l & 3] ? 0u : 1u);
                      first[l & 3] = false;
                    }
              };
              bool first[4] = {fst, fst, fst, fst};
              if (!ready(0) || !ready(1)) { ok = false; break; }
              tc_fence_after();
              if (sweep == 0) {
                group(sa[0], sa[1], 0, 0, 4, 7, first);
                if (!ready(2)) { ok = false; break; }
                tc_fence_after();
                group(sa[0], sa[2], 0, 4, 4, 7, first);
                tc_commit(&empty[n % F8_SLOTS]);
                tc_commit(&empty[(n + 2) % F8_SLOTS]);
                if (!ready(3)) { ok = false; break; }
                tc_fence_after();
                group(sa[3], sa[1], 4, 0, 4, 7, first);
                tc_commit(&empty[(n + 1) % F8_SLOTS]);
                tc_commit(&empty[(n + 3) % F8_SLOTS]);
                n += 4;
              } else {
                group(sa[0], sa[1], 0, 0, 0, 3, first);
                tc_commit(&empty[n % F8_SLOTS]);
                tc_commit(&empty[(n + 1) % F8_SLOTS]);
                n += 2;
              }
            }
            if (!ok) break;
            tc_commit(accfull);
            ++set;
          }
        }
      }
      if (!ok) {
        if (!*abort_flag) atomicExch(p.status, MG_DEV_TIMEOUT);
        *abort_flag = 1;
      }
      // no MMA stays in flight when TMEM is freed
      tc_commit(mmadone);
      const uint64_t t0 = global_ns();
      while (!mbar_try_wait(mmadone, 0) && global_ns() - t0 < 4000000000ull) {
      }
    }
  } else if constexpr (CPLX) {
    // ---------------- warps 2, 3: does any tile run in FP64 arithmetic? ----------------
    bool any = false;
    for (int b = threadIdx.x - 64; b < p.batch; b += 64) any |= (p.bad_a[b] | p.bad_b[b]) != 0 && !f8_done(p, b);
    if (p.weak)
      for (long long t = threadIdx.x - 64; t < tiles; t += 64) any |= p.weak[t] != 0;
    if (any) *pipe_flag = 1;
  }
  } else {
    // ---------------- epilogue (warps 4..19) ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(F8_REGS_EPI));
    const int q = warp & 3;                    // TMEM lane quarter of this warp
    constexpr int WC = CPLX ? 16 : 32;         // columns per warp, four warps to a tile's row
    const int c0 = ((warp - 4) >> 2) * WC;
    const int et = threadIdx.x - 128;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + c0;
    uint32_t* scratch = p.scratch + (long long)blockIdx.x * F8_VALS * F8_EPI + et;
    double2* stg = staging + (warp - 4) * 128;
    uint32_t set = 0;
    bool ok = true;
    long long t = blockIdx.x;
    for (; t < tiles; t += gridDim.x) {
      const int b = (int)(t / per_item);
      int mt, nt;
      f8_tile<CPLX>(p, (int)(t % per_item), mt, nt);
      const int row0 = mt * F8_BM + q * 32, col0 = nt * 4 * WC + c0;
      if (f8_skip(p, b, t)) continue;
      // uniform over the warp; a real tile's columns right of all its rows are not needed
      const bool live = row0 < p.d && col0 < p.d && (CPLX || col0 <= row0 + 31);
      long long acc[F8_VALS];
#pragma unroll
      for (int v = 0; v < F8_VALS; ++v) acc[v] = 0;
      for (int sweep = 0; sweep < 2 && ok; ++sweep) {
        const int ns = segments(b, sweep);
        for (int sg = 0; sg < ns; ++sg) {
          bool got = true;
          if (lane == 0) got = f8_wait(accfull, set & 1, p.wait_ns, abort_flag);
          got = __shfl_sync(0xffffffffu, (int)got, 0) != 0;
          if (!got) { ok = false; break; }
          tc_fence_after();
          if (live) f8_drain<CPLX>(tbase, sweep == 0 ? 4 : 0, acc);
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(accempty)) : "memory");
          ++set;
        }
        if (sweep == 0 && ok && live) {
          // the levels 4..7, in units of 2^-56: the sums of levels 0..3, in units of 2^-24, go
          // on from their high words; the low words wait in the scratch
#pragma unroll
          for (int v = 0; v < F8_VALS; ++v) {
            scratch[v * F8_EPI] = (uint32_t)acc[v];
            acc[v] >>= 32;
          }
          if (p.add_n > 0) {   // the tile's addends into L2 (128-byte lines)
            const int lines = 2, n = p.add_n * 32 * lines;
            const int r0 = CPLX ? row0 : col0, q0 = CPLX ? col0 : row0;   // real addends are read as columns
            for (int i = lane; i < n; i += 32) {
              const int m = i / (32 * lines), r = r0 + i / lines % 32, c = q0 + (i % lines) * (CPLX ? 8 : 16);
              if (r < p.d && c < p.d)
                asm volatile("prefetch.global.L2 [%0];" ::"l"((m == 0 ? p.add_src[0] : m == 1 ? p.add_src[1] : p.add_src[2]) +
                                                              b * p.add_stride + ((long long)r * p.d + c) * (CPLX ? 2 : 1)));
            }
          }
        }
      }
      if (!ok) break;
      if (!live) continue;
      const int row = row0 + lane;
      const int Ea = row < p.d ? f8_exponent(p.ea[(long long)b * p.d + row]) : 0;
      if constexpr (!CPLX) {
        // entry (row, col) goes to both sides of the diagonal: (col, row) straight from the
        // registers (lanes are consecutive rows), (row, col) through the warp's staging
        double* Cr = p.C + b * p.sC;
        double* stg8 = reinterpret_cast<double*>(stg);
        const int* ebp = p.eb + (long long)b * p.d;
        uint32_t lo[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) lo[v] = scratch[v * F8_EPI];
#pragma unroll
        for (int c = 0; c < F8_VALS; c += 8) {
          uint32_t w[8];
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            w[v] = lo[v];
            if (c + 8 < F8_VALS) lo[v] = scratch[(c + 8 + v) * F8_EPI];   // one round ahead
          }
          if (col0 + c < p.d && col0 + c <= row0 + 31) {
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              const int col = col0 + c + v;
              const int k = Ea + (col < p.d ? f8_exponent(ebp[col]) : 0) - 68 + p.scale2;
              double x = v % 4 == 3 ? f8_value_fp64(acc[c + v], w[v], k) : f8_value<true>(acc[c + v], w[v], k);
              if (row < p.d && col <= row) {
                const long long off = (long long)col * p.d + row;
#pragma unroll
                for (int m = 0; m < 3; ++m)
                  if (m < p.add_n) x = fma(p.add_coef[m], p.add_src[m][b * p.add_stride + off], x);
                if (col == row) x += p.diag;
                Cr[off] = x;
              }
              stg8[lane * 8 + (v ^ (lane & 7))] = x;
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = i * 4 + (lane >> 3), cc = lane & 7;
              const int grow = row0 + r, gcol = col0 + c + cc;
              if (grow < p.d && gcol < grow) Cr[(long long)grow * p.d + gcol] = stg8[r * 8 + (cc ^ (r & 7))];
            }
            __syncwarp();
          }
        }
      } else {
      const int Eb = col0 + lane < p.d ? f8_exponent(p.eb[(long long)b * p.d + col0 + lane]) : 0;
      const double2* addp[3];
#pragma unroll
      for (int m = 0; m < 3; ++m)
        addp[m] = reinterpret_cast<const double2*>(m < p.add_n ? p.add_src[m] + b * p.add_stride : nullptr);
      double2* Cb = reinterpret_cast<double2*>(p.C + b * p.sC);
      uint32_t lre[4], lim[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        lre[v] = scratch[v * F8_EPI];
        lim[v] = scratch[(WC + v) * F8_EPI];
      }
#pragma unroll
      for (int c = 0; c < WC; c += 4) {   // 4 columns at a time through the warp's staging
        uint32_t wre[4], wim[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          wre[v] = lre[v];
          wim[v] = lim[v];
          if (c + 4 < WC) {   // one round ahead
            lre[v] = scratch[(c + 4 + v) * F8_EPI];
            lim[v] = scratch[(WC + 4 + c + v) * F8_EPI];
          }
        }
        if (col0 + c < p.d) {
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            // the value is (sum 2^32 + low word) 2^{Ea + Eb - 68}, in units of 2^-56; every
            // fourth goes over the FP64 pipe
            const int k = Ea + __shfl_sync(0xffffffffu, Eb, c + v) - 68;
            const double re = f8_value<false>(acc[c + v], wre[v], k);
            const double im = v & 1 ? f8_value_fp64(acc[WC + c + v], wim[v], k) : f8_value<false>(acc[WC + c + v], wim[v], k);
            stg[lane * 4 + (v ^ ((lane >> 1) & 3))] = make_double2(re, im);
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = i * 8 + (lane >> 2), cc = lane & 3;
            const int grow = row0 + r, gcol = col0 + c + cc;
            if (grow < p.d && gcol < p.d) {
              double2 v = stg[r * 4 + (cc ^ ((r >> 1) & 3))];
              const long long off = (long long)grow * p.d + gcol;
#pragma unroll
              for (int m = 0; m < 3; ++m)
                if (m < p.add_n) {
                  const double2 a = addp[m][off];
                  v.x = fma(p.add_coef[m], a.x, v.x);
                  v.y = fma(p.add_coef[m], a.y, v.y);
                }
              if (grow == gcol) v.x += p.diag;
              Cb[off] = v;
            }
          }
          __syncwarp();
        }
      }
      }
    }
    if (!ok) {
      if (lane == 0) {
        if (!*abort_flag) atomicExch(p.status, MG_DEV_TIMEOUT);
        *abort_flag = 1;
      }
      // the tiles this CTA leaves unfinished are not left looking like a result (marked items
      // are computed below)
      const double nan = __longlong_as_double(0x7FF8000000000000ll);
      for (; t < tiles; t += gridDim.x) {
        const int b = (int)(t / per_item);
        int mt, nt;
        f8_tile<CPLX>(p, (int)(t % per_item), mt, nt);
        const int row = mt * F8_BM + q * 32 + lane;
        if (f8_skip(p, b, t) || row >= p.d) continue;
        const int n0 = nt * 4 * WC + c0;
        for (int c = n0; c < min(p.d, n0 + WC); ++c) {
          if constexpr (CPLX) reinterpret_cast<double2*>(p.C + b * p.sC)[(long long)row * p.d + c] = make_double2(nan, nan);
          else p.C[b * p.sC + (long long)row * p.d + c] = p.C[b * p.sC + (long long)c * p.d + row] = nan;
        }
      }
    }
    tc_fence_before();
  }
  __syncwarp();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if constexpr (CPLX)
    if (warp >= 4 && *pipe_flag) f8_pipe_tiles(p, staging, threadIdx.x - 128);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct F8Buf {
  __nv_bfloat16* dig;
  int* e;
  int* bad;
  uint32_t* energy;
};
static F8Buf f8_buf(void* buf, long long elems, int d, int batch) {
  F8Buf r;
  r.dig = reinterpret_cast<__nv_bfloat16*>(buf);
  r.e = reinterpret_cast<int*>(r.dig + elems * batch);
  r.bad = r.e + (long long)d * batch;
  r.energy = reinterpret_cast<uint32_t*>(r.bad + batch);
  return r;
}

int f64d_slice_a(int d, int batch, const double* A, long long sA, int opA, void* buf, cudaStream_t s,
                 const SplitCtl& ctl) {
  if (batch > 65535) return MG_EUNSUPPORTED;
  const F8Geom g = f8_geom(d);
  const F8Buf o = f8_buf(buf, g.a_elems, d, batch);
  const double2* A2 = reinterpret_cast<const double2*>(A);
  if (opA == 0) {
    MG_CUDA_TRY(cudaMemsetAsync(o.bad, 0, 3 * sizeof(int) * (size_t)batch, s));
    f64d_slice_a_kernel<<<dim3(ceil_div(d, 8), batch), 256, 0, s>>>(d, g.Kp, A2, sA / 2, o.dig, g.a_elems, o.e, o.bad,
                                                                    o.energy, ctl.item_sq, ctl.sq_step);
    return check_launch("f64d_slice_a_kernel");
  }
  MG_CUDA_TRY(cudaMemsetAsync(o.e, 0, sizeof(int) * (size_t)(d + 3) * batch, s));   // exponents, marks, energies
  f64d_col_exponent_kernel<<<dim3(ceil_div(d, 64), ceil_div(d, 64), batch), 256, 0, s>>>(d, A2, sA / 2, o.e,
                                                                                          ctl.item_sq, ctl.sq_step);
  MG_TRY(check_launch("f64d_col_exponent_kernel"));
  f64d_slice_col_kernel<true><<<dim3(ceil_div(d, 64), g.Kh / 32, batch), 256, 0, s>>>(
      d, g.Kp, A2, sA / 2, o.dig, g.a_elems, o.e, o.bad, o.energy, ctl.item_sq, ctl.sq_step);
  return check_launch("f64d_slice_col_kernel");
}

int f64d_slice_b(int d, int batch, const double* B, long long sB, void* buf, cudaStream_t s, const SplitCtl& ctl) {
  if (batch > 65535) return MG_EUNSUPPORTED;
  const F8Geom g = f8_geom(d);
  const F8Buf o = f8_buf(buf, g.b_elems, d, batch);
  const double2* B2 = reinterpret_cast<const double2*>(B);
  MG_CUDA_TRY(cudaMemsetAsync(o.e, 0, sizeof(int) * (size_t)(d + 3) * batch, s));   // exponents, marks, energies
  f64d_col_exponent_kernel<<<dim3(ceil_div(d, 64), ceil_div(d, 64), batch), 256, 0, s>>>(d, B2, sB / 2, o.e,
                                                                                          ctl.item_sq, ctl.sq_step);
  MG_TRY(check_launch("f64d_col_exponent_kernel"));
  f64d_slice_col_kernel<false><<<dim3(ceil_div(d, 64), g.Kh / 32, batch), 256, 0, s>>>(
      d, g.Kp, B2, sB / 2, o.dig, g.b_elems, o.e, o.bad, o.energy, ctl.item_sq, ctl.sq_step);
  return check_launch("f64d_slice_col_kernel");
}

// scratch of the product: the low words between the sweeps, one block per SM, then a byte per
// tile (f64d_weak_kernel)
static size_t f8_low_words_bytes(int sms) { return (size_t)sms * F8_VALS * F8_EPI * sizeof(uint32_t); }
size_t f64d_scratch_bytes(int sms, int d, int batch) {
  return f8_low_words_bytes(sms) + (size_t)ceil_div(d, F8_BM) * ceil_div(d, F8_BN) * batch;
}

int f64d_gemm(int d, int batch, int opA, const double* A, long long sA, const void* abuf, const double* B,
              long long sB, const void* bbuf, double* C, long long sC, const AddTerms& add, void* scratch, int sms,
              bool entrywise, int* status, cudaStream_t s, const SplitCtl& ctl) {
  if (batch <= 0) return MG_OK;
  if (batch > 65535) return MG_EUNSUPPORTED;
  if (add.scale != 1.0) return MG_EINVAL;
  const F8Geom g = f8_geom(d);
  const F8Buf a = f8_buf(const_cast<void*>(abuf), g.a_elems, d, batch);
  const F8Buf b = f8_buf(const_cast<void*>(bbuf), g.b_elems, d, batch);
  CUtensorMap ma, mb;
  MG_TRY(make_digit_map(&ma, a.dig, g.Kp, d, d, F8_L, batch, F8_BK, F8_BM, 4));
  MG_TRY(make_bplane_map(&mb, b.dig, g.Kh, d, d, F8_L, batch, 2, 4, F8_BK));
  F8Args p{};
  p.A = A;
  p.B = B;
  p.sA = sA;
  p.sB = sB;
  p.opA = opA;
  p.d = d;
  p.Kp = g.Kp;
  p.batch = batch;
  p.ntn = ceil_div(d, F8_BN);
  p.ntm = ceil_div(d, F8_BM);
  p.ea = a.e;
  p.eb = b.e;
  p.bad_a = a.bad;
  p.bad_b = b.bad;
  p.en_a = a.energy;
  p.en_b = b.energy;
  p.C = C;
  p.sC = sC;
  p.add_n = add.n;
  for (int m = 0; m < 3; ++m) { p.add_src[m] = add.src[m]; p.add_coef[m] = add.coef[m]; }
  p.add_stride = add.stride;
  p.diag = add.diag;
  p.scratch = reinterpret_cast<uint32_t*>(scratch);
  p.status = status;
  p.item_sq = ctl.item_sq;
  p.sq_step = ctl.sq_step;
  p.stall = ctl.stall;
  p.wait_ns = std::min<unsigned long long>(ctl.wait_ns, 4000000000ull);
  if (entrywise) {
    unsigned char* weak = static_cast<unsigned char*>(scratch) + f8_low_words_bytes(sms);
    const float least = ldexpf(1.0f, 114 - 8) / sqrtf((float)d);
    f64d_weak_kernel<<<dim3(p.ntm * p.ntn, batch), F8_WEAK_THREADS, 0, s>>>(p, least, weak);
    MG_TRY(check_launch("f64d_weak_kernel"));
    p.weak = weak;
  }
  // one CTA per tile up to one per SM, and no fewer than marked items' 16 x 16 tiles would fill
  const long long tiles = (long long)p.ntn * p.ntm * batch, sub = ceil_div(d, 16);
  const int grid = (int)std::min<long long>(std::max(tiles, (sub * sub * batch + 1) / 2), sms);
  const size_t smem = (size_t)F8_SLOTS * F8_SLOT_BYTES + F8_STAGE_BYTES + 256 + 1024;
  MG_TRY(ensure_smem_limit(reinterpret_cast<const void*>(f64d_gemm_kernel<true>), (int)smem));
  MG_TRY(f8_check_registers(reinterpret_cast<const void*>(f64d_gemm_kernel<true>), f8_checked[0]));
  f64d_gemm_kernel<true><<<grid, F8_THREADS, smem, s>>>(ma, mb, p);
  MG_TRY(check_launch("f64d_gemm_kernel"));
  return MG_OK;
}

// ---------------------------------------------------------------------------
// exponentials of real symmetric exponents
// ---------------------------------------------------------------------------
static long long f64r_elems(int d) { return (long long)F8_L * d * ceil_div(d, F8_BK) * F8_BK; }
size_t f64r_bytes(int d, int batch) {
  return (((size_t)f64r_elems(d) * 2 + (size_t)d * 4 + 8) * batch + 255) / 256 * 256;
}

// U_b = e^{-i tau_b} (cos A_b - i sin A_b)^(2^s) with A_b = 2^{-s} W_b, W_b = Hbar_b - tau_b I
// real and symmetric (held as complex).  The degree-m Taylor polynomial of exp(-i A) splits
// exactly into C = sum (-1)^k Y^k / (2k)! and S = A sum (-1)^k Y^k / (2k+1)!, Y = A^2; powers up
// to Y^p with 2 p >= m / 2 leave one product to each series, and a squaring takes two,
// C' = (C + S)(C - S) and S' = 2 S C.  All are symmetric: d^2 (d + 1) flops a product against
// 8 d^3 of the complex form (degree 16: 7 + 2 s such products against 6 + s).  U(T) of 20
// intervals of the d = 729 chain (s = 3): 22.5 ms with complex products from digits, 9.7 ms so.
// mats: eight d x d real matrices per item (Y1..Y4, T1, T2, C, S), digs: four digit buffers of
// f64r_bytes.  sq_dev: per-item squaring counts (at most sq), else sq for every item.
int f64r_expm(int d, int batch, const double* W, const double* tau, int m, int sq, const int* sq_dev, double* const* mats,
              void* const* digs, double* U, void* scratch, int sms, int* status, cudaStream_t s, const SplitCtl& ctl0) {
  if (batch <= 0) return MG_OK;
  if (batch > 65535) return MG_EUNSUPPORTED;
  const int Kh = ceil_div(d, F8_BK) * F8_BK;
  const long long elems = f64r_elems(d), dd = (long long)d * d;
  SplitCtl ctl = ctl0;
  ctl.item_sq = nullptr;
  struct Dig {
    __nv_bfloat16* dig;
    int* e;
    uint32_t* energy;   // largest over the matrices that pass through the buffer
    CUtensorMap map;
  } D[4];
  for (int q = 0; q < 4; ++q) {
    D[q].dig = reinterpret_cast<__nv_bfloat16*>(digs[q]);
    D[q].e = reinterpret_cast<int*>(D[q].dig + elems * batch);
    D[q].energy = reinterpret_cast<uint32_t*>(D[q].e + (long long)d * batch);
    MG_CUDA_TRY(cudaMemsetAsync(D[q].energy, 0, 2 * sizeof(uint32_t) * (size_t)batch, s));
    MG_TRY(make_digit_map(&D[q].map, D[q].dig, Kh, d, d, F8_L, batch, F8_BK, F8_BM, 4));
  }
  auto slice = [&](int q, const double* X, const double* Z, double sz) {
    f64r_slice_kernel<false><<<dim3(ceil_div(d, 8), batch), 256, 0, s>>>(d, Kh, X, Z, sz, dd, 0, nullptr, D[q].dig, elems,
                                                                         D[q].e, D[q].energy, ctl.item_sq, ctl.sq_step);
    return check_launch("f64r_slice_kernel");
  };
  const int ntm = ceil_div(d, F8_BM);
  const size_t smem = (size_t)F8_SLOTS * F8_SLOT_BYTES + F8_STAGE_BYTES + 256 + 1024;
  MG_TRY(ensure_smem_limit(reinterpret_cast<const void*>(f64d_gemm_kernel<false>), (int)smem));
  MG_TRY(f8_check_registers(reinterpret_cast<const void*>(f64d_gemm_kernel<false>), f8_checked[1]));
  // dst = 2^scale2 D[x] D[y] + sum_m coef_m src_m + diag I
  auto mul = [&](int x, int y, double* dst, int n, const double* const* src, const double* coef, double diag,
                 int scale2) {
    F8Args p{};
    p.d = d;
    p.Kp = Kh;
    p.batch = batch;
    p.ntn = p.ntm = ntm;
    p.ea = D[x].e;
    p.eb = D[y].e;
    p.en_a = D[x].energy;
    p.en_b = D[y].energy;
    p.C = dst;
    p.sC = dd;
    p.add_n = n;
    for (int q = 0; q < n; ++q) { p.add_src[q] = src[q]; p.add_coef[q] = coef[q]; }
    p.add_stride = dd;
    p.diag = diag;
    p.scale2 = scale2;
    p.scratch = reinterpret_cast<uint32_t*>(scratch);
    p.status = status;
    p.item_sq = ctl.item_sq;
    p.sq_step = ctl.sq_step;
    p.stall = ctl.stall;
    p.wait_ns = std::min<unsigned long long>(ctl.wait_ns, 4000000000ull);
    const long long tiles = (long long)ntm * (ntm + 1) / 2 * batch;
    f64d_gemm_kernel<false><<<(int)std::min<long long>(tiles, sms), F8_THREADS, smem, s>>>(D[x].map, D[y].map, p);
    return check_launch("f64d_gemm_kernel (real)");
  };
  double f[18], cc[9], ss[9];
  f[0] = 1.0;
  for (int j = 1; j < 18; ++j) f[j] = f[j - 1] / j;
  const int kc = m / 2, ks = (m - 1) / 2, p = (kc + 1) / 2;
  for (int k = 0; k < 9; ++k) {
    cc[k] = k <= kc ? ((k & 1) ? -f[2 * k] : f[2 * k]) : 0.0;
    ss[k] = k <= ks ? ((k & 1) ? -f[2 * k + 1] : f[2 * k + 1]) : 0.0;
  }
  double* const* Y = mats;   // Y[q - 1] = Y^q
  double *T1 = mats[4], *T2 = mats[5], *C = mats[6], *S = mats[7];
  const bool hc = kc > p, hs = ks > p;
  // D0: A; D1: Y, then the high part's digits; D2: Y^2, then Y^p; D3: sine's sum
  f64r_slice_kernel<true><<<dim3(ceil_div(d, 8), batch), 256, 0, s>>>(d, Kh, W, nullptr, 0.0, 2 * dd, sq, sq_dev, D[0].dig,
                                                                      elems, D[0].e, D[0].energy, nullptr, 0);
  MG_TRY(check_launch("f64r_slice_kernel"));
  MG_TRY(mul(0, 0, Y[0], 0, nullptr, nullptr, 0.0, 0));
  int dp = 1;   // digits of Y^p
  if (p >= 2 || hc || hs) MG_TRY(slice(1, Y[0], nullptr, 0.0));
  if (p >= 2) {
    MG_TRY(mul(1, 1, Y[1], 0, nullptr, nullptr, 0.0, 0));
    MG_TRY(slice(2, Y[1], nullptr, 0.0));
    dp = 2;
  }
  if (p >= 3) MG_TRY(mul(2, 1, Y[2], 0, nullptr, nullptr, 0.0, 0));
  if (p >= 4) MG_TRY(mul(2, 2, Y[3], 0, nullptr, nullptr, 0.0, 0));
  if (p >= 3) MG_TRY(slice(2, Y[p - 1], nullptr, 0.0));
  RealComb a{};
  a.n = p;
  for (int q = 0; q < p; ++q) {
    a.src[q] = Y[q];
    a.coef[0][q] = hc ? (p + 1 + q <= kc ? cc[p + 1 + q] : 0.0) : cc[1 + q];
    a.coef[1][q] = hs ? (p + 1 + q <= ks ? ss[p + 1 + q] : 0.0) : ss[1 + q];
  }
  a.diag[0] = hc ? cc[p] : cc[0];
  a.diag[1] = hs ? ss[p] : ss[0];
  a.dst[0] = hc ? T1 : C;
  a.dst[1] = T2;   // sine's high part, or its whole sum
  const long long total = dd * batch;
  f64r_lincomb_kernel<<<(int)std::min<long long>((total + 255) / 256, (long long)sms * 16), 256, 0, s>>>(d, total, a);
  MG_TRY(check_launch("f64r_lincomb_kernel"));
  const double* low[3] = {Y[0], Y[1], Y[2]};
  const int hd = dp == 1 ? 3 : 1;   // where the high part's digits go
  if (hc) {
    MG_TRY(slice(hd, T1, nullptr, 0.0));
    MG_TRY(mul(hd, dp, C, p - 1, low, cc + 1, cc[0], 0));
  }
  double* sine = T2;
  if (hs) {
    MG_TRY(slice(hd, T2, nullptr, 0.0));
    MG_TRY(mul(hd, dp, S, p - 1, low, ss + 1, ss[0], 0));
    sine = S;
  }
  MG_TRY(slice(3, sine, nullptr, 0.0));
  MG_TRY(mul(0, 3, S, 0, nullptr, nullptr, 0.0, 0));   // sin = A (sum)
  for (int k = 0; k < sq; ++k) {
    ctl.item_sq = sq_dev;   // items whose count is reached keep their matrices
    ctl.sq_step = k;
    MG_TRY(slice(0, C, S, 1.0));
    MG_TRY(slice(1, C, S, -1.0));
    MG_TRY(slice(2, S, nullptr, 0.0));
    MG_TRY(slice(3, C, nullptr, 0.0));
    MG_TRY(mul(0, 1, C, 0, nullptr, nullptr, 0.0, 0));
    MG_TRY(mul(2, 3, S, 0, nullptr, nullptr, 0.0, 1));
  }
  f64r_phase_kernel<<<dim3((unsigned)std::min<long long>((dd + 1023) / 1024, 64), batch), 256, 0, s>>>(
      dd, tau, C, S, reinterpret_cast<double2*>(U));
  return check_launch("f64r_phase_kernel");
}

}  // namespace mg
