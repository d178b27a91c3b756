// FP64 complex matrix products on the tcgen05 tensor cores, to FP64 accuracy.
//
//   C[b] = opA(A[b]) B[b] + sum_m coef_m P_m[b] + diag I        (FP64 in, FP64 out)
//
// GB300's FP64 pipe gives 1.1 TFLOP/s, its BF16 tensor cores 1900.  A product of the
// exponential or of the propagators (MG_PREC_FP64) is therefore formed from integer digits
// whose products the tensor cores accumulate exactly (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump, Numerical Algorithms 59, 2012):
//   * Every row of A (column of B) is scaled by the power of two 2^E that bounds it and
//     rounded to 56-bit fixed point: an entry a becomes F = rint(a 2^{55 - E}), |F| < 2^55,
//     and F = sum_{s<8} q_s 2^{7 (7 - s)} with balanced base-128 digits |q_s| <= 64, each
//     exact in BF16 (stored as q_s 2^{-7 s}).  Entries of the row's own binade keep all 53
//     bits of their mantissa.
//   * Digit products q_s q_t with s + t <= 8 (43 of 64; the rest lie 2^-7 below the rounding
//     of F) are summed by level l = s + t in FP32 TMEM accumulators.  A product is at most
//     2^12, so (l + 1) K products stay below 2^24, an exact integer, while
//     (l + 1) K <= 4096: the accumulators are drained into 64-bit integer registers every
//     KSEG positions of K (1024 for levels 0..3, 576 for levels 4..7).  Level 8 shares level
//     7's accumulator; their sum, 2^-49 below the leading digit product, is the only one
//     that FP32 rounds (to 2^-7 of level 7's unit while it is below 2^17).
//   * The two 64-bit sums (levels 0..3 and 4..8) are joined by one FP64 FMA, the product's
//     only rounding beside that of F.
// The error is about 2^-57 sqrt(K) of (largest entry of the row of A) x (rms entry of the
// column of B) and the same with A and B exchanged: for the exponential's matrices no
// larger than that of FP64 arithmetic, whose K roundings accumulate.  (Without level 8 the
// dropped digit products weigh 2^-56 sqrt(K) of the largest entries on both sides, which
// near-diagonal matrices show: 1.6e-14 of a row's norm at d = 729 against FP64's 2e-15.)  Operands that the scheme does not cover -- a NaN, an
// infinity, a row or column whose largest entry lies outside 2^-400 .. 2^400 -- are marked
// by the slicers; such an item is left to the FP64-pipe product, which is launched behind
// and returns at once for all others.
//
// Structure of the product kernel (persistent, one CTA of 320 threads per SM, 128 x 64
// complex output tiles; every tile makes two sweeps over K, levels 4..7 first):
//   warp 0      TMA producer: 32 KiB slots (4 digits of the A or B tile, K = 32, SWIZZLE_64B)
//               in a ring of six.  Levels 0..3 need the digits 0..3 of A and B (two slots per
//               K step), levels 4..7 all eight (four slots).
//   warp 1      MMA issuer: M = 128, N = 128 (64 real, 64 imaginary columns), K = 16; four
//               levels fill the 512 TMEM columns.  In the sweep of levels 4..8 the order
//               (A 0..3, B 0..3), (A 0..3, B 4..7), (A 4..7, B 4..7), (A 4..7, B 0..3) frees
//               two slots while 13 digit pairs are still to be multiplied, so a ring of 1.5 K
//               steps keeps loads in flight.
//   warps 2..9  drains: tcgen05.ld, float -> int, 64-bit accumulation in registers (64 sums
//               per thread).  The sums of levels 4..7 wait in a per-CTA scratch (L2) while
//               levels 0..3 are swept.  Conversion to FP64, scaling, addends and stores run
//               while the next tile's MMAs are issued: the FP64 pipe (4 operations per output)
//               is idle otherwise.
// Measured (GB300, one product of a batch, slicing included): d = 729 2804 us on the FP64
// pipe -> 110 us (28 TFLOP/s of the product's 8 d^3); d = 256 112 -> 8.3 us; d = 81 8.9 ->
// 1.5 us.  At d = 729 the slicers take 12% (HBM-bound), the tensor pipe is active 67% of
// the product's cycles: the rest goes to the drains (five per tile, ~4000 cycles of
// float-to-int conversions each) and to operand delivery (single CTAs load 43 bytes per
// cycle and SM).
// Every wait is bounded (SplitCtl::wait_ns, at most 4 s): a wait that gives up records
// MG_DEV_TIMEOUT, the CTA's unfinished tiles become NaN, and it leaves once its own copies
// and MMAs have completed.
#include "common.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace mg {

constexpr int F8_L = 8;                 // digits
constexpr int F8_BM = 128;              // output rows per tile
constexpr int F8_BN = 64;               // complex output columns per tile
constexpr int F8_BK = 32;               // K per slot
constexpr int F8_SLOTS = 6;
constexpr int F8_SLOT_BYTES = 4 * F8_BM * F8_BK * 2;
constexpr int F8_THREADS = 320;
constexpr int F8_EPI_WARPS = 8;
constexpr int F8_SEG_LO = 18;           // K steps per drain of levels 4..7 (576 positions of K)
constexpr int F8_SEG_HI = 32;           // and of levels 0..3 (1024)
constexpr int F8_VALS = 64;             // sums per epilogue thread
constexpr int F8_STAGE_BYTES = F8_EPI_WARPS * 32 * 8 * 16;   // epilogue staging: 32 rows x 8 columns per warp
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

// operand buffer: digits of all items, then row (column) exponents, then the items' marks
size_t f64d_a_bytes(int d, int batch) {
  return ((size_t)f8_geom(d).a_elems * 2 + (size_t)d * 4 + 4) * batch;
}
size_t f64d_b_bytes(int d, int batch) {
  return ((size_t)f8_geom(d).b_elems * 2 + (size_t)d * 4 + 4) * batch;
}

// ---------------------------------------------------------------------------
// slicers
// ---------------------------------------------------------------------------
// E with |a| < 2^E; zero and subnormals -> -2^29; NaN and infinities -> 1025
__device__ __forceinline__ int f8_exp(double a) {
  const int bexp = (__double2hiint(a) >> 20) & 0x7FF;
  return bexp == 0 ? -(1 << 29) : bexp - 1022;
}
__device__ __forceinline__ bool f8_marked(int E) { return E > F8_EXP_MAX || (E < -F8_EXP_MAX && E > -(1 << 28)); }

constexpr unsigned long long F8_BIAS = 0x0102040810204081ull * 64;   // 64 in every base-128 position 0..8
// F + bias for F = rint(a 2^{55 - E}): digit s is ((F + bias) >> 7 (7 - s)) mod 128 - 64, the
// top one without the mod.  The fixed-point value is formed on the integer pipe.
__device__ __forceinline__ unsigned long long f8_fixed(double a, int E) {
  const long long bits = __double_as_longlong(a);
  const int bexp = (int)((bits >> 52) & 0x7FF);
  const int sh = bexp - 1075 + 55 - E;                       // <= 2
  unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  if (sh >= 0) m <<= min(sh, 2);
  else if (sh > -56) m = (m + (1ull << (-sh - 1))) >> -sh;
  else m = 0;
  if (bexp == 0) m = 0;                                      // zero (a subnormal is below any kept bit)
  const unsigned long long f = bits < 0 ? 0ull - m : m;
  return f + (F8_BIAS & 0x00FFFFFFFFFFFFFFull);
}
// q_s 2^{-7 s} of a biased value as FP32 (exact): the field in the low mantissa bits of
// 2^{23 - 7 s}, less (2^23 + 64) 2^{-7 s}
__device__ __forceinline__ float f8_digit(unsigned long long f, int s) {
  uint32_t q = (uint32_t)(f >> (7 * (7 - s)));
  q = s == 0 ? (q & 0xFFu) : (q & 0x7Fu);
  const uint32_t magic = 0x4B000000u - ((uint32_t)(7 * s) << 23);
  return __uint_as_float(magic | q) - __uint_as_float(magic | 64u);
}
// BF16 pair (lo in the low half); the digits are exact in the high 16 bits of their FP32 form
__device__ __forceinline__ uint32_t f8_pack(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// A digits, one warp per row: row exponent, then 4 consecutive elements per lane and step.
// grid (ceil(d / 8), batch), block 256.  Bound by the digit stores (32 bytes per complex
// entry written, 16 read).
__global__ void __launch_bounds__(256)
f64d_slice_a_kernel(int d, int Kp, const double2* __restrict__ A, long long sA2, __nv_bfloat16* __restrict__ out,
                    long long item_elems, int* __restrict__ ea, int* __restrict__ bad,
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
    ea[(long long)b * d + row] = E;
    if (mark) atomicOr(bad + b, 1);
  }
  __nv_bfloat16* o = out + b * item_elems + (long long)row * Kp;
  const long long ds = (long long)d * Kp;
  for (int k = 4 * lane; k < Kh; k += 128) {
    unsigned long long re[4], im[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 v = k + q < d ? a[k + q] : make_double2(0.0, 0.0);
      re[q] = f8_fixed(v.x, E);
      im[q] = f8_fixed(v.y, E);
    }
#pragma unroll
    for (int s = 0; s < F8_L; ++s) {
      *reinterpret_cast<uint2*>(o + s * ds + k) =
          make_uint2(f8_pack(f8_digit(re[0], s), f8_digit(re[1], s)), f8_pack(f8_digit(re[2], s), f8_digit(re[3], s)));
      *reinterpret_cast<uint2*>(o + s * ds + Kh + k) =
          make_uint2(f8_pack(f8_digit(im[0], s), f8_digit(im[1], s)), f8_pack(f8_digit(im[2], s), f8_digit(im[3], s)));
    }
  }
}

// Column exponents (preset to byte 0x80): grid (ceil(d/64), ceil(d/64), batch), block 256.
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
  if (g == 0 && j0 + c < d)
    atomicMax(eb + (long long)b * d + j0 + c, max(max(red[0][c], red[1][c]), max(red[2][c], red[3][c])));
}

// Column digits of a 32 (k) x 64 (j) block, staged in shared memory.  ADJ = false: B planes
// (-Im, Re, Im; row j of a plane is column j along k).  ADJ = true: the same columns written
// as A rows of the adjoint, [Re | -Im].  grid (ceil(d/64), Kh/32, batch), block 256.
template <bool ADJ>
__global__ void __launch_bounds__(256)
f64d_slice_col_kernel(int d, int Kp, const double2* __restrict__ B, long long sB2, __nv_bfloat16* __restrict__ out,
                      long long item_elems, int* __restrict__ eb, int* __restrict__ bad,
                      const int* __restrict__ item_sq, int sq_step) {
  __shared__ double2 tile[32][65];
  __shared__ int ex[64];
  const int b = blockIdx.z;
  if (item_sq && item_sq[b] <= sq_step) return;
  const int j0 = blockIdx.x * 64, k0 = blockIdx.y * 32, tid = threadIdx.x, Kh = Kp / 2;
  const double2* Bb = B + b * sB2;
  if (tid < 64) {
    int E = j0 + tid < d ? eb[(long long)b * d + j0 + tid] : 0;
    if (f8_marked(E)) atomicOr(bad + b, 1);
    ex[tid] = E < -(1 << 28) ? 0 : E;   // all-zero column
  }
  for (int e = tid; e < 32 * 64; e += 256) {
    const int kk = e >> 6, c = e & 63;
    tile[kk][c] = (k0 + kk < d && j0 + c < d) ? Bb[(long long)(k0 + kk) * d + j0 + c] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int e = tid; e < 8 * 64; e += 256) {
    const int g = e & 7, r = e >> 3, j = j0 + r, k = k0 + 4 * g;
    if (j >= d) continue;
    const int E = ex[r];
    unsigned long long re[4], im[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 v = tile[4 * g + q][r];
      re[q] = f8_fixed(v.x, E);
      im[q] = f8_fixed(ADJ ? -v.y : v.y, E);
    }
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
  // the exponents of all-zero columns stay preset; the product reads them as 0
}

// ---------------------------------------------------------------------------
// product
// ---------------------------------------------------------------------------
struct F8Args {
  int d, Kp, batch, ntn, ntm;
  const int* ea;
  const int* eb;
  const int* bad_a;
  const int* bad_b;
  double* C;
  long long sC;               // doubles
  const double* add_src[3];
  double add_coef[3];
  long long add_stride;       // doubles
  int add_n;
  double diag;
  long long* scratch;         // per CTA: F8_VALS x 256 sums of levels 4..7
  int* status;
  const int* item_sq;
  int sq_step;
  unsigned long long wait_ns;
  int stall;                  // test only: the MMA issuer waits on a barrier nothing completes
};

__device__ __forceinline__ bool f8_skip(const F8Args& p, int b) {
  return (p.bad_a[b] | p.bad_b[b]) != 0 || (p.item_sq && p.item_sq[b] <= p.sq_step);
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

// 64-bit integer |x| < 2^51 as FP64 (exact): the bits of 1.5 2^52 + x
__device__ __forceinline__ double f8_to_double(long long x) {
  return __longlong_as_double(x + 0x4338000000000000ll) - 6755399441055744.0;
}

// Drain of one accumulator set (levels l0 .. l0 + 3) into the thread's sums, in units of
// 2^{-7 (l0 + 3)}.  With KSEG as above |G_l| 128 + |G_{l+1}| fits 32 bits for the integers
// G_l = 2^{7 l} g_l.
__device__ __forceinline__ void f8_drain(uint32_t tbase, int l0, long long (&acc)[F8_VALS]) {
  const float m0 = l0 ? 268435456.0f : 1.0f;   // 2^{7 l0}
  const float m1 = m0 * 128.0f, m2 = m0 * 16384.0f, m3 = m0 * 2097152.0f;
#pragma unroll
  for (int c = 0; c < F8_VALS; c += 8) {
    // values 0..31: real parts of the thread's 32 columns, 32..63: imaginary parts
    const uint32_t col = tbase + (c < 32 ? c : F8_BN + c - 32);
    uint32_t g[4][8];
#pragma unroll
    for (int l = 0; l < 4; ++l) tmem_ld8(col + l * 128, g[l]);
    tmem_wait_ld();
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int i01 = __float2int_rn(__uint_as_float(g[0][v]) * m0) * 128 +
                      __float2int_rn(__uint_as_float(g[1][v]) * m1);
      const int i23 = __float2int_rn(__uint_as_float(g[2][v]) * m2) * 128 +
                      __float2int_rn(__uint_as_float(g[3][v]) * m3);
      acc[c + v] += (long long)i01 * 16384 + i23;
    }
  }
}

constexpr uint32_t kF8Idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

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
  const int per_item = p.ntn * p.ntm;
  const long long tiles = (long long)per_item * p.batch;
  const int nseg[2] = {(steps + F8_SEG_LO - 1) / F8_SEG_LO, (steps + F8_SEG_HI - 1) / F8_SEG_HI};   // levels 4..7, 0..3

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      long long n = 0;   // slots filled
      bool ok = true;
      for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
        const int b = (int)(t / per_item), rem = (int)(t % per_item), mt = rem / p.ntn, nt = rem % p.ntn;
        if (f8_skip(p, b)) continue;
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
        if (f8_skip(p, (int)(t / per_item))) continue;
        for (int sweep = 0; sweep < 2 && ok; ++sweep) {
          const int ns = nseg[sweep];
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
                      int l = s0 + s + t0 + u;
                      if (l < lmin || l > lmax) continue;
                      l = min(l, lmin + 3);   // level 8 with level 7
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
                group(sa[0], sa[1], 0, 0, 4, 8, first);
                if (!ready(2)) { ok = false; break; }
                tc_fence_after();
                group(sa[0], sa[2], 0, 4, 4, 8, first);
                tc_commit(&empty[n % F8_SLOTS]);
                if (!ready(3)) { ok = false; break; }
                tc_fence_after();
                group(sa[3], sa[2], 4, 4, 4, 8, first);
                tc_commit(&empty[(n + 2) % F8_SLOTS]);
                group(sa[3], sa[1], 4, 0, 4, 8, first);
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
  } else {
    // ---------------- epilogue (warps 2..9) ----------------
    const int q = warp & 3;                    // TMEM lane quarter of this warp
    const int c0 = ((warp - 2) >> 2) * 32;     // first of its 32 complex columns
    const int et = threadIdx.x - 64;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + c0;
    long long* scratch = p.scratch + (long long)blockIdx.x * F8_VALS * 256 + et;
    double2* stg = staging + (warp - 2) * 256;
    uint32_t set = 0;
    bool ok = true;
    long long t = blockIdx.x;
    for (; t < tiles; t += gridDim.x) {
      const int b = (int)(t / per_item), rem = (int)(t % per_item), mt = rem / p.ntn, nt = rem % p.ntn;
      if (f8_skip(p, b)) continue;
      const int row0 = mt * F8_BM + q * 32, col0 = nt * F8_BN + c0;
      const bool live = row0 < p.d && col0 < p.d;   // uniform over the warp
      long long acc[F8_VALS];
      for (int sweep = 0; sweep < 2 && ok; ++sweep) {
#pragma unroll
        for (int v = 0; v < F8_VALS; ++v) acc[v] = 0;
        for (int sg = 0; sg < nseg[sweep]; ++sg) {
          bool got = true;
          if (lane == 0) got = f8_wait(accfull, set & 1, p.wait_ns, abort_flag);
          got = __shfl_sync(0xffffffffu, (int)got, 0) != 0;
          if (!got) { ok = false; break; }
          tc_fence_after();
          if (live) f8_drain(tbase, sweep == 0 ? 4 : 0, acc);
          tc_fence_before();
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(accempty)) : "memory");
          ++set;
        }
        if (sweep == 0 && ok && live) {
#pragma unroll
          for (int v = 0; v < F8_VALS; ++v) scratch[v * 256] = acc[v];
        }
      }
      if (!ok) break;
      if (!live) continue;
      const int row = row0 + lane;
      const int Ea = row < p.d ? p.ea[(long long)b * p.d + row] : 0;
      int Eb = col0 + lane < p.d ? p.eb[(long long)b * p.d + col0 + lane] : 0;
      if (Eb < -(1 << 28)) Eb = 0;   // all-zero column
      const double2* addp[3];
#pragma unroll
      for (int m = 0; m < 3; ++m)
        addp[m] = reinterpret_cast<const double2*>(m < p.add_n ? p.add_src[m] + b * p.add_stride : nullptr);
      double2* Cb = reinterpret_cast<double2*>(p.C + b * p.sC);
#pragma unroll
      for (int c = 0; c < 32; c += 8) {   // 8 columns at a time through the warp's staging
        if (col0 + c < p.d) {
          long long lre[8], lim[8];
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            lre[v] = scratch[(c + v) * 256];
            lim[v] = scratch[(32 + c + v) * 256];
          }
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            // the value is T 2^{Ea + Eb - 61}, T = hi 2^28 + lo in units of 2^-49
            const int k = Ea + __shfl_sync(0xffffffffu, Eb, c + v) - 61;
            const double sc = __hiloint2double((k + 1023) << 20, 0);
            const double re = fma(f8_to_double(acc[c + v]), 268435456.0, f8_to_double(lre[v])) * sc;
            const double im = fma(f8_to_double(acc[32 + c + v]), 268435456.0, f8_to_double(lim[v])) * sc;
            stg[lane * 8 + (v ^ (lane & 7))] = make_double2(re, im);
          }
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = i * 4 + (lane >> 3), cc = lane & 7;
            const int grow = row0 + r, gcol = col0 + c + cc;
            if (grow < p.d && gcol < p.d) {
              double2 v = stg[r * 8 + (cc ^ (r & 7))];
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
    if (!ok) {
      if (lane == 0) {
        if (!*abort_flag) atomicExch(p.status, MG_DEV_TIMEOUT);
        *abort_flag = 1;
      }
      // the tiles this CTA leaves unfinished are not left looking like a result
      const double nan = __longlong_as_double(0x7FF8000000000000ll);
      for (; t < tiles; t += gridDim.x) {
        const int b = (int)(t / per_item), rem = (int)(t % per_item), mt = rem / p.ntn, nt = rem % p.ntn;
        const int row = mt * F8_BM + q * 32 + lane;
        if (f8_skip(p, b) || row >= p.d) continue;
        for (int c = nt * F8_BN + c0; c < min(p.d, nt * F8_BN + c0 + 32); ++c)
          reinterpret_cast<double2*>(p.C + b * p.sC)[(long long)row * p.d + c] = make_double2(nan, nan);
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
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct F8Buf {
  __nv_bfloat16* dig;
  int* e;
  int* bad;
};
static F8Buf f8_buf(void* buf, long long elems, int d, int batch) {
  F8Buf r;
  r.dig = reinterpret_cast<__nv_bfloat16*>(buf);
  r.e = reinterpret_cast<int*>(r.dig + elems * batch);
  r.bad = r.e + (long long)d * batch;
  return r;
}

int f64d_slice_a(int d, int batch, const double* A, long long sA, int opA, void* buf, cudaStream_t s,
                 const SplitCtl& ctl) {
  if (batch > 65535) return MG_EUNSUPPORTED;
  const F8Geom g = f8_geom(d);
  const F8Buf o = f8_buf(buf, g.a_elems, d, batch);
  const double2* A2 = reinterpret_cast<const double2*>(A);
  if (opA == 0) {
    MG_CUDA_TRY(cudaMemsetAsync(o.bad, 0, sizeof(int) * (size_t)batch, s));
    f64d_slice_a_kernel<<<dim3(ceil_div(d, 8), batch), 256, 0, s>>>(d, g.Kp, A2, sA / 2, o.dig, g.a_elems, o.e, o.bad,
                                                                    ctl.item_sq, ctl.sq_step);
    return check_launch("f64d_slice_a_kernel");
  }
  MG_CUDA_TRY(cudaMemsetAsync(o.e, 0x80, sizeof(int) * (size_t)d * batch, s));
  MG_CUDA_TRY(cudaMemsetAsync(o.bad, 0, sizeof(int) * (size_t)batch, s));
  f64d_col_exponent_kernel<<<dim3(ceil_div(d, 64), ceil_div(d, 64), batch), 256, 0, s>>>(d, A2, sA / 2, o.e,
                                                                                          ctl.item_sq, ctl.sq_step);
  MG_TRY(check_launch("f64d_col_exponent_kernel"));
  f64d_slice_col_kernel<true><<<dim3(ceil_div(d, 64), g.Kh / 32, batch), 256, 0, s>>>(
      d, g.Kp, A2, sA / 2, o.dig, g.a_elems, o.e, o.bad, ctl.item_sq, ctl.sq_step);
  return check_launch("f64d_slice_col_kernel");
}

int f64d_slice_b(int d, int batch, const double* B, long long sB, void* buf, cudaStream_t s, const SplitCtl& ctl) {
  if (batch > 65535) return MG_EUNSUPPORTED;
  const F8Geom g = f8_geom(d);
  const F8Buf o = f8_buf(buf, g.b_elems, d, batch);
  const double2* B2 = reinterpret_cast<const double2*>(B);
  MG_CUDA_TRY(cudaMemsetAsync(o.e, 0x80, sizeof(int) * (size_t)d * batch, s));
  MG_CUDA_TRY(cudaMemsetAsync(o.bad, 0, sizeof(int) * (size_t)batch, s));
  f64d_col_exponent_kernel<<<dim3(ceil_div(d, 64), ceil_div(d, 64), batch), 256, 0, s>>>(d, B2, sB / 2, o.e,
                                                                                          ctl.item_sq, ctl.sq_step);
  MG_TRY(check_launch("f64d_col_exponent_kernel"));
  f64d_slice_col_kernel<false><<<dim3(ceil_div(d, 64), g.Kh / 32, batch), 256, 0, s>>>(
      d, g.Kp, B2, sB / 2, o.dig, g.b_elems, o.e, o.bad, ctl.item_sq, ctl.sq_step);
  return check_launch("f64d_slice_col_kernel");
}

// scratch of the product (sums of levels 4..7 between the sweeps): one block per SM
size_t f64d_scratch_bytes(int sms) { return (size_t)sms * F8_VALS * 256 * sizeof(long long); }

int f64d_gemm(int d, int batch, int opA, const double* A, long long sA, const void* abuf, const double* B,
              long long sB, const void* bbuf, double* C, long long sC, const AddTerms& add, void* scratch, int sms,
              int* status, cudaStream_t s, const SplitCtl& ctl) {
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
  p.d = d;
  p.Kp = g.Kp;
  p.batch = batch;
  p.ntn = ceil_div(d, F8_BN);
  p.ntm = ceil_div(d, F8_BM);
  p.ea = a.e;
  p.eb = b.e;
  p.bad_a = a.bad;
  p.bad_b = b.bad;
  p.C = C;
  p.sC = sC;
  p.add_n = add.n;
  for (int m = 0; m < 3; ++m) { p.add_src[m] = add.src[m]; p.add_coef[m] = add.coef[m]; }
  p.add_stride = add.stride;
  p.diag = add.diag;
  p.scratch = reinterpret_cast<long long*>(scratch);
  p.status = status;
  p.item_sq = ctl.item_sq;
  p.sq_step = ctl.sq_step;
  p.stall = ctl.stall;
  p.wait_ns = std::min<unsigned long long>(ctl.wait_ns, 4000000000ull);
  const long long tiles = (long long)p.ntn * p.ntm * batch;
  const int grid = (int)std::min<long long>(tiles, sms);
  const size_t smem = (size_t)F8_SLOTS * F8_SLOT_BYTES + F8_STAGE_BYTES + 256 + 1024;
  MG_TRY(ensure_smem_limit(reinterpret_cast<const void*>(f64d_gemm_kernel), (int)smem));
  f64d_gemm_kernel<<<grid, F8_THREADS, smem, s>>>(ma, mb, p);
  MG_TRY(check_launch("f64d_gemm_kernel"));
  // items the slicers marked (usually none: the launch returns at once)
  AddTerms rest = add;
  rest.item_sq = ctl.item_sq;
  rest.sq_step = ctl.sq_step;
  return launch_cgemm_f64_marked(batch, d, A, sA, opA, B, sB, C, sC, rest, a.bad, b.bad, sms, s);
}

}  // namespace mg
