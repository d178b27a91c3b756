// Sequential state propagation psi_{n+1} = U_n psi_n (the state form of the
// product U_{N-1} ... U_0 psi0), with the optional FP64 renormalisation
// psi <- psi / |psi| every R intervals.
//
// d <= 256: a cluster of C CTAs (one CTA for d <= 32) carries the state through all
// intervals of a chunk and shares its rows; every CTA holds all of psi in shared memory, and
// a finished row is written into every CTA's copy (chain_cluster_kernel).  Where more states
// run at once than their clusters fit, one CTA per state, a warp per row.
// Large d: one multi-CTA matrix-vector launch per interval (HBM-bound).
#include "common.cuh"

#include <mutex>

namespace mg {

constexpr int CHAIN_THREADS = 1024;

// One CTA carries psi (d complex, global) through n_steps propagators.
// traj (may be null): psi after every step is also written to traj + (step_offset + n + 1) d.
__device__ void chain_body(int n_steps, int d, const double* __restrict__ U, long long sU,
                           double* __restrict__ psi, int reorth_every, int step_offset, double2* sh,
                           double* red, double* __restrict__ traj) {
  double2* cur = sh;
  double2* nxt = sh + d;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i = threadIdx.x; i < d; i += blockDim.x) cur[i] = reinterpret_cast<double2*>(psi)[i];
  __syncthreads();
  for (int n = 0; n < n_steps; ++n) {
    const double2* Un = reinterpret_cast<const double2*>(U + n * sU);
    for (int i = warp; i < d; i += nw) {
      const double2* row = Un + (long long)i * d;
      double re = 0.0, im = 0.0;
      for (int j = lane; j < d; j += 32) {
        double2 u = row[j], v = cur[j];
        re = fma(u.x, v.x, re);
        re = fma(-u.y, v.y, re);
        im = fma(u.x, v.y, im);
        im = fma(u.y, v.x, im);
      }
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) nxt[i] = make_double2(re, im);
    }
    __syncthreads();
    double2* t = cur; cur = nxt; nxt = t;
    const int done = step_offset + n + 1;
    if (reorth_every > 0 && done % reorth_every == 0) {
      double s = 0.0;
      for (int i = threadIdx.x; i < d; i += blockDim.x) s += cur[i].x * cur[i].x + cur[i].y * cur[i].y;
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) red[warp] = s;
      __syncthreads();
      if (warp == 0) {
        double v = lane < nw ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[0] = v;
      }
      __syncthreads();
      const double inv = 1.0 / sqrt(red[0]);
      for (int i = threadIdx.x; i < d; i += blockDim.x) { cur[i].x *= inv; cur[i].y *= inv; }
      __syncthreads();
    }
    if (traj) {
      double2* t_out = reinterpret_cast<double2*>(traj) + (long long)done * d;
      for (int i = threadIdx.x; i < d; i += blockDim.x) t_out[i] = cur[i];
    }
  }
  for (int i = threadIdx.x; i < d; i += blockDim.x) reinterpret_cast<double2*>(psi)[i] = cur[i];
}

__global__ void __launch_bounds__(CHAIN_THREADS)
state_chain_kernel(int n_steps, int d, const double* __restrict__ U, long long sU,
                   double* __restrict__ psi, int reorth_every, int step_offset, double* __restrict__ traj) {
  extern __shared__ double2 sh[];
  __shared__ double red[CHAIN_THREADS / 32];
  chain_body(n_steps, d, U, sU, psi, reorth_every, step_offset, sh, red, traj);
}

// Many jobs at once: CTA b carries job segs[b].job through its segment of the chunk.
__global__ void __launch_bounds__(CHAIN_THREADS)
multi_chain_kernel(int d, const ChainSeg* __restrict__ segs, const double* __restrict__ U, long long sU,
                   double* const* __restrict__ psi, int reorth_every) {
  extern __shared__ double2 sh[];
  __shared__ double red[CHAIN_THREADS / 32];
  const ChainSeg g = segs[blockIdx.x];
  chain_body(g.count, d, U + g.first * sU, sU, psi[g.job], reorth_every, g.done_before, sh, red, nullptr);
}

// The chain of one job on a cluster (C = 1: one CTA): CTA r of C holds rows [r d / C,
// (r + 1) d / C), T lanes per row, and a copy of psi.  A row is read from U_n into registers
// AHEAD intervals early (the loads do not depend on psi), multiplied, summed over its T lanes
// and stored into all C copies through distributed shared memory; one barrier per interval.
// Bound by the FP64 pipe of the SMs, where a warp's instruction takes about 64 cycles of its
// quarter: 4 d / T FMAs and 2 log2 T additions per lane.  On one CTA (d <= 32) a warp per row
// spent as much on the sums as on the products, 6.2 us per interval at d = 30; T = 4 takes
// 1.7.  On clusters T = 32 is as fast as T = 8 (its loads coalesce better).  At d <= 8 the
// loads' latency is what an interval takes (0.85 us at d = 2 with one interval ahead), hence
// AHEAD.  C: rows per CTA down to 8-16, where the barrier (~0.7 us) weighs as much as the rows
// (one CTA took 88 us per interval at d = 256, of which 16 leave 5).
template <int T, int Q, int AHEAD>
__global__ void __launch_bounds__(T == 32 ? 512 : 128)
chain_cluster_kernel(int d, int n_steps, const ChainSeg* __restrict__ segs, const double* __restrict__ U, long long sU,
                     double* psi_one, double* const* __restrict__ psi_many, int reorth_every, int step_offset,
                     double* __restrict__ traj) {
  __shared__ double2 buf[2][T * Q];
  __shared__ double red[16];
  uint32_t rank, C;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
  double* psi = psi_one;
  if (segs) {
    const ChainSeg g = segs[blockIdx.x / C];
    n_steps = g.count;
    U += g.first * sU;
    psi = psi_many[g.job];
    step_offset = g.done_before;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int sub = threadIdx.x % T, nrow = blockDim.x / T;
  const int r0 = (int)((long long)d * rank / C), r1 = (int)((long long)d * (rank + 1) / C);
  const int first = r0 + threadIdx.x / T;
  auto sync = [&]() {
    if (C > 1)
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
      __syncthreads();
  };
  for (int i = threadIdx.x; i < d; i += blockDim.x) buf[0][i] = reinterpret_cast<double2*>(psi)[i];
  double2 ring[AHEAD][Q];   // this lane's part of its first row: columns sub, sub + T, ...
  auto fetch = [&](int n, double2 (&u)[Q]) {
    if (n >= n_steps) return;
    const double2* row = reinterpret_cast<const double2*>(U + n * sU) + (long long)first * d;
#pragma unroll
    for (int q = 0; q < Q; ++q) u[q] = (first < r1 && q * T + sub < d) ? row[q * T + sub] : make_double2(0.0, 0.0);
  };
#pragma unroll
  for (int a = 0; a < AHEAD; ++a) fetch(a, ring[a]);
  // every CTA has read psi before any may write it back, and has started before a remote store
  sync();
  int cur = 0;
  for (int nb = 0; nb < n_steps; nb += AHEAD)
#pragma unroll
  for (int a = 0; a < AHEAD; ++a) {
    const int n = nb + a;
    if (n >= n_steps) break;   // uniform over the cluster
    double2 (&u)[Q] = ring[a];
    for (int i0 = r0; i0 < r1; i0 += nrow) {   // one round, more only where few CTAs were to be had
      const int i = i0 + threadIdx.x / T;
      double re = 0.0, im = 0.0;
      if (i0 == r0) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          if (q * T < d) {   // uniform; lanes beyond d hold zeros (and read a slot of psi below T Q)
            const double2 v = q * T + sub < d ? buf[cur][q * T + sub] : make_double2(0.0, 0.0);
            re = fma(u[q].x, v.x, re);
            re = fma(-u[q].y, v.y, re);
            im = fma(u[q].x, v.y, im);
            im = fma(u[q].y, v.x, im);
          }
        }
        fetch(n + AHEAD, u);
      } else if (i < r1) {
        const double2* row = reinterpret_cast<const double2*>(U + n * sU) + (long long)i * d;
        for (int j = sub; j < d; j += T) {
          const double2 w = row[j], v = buf[cur][j];
          re = fma(w.x, v.x, re);
          re = fma(-w.y, v.y, re);
          im = fma(w.x, v.y, im);
          im = fma(w.y, v.x, im);
        }
      }
#pragma unroll
      for (int o = T / 2; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (i < r1) {
        if (C == 1) {
          if (sub == 0) buf[cur ^ 1][i] = make_double2(re, im);
        } else {
          for (int q = sub; q < (int)C; q += T) {   // the row's lanes share the copies
            const uint32_t a = (uint32_t)__cvta_generic_to_shared(&buf[cur ^ 1][i]);
            uint32_t ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"((uint32_t)q));
            asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(ra), "d"(re), "d"(im) : "memory");
          }
        }
      }
    }
    sync();
    cur ^= 1;
    const int done = step_offset + n + 1;
    if (reorth_every > 0 && done % reorth_every == 0) {   // every CTA on its own copy
      double s = 0.0;
      for (int i = threadIdx.x; i < d; i += blockDim.x) s += buf[cur][i].x * buf[cur][i].x + buf[cur][i].y * buf[cur][i].y;
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) red[warp] = s;
      __syncthreads();
      double v = 0.0;
      for (int w = 0; w < nw; ++w) v += red[w];
      const double inv = 1.0 / sqrt(v);
      for (int i = threadIdx.x; i < d; i += blockDim.x) { buf[cur][i].x *= inv; buf[cur][i].y *= inv; }
      __syncthreads();
    }
    if (traj) {
      double2* t_out = reinterpret_cast<double2*>(traj) + (long long)done * d;
      for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) t_out[i] = buf[cur][i];
    }
  }
  for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) reinterpret_cast<double2*>(psi)[i] = buf[cur][i];
}

// out = U psi (one interval), rows split over CTAs: 8 warps per CTA, one row per warp.
__global__ void __launch_bounds__(256)
matvec_kernel(int d, const double* __restrict__ U, const double* __restrict__ in, double* __restrict__ out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 8 + warp;
  if (i >= d) return;
  const double2* row = reinterpret_cast<const double2*>(U) + (long long)i * d;
  const double2* v = reinterpret_cast<const double2*>(in);
  double re = 0.0, im = 0.0;
  for (int j = lane; j < d; j += 32) {
    double2 u = row[j], x = v[j];
    re = fma(u.x, x.x, re);
    re = fma(-u.y, x.y, re);
    im = fma(u.x, x.y, im);
    im = fma(u.y, x.x, im);
  }
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if (lane == 0) reinterpret_cast<double2*>(out)[i] = make_double2(re, im);
}

__global__ void normalize_kernel(int d, double* __restrict__ psi) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < d; i += blockDim.x) s += psi[2 * i] * psi[2 * i] + psi[2 * i + 1] * psi[2 * i + 1];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  const double inv = 1.0 / sqrt(red[0]);
  for (int i = threadIdx.x; i < 2 * d; i += blockDim.x) psi[i] *= inv;
}

__global__ void norm_defect_kernel(int d, const double* __restrict__ psi, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < d; i += blockDim.x) s += psi[2 * i] * psi[2 * i] + psi[2 * i + 1] * psi[2 * i + 1];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w];
    *out = fabs(sqrt(v) - 1.0);
  }
}

using ChainKernel = void (*)(int, int, const ChainSeg*, const double*, long long, double*, double* const*, int, int,
                             double*);
// lanes per row, columns per lane and intervals ahead by d
static ChainKernel chain_kernel(int d) {
  return d <= 4 ? chain_cluster_kernel<4, 1, 8>
                : d <= 8 ? chain_cluster_kernel<4, 2, 4>
                         : d <= 32 ? chain_cluster_kernel<4, 8, 1> : chain_cluster_kernel<32, 8, 1>;
}

static void chain_cluster_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int d, int C, int nseg,
                                 cudaStream_t s) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)(nseg * C), 1, 1);
  const int lanes = (d <= 32 ? 4 : 32) * ceil_div(d, C);
  cfg->blockDim = dim3(lanes >= 512 ? 512 : (lanes + 31) / 32 * 32, 1, 1);
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// CTAs per state for nseg states of dimension d (32 < d <= 256): about 12 rows per CTA,
// fewer CTAs where that many clusters do not run at once.  The clusters that fit are asked
// for once per device and size.
static int chain_cluster_size(int d, int nseg) {
  static std::mutex mu;
  static int fits[64][5];   // clusters of 1 << q CTAs that fit at once, + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  int want = 2;
  while (want < 16 && want * 12 < d) want *= 2;
  std::lock_guard<std::mutex> lock(mu);
  for (int q = 4; q >= 1; --q) {
    const int C = 1 << q;
    if (C > want) continue;
    if (fits[dev][q] == 0) {
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attr[1];
      // asked of the form with most registers and threads, d = 256
      const void* k = reinterpret_cast<const void*>(chain_kernel(256));
      chain_cluster_config(&cfg, attr, 256, C, 1, nullptr);
      int n = 0;
      if (ensure_func_attr(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != MG_OK ||
          cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      fits[dev][q] = 1 + n;
    }
    if (fits[dev][q] - 1 >= nseg) return C;
  }
  return 1;
}

static int launch_chain_cluster(int C, int nseg, int d, int n_steps, const ChainSeg* segs, const double* U, long long sU,
                                double* psi, double* const* psi_many, int reorth_every, int step_offset, double* traj,
                                cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  chain_cluster_config(&cfg, attr, d, C, nseg, s);
  const ChainKernel k = chain_kernel(d);
  MG_TRY(ensure_func_attr(reinterpret_cast<const void*>(k), cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k, d, n_steps, segs, U, sU, psi, psi_many,
                                           reorth_every, step_offset, traj);
  if (e != cudaSuccess) {
    set_last_cuda_error(e, "cudaLaunchKernelEx(chain_cluster_kernel)", __FILE__, __LINE__);
    return MG_ECUDA;
  }
  return check_launch("chain_cluster_kernel");
}

// psi (device, d complex) is carried through n_steps propagators U (stride sU doubles).
// tmp: d complex of scratch for the large-d path.  traj (may be null): the state
// after step n is also written to traj + (step_offset + n + 1) d complex.
int launch_state_chain(int n_steps, int d, const double* U, long long sU, double* psi, double* tmp,
                       int reorth_every, int step_offset, cudaStream_t s, double* traj) {
  if (n_steps <= 0) return MG_OK;
  const int C = d > 32 && d <= 256 && n_steps > 1 ? chain_cluster_size(d, 1) : 1;
  if (C > 1 || d <= 32)
    return launch_chain_cluster(C, 1, d, n_steps, nullptr, U, sU, psi, nullptr, reorth_every, step_offset, traj, s);
  if (d <= 256) {   // one step, or no cluster to be had
    size_t smem = sizeof(double2) * 2 * d;
    state_chain_kernel<<<1, CHAIN_THREADS, smem, s>>>(n_steps, d, U, sU, psi, reorth_every, step_offset, traj);
    return check_launch("state_chain_kernel");
  }
  double* a = psi;
  double* b = tmp;
  for (int n = 0; n < n_steps; ++n) {
    matvec_kernel<<<ceil_div(d, 8), 256, 0, s>>>(d, U + n * sU, a, b);
    MG_TRY(check_launch("matvec_kernel"));
    double* t = a; a = b; b = t;
    const int done = step_offset + n + 1;
    if (reorth_every > 0 && done % reorth_every == 0) {
      normalize_kernel<<<1, 1024, 0, s>>>(d, a);
      MG_TRY(check_launch("normalize_kernel"));
    }
    if (traj)
      MG_CUDA_TRY(cudaMemcpyAsync(traj + (long long)done * 2 * d, a, sizeof(double) * 2 * d,
                                  cudaMemcpyDeviceToDevice, s));
  }
  if (a != psi) MG_CUDA_TRY(cudaMemcpyAsync(psi, a, sizeof(double) * 2 * d, cudaMemcpyDeviceToDevice, s));
  return MG_OK;
}

int launch_multi_chain(int nseg, int d, const ChainSeg* segs_dev, const double* U, long long sU,
                       double* const* psi_dev, int reorth_every, cudaStream_t s) {
  if (nseg <= 0) return MG_OK;
  if (d > 256) return MG_EUNSUPPORTED;
  // clusters while all states' clusters run at once; beyond, one CTA per state keeps the
  // device as busy without the barriers
  const int C = d > 32 ? chain_cluster_size(d, nseg) : 1;
  if (C > 1 || d <= 32)
    return launch_chain_cluster(C, nseg, d, 0, segs_dev, U, sU, nullptr, psi_dev, reorth_every, 0, nullptr, s);
  multi_chain_kernel<<<nseg, CHAIN_THREADS, sizeof(double2) * 2 * d, s>>>(d, segs_dev, U, sU, psi_dev, reorth_every);
  return check_launch("multi_chain_kernel");
}

int launch_norm_defect(int d, const double* psi, double* out, cudaStream_t s) {
  norm_defect_kernel<<<1, 1024, 0, s>>>(d, psi, out);
  return check_launch("norm_defect_kernel");
}

}  // namespace mg
