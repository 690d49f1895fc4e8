// a3: spectral bounds [e_min, e_max] of H by FP64 Lanczos (the paper maps the spectral interval
// onto [-1, 1] before the Chebyshev expansion, Sec. II.B.1).  The Lanczos scalars stay on the
// device; the host reads the tridiagonal matrix once at the end and takes its extreme
// eigenvalues (Sturm bisection) and eigenvector end components (inverse iteration).
#include <algorithm>
#include <cmath>
#include <vector>

#include "bulk.cuh"
#include "common.cuh"

namespace tbk {

// w = H v - beta * vprev (beta read from the device; vprev may be NULL), and per-CTA partial
// sums of w . v.  One thread per orbital row.
__device__ __forceinline__ void lz_spmv_cta(int cta, int n_atoms, int B, const int32_t* __restrict__ row_ptr,
                                            const int32_t* __restrict__ col, const double* __restrict__ H,
                                            const double* __restrict__ v, const double* __restrict__ vprev,
                                            const double* __restrict__ beta, double* __restrict__ w,
                                            double* __restrict__ part) {
  __shared__ double red[32];
  const int64_t n = (int64_t)n_atoms * B;
  const int64_t row = (int64_t)cta * blockDim.x + threadIdx.x;
  double d = 0.0;
  if (row < n) {
    const int a = (int)(row / B), i = (int)(row - (int64_t)a * B);
    double acc = 0.0;
    for (int k = row_ptr[a]; k < row_ptr[a + 1]; ++k) {
      const int b = col[k];
      const double* h = H + (int64_t)k * B * B + i * B;
      for (int l = 0; l < B; ++l) acc += h[l] * v[(int64_t)b * B + l];
    }
    if (vprev) acc -= (*beta) * vprev[row];
    w[row] = acc;
    d = acc * v[row];
  }
  double t = tbk_block_sum(d, red);
  if (threadIdx.x == 0) part[cta] = t;
}

// w -= alpha v; per-CTA partial sums of w . w.
__device__ __forceinline__ void lz_orth_cta(int cta, int64_t n, const double* __restrict__ v,
                                            const double* __restrict__ alpha, double* __restrict__ w,
                                            double* __restrict__ part) {
  __shared__ double red[32];
  const int64_t i = (int64_t)cta * blockDim.x + threadIdx.x;
  double d = 0.0;
  if (i < n) {
    double x = w[i] - (*alpha) * v[i];
    w[i] = x;
    d = x * x;
  }
  double t = tbk_block_sum(d, red);
  if (threadIdx.x == 0) part[cta] = t;
}

// out = sum(part) (take_sqrt: sqrt of it), single block, fixed order.
__device__ __forceinline__ void lz_reduce_block(const double* __restrict__ part, int m, int take_sqrt,
                                                double* __restrict__ out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < m; i += blockDim.x) s += part[i];
  double t = tbk_block_sum(s, red);
  if (threadIdx.x == 0) *out = take_sqrt ? sqrt(t) : t;
}

__global__ void lz_start(int64_t n, uint64_t seed, double* __restrict__ v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = (double)tbk_probe_sign(seed, i, 0) / sqrt((double)n);
}

// ---- one operator: all steps in one cooperative launch -----------------------------------------
//
// A warp owns 32 consecutive rows (a unit); units are dealt over the CTAs first, so that a small
// operator still uses one warp on many SMs.  A step is H v - beta v_prev with the partial sums of
// alpha, then w - alpha v with those of beta, then w / beta, each ended by a barrier over the grid;
// the CTA that arrives last adds the units' partial sums (in every CTA the additions took a quarter
// of all FP64 issue at 10,000 atoms).  The sums keep one order: rows in groups of 256, a tree per
// group, 256 strided chains of groups, a tree; that of lz_reduce_block.
//
// An FP64 operation takes 64 cycles and a row of 19 blocks is a chain of 171: 5.3 us a step,
// while five launches a step took 57 us on 147 atoms (41 us of it in the product, whose rows sat on
// 6 SMs) and 66 us on 10,000 atoms, where the FP64 issue rate allows 27.  Now 23 us a step on 1,000
// atoms and 47 us on 10,000.
// TR: blocks stored transposed (lz_transpose), so that the rows of an atom read neighbouring words.
// PF: the next block is loaded ahead, for operators with few warps per SM.
constexpr int LZ_CHAINS = 256;
constexpr size_t LZ_TRANSPOSE_MAX = (size_t)128 << 20;

struct LzSync {
  unsigned arrived, gen;  // arrivals at the barrier, finished barriers
  double sum[2];          // the sums of the last two reducing barriers
};

__device__ __forceinline__ double lz_warp_sum(double d) {
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  return d;
}

// Sum of the units' partial sums over the CTA, valid in thread 0.
__device__ __forceinline__ double lz_units_sum(const double* part, int nb, double* red) {
  double s = 0.0;
  for (int g = threadIdx.x; g < nb && threadIdx.x < LZ_CHAINS; g += LZ_CHAINS) {
    double2 p[4];
    for (int q = 0; q < 4; ++q) p[q] = __ldcg(reinterpret_cast<const double2*>(part + 8 * (size_t)g) + q);
    s += ((p[0].x + p[2].x) + (p[1].x + p[3].x)) + ((p[0].y + p[2].y) + (p[1].y + p[3].y));
  }
  if (nb <= 32) return threadIdx.x < 32 ? lz_warp_sum(s) : 0.0;  // the other warps hold zeros
  s = lz_warp_sum(s);
  if ((threadIdx.x & 31) == 0 && threadIdx.x < LZ_CHAINS) red[threadIdx.x >> 5] = s;
  __syncthreads();
  return ((red[0] + red[4]) + (red[2] + red[6])) + ((red[1] + red[5]) + (red[3] + red[7]));
}

// Barrier of the grid (co-resident CTAs), number `gen` from 1 on; with part, the last CTA to arrive
// leaves the sum of the partial sums in sy->sum[gen & 1] first.  Bounded like tbk_grid_wait.
__device__ __forceinline__ bool lz_barrier(LzSync* sy, unsigned gen, const double* part, int nb, double* red) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&sy->arrived) : "memory");
    last = old == gen * gridDim.x - 1;
  }
  __syncthreads();
  int ok = 1;
  if (last) {
    double t = 0.0;
    if (part) t = lz_units_sum(part, nb, red);
    if (threadIdx.x == 0) {
      if (part) __stcg(&sy->sum[gen & 1], t);
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&sy->gen), "r"(gen) : "memory");
    }
  } else if (threadIdx.x == 0) {
    ok = tbk_spin_until(&sy->gen, gen);
  }
  return __syncthreads_and(ok) != 0;
}

// Threads per CTA: one CTA per SM, so that a barrier has few arrivals.
template <bool PF> constexpr int lz_threads() { return PF ? 256 : 768; }

template <int B, bool TR, bool PF>
__global__ void __launch_bounds__(lz_threads<PF>(), 1)
lz_run(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
       const double* __restrict__ H, int m, double* vecs, double* part, double* __restrict__ alpha,
       double* __restrict__ beta, LzSync* sy, double* __restrict__ fail) {
  __shared__ double red[8];
  const int64_t n = (int64_t)n_atoms * B;
  const int nb = (int)((n + 255) / 256), units = 8 * nb;
  const int lane = threadIdx.x & 31, stride = gridDim.x * (lz_threads<PF>() / 32);
  const int first = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  unsigned gen = 0;
  bool ok = true;
  // with p: returns the sum of the partial sums
  auto wait = [&](const double* p) {
    ok = lz_barrier(sy, ++gen, p, nb, red) && ok;
    return p ? __ldcg(&sy->sum[gen & 1]) : 0.0;
  };
  double bj = 0.0;
  for (int j = 0; j < m && ok; ++j) {
    // v_{j-1}, v_j and w rotate through three vectors
    const double* vp = vecs + (j % 3) * n;
    double* v = vecs + ((j + 1) % 3) * n;
    double* w = vecs + ((j + 2) % 3) * n;
    double own = 0.0, vown = 0.0;  // this thread's row of the warp's first unit
    for (int u = first; u < units; u += stride) {
      const int64_t row = (int64_t)u * 32 + lane;
      double d = 0.0;
      if (row < n) {
        const int a = (int)(row / B), i = (int)(row - (int64_t)a * B);
        double acc = 0.0;
        const int k1 = __ldg(row_ptr + a + 1);
        int k = __ldg(row_ptr + a);
        double h[B], x[B];
        auto fetch = [&](int kk, double (&hh)[B], double (&xx)[B]) {
          const double* xb = v + (int64_t)__ldg(col + kk) * B;
          const double* hb = H + (int64_t)kk * B * B + (TR ? i : i * B);
#pragma unroll
          for (int l = 0; l < B; ++l) {
            hh[l] = __ldg(hb + (TR ? l * B : l));
            xx[l] = xb[l];
          }
        };
        if (PF && k < k1) fetch(k, h, x);
        for (; k < k1; ++k) {
          double hn[B], xn[B];
          if constexpr (PF) {
            if (k + 1 < k1) fetch(k + 1, hn, xn);
          } else {
            fetch(k, h, x);
          }
#pragma unroll
          for (int l = 0; l < B; ++l) acc += h[l] * x[l];
          if constexpr (PF) {
#pragma unroll
            for (int l = 0; l < B; ++l) {
              h[l] = hn[l];
              x[l] = xn[l];
            }
          }
        }
        if (j) acc -= bj * vp[row];
        const double vr = v[row];
        if (u == first) {
          own = acc;
          vown = vr;
        } else {
          w[row] = acc;
        }
        d = acc * vr;
      }
      d = lz_warp_sum(d);
      if (lane == 0) __stcg(part + u, d);
    }
    const double aj = wait(part);
    for (int u = first; u < units; u += stride) {
      const int64_t row = (int64_t)u * 32 + lane;
      double d = 0.0;
      if (row < n) {
        const double x = (u == first ? own : w[row]) - aj * (u == first ? vown : v[row]);
        if (u == first) own = x; else w[row] = x;
        d = x * x;
      }
      d = lz_warp_sum(d);
      if (lane == 0) __stcg(part + units + u, d);
    }
    bj = sqrt(wait(part + units));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      alpha[j] = aj;
      beta[j + 1] = bj;
    }
    if (j + 1 == m) break;
    for (int u = first; u < units; u += stride) {
      const int64_t row = (int64_t)u * 32 + lane;
      if (row < n) w[row] = bj > 0.0 ? (u == first ? own : w[row]) / bj : 0.0;
    }
    wait(nullptr);
  }
  if (!ok && threadIdx.x == 0) *fail = 1.0;
}

// out[k][l][i] = H[k][i][l], 9x9 blocks
__global__ void lz_transpose(int64_t n, const double* __restrict__ H, double* __restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int64_t k = t / 81;
  const int e = (int)(t - k * 81), l = e / 9, i = e - 9 * l;
  out[t] = __ldg(H + k * 81 + i * 9 + l);
}

// ---- a small operator: one thread-block cluster, the vectors in shared memory and registers ----------
//
// The same sums with a cluster of CL CTAs, one unit per warp: v is copied into every CTA's shared memory, a
// thread keeps its row of v_prev, v and w (and of H, as far as shared memory goes), and partial sums go to
// every CTA, where each warp adds them itself.  The hardware barrier of a cluster takes ~0.2 us where one over
// the grid takes ~2 with its sum: what is left of a step is the row's chain of 171 operations, 64 cycles each
// up to three warps per SM and 19 per warp beyond (the SM's FP64 units are shared), and about 6 us of sums,
// square root, division and barriers.  147 atoms: 21.9 us a step over the grid,
// 15.5 with 8 CTAs, 11.7 with 16 (where the device takes such clusters).  With 16: 340 atoms 14.1, 455 atoms
// 17.4; the grid takes 21.1 at 456 atoms and 22.6 at 1,000, most of it its barriers (with H and the gathered v
// in shared memory there the same).  Longer rows do not turn it: cluster / grid at 147 atoms 38 / 53 with 44 blocks a
// row, 68 / 90 with 79; at 455 atoms 48 / 57 with 53 and 101 / 117 with 108.
constexpr int LZ_CL_UNITS = 128;

template <int B, int CL>
__global__ void __launch_bounds__(32 * LZ_CL_UNITS / CL)
lz_run_cluster(int n_atoms, int cap, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const double* __restrict__ H, int m, uint64_t seed, double* __restrict__ alpha,
               double* __restrict__ beta) {
  __shared__ double vs[32 * LZ_CL_UNITS];
  __shared__ double part[2][LZ_CL_UNITS];
  const int n = n_atoms * B, nb = (n + 255) / 256, units = 8 * nb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int u = warp * CL + blockIdx.x, row = 32 * u + lane, T = blockDim.x;
  const bool has = row < n;
  // the thread's row of the first `cap` blocks, and where their v lies
  extern __shared__ double lz_smem[];
  double* hs = lz_smem + threadIdx.x;
  int* cs = reinterpret_cast<int*>(lz_smem + (int64_t)cap * B * T) + threadIdx.x;
  for (int i = threadIdx.x; i < n; i += blockDim.x) vs[i] = (double)tbk_probe_sign(seed, i, 0) / sqrt((double)n);
  for (int i = threadIdx.x; i < 2 * LZ_CL_UNITS; i += blockDim.x) part[0][i] = 0.0;
  cluster_barrier();
  // the sum of the units' values d, in every thread
  auto total = [&](int set, double d) {
    d = lz_warp_sum(d);
    if (u < units && lane < CL) store_cluster(&part[set][u], lane, d);
    cluster_barrier();
    double s = 0.0;
    if (lane < nb) {
      const double* p = part[set] + 8 * lane;
      s = ((p[0] + p[4]) + (p[2] + p[6])) + ((p[1] + p[5]) + (p[3] + p[7]));
    }
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);  // nb <= 16
    return __shfl_sync(0xffffffffu, s, 0);
  };
  const int a = has ? row / B : 0, i = row - a * B;
  const int k0 = has ? __ldg(row_ptr + a) : 0, k1 = has ? __ldg(row_ptr + a + 1) : 0;
  const int ks = min(k1 - k0, cap);
  for (int k = 0; k < ks; ++k) {
    cs[k * T] = __ldg(col + k0 + k) * B;
#pragma unroll
    for (int l = 0; l < B; ++l) hs[(int64_t)(k * B + l) * T] = __ldg(H + (int64_t)(k0 + k) * B * B + l * B + i);
  }
  double vprev = 0.0, v = has ? vs[row] : 0.0, bj = 0.0;
  for (int j = 0; j < m; ++j) {
    double acc = 0.0;
#pragma unroll 2
    for (int k = 0; k < ks; ++k) {
      const double *h = hs + (int64_t)k * B * T, *x = vs + cs[k * T];
#pragma unroll
      for (int l = 0; l < B; ++l) acc += h[l * T] * x[l];
    }
    for (int k = k0 + ks; k < k1; ++k) {
      const double *h = H + (int64_t)k * B * B + i, *x = vs + __ldg(col + k) * B;
#pragma unroll
      for (int l = 0; l < B; ++l) acc += __ldg(h + l * B) * x[l];
    }
    if (j) acc -= bj * vprev;
    const double aj = total(0, has ? acc * v : 0.0);
    const double x = acc - aj * v;
    bj = sqrt(total(1, has ? x * x : 0.0));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      alpha[j] = aj;
      beta[j + 1] = bj;
    }
    if (j + 1 == m) break;
    vprev = v;
    v = has && bj > 0.0 ? x / bj : 0.0;
    if (has)
      for (int r = 0; r < CL; ++r) store_cluster(vs + row, r, v);
    cluster_barrier();
  }
  cluster_barrier();  // no CTA leaves while another may still write to it
}

template <int B, bool TR, bool PF>
static void lz_launch_pf(tbk_ctx* ctx, const tbk_bsr* H, const double* val, int m, double* vecs, double* part,
                         double* alpha, double* beta, LzSync* sy, double* fail) {
  constexpr int T = lz_threads<PF>();
  const int units = 8 * ceil_div((int64_t)H->n_atoms * B, 256);
  const int grid = std::min(units, ctx->num_sms);
  int n_atoms = H->n_atoms;
  const int32_t *rp = H->row_ptr, *cl = H->col;
  void* args[] = {&n_atoms, &rp, &cl, &val, &m, &vecs, &part, &alpha, &beta, &sy, &fail};
  TBK_CUDA(cudaLaunchCooperativeKernel((const void*)lz_run<B, TR, PF>, dim3(grid), dim3(T), args, 0, ctx->stream));
  post_launch(ctx, "lz_run");
}

template <int B, int CL>
static cudaLaunchConfig_t lz_cluster_config(tbk_ctx* ctx, int units, int64_t blocks, cudaLaunchAttribute* at, int* cap) {
  cudaLaunchConfig_t cfg{};
  const int T = 32 * ceil_div(units, CL);
  const int64_t most = 180 << 10;  // beside 34 KB of vectors
  *cap = (int)std::min<int64_t>(blocks, most / ((8 * B + 4) * T));
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(T);
  cfg.dynamicSmemBytes = (size_t)(8 * B + 4) * T * *cap;
  cfg.stream = ctx->stream;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = CL;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

template <int B, int CL>
static void lz_cluster_attributes() {
  TBK_CUDA(cudaFuncSetAttribute(lz_run_cluster<B, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, 180 << 10));
  if (CL > 8) TBK_CUDA(cudaFuncSetAttribute(lz_run_cluster<B, CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
}

// Whether the device takes clusters of 16 with the largest shared memory and block used.
template <int B>
static bool lz_wide_clusters(tbk_ctx* ctx) {
  static int known[64] = {0};
  int& k = known[ctx->device & 63];
  if (!k) {
    lz_cluster_attributes<B, 16>();
    cudaLaunchAttribute at{};
    int cap, clusters = 0;
    const cudaLaunchConfig_t cfg = lz_cluster_config<B, 16>(ctx, LZ_CL_UNITS, 1 << 20, &at, &cap);
    if (cudaOccupancyMaxActiveClusters(&clusters, lz_run_cluster<B, 16>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    k = clusters > 0 ? 1 : 2;
  }
  return k == 1;
}

template <int B, int CL>
static void lz_launch_cluster(tbk_ctx* ctx, const tbk_bsr* H, const double* val, int m, uint64_t seed, double* alpha,
                              double* beta) {
  const int units = 8 * ceil_div((int64_t)H->n_atoms * B, 256);
  lz_cluster_attributes<B, CL>();
  cudaLaunchAttribute at{};
  int cap;
  // up to four times the average row in shared memory
  const cudaLaunchConfig_t cfg =
      lz_cluster_config<B, CL>(ctx, units, 4 * (int64_t)ceil_div(H->nnzb, H->n_atoms), &at, &cap);
  TBK_CUDA(cudaLaunchKernelEx(&cfg, lz_run_cluster<B, CL>, (int)H->n_atoms, cap, H->row_ptr, H->col, val, m, seed, alpha,
                              beta));
  post_launch(ctx, "lz_run_cluster");
}

// val: the blocks, transposed (TR) or as given
template <int B, bool TR>
static void lz_launch(tbk_ctx* ctx, const tbk_bsr* H, const double* val, int m, uint64_t seed, double* vecs,
                      double* part, double* alpha, double* beta, LzSync* sy, double* fail) {
  const int64_t n = (int64_t)H->n_atoms * B;
  const int64_t units = 8 * (int64_t)ceil_div(n, 256);
  if ((TR || B == 1) && units <= LZ_CL_UNITS) {
    if (lz_wide_clusters<B>(ctx)) lz_launch_cluster<B, 16>(ctx, H, val, m, seed, alpha, beta);
    else lz_launch_cluster<B, 8>(ctx, H, val, m, seed, alpha, beta);
    return;
  }
  lz_start<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(n, seed, vecs + n);
  post_launch(ctx, "lz_start");
  // up to 8 warps per SM the loads ahead hide the latency, beyond that the warps do
  if (n <= (int64_t)ctx->num_sms * 8 * 32)
    lz_launch_pf<B, TR, true>(ctx, H, val, m, vecs, part, alpha, beta, sy, fail);
  else
    lz_launch_pf<B, TR, false>(ctx, H, val, m, vecs, part, alpha, beta, sy, fail);
}

// ---- many clusters: the same kernels, blockIdx.y = cluster ---------------------------------
struct LzJob {
  int n_atoms, B, nb, m;
  const int32_t* row_ptr;
  const int32_t* col;
  const double* H;
  double* vecs;  // vp, v, w (n each), part (nb), alpha (m + 2), beta (m + 2)
  int64_t n;
  uint64_t seed;
};

__device__ __forceinline__ void lz_ptrs(const LzJob& j, int step, double*& vp, double*& v, double*& w) {
  // the rotation vp <- v, v <- w, w <- old vp of the single-cluster loop, by step parity mod 3
  double* base[3] = {j.vecs, j.vecs + j.n, j.vecs + 2 * j.n};
  vp = base[step % 3];
  v = base[(step + 1) % 3];
  w = base[(step + 2) % 3];
}

__global__ void lzb_start(const LzJob* __restrict__ jobs) {
  const LzJob j = jobs[blockIdx.y];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < j.n) j.vecs[j.n + i] = (double)tbk_probe_sign(j.seed, i, 0) / sqrt((double)j.n);
}

__global__ void lzb_spmv(const LzJob* __restrict__ jobs, int step) {
  const LzJob j = jobs[blockIdx.y];
  if (step >= j.m || (int)blockIdx.x >= j.nb) return;
  double *vp, *v, *w;
  lz_ptrs(j, step, vp, v, w);
  double* part = j.vecs + 3 * j.n;
  double* beta = part + j.nb + (j.m + 2);
  lz_spmv_cta(blockIdx.x, j.n_atoms, j.B, j.row_ptr, j.col, j.H, v, step ? vp : nullptr, beta + step, w, part);
}

__global__ void lzb_reduce(const LzJob* __restrict__ jobs, int step, int take_sqrt) {
  const LzJob j = jobs[blockIdx.y];
  if (step >= j.m) return;
  double* part = j.vecs + 3 * j.n;
  double* alpha = part + j.nb;
  double* beta = alpha + (j.m + 2);
  lz_reduce_block(part, j.nb, take_sqrt, take_sqrt ? beta + step + 1 : alpha + step);
}

__global__ void lzb_orth(const LzJob* __restrict__ jobs, int step) {
  const LzJob j = jobs[blockIdx.y];
  if (step >= j.m || (int)blockIdx.x >= j.nb) return;
  double *vp, *v, *w;
  lz_ptrs(j, step, vp, v, w);
  double* part = j.vecs + 3 * j.n;
  lz_orth_cta(blockIdx.x, j.n, v, part + j.nb + step, w, part);
}

__global__ void lzb_scale(const LzJob* __restrict__ jobs, int step) {
  const LzJob j = jobs[blockIdx.y];
  if (step >= j.m) return;
  double *vp, *v, *w;
  lz_ptrs(j, step, vp, v, w);
  const double* beta = j.vecs + 3 * j.n + j.nb + (j.m + 2);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const double b = beta[step + 1];
  if (i < j.n) w[i] = b > 0.0 ? w[i] / b : 0.0;
}

// ---- host: tridiagonal eigen-analysis -------------------------------------------------------

// Number of eigenvalues of the tridiagonal (a, b) below x (Sturm sequence).
static int sturm_count(const std::vector<double>& a, const std::vector<double>& b, double x) {
  int cnt = 0;
  double q = 1.0;
  const double tiny = 1e-300;
  for (size_t i = 0; i < a.size(); ++i) {
    const double bb = i ? b[i - 1] * b[i - 1] : 0.0;
    q = (a[i] - x) - (i ? bb / q : 0.0);
    if (q == 0.0) q = -tiny;
    if (q < 0.0) ++cnt;
  }
  return cnt;
}

// k-th smallest eigenvalue (0-based) by bisection.
static double tri_eig(const std::vector<double>& a, const std::vector<double>& b, int k) {
  const size_t m = a.size();
  double lo = INFINITY, hi = -INFINITY;
  for (size_t i = 0; i < m; ++i) {
    const double r = (i ? fabs(b[i - 1]) : 0.0) + (i + 1 < m ? fabs(b[i]) : 0.0);
    lo = std::min(lo, a[i] - r);
    hi = std::max(hi, a[i] + r);
  }
  const double scale = std::max(fabs(lo), fabs(hi)) + 1e-300;
  for (int it = 0; it < 200 && hi - lo > 4e-16 * scale; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (sturm_count(a, b, mid) > k) hi = mid; else lo = mid;
  }
  return 0.5 * (lo + hi);
}

// |last component| of the unit eigenvector of the tridiagonal for eigenvalue theta, by three
// steps of inverse iteration with a slightly shifted theta (Gaussian elimination with partial
// pivoting on the tridiagonal system).
static double tri_last_component(const std::vector<double>& a, const std::vector<double>& b, double theta) {
  const int m = (int)a.size();
  if (m == 1) return 1.0;
  double scale = 0.0;
  for (int i = 0; i < m; ++i) scale = std::max(scale, fabs(a[i]) + (i < m - 1 ? fabs(b[i]) : 0.0));
  const double sigma = theta + 1e-10 * (scale + 1e-300);
  std::vector<double> z(m, 1.0 / std::sqrt((double)m));
  for (int rep = 0; rep < 3; ++rep) {
    // rows: dl (sub), d (diag), du (super), du2 (fill-in)
    std::vector<double> dl(m, 0.0), d(m), du(m, 0.0), du2(m, 0.0), rhs = z;
    for (int i = 0; i < m; ++i) {
      d[i] = a[i] - sigma;
      if (i < m - 1) { du[i] = b[i]; dl[i] = b[i]; }
    }
    for (int i = 0; i < m - 1; ++i) {
      if (fabs(d[i]) >= fabs(dl[i])) {
        if (d[i] == 0.0) d[i] = 1e-300;
        const double f = dl[i] / d[i];
        d[i + 1] -= f * du[i];
        if (i < m - 2) du2[i] = 0.0;
        rhs[i + 1] -= f * rhs[i];
      } else {
        // swap rows i and i+1, then eliminate: the pivot row gains a second superdiagonal
        const double f = d[i] / dl[i];
        const double old_dnext = d[i + 1], old_du = du[i];
        d[i] = dl[i];
        du[i] = old_dnext;
        d[i + 1] = old_du - f * old_dnext;
        if (i < m - 2) {
          du2[i] = du[i + 1];
          du[i + 1] = -f * du2[i];
        }
        std::swap(rhs[i], rhs[i + 1]);
        rhs[i + 1] -= f * rhs[i];
      }
    }
    if (d[m - 1] == 0.0) d[m - 1] = 1e-300;
    std::vector<double> x(m);
    x[m - 1] = rhs[m - 1] / d[m - 1];
    if (m >= 2) x[m - 2] = (rhs[m - 2] - du[m - 2] * x[m - 1]) / d[m - 2];
    for (int i = m - 3; i >= 0; --i) x[i] = (rhs[i] - du[i] * x[i + 1] - du2[i] * x[i + 2]) / d[i];
    double nrm = 0.0;
    for (double v : x) nrm += v * v;
    nrm = std::sqrt(nrm);
    if (!(nrm > 0.0) || !std::isfinite(nrm)) return 1.0;
    for (int i = 0; i < m; ++i) z[i] = x[i] / nrm;
  }
  return fabs(z[m - 1]);
}

void bounds_from_tridiagonal(const std::vector<double>& ha, const std::vector<double>& hb, int m,
                             double rel_margin, double* emin, double* emax);

}  // namespace tbk

using namespace tbk;

extern "C" int tbk_spectral_bounds(tbk_ctx* ctx, const tbk_bsr* H, int32_t steps,
                                   double rel_margin, uint64_t seed, double* emin, double* emax) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx && H && emin && emax, "NULL argument");
  TBK_CHECK_ARG(H->n_orb == 1 || H->n_orb == 9, "n_orb must be 1 or 9");
  TBK_CHECK_ARG(H->n_atoms >= 1 && H->row_ptr && H->col && H->val, "empty or NULL matrix");
  TBK_CHECK_ARG(steps >= 1 && steps <= 10000, "steps must be in [1, 10000]");
  TBK_CHECK_ARG(rel_margin >= 0.0 && std::isfinite(rel_margin), "rel_margin must be >= 0");
  DeviceGuard dg(ctx);
  const int64_t n = (int64_t)H->n_atoms * H->n_orb;
  const int m = (int)std::min<int64_t>(steps, n);
  const int nb = ceil_div(n, 256), units = 8 * nb;
  // transposed blocks as long as the copy stays in L2 between the steps (10,000 atoms: 115 MB)
  const bool tr = H->n_orb == 9 && H->nnzb >= H->n_atoms && (size_t)H->nnzb * 648 <= LZ_TRANSPOSE_MAX;
  // vectors | partial sums | alpha (m + 2) | beta (m + 2) | barrier | failure flag | H^T
  const size_t nvec = (3 * (size_t)n + 1) & ~(size_t)1, nred = 2 * (size_t)units, nab = 2 * ((size_t)m + 2) + 4;
  double* vecs = (double*)scratch(ctx, WS_LANCZOS, sizeof(double) * (nvec + nred + nab + (tr ? 81 * (size_t)H->nnzb : 0)));
  double* part = vecs + nvec;
  double* alpha = part + nred;        // alpha[j], j < m
  double* beta = alpha + (m + 2);     // beta[j]: beta[0] = 0, beta[j+1] = ||w_j||
  LzSync* sy = (LzSync*)(beta + (m + 2));
  double* fail = beta + (m + 2) + 3;
  TBK_CUDA(cudaMemsetAsync(alpha, 0, sizeof(double) * nab, ctx->stream));
  if (tr) {
    double* ht = alpha + nab;
    lz_transpose<<<(unsigned)((81 * H->nnzb + 255) / 256), 256, 0, ctx->stream>>>(81 * H->nnzb, H->val, ht);
    post_launch(ctx, "lz_transpose");
    lz_launch<9, true>(ctx, H, ht, m, seed, vecs, part, alpha, beta, sy, fail);
  } else if (H->n_orb == 9) {
    lz_launch<9, false>(ctx, H, H->val, m, seed, vecs, part, alpha, beta, sy, fail);
  } else {
    lz_launch<1, false>(ctx, H, H->val, m, seed, vecs, part, alpha, beta, sy, fail);
  }
  std::vector<double> hab(nab);
  TBK_CUDA(cudaMemcpyAsync(hab.data(), alpha, sizeof(double) * nab, cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  if (hab[nab - 1] != 0.0) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the Lanczos kernel expired");
  const std::vector<double> ha(hab.begin(), hab.begin() + m), hb(hab.begin() + m + 2, hab.begin() + 2 * m + 3);
  bounds_from_tridiagonal(ha, hb, m, rel_margin, emin, emax);
  TBK_API_END
}

namespace tbk {
// Extreme Ritz values of the Lanczos tridiagonal (alpha ha[0..m), beta hb[1..m]) widened by their
// residual norms, then by rel_margin of the width on each side.
void bounds_from_tridiagonal(const std::vector<double>& ha, const std::vector<double>& hb, int m,
                             double rel_margin, double* emin, double* emax) {
  // Stop at the first (numerically) vanishing beta: the Krylov space is invariant there.
  int mm = m;
  double scale = 0.0;
  for (int j = 0; j < m; ++j) scale = std::max(scale, fabs(ha[j]) + fabs(hb[j + 1]));
  for (int j = 1; j < m; ++j)
    if (hb[j] <= 1e-14 * (scale + 1e-300)) { mm = j; break; }
  std::vector<double> a(ha.begin(), ha.begin() + mm), b(hb.begin() + 1, hb.begin() + mm);
  for (double x : a) TBK_CHECK_ARG(std::isfinite(x), "Lanczos produced a non-finite value");
  const double tmin = tri_eig(a, b, 0), tmax = tri_eig(a, b, mm - 1);
  const double bm = hb[mm];  // residual coupling of the last Lanczos vector
  const double rmin = fabs(bm) * tri_last_component(a, b, tmin);
  const double rmax = fabs(bm) * tri_last_component(a, b, tmax);
  double lo = tmin - rmin, hi = tmax + rmax;
  const double width = std::max(hi - lo, 1e-12 * std::max(1.0, std::max(fabs(lo), fabs(hi))));
  *emin = lo - rel_margin * width;
  *emax = hi + rel_margin * width;
  if (!(*emax > *emin)) *emax = *emin + 1e-12;
}
}  // namespace tbk

extern "C" int tbk_batched_spectral_bounds(tbk_ctx* ctx, int32_t n_clusters, const tbk_bsr* H,
                                           int32_t steps, double rel_margin, uint64_t seed,
                                           double* emin, double* emax) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx && H && emin && emax, "NULL argument");
  TBK_CHECK_ARG(n_clusters >= 1, "n_clusters must be >= 1");
  TBK_CHECK_ARG(steps >= 1 && steps <= 10000, "steps must be in [1, 10000]");
  TBK_CHECK_ARG(rel_margin >= 0.0 && std::isfinite(rel_margin), "rel_margin must be >= 0");
  DeviceGuard dg(ctx);
  std::vector<LzJob> jobs(n_clusters);
  size_t tot = 0;
  int nb_max = 1, m_max = 1;
  for (int c = 0; c < n_clusters; ++c) {
    TBK_CHECK_ARG(H[c].n_orb == 1 || H[c].n_orb == 9, "n_orb must be 1 or 9");
    TBK_CHECK_ARG(H[c].n_atoms >= 1 && H[c].row_ptr && H[c].col && H[c].val, "empty or NULL matrix");
    LzJob& j = jobs[c];
    j.n_atoms = H[c].n_atoms;
    j.B = H[c].n_orb;
    j.n = (int64_t)j.n_atoms * j.B;
    j.m = (int)std::min<int64_t>(steps, j.n);
    j.nb = ceil_div(j.n, 256);
    j.row_ptr = H[c].row_ptr;
    j.col = H[c].col;
    j.H = H[c].val;
    j.seed = seed;
    j.vecs = nullptr;
    tot += (size_t)(3 * j.n + j.nb + 2 * (j.m + 2));
    nb_max = std::max(nb_max, j.nb);
    m_max = std::max(m_max, j.m);
  }
  double* vecs = (double*)scratch(ctx, WS_LANCZOS, sizeof(double) * tot);
  LzJob* d_jobs = (LzJob*)scratch(ctx, WS_MISC, sizeof(LzJob) * (size_t)n_clusters);
  size_t off = 0;
  for (int c = 0; c < n_clusters; ++c) {
    LzJob& j = jobs[c];
    j.vecs = vecs + off;
    off += (size_t)(3 * j.n + j.nb + 2 * (j.m + 2));
    // beta[0] = 0 (the first step has no previous vector)
    TBK_CUDA(cudaMemsetAsync(j.vecs + 3 * j.n + j.nb + (j.m + 2), 0, sizeof(double) * (j.m + 2), ctx->stream));
  }
  TBK_CUDA(cudaMemcpyAsync(d_jobs, jobs.data(), sizeof(LzJob) * n_clusters, cudaMemcpyHostToDevice, ctx->stream));
  const dim3 g(nb_max, n_clusters), g1(1, n_clusters);
  lzb_start<<<g, 256, 0, ctx->stream>>>(d_jobs);
  post_launch(ctx, "lzb_start");
  for (int step = 0; step < m_max; ++step) {
    lzb_spmv<<<g, 256, 0, ctx->stream>>>(d_jobs, step);
    post_launch(ctx, "lzb_spmv");
    lzb_reduce<<<g1, 256, 0, ctx->stream>>>(d_jobs, step, 0);
    post_launch(ctx, "lzb_reduce");
    lzb_orth<<<g, 256, 0, ctx->stream>>>(d_jobs, step);
    post_launch(ctx, "lzb_orth");
    lzb_reduce<<<g1, 256, 0, ctx->stream>>>(d_jobs, step, 1);
    post_launch(ctx, "lzb_reduce");
    lzb_scale<<<g, 256, 0, ctx->stream>>>(d_jobs, step);
    post_launch(ctx, "lzb_scale");
  }
  std::vector<std::vector<double>> ha(n_clusters), hb(n_clusters);
  for (int c = 0; c < n_clusters; ++c) {
    const LzJob& j = jobs[c];
    ha[c].resize(j.m);
    hb[c].resize(j.m + 1);
    const double* alpha = j.vecs + 3 * j.n + j.nb;
    TBK_CUDA(cudaMemcpyAsync(ha[c].data(), alpha, sizeof(double) * j.m, cudaMemcpyDeviceToHost, ctx->stream));
    TBK_CUDA(cudaMemcpyAsync(hb[c].data(), alpha + (j.m + 2), sizeof(double) * (j.m + 1), cudaMemcpyDeviceToHost,
                             ctx->stream));
  }
  sync(ctx);
  for (int c = 0; c < n_clusters; ++c)
    bounds_from_tridiagonal(ha[c], hb[c], jobs[c].m, rel_margin, emin + c, emax + c);
  TBK_API_END
}
