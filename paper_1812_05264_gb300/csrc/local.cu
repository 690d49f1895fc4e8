// f3: the local approximation of the sampled density and energy-density matrices (Sec. II.C.1,
// Eq. local_density, S = I).
//
// For each atom a, the region R_a = the atoms within r_max of a (the mask M_L(r_max) of the
// paper; a included) defines the local operator H_a = L_a^T H L_a.  All n_orb functions of a share
// its centre and so its region: one local problem per atom gives the n_orb columns of a, which
// are P~_L[:, a] = L_a p_f(H_a) L_a^T E_a and Q~_L[:, a] = L_a H_a p_f(H_a) L_a^T E_a, E_a the unit
// vectors of a's functions, p_f the order-term Chebyshev expansion of the Fermi function on the
// global bounds [emin, emax] (every local spectrum lies inside them: a principal submatrix's
// eigenvalues interlace H's).  The result is kept on the pattern M of H: block (b, a) of the output
// is rows b of column block a.  Columns come from different local problems, so the result is not
// symmetric.
//
// All local problems run together as one block-diagonal operator: the regions' atoms are listed
// one region after another (region a's atom i at merged index rs[a] + i), the local pattern is M
// restricted to each region, and each local block is a copy of the mapped global block
// (H^ of the global bounds restricted to the region is the region's own mapped operator).  X =
// p_f(H^_loc) E is formed by the backward (Clenshaw) form of the sum on the recurrence kernels,
// with the unit-vector source added by a scatter after each step; H X is one more product with
// the local copies of H itself.
//
// FP32 with 9 orbitals: local_clenshaw runs all steps of a region inside one CTA (below).  FP64, one
// orbital, or a region whose panels exceed shared memory: one recurrence launch per step over all regions.
#include <algorithm>
#include <numeric>
#include <vector>

#include "cheb.cuh"
#include "scan.cuh"

namespace tbk {

// Position of value v in the ascending list c[lo .. hi), or -1.
__device__ __forceinline__ int find_in(const int32_t* __restrict__ c, int lo, int hi, int v) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    const int x = c[mid];
    if (x == v) return mid;
    if (x < v) lo = mid + 1; else hi = mid;
  }
  return -1;
}

// Region of merged index t: the a with rs[a] <= t < rs[a + 1].
__device__ __forceinline__ int region_of(const int32_t* __restrict__ rs, int n_atoms, int64_t t) {
  int lo = 0, hi = n_atoms;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (rs[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// Pass 1 (fill = false): cnt[t] = stored blocks of merged row t inside its region.  Pass 2 (fill):
// their local columns (merged indices) and global block indices, at lrp[t].
template <bool FILL>
__global__ void local_pattern(int n_atoms, int64_t n_loc, const int32_t* __restrict__ rs, const int32_t* __restrict__ rcol,
                              const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                              int32_t* __restrict__ cnt, const int64_t* __restrict__ lrp, int32_t* __restrict__ lrow,
                              int32_t* __restrict__ lcol, int32_t* __restrict__ lblk) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_loc) return;
  const int a = region_of(rs, n_atoms, t);
  const int r0 = rs[a], r1 = rs[a + 1];
  const int g = rcol[t];
  int n = 0;
  int64_t o = FILL ? lrp[t] : 0;
  if (FILL) {
    lrow[t] = (int32_t)o;
    if (t == n_loc - 1) lrow[n_loc] = (int32_t)lrp[n_loc];
  }
  for (int k = rp[g]; k < rp[g + 1]; ++k) {
    const int j = find_in(rcol, r0, r1, col[k]);
    if (j < 0) continue;
    if (FILL) {
      lcol[o] = j;
      lblk[o] = k;
      ++o;
    }
    ++n;
  }
  if (!FILL) cnt[t] = n;
}

// size[a] = (atoms, stored blocks) of region a.
__global__ void region_sizes(int n_atoms, const int32_t* __restrict__ rs, const int64_t* __restrict__ lrp,
                             int64_t* __restrict__ size) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_atoms) return;
  size[2 * a] = rs[a + 1] - rs[a];
  size[2 * a + 1] = lrp[rs[a + 1]] - lrp[rs[a]];
}

// ---- all steps of a region in one CTA (FP32, 9 orbitals) ------------------------------------------
//
// b_k = 2 H^ b_{k+1} - b_{k+2} + c_k E, X = H^ b_1 - b_2 + c_0 E, Y = H X for one region after another:
// the two panels and as many mapped blocks as fit stay in shared memory, the other blocks come from L2 (the
// same share of every row, so that all warps read both; the longest rows first, so that a warp's ten have
// about one length).  Three lanes form an atom's 9 x 9 tile, 9 x 3 entries each: 12 reads serve 27 FMAs.
// What binds are these reads: L1 delivers 32 floats a cycle and SM, whatever lanes they go to, and looks up
// ten atoms' blocks one after the other.  Each entry adds its blocks in the order of the step kernel and
// rounds where it does.  One launch per step reads copies of the blocks (140 MB) and the panels of all
// regions instead.  500 atoms, 6 A, 126 terms: 10.9 ms so, 4.9 ms here; other tiles: 3 x 3 entries per lane
// 5.5 ms, 1 x 9 7.1 ms, 5 x 3 7.1 ms, 1 x 3 (one atom per warp) 8.0 ms.
constexpr int LC_THREADS = 256, LC_ATOMS = 10, LC_HB = Layout<float, 9>::BS, LC_BS = 81, LC_ROW = 9;

struct LocalArgs {
  int n_atoms, p, max_m, max_nnz, n_stage;  // n_stage: blocks in shared memory
  const int32_t *order, *rs, *lrow, *lcol, *lblk, *own;
  const float *hv, *h1;                     // mapped blocks; H itself (NULL: no Y)
  const double* coef;
  float *X, *Y;
  int* next;
};

__device__ __forceinline__ void local_stage(const LocalArgs& A, const float* __restrict__ hv, float* hs, const int2* stage,
                                            int r0, int m) {
  for (int t = threadIdx.x >> 5; t < m; t += LC_THREADS / 32) {
    const int kb = A.lrow[r0 + t];
    for (int e = threadIdx.x & 31; e < stage[t].y * LC_BS; e += 32) {
      const int k = e / LC_BS, j = e - k * LC_BS, l = j / 9;
      hs[stage[t].x * LC_BS + e] = __ldg(hv + (int64_t)__ldg(A.lblk + kb + k) * LC_HB + j + 3 * l);
    }
  }
}

// out = alpha h in - out (SUB) or alpha h in, + c at the unit vectors of the atom at position o.
template <bool SUB>
__device__ __forceinline__ void local_step(const LocalArgs& A, const float* __restrict__ hv, const float* hs,
                                           const int* idx, const int* perm, const int2* stage, int r0, int m,
                                           int k0, const float* in, float* out, float alpha, double c, int o) {
  const int lane = threadIdx.x & 31, sub = lane / 3, gc = lane - 3 * sub;
  for (int q = LC_ATOMS * (threadIdx.x >> 5) + sub; q < m && sub < LC_ATOMS; q += LC_ATOMS * (LC_THREADS / 32)) {
    const int t = perm[q];
    const int kb = __ldg(A.lrow + r0 + t) - k0, ke = __ldg(A.lrow + r0 + t + 1) - k0;
    float acc[9][3];
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
      for (int v = 0; v < 3; ++v) acc[i][v] = 0.f;
    auto block = [&](const float* x, auto&& column) {
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        const float u[3] = {x[l * 9], x[l * 9 + 1], x[l * 9 + 2]};
        float h[9];
        column(l, h);
#pragma unroll
        for (int i = 0; i < 9; ++i)
#pragma unroll
          for (int v = 0; v < 3; ++v) acc[i][v] = fmaf(h[i], u[v], acc[i][v]);
      }
    };
    int k = kb;
    const int2 st = stage[t];  // its blocks in shared memory: first slot, number
    const float* p = hs + st.x * LC_BS;
    for (const int ks = kb + st.y; k < ks; ++k, p += LC_BS)
      block(in + idx[k] + 3 * gc, [&](int l, float (&h)[9]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = p[l * 9 + i];
      });
    for (; k < ke; ++k) {
      const float* g = hv + (int64_t)__ldg(A.lblk + k0 + k) * LC_HB;
      block(in + idx[k] + 3 * gc, [&](int l, float (&h)[9]) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(g + l * 12)), b = __ldg(reinterpret_cast<const float4*>(g + l * 12 + 4));
        h[0] = a.x; h[1] = a.y; h[2] = a.z; h[3] = a.w;
        h[4] = b.x; h[5] = b.y; h[6] = b.z; h[7] = b.w;
        h[8] = __ldg(g + l * 12 + 8);
      });
    }
    float* y = out + t * 81 + 3 * gc;
#pragma unroll
    for (int j = 0; j < 9; ++j)
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        float r = alpha * acc[j][v];
        if (SUB) r -= y[j * 9 + v];
        if (t == o && j == 3 * gc + v && c != 0.0) r = (float)((double)r + c);
        y[j * 9 + v] = r;
      }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(LC_THREADS, 2) local_clenshaw(const __grid_constant__ LocalArgs A) {
  extern __shared__ __align__(16) float lsm[];
  float* pa = lsm;
  float* pb = pa + A.max_m * 9 * LC_ROW;
  float* hs = pb + A.max_m * 9 * LC_ROW;
  int2* stage = reinterpret_cast<int2*>(hs + (((int64_t)A.n_stage * LC_BS + 1) & ~(int64_t)1));
  int* perm = reinterpret_cast<int*>(stage + A.max_m);
  int* idx = perm + A.max_m;
  __shared__ int job, slots;
  for (;;) {
    if (threadIdx.x == 0) {
      job = atomicAdd(A.next, 1);
      slots = 0;
    }
    __syncthreads();
    const int q = job;
    if (q >= A.n_atoms) return;
    const int r = A.order[q], r0 = A.rs[r], m = A.rs[r + 1] - r0;
    const int k0 = A.lrow[r0], nnz = A.lrow[r0 + m] - k0, o = A.own[r] - r0;
    const int n_el = m * 9 * LC_ROW;
    // idx: a block's column offset in the panels; perm: the rows, the longest first; stage: the share of
    // a row's blocks that lies in shared memory (the same for every row: all warps read both spaces)
    const int64_t share = (int64_t)min(A.n_stage, nnz) * 65536 / max(nnz, 1);
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < nnz; k += LC_THREADS) idx[k] = (A.lcol[k0 + k] - r0) * 9 * LC_ROW;
    for (int t = threadIdx.x >> 5; t < m; t += LC_THREADS / 32) {
      const int len = A.lrow[r0 + t + 1] - A.lrow[r0 + t];
      int rank = 0;
      if (lane == 0) {
        const int n = (int)(len * share >> 16);
        stage[t] = make_int2(atomicAdd(&slots, n), n);
      }
      for (int u = lane; u < m; u += 32) {
        const int lu = A.lrow[r0 + u + 1] - A.lrow[r0 + u];
        rank += lu > len || (lu == len && u < t);
      }
      rank = __reduce_add_sync(0xffffffffu, rank);
      if (lane == 0) perm[rank] = t;
    }
    for (int e = threadIdx.x; e < n_el; e += LC_THREADS) pa[e] = pb[e] = 0.f;
    __syncthreads();
    local_stage(A, A.hv, hs, stage, r0, m);
    if (threadIdx.x < 9) pa[(o * 9 + threadIdx.x) * LC_ROW + threadIdx.x] = (float)A.coef[A.p - 1];
    __syncthreads();
    float *b1 = pa, *b2 = pb;
    for (int k = A.p - 2; k >= 0; --k) {
      local_step<true>(A, A.hv, hs, idx, perm, stage, r0, m, k0, b1, b2, k ? 2.f : 1.f, A.coef[k], o);
      float* t = b1;
      b1 = b2;
      b2 = t;
    }
    auto store = [&](const float* v, float* dst) {
      for (int e = threadIdx.x; e < n_el; e += LC_THREADS)
        dst[((int64_t)r0 * 9 + e / 9) * 12 + e % 9] = v[e];  // panel rows of 12
    };
    store(b1, A.X);
    if (A.h1) {
      local_stage(A, A.h1, hs, stage, r0, m);
      __syncthreads();
      local_step<false>(A, A.h1, hs, idx, perm, stage, r0, m, k0, b1, b2, 1.f, 0.0, o);
      store(b2, A.Y);
    }
    __syncthreads();  // the next region overwrites the panels
  }
}

// The local copy of every mapped block: dst[k] = src[blk[k]] (BS elements each).
template <typename T>
__global__ void gather_blocks(int64_t nnz, int BS, const int32_t* __restrict__ blk, const T* __restrict__ src,
                              T* __restrict__ dst) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nnz * BS) return;
  const int64_t k = i / BS;
  dst[i] = src[(int64_t)blk[k] * BS + (i - k * BS)];
}

// own[a] = merged index of atom a inside its own region.
__global__ void own_index(int n_atoms, const int32_t* __restrict__ rs, const int32_t* __restrict__ rcol,
                          int32_t* __restrict__ own, int* __restrict__ err) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_atoms) return;
  const int j = find_in(rcol, rs[a], rs[a + 1], a);
  if (j < 0) atomicOr(err, 1);
  own[a] = j < 0 ? rs[a] : j;
}

// panel[(own[a] B + c) S + c] += alpha for every atom a and c < B (the unit vectors E).
template <typename T>
__global__ void add_units(int n_atoms, int B, int S, const int32_t* __restrict__ own, double alpha,
                          T* __restrict__ panel) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)n_atoms * B) return;
  const int a = (int)(i / B), c = (int)(i - (int64_t)a * B);
  T* p = panel + ((int64_t)own[a] * B + c) * S + c;
  *p = (T)((double)*p + alpha);
}

// out[k][l][c] = X[(loc B + l) S + c] for every stored block k = (b, a) of M, loc = the merged
// index of b in a's region: rows b of column block a.
template <typename T>
__global__ void local_extract(int n_atoms, int B, int S, const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                              const int32_t* __restrict__ rs, const int32_t* __restrict__ rcol,
                              const T* __restrict__ X, double* __restrict__ out, int* __restrict__ err) {
  const int b = blockIdx.x * blockDim.y + threadIdx.y;
  if (b >= n_atoms) return;
  for (int k = rp[b]; k < rp[b + 1]; ++k) {
    const int a = col[k];
    const int loc = find_in(rcol, rs[a], rs[a + 1], b);
    for (int e = threadIdx.x; e < B * B; e += blockDim.x) {
      const int l = e / B, c = e - l * B;
      double v = 0.0;
      if (loc < 0) {
        if (e == 0) atomicOr(err, 1);
      } else {
        v = (double)X[((int64_t)loc * B + l) * S + c];
      }
      out[(int64_t)k * B * B + e] = v;
    }
  }
}

}  // namespace tbk

using namespace tbk;

extern "C" int tbk_local_density(tbk_ctx* ctx, const tbk_bsr* H, const double* pos, const double* box,
                                 double r_max, double emin, double emax, int32_t order, double mu, double kT,
                                 int32_t damping, int32_t flags, double* P, double* Q) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr && H != nullptr && pos != nullptr, "NULL argument");
  TBK_CHECK_ARG(P || Q, "nothing to compute: P and Q are both NULL");
  TBK_CHECK_ARG(order >= 1, "order must be >= 1");
  TBK_CHECK_ARG(r_max > 0.0, "r_max must be positive");
  TBK_CHECK_ARG((flags & ~TBK_FP64) == 0, "unknown flag");
  TBK_CHECK_ARG(kT > 0.0, "kT must be positive");
  DeviceGuard dg(ctx);
  const int prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  const int n = H->n_atoms, B = H->n_orb, p = order;
  const int S = 4 * ((B + 3) / 4);                 // panel width: the B unit vectors, padded

  // 1. regions: the atoms within r_max of each atom (CSR, ascending)
  int32_t* rs = (int32_t*)scratch(ctx, WS_LOCAL0, sizeof(int32_t) * ((size_t)n + 1));
  int64_t n_loc = 0;
  int rc = tbk_build_neighbors(ctx, pos, n, box, r_max, rs, nullptr, 0, &n_loc);
  if (rc != TBK_OK) throw Error(rc, tbk_last_error());
  TBK_CHECK_ARG(n_loc < INT32_MAX, "the regions hold too many atoms");
  int32_t* rcol = (int32_t*)scratch(ctx, WS_LOCAL1, sizeof(int32_t) * (size_t)std::max<int64_t>(1, n_loc));
  rc = tbk_build_neighbors(ctx, pos, n, box, r_max, rs, rcol, n_loc, &n_loc);
  if (rc != TBK_OK) throw Error(rc, tbk_last_error());

  int* err = (int*)scratch(ctx, WS_FLAGS, 64);
  TBK_CUDA(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
  // 2. the local pattern: M restricted to each region, merged
  int32_t* cnt = (int32_t*)scratch(ctx, WS_LOCAL2, sizeof(int32_t) * ((size_t)n_loc + 2 * (size_t)n) + 64);
  int32_t* own = cnt + n_loc;
  int32_t* d_order = own + n;  // and the counter of regions taken
  local_pattern<false><<<ceil_div(n_loc, 256), 256, 0, ctx->stream>>>(n, n_loc, rs, rcol, H->row_ptr, H->col, cnt,
                                                                       nullptr, nullptr, nullptr, nullptr);
  post_launch(ctx, "local_pattern");
  const size_t scan_n = (size_t)n_loc + 1 + scan_tmp_elems(n_loc);
  int64_t* lrp = (int64_t*)scratch(ctx, WS_LOCAL3, sizeof(int64_t) * (scan_n + 2 * (size_t)n));
  int64_t* d_size = lrp + scan_n;
  exclusive_scan_i32(ctx, cnt, lrp, n_loc, lrp + n_loc + 1);
  region_sizes<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(n, rs, lrp, d_size);
  post_launch(ctx, "region_sizes");
  int64_t nnz_loc = 0;
  std::vector<int64_t> size(2 * (size_t)n);
  TBK_CUDA(cudaMemcpyAsync(&nnz_loc, lrp + n_loc, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
  TBK_CUDA(cudaMemcpyAsync(size.data(), d_size, sizeof(int64_t) * size.size(), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  TBK_CHECK_ARG(nnz_loc < INT32_MAX, "the local operators hold too many blocks");
  int32_t* lrow = (int32_t*)scratch(ctx, WS_LOCAL4, sizeof(int32_t) * ((size_t)n_loc + 1 + 2 * (size_t)nnz_loc));
  int32_t* lcol = lrow + n_loc + 1;
  int32_t* lblk = lcol + nnz_loc;
  local_pattern<true><<<ceil_div(n_loc, 256), 256, 0, ctx->stream>>>(n, n_loc, rs, rcol, H->row_ptr, H->col, nullptr,
                                                                      lrp, lrow, lcol, lblk);
  post_launch(ctx, "local_pattern");
  own_index<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(n, rs, rcol, own, err);
  post_launch(ctx, "own_index");

  const dim3 eb(32, 8);
  auto extract = [&](const void* Y, double* out) {
    if (prec == TBK_MIXED)
      local_extract<float><<<ceil_div(n, 8), eb, 0, ctx->stream>>>(n, B, S, H->row_ptr, H->col, rs, rcol,
                                                                   (const float*)Y, out, err);
    else
      local_extract<double><<<ceil_div(n, 8), eb, 0, ctx->stream>>>(n, B, S, H->row_ptr, H->col, rs, rcol,
                                                                    (const double*)Y, out, err);
    post_launch(ctx, "local_extract");
  };
  double* dcoef = (double*)scratch(ctx, WS_COEF, sizeof(double) * (size_t)p);
  coefficients(ctx, TBK_FN_FERMI, p, emin, emax, mu, kT, damping, dcoef);
  const size_t esz = prec == TBK_MIXED ? 4 : 8;
  const size_t panel = (size_t)n_loc * B * S * esz;

  // 3a. FP32, 9 orbitals, panels and block list in shared memory: whole regions per CTA, the largest first
  LocalArgs la{};
  for (int a = 0; a < n; ++a) {
    la.max_m = std::max(la.max_m, (int)std::min<int64_t>(size[2 * a], 1 << 20));
    la.max_nnz = std::max(la.max_nnz, (int)std::min<int64_t>(size[2 * a + 1], 1 << 24));
  }
  const int64_t smem_fix = 2 * (int64_t)la.max_m * 9 * LC_ROW * 4 + ((int64_t)la.max_nnz + 3 * (int64_t)la.max_m) * 4;
  // two CTAs per SM where their panels fit (500 atoms, 6 A: 4.9 ms; one with more blocks in shared memory 5.7)
  const int per_sm = smem_fix <= (110 << 10) ? 2 : 1;
  const int64_t smem_max = per_sm == 2 ? 110 << 10 : 226 << 10;
  if (prec == TBK_MIXED && B == 9 && smem_fix <= smem_max) {
    std::vector<int32_t> ord((size_t)n + 1);
    std::iota(ord.begin(), ord.end() - 1, 0);
    std::stable_sort(ord.begin(), ord.end() - 1, [&](int a, int b) { return size[2 * a + 1] > size[2 * b + 1]; });
    ord[n] = 0;
    TBK_CUDA(cudaMemcpyAsync(d_order, ord.data(), sizeof(int32_t) * ord.size(), cudaMemcpyHostToDevice, ctx->stream));
    la.n_atoms = n;
    la.p = p;
    la.n_stage = (int)std::min<int64_t>(la.max_nnz, (smem_max - smem_fix) / (LC_BS * 4));
    la.order = d_order;
    la.next = d_order + n;
    la.rs = rs;
    la.lrow = lrow;
    la.lcol = lcol;
    la.lblk = lblk;
    la.own = own;
    la.hv = (const float*)prepare_hop(ctx, H, emin, emax, prec, WS_HHAT, err).hv;
    la.h1 = Q ? (const float*)prepare_hop(ctx, H, -1.0, 1.0, prec, WS_SEGMENT, err).hv : nullptr;
    la.coef = dcoef;
    la.X = (float*)scratch(ctx, WS_CHECKPOINTS, 2 * panel);
    la.Y = la.X + panel / 4;
    const int smem = (int)(smem_fix + (int64_t)la.n_stage * LC_BS * 4) + 16;
    TBK_CUDA(cudaFuncSetAttribute(local_clenshaw, cudaFuncAttributeMaxDynamicSharedMemorySize, (226 << 10) + 16));
    local_clenshaw<<<std::min(n, per_sm * ctx->num_sms), LC_THREADS, smem, ctx->stream>>>(la);
    post_launch(ctx, "local_clenshaw");
    if (P) extract(la.X, P);
    if (Q) extract(la.Y, Q);
    int herr = 0;
    TBK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    sync(ctx);  // also: ord stays until its copy is done
    check_diagonal_flag(herr);
    TBK_CHECK_ARG(herr == 0, "a stored block of H joins atoms farther apart than r_max");
    return TBK_OK;
  }

  // 3b. local copies of the mapped blocks (H^ for X; H itself, the bounds [-1, 1], for H X)
  const int BS = prec == TBK_MIXED ? (B == 1 ? Layout<float, 1>::BS : Layout<float, 9>::BS)
                                   : (B == 1 ? Layout<double, 1>::BS : Layout<double, 9>::BS);
  void* hv_loc = scratch(ctx, WS_SEGMENT, (size_t)nnz_loc * BS * esz);
  auto local_operator = [&](double lo, double hi) {
    HOp g = prepare_hop(ctx, H, lo, hi, prec, WS_HHAT, err);
    const int64_t tot = nnz_loc * BS;
    if (prec == TBK_MIXED)
      gather_blocks<float><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(nnz_loc, BS, lblk, (const float*)g.hv,
                                                                                  (float*)hv_loc);
    else
      gather_blocks<double><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(nnz_loc, BS, lblk, (const double*)g.hv,
                                                                                   (double*)hv_loc);
    post_launch(ctx, "gather_blocks");
    HOp o;
    o.n_atoms = (int)n_loc;
    o.B = B;
    o.prec = prec;
    o.nnzb = nnz_loc;
    o.n_rows = n_loc * B;
    o.row_ptr = lrow;
    o.col = lcol;
    o.hv = hv_loc;
    return o;
  };
  HOp op = local_operator(emin, emax);

  // 4. coefficients of p_f, then X = p_f(H^) E by the Clenshaw form with unit-vector sources
  std::vector<double> c(p);
  TBK_CUDA(cudaMemcpyAsync(c.data(), dcoef, sizeof(double) * p, cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  char* base = (char*)scratch(ctx, WS_CHECKPOINTS, 3 * panel);
  void* B1 = base;
  void* B2 = base + panel;
  void* X = base + 2 * panel;
  auto add_e = [&](void* pnl, double alpha) {
    if (alpha == 0.0) return;
    const int64_t tot = (int64_t)n * B;
    if (prec == TBK_MIXED)
      add_units<float><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(n, B, S, own, alpha, (float*)pnl);
    else
      add_units<double><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(n, B, S, own, alpha, (double*)pnl);
    post_launch(ctx, "add_units");
  };
  auto step = [&](const HOp& o, const void* yin, void* yprev, void* yout, double alpha) {
    StepArgs a;
    a.yin = yin;
    a.yprev = yprev;
    a.yout = yout;
    a.alpha = alpha;
    a.s = S;
    a.err = err;
    a.force_simple = 1;
    launch_step(ctx, o, a);
  };
  TBK_CUDA(cudaMemsetAsync(X, 0, panel, ctx->stream));
  if (p == 1) {
    add_e(X, c[0]);
  } else {
    TBK_CUDA(cudaMemsetAsync(B1, 0, panel, ctx->stream));
    add_e(B1, c[p - 1]);                           // b_{p-1} = alpha_{p-1} E
    void *bk1 = B1, *bk2 = nullptr;
    for (int k = p - 2; k >= 1; --k) {
      void* out = bk2 ? bk2 : B2;
      step(op, bk1, bk2, out, 2.0);                // 2 H^ b_{k+1} - b_{k+2}
      add_e(out, c[k]);                            // + alpha_k E
      bk2 = bk1;
      bk1 = out;
    }
    step(op, bk1, bk2, X, 1.0);                    // X = H^ b_1 - b_2 + alpha_0 E
    add_e(X, c[0]);
  }
  if (P) extract(X, P);
  if (Q) {
    HOp h1 = local_operator(-1.0, 1.0);
    step(h1, X, nullptr, B1, 1.0);                 // H X
    extract(B1, Q);
  }
  int herr = 0;
  TBK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  check_diagonal_flag(herr);
  TBK_CHECK_ARG(herr == 0, "a stored block of H joins atoms farther apart than r_max");
  TBK_API_END
}
