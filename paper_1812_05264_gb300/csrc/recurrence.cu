// a5-a7: the fused block-SpMM Chebyshev recurrence with in-kernel probe generation and moment
// partial sums (Sec. II.B.1 Eq. poly_PQ with S = I; Sec. II.C.2 random approximation).
#include <algorithm>
#include <cmath>
#include <mutex>

#include "bulk.cuh"
#include "cheb.cuh"
#include "sums.cuh"

namespace tbk {

template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; static constexpr int N = 4; };
template <> struct Vec16<double> { using type = double2; static constexpr int N = 2; };

template <typename T>
__device__ __forceinline__ void ld16(const T* p, T* x) {
  if constexpr (sizeof(T) == 4) {
    float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  } else {
    double2 v = *reinterpret_cast<const double2*>(p);
    x[0] = v.x; x[1] = v.y;
  }
}
template <typename T>
__device__ __forceinline__ void ldg16(const T* p, T* x) {
  if constexpr (sizeof(T) == 4) {
    float4 v = __ldg(reinterpret_cast<const float4*>(p));
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  } else {
    double2 v = __ldg(reinterpret_cast<const double2*>(p));
    x[0] = v.x; x[1] = v.y;
  }
}
template <typename T>
__device__ __forceinline__ void st16(T* p, const T* x) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
  }
}

// ---- H^ in the padded kernel layout --------------------------------------------------------

// One warp per block row, element by element (lanes over a block's 81; 1 x 1 blocks: eight lanes over the row, whose
// seven blocks leave most of a warp idle):
// reads are coalesced and the FP64 product and conversion, the two that bind (an SM takes about 19
// cycles for a warp's), run for stored elements only.  One thread per block: 34 us at 1,000 atoms, 188 at
// 10,000; so 18 and 99.
constexpr int MAP_THREADS = 128;
template <int B>
constexpr int map_lanes() { return B == 1 ? 8 : 32; }
static int map_grid(const HOp& op) { return ceil_div(op.n_atoms, MAP_THREADS / (op.B == 1 ? map_lanes<1>() : map_lanes<9>())); }

template <typename T, int B>
__global__ void __launch_bounds__(MAP_THREADS)
map_h_kernel(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
             const double* __restrict__ H, double shift, double inv_half_w, T* __restrict__ out, int* __restrict__ err) {
  constexpr int RS = Layout<T, B>::RS, BS = Layout<T, B>::BS;
  constexpr int L = map_lanes<B>();
  const int a = blockIdx.x * (MAP_THREADS / L) + threadIdx.x / L, lane = threadIdx.x % L;
  if (a >= n_atoms) return;
  bool has_diag = false;
  const int k1 = row_ptr[a + 1];
  if constexpr (B == 1) {
    for (int k = row_ptr[a] + lane; k < k1; k += L) {
      const bool diag = col[k] == a;
      has_diag |= diag;
      double v = H[k];
      if (diag) v -= shift;
      out[k] = (T)(v * inv_half_w);
    }
  } else {
#pragma unroll 4
    for (int k = row_ptr[a]; k < k1; ++k) {
      const bool diag = col[k] == a;
      has_diag |= diag;
      T* o = out + (int64_t)k * BS;
#pragma unroll
      for (int e = lane; e < 96; e += 32) {
        if (e >= B * B) continue;
        const int i = e / B, j = e - i * B;
        double v = H[(int64_t)k * (B * B) + e];
        if (diag && i == j) v -= shift;
        // H^[i][j] row-major, or column-major
        o[Layout<T, B>::COLMAJOR ? j * RS + i : i * RS + j] = (T)(v * inv_half_w);
      }
      if (lane < B * (RS - B)) o[lane / (RS - B) * RS + B + lane % (RS - B)] = T(0);
    }
  }
  const unsigned row_mask = L == 32 ? 0xffffffffu : ((1u << L) - 1) << (threadIdx.x & 31 & ~(L - 1));
  if (!__any_sync(row_mask, has_diag) && lane == 0) atomicOr(err, ERR_NO_DIAGONAL);
}

HOp prepare_hop(tbk_ctx* ctx, const tbk_bsr* H, double emin, double emax, int prec, Slot slot, int* err) {
  TBK_CHECK_ARG(H != nullptr, "H is NULL");
  TBK_CHECK_ARG(H->n_orb == 1 || H->n_orb == 9, "n_orb must be 1 or 9");
  TBK_CHECK_ARG(H->n_atoms >= 1 && H->nnzb >= H->n_atoms, "empty or inconsistent matrix");
  TBK_CHECK_ARG(H->row_ptr && H->col && H->val, "NULL matrix array");
  TBK_CHECK_ARG(H->nnzb < INT32_MAX, "nnzb must be below 2^31");
  TBK_CHECK_ARG(std::isfinite(emin) && std::isfinite(emax) && emax > emin, "need emax > emin");
  TBK_CHECK_ARG(prec == TBK_MIXED || prec == TBK_FP64, "unknown precision");
  HOp op;
  op.n_atoms = H->n_atoms;
  op.B = H->n_orb;
  op.prec = prec;
  op.nnzb = H->nnzb;
  op.n_rows = (int64_t)H->n_atoms * H->n_orb;
  op.row_ptr = H->row_ptr;
  op.col = H->col;
  const double shift = 0.5 * (emax + emin), inv = 2.0 / (emax - emin);
  const int blk = MAP_THREADS, grid = map_grid(op);
#define TBK_MAP(TT, BB)                                                                        \
  {                                                                                            \
    TT* out = (TT*)scratch(ctx, slot, sizeof(TT) * (size_t)op.nnzb * Layout<TT, BB>::BS);      \
    map_h_kernel<TT, BB><<<grid, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, H->val, \
                                                        shift, inv, out, err);                 \
    post_launch(ctx, "map_h_kernel");                                                          \
    op.hv = out;                                                                               \
  }
  if (prec == TBK_MIXED) {
    if (op.B == 9) TBK_MAP(float, 9) else TBK_MAP(float, 1)
  } else {
    if (op.B == 9) TBK_MAP(double, 9) else TBK_MAP(double, 1)
  }
#undef TBK_MAP
  return op;
}

// ---- the fused step --------------------------------------------------------------------------

constexpr int STEP_THREADS = 128;

// Further own-row terms of a step: sum_e c[e] p[e] (p[e] NULL: none).
template <typename T>
struct StepSources {
  const T* p[3];
  T c[3];
};

// SRC: with the further own-row terms.  Where none is asked for, the tests for them alone made FP64 steps of 1x1
// blocks, whose rows are short, 20 % slower (10,648 sites x 512 probes 138 -> 166 us).
template <typename T, int B, bool PROBE_IN, bool SRC>
__global__ void __launch_bounds__(STEP_THREADS)
cheb_step_kernel(const int n_atoms, const int32_t* __restrict__ row_ptr,
                 const int32_t* __restrict__ col, const T* __restrict__ hv,
                 const T* __restrict__ yin, const T* yprev, T* yout, const T alpha,
                 const T c_r, const uint64_t seed, const int s, const int direct, const StepSources<T> src,
                 double* __restrict__ partials) {
  constexpr int VEC = Vec16<T>::N;
  constexpr int RS = Layout<T, B>::RS, BS = Layout<T, B>::BS;
  // tasks: (row group, probe chunk) with chunk fastest; CTAs stride over tasks
  const int chunk_w = blockDim.x * VEC;
  const int n_chunks = (s + chunk_w - 1) / chunk_w;
  const int n_groups = (n_atoms + blockDim.y - 1) / blockDim.y;
  double sum0 = 0.0, sum1 = 0.0;
  for (int task = blockIdx.x; task < n_groups * n_chunks; task += gridDim.x) {
    const int grp = task / n_chunks, chunk = task - grp * n_chunks;
    const int p0 = chunk * chunk_w + threadIdx.x * VEC;
    const int a = grp * blockDim.y + threadIdx.y;
    if (p0 < s && a < n_atoms) {
      T acc[B][VEC];
#pragma unroll
      for (int i = 0; i < B; ++i)
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[i][v] = T(0);
      const int k1 = __ldg(row_ptr + a + 1);
      for (int k = __ldg(row_ptr + a); k < k1; ++k) {
        const int b = __ldg(col + k);
        T x[B][VEC];
#pragma unroll
        for (int l = 0; l < B; ++l) {
          const int64_t row = (int64_t)b * B + l;
          if constexpr (PROBE_IN) {
#pragma unroll
            for (int v = 0; v < VEC; ++v) x[l][v] = (T)tbk_probe_sign(seed, row, p0 + v);
          } else {
            ldg16(yin + row * s + p0, x[l]);
          }
        }
        const T* h = hv + (int64_t)k * BS;
        if constexpr (Layout<T, B>::COLMAJOR) {
          // column l of the block against row l of the tile; each acc[i] still sums l = 0..8
#pragma unroll
          for (int l = 0; l < B; ++l) {
            T hc[RS];
#pragma unroll
            for (int j = 0; j < RS; j += VEC) ldg16(h + l * RS + j, hc + j);
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
              for (int v = 0; v < VEC; ++v) acc[i][v] = fma(hc[i], x[l][v], acc[i][v]);
          }
        } else {
#pragma unroll
          for (int i = 0; i < B; ++i) {
            T hr[RS];
            if constexpr (B == 1) {
              hr[0] = __ldg(h);
            } else {
#pragma unroll
              for (int j = 0; j < RS; j += VEC) ldg16(h + i * RS + j, hr + j);
            }
#pragma unroll
            for (int l = 0; l < B; ++l)
#pragma unroll
              for (int v = 0; v < VEC; ++v) acc[i][v] = fma(hr[l], x[l][v], acc[i][v]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < B; ++i) {
        const int64_t row = (int64_t)a * B + i;
        const int64_t off = row * s + p0;
        T yo[VEC], r[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) yo[v] = alpha * acc[i][v];
        if (c_r != T(0) || direct || PROBE_IN) {
#pragma unroll
          for (int v = 0; v < VEC; ++v) r[v] = (T)tbk_probe_sign(seed, row, p0 + v);
        }
        if (c_r != T(0)) {
#pragma unroll
          for (int v = 0; v < VEC; ++v) yo[v] = fma(c_r, r[v], yo[v]);
        }
        if (yprev) {
          T t[VEC];
          ld16(yprev + off, t);
#pragma unroll
          for (int v = 0; v < VEC; ++v) yo[v] -= t[v];
        }
        if constexpr (SRC) {
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (src.p[e]) {
              T t[VEC];
              ldg16(src.p[e] + off, t);
#pragma unroll
              for (int v = 0; v < VEC; ++v) yo[v] = fma(src.c[e], t[v], yo[v]);
            }
        }
        st16(yout + off, yo);
        if (partials) {
          T xin[VEC];
          if (direct || PROBE_IN) {
#pragma unroll
            for (int v = 0; v < VEC; ++v) xin[v] = r[v];
          } else {
            ldg16(yin + off, xin);
          }
          T q0 = T(0), q1 = T(0);
#pragma unroll
          for (int v = 0; v < VEC; ++v) {
            q0 = fma(yo[v], xin[v], q0);
            q1 = fma(yo[v], yo[v], q1);
          }
          sum0 += (double)q0;
          sum1 += (double)q1;
        }
      }
    }
  }
  if (partials) {
    __shared__ double red[2][STEP_THREADS / 32];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nthreads = blockDim.x * blockDim.y;
    for (int o = 16; o > 0; o >>= 1) {
      sum0 += __shfl_xor_sync(0xffffffffu, sum0, o);
      sum1 += __shfl_xor_sync(0xffffffffu, sum1, o);
    }
    if ((tid & 31) == 0) {
      red[0][tid >> 5] = sum0;
      red[1][tid >> 5] = sum1;
    }
    __syncthreads();
    if (tid == 0) {
      double a0 = 0.0, a1 = 0.0;
      for (int w = 0; w < (nthreads + 31) / 32; ++w) {
        a0 += red[0][w];
        a1 += red[1][w];
      }
      partials[2 * blockIdx.x] = a0;
      partials[2 * blockIdx.x + 1] = a1;
    }
  }
}

// ---- TMA-fed step (FP32, 9x9 blocks, panel input) -------------------------------------------
//
// CTA = CW consumer warps + 1 producer warp.  A task is one block row a and a chunk of
// P = 128 CW probes (each consumer thread owns 4 consecutive probes).  The producer streams, for
// every neighbour block k = (a, b) of the task, the 9 x P tile of y_in rows 9b..9b+8 and the
// block H^_ab through a (D + 1)-stage shared-memory ring with cp.async.bulk copies completing on
// mbarriers, in stored order, then the row's own y_in tile a second time (when the moment sums
// need it) and the y_prev tile.  The consumers keep those last two stages until the epilogue
// has read them, so the epilogue reads nothing from global memory but the probe signs it
// regenerates (the second copy of the own tile is normally an L2 hit; holding the first one
// instead would stall the ring in the middle of the row).  Every wait is bounded: on expiry the
// CTA raises *err = 2 and leaves the loop, and the producer waits (bounded) for the copies it
// issued before returning.

template <int CW, int D>
struct BulkCfg {
  static constexpr int P = 128 * CW;                       // probes per task
  static constexpr int XB = 9 * P * 4;                      // tile bytes
  static constexpr int HB = Layout<float, 9>::BS * 4;       // 432 bytes
  static constexpr int SB = ((XB + HB + 127) / 128) * 128;  // stage bytes
  static constexpr int SMEM = (D + 1) * SB + 8 * (2 * D + 4);
  static constexpr int THREADS = 32 * (CW + 1);
};

// DENSE: seven CTAs per SM (80 registers).
template <int CW, int D, bool DENSE = false>
__global__ void __launch_bounds__(32 * (CW + 1), DENSE ? 7 : 4)
cheb_step_bulk(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const float* __restrict__ hv, const float* __restrict__ yin, const float* yprev,
               float* yout, const float alpha, const float c_r, const uint64_t seed, const int s,
               const int direct, double* __restrict__ partials, int* __restrict__ err,
               const BatchRows batch, const int per_task, const int stall) {
  using C = BulkCfg<CW, D>;
  // every tile, the diagonal one included, streams through a ring of R = D + 1 stages (R >= 2:
  // the epilogue holds two)
  constexpr int R = D + 1;
  static_assert(R >= 2, "the epilogue holds two stages");
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + R * C::SB);
  // bars: full[0..R), empty[R..2R)
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (R + i); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_chunks = s / C::P;
  const int n_tasks = n_atoms * n_chunks;
  const bool has_prev = yprev != nullptr;
  const bool own = partials != nullptr && !direct;  // the moment sums read the row's own y_in
  if (threadIdx.x == 0) {
    for (int i = 0; i < R; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), CW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();

  if (warp == CW) {
    // ---------------- producer ----------------
    // (stall: a test of the bounded waits; nothing is copied, the consumers give up and report)
    if (lane == 0 && !stall) {
      int it = 0;
      bool ok = true;
      for (int task = blockIdx.x; task < n_tasks && ok; task += gridDim.x) {
        const int a = task / n_chunks, ch = task - a * n_chunks;
        const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
        const int nb = k1 - k0;
        const int nt = nb + (own ? 1 : 0) + (has_prev ? 1 : 0);
        for (int q = 0; q < nt && ok; ++q) {
          // tiles: the nb neighbour tiles with their blocks, then the row's own y_in tile again
          // (own: for the moment sums), then y_prev
          const bool is_nb = q < nb, is_prev = q == nt - 1 && has_prev;
          const int k = k0 + q;
          const int b = is_nb ? __ldg(col + k) : a;
          const int st = it % R;
          ok = mbar_wait(empty(st), ((it / R) & 1) ^ 1);
          if (!ok) break;
          const uint32_t dst = smem_u32(smem + st * C::SB), bar = full(st);
          ++it;
          const float* src = (is_prev ? yprev : yin) + (int64_t)9 * b * s + (int64_t)ch * C::P;
          mbar_expect_tx(bar, C::XB + (is_nb ? C::HB : 0));
          if (C::P == s) {
            bulk_g2s(dst, src, C::XB, bar);
          } else {
            for (int l = 0; l < 9; ++l) bulk_g2s(dst + l * C::P * 4, src + (int64_t)l * s, C::P * 4, bar);
          }
          if (is_nb) bulk_g2s(dst + C::XB, hv + (int64_t)k * Layout<float, 9>::BS, C::HB, bar);
        }
      }
      if (!ok) {
        atomicOr(err, 2);
        // wait (bounded) for copies still in flight into the ring before leaving
        for (int j = (it > R ? it - R : 0); j < it; ++j) mbar_wait(full(j % R), (j / R) & 1);
      }
    }
    return;
  }

  // ---------------- consumers ----------------
  // After the neighbour tiles come the row's own y_k tile (own) and the y_prev tile: both stay in
  // the ring (their stages are released after the epilogue, in order) and the epilogue reads them
  // from shared memory.
  double sum0 = 0.0, sum1 = 0.0;
  int it = 0;
  bool ok = true;
  uint32_t rdy = 0;  // stage it % R was found ready by the early test
  for (int task = blockIdx.x; task < n_tasks && ok; task += gridDim.x) {
    const int a = task / n_chunks, ch = task - a * n_chunks;
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    const int nb = k1 - k0;
    const int pl = 4 * threadIdx.x;  // probe offset inside the chunk
    float2 acc[9][2];  // row i, probe v: acc_at(acc, i, v)
#pragma unroll
    for (int i = 0; i < 9; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    int held = 0;  // stages held for the epilogue, starting at it - held
    for (int q = 0; q < nb; ++q) {
      const int st = it % R;
      if (!rdy) ok = mbar_wait(full(st), (it / R) & 1);
      ok = __all_sync(0xffffffffu, ok);  // one decision per warp: the warps meet at a barrier below
      if (!ok) break;
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      const unsigned char* base = smem + st * C::SB;
      const float* X = reinterpret_cast<const float*>(base);
      const float* Hs = reinterpret_cast<const float*>(base + C::XB);
      spmm_tile_f2(X, Hs, C::P, pl, acc);
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(st));
      ++it;
    }
    if (!ok) break;
    const float* Xown = nullptr;
    const float* Xprev = nullptr;
    if (own) {
      const int st = it % R;
      if (!rdy) ok = mbar_wait(full(st), (it / R) & 1);
      ok = __all_sync(0xffffffffu, ok);  // one decision per warp: the warps meet at a barrier below
      if (!ok) break;
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      Xown = reinterpret_cast<const float*>(smem + st * C::SB);
      ++held;
      ++it;
    }
    if (has_prev) {
      const int st = it % R;
      if (!rdy) ok = mbar_wait(full(st), (it / R) & 1);
      ok = __all_sync(0xffffffffu, ok);  // one decision per warp: the warps meet at a barrier below
      if (!ok) break;
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      Xprev = reinterpret_cast<const float*>(smem + st * C::SB);
      ++held;
      ++it;
    }
    // epilogue: y_out = alpha acc + c_r r - y_prev, moment partial sums
    const int p0 = ch * C::P + pl;
    uint64_t sd = seed;          // probe stream and row index within the cluster
    int64_t rloc = (int64_t)9 * a;
    if (batch.atom_cl) {
      const int cl = __ldg(batch.atom_cl + a);
      sd = __ldg(batch.seed + cl);
      rloc = (int64_t)9 * (a - __ldg(batch.atom0 + cl));
    }
    float cs0 = 0.f, cc0 = 0.f, cs1 = 0.f, cc1 = 0.f;  // the task's compensated partial sums
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int64_t row = (int64_t)9 * a + i;
      float yo[4], r[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) yo[v] = alpha * acc_at(acc, i, v);
      if (c_r != 0.f || direct) {
#pragma unroll
        for (int v = 0; v < 4; ++v) r[v] = tbk_probe_sign(sd, rloc + i, p0 + v);
      }
      if (c_r != 0.f) {
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[v] = fmaf(c_r, r[v], yo[v]);
      }
      if (Xprev) {
        const float4 t = *reinterpret_cast<const float4*>(Xprev + i * C::P + pl);
        yo[0] -= t.x; yo[1] -= t.y; yo[2] -= t.z; yo[3] -= t.w;
      }
      *reinterpret_cast<float4*>(yout + row * s + p0) = make_float4(yo[0], yo[1], yo[2], yo[3]);
      if (partials) {
        float xin[4];
        if (direct) {
#pragma unroll
          for (int v = 0; v < 4; ++v) xin[v] = r[v];
        } else {
          // the row's own y_k from its held tile (Xown is set whenever these sums run: the global
          // read is never taken, but with it the kernel compiles to 96 registers without spills)
          const float4 t = Xown ? *reinterpret_cast<const float4*>(Xown + i * C::P + pl)
                                : __ldg(reinterpret_cast<const float4*>(yin + row * s + p0));
          xin[0] = t.x; xin[1] = t.y; xin[2] = t.z; xin[3] = t.w;
        }
        float q0 = 0.f, q1 = 0.f;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          q0 = fmaf(yo[v], xin[v], q0);
          q1 = fmaf(yo[v], yo[v], q1);
        }
        two_sum_acc(cs0, cc0, q0);
        two_sum_acc(cs1, cc1, q1);
      }
    }
    if (partials) {
      sum0 += (double)cs0 + (double)cc0;
      sum1 += (double)cs1 + (double)cc1;
    }
    // release the held stages in ring order
    __syncwarp();
    if (lane == 0)
      for (int h = held; h > 0; --h) mbar_arrive(empty((it - h) % R));
    if (per_task && partials) {
      // per (atom, warp) partial sums: no barrier between warps is needed
      for (int o = 16; o > 0; o >>= 1) {
        sum0 += __shfl_xor_sync(0xffffffffu, sum0, o);
        sum1 += __shfl_xor_sync(0xffffffffu, sum1, o);
      }
      if (lane == 0) {
        partials[2 * ((int64_t)a * CW + warp)] = sum0;
        partials[2 * ((int64_t)a * CW + warp) + 1] = sum1;
      }
      sum0 = sum1 = 0.0;
    }
  }
  if (!ok) atomicOr(err, 2);
  if (partials && !per_task) {
    __shared__ double red[2][8];
    for (int o = 16; o > 0; o >>= 1) {
      sum0 += __shfl_xor_sync(0xffffffffu, sum0, o);
      sum1 += __shfl_xor_sync(0xffffffffu, sum1, o);
    }
    if (lane == 0) {
      red[0][warp] = sum0;
      red[1][warp] = sum1;
    }
    // named barrier over the consumer warps only (the producer warp has returned)
    asm volatile("bar.sync 1, %0;" ::"r"(32 * CW) : "memory");
    if (threadIdx.x == 0) {
      double a0 = 0.0, a1 = 0.0;
      for (int w = 0; w < CW; ++w) {
        a0 += red[0][w];
        a1 += red[1][w];
      }
      partials[2 * blockIdx.x] = a0;
      partials[2 * blockIdx.x + 1] = a1;
    }
  }
}

// The lanes' sums of s0, in lanes 0..15, and of s1, in lanes 16..31: half the FP64 instructions of two butterflies.
__device__ __forceinline__ double lanes_sum2(double s0, double s1, int lane) {
  double a = lane < 16 ? s0 : s1;
  a += __shfl_xor_sync(0xffffffffu, lane < 16 ? s1 : s0, 16);
  for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// ---- self-fed step for 128-probe tasks ---------------------------------------------------------
//
// The same step as cheb_step_bulk<1, D> with one warp per CTA and no producer warp: lane 0 keeps
// R tiles in flight and, as soon as the warp has finished with a stage, refills it with the tile
// R positions ahead in the CTA's tile sequence (its tasks' neighbour tiles, then the y_prev tile
// of each task).  With 128 probes a task is quickly done, so a CTA that spends half its warps
// and registers on a producer limits how many consumers an SM holds.  NARROW: fewer than 128 probes, one
// narrower task a row (its tile is one contiguous copy); the lanes past the end compute on what the ring holds
// and store nothing.  Wider counts that are no multiple of 128 take the lane kernel.
template <int R>
struct SelfCfg {
  static constexpr int P = 128;
  static constexpr int XB = 9 * P * 4;
  static constexpr int HB = Layout<float, 9>::BS * 4;
  static constexpr int SB = ((XB + HB + 127) / 128) * 128;
  static constexpr int SMEM = R * SB + 8 * R;
};

template <int R, bool NARROW>
__global__ void __launch_bounds__(32)
cheb_step_self(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const float* __restrict__ hv, const float* __restrict__ yin, const float* yprev,
               float* yout, const float alpha, const float c_r, const uint64_t seed, const int s,
               const int direct, double* __restrict__ partials, int* __restrict__ err,
               const BatchRows batch, const int per_task, const int stall) {
  using C = SelfCfg<R>;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t bar0 = smem_u32(smem + R * C::SB);
  auto full = [&](int i) { return bar0 + 8u * i; };
  const int lane = threadIdx.x;
  const int n_chunks = NARROW ? 1 : s / C::P;
  const int P = NARROW ? s : C::P;  // floats between the rows of a tile
  const int n_tasks = n_atoms * n_chunks;
  const bool has_prev = yprev != nullptr;
  if (lane == 0) {
    for (int i = 0; i < R; ++i) mbar_init(full(i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  pdl_wait();
  // producer cursor (lane 0): the next tile to issue, as (task, tile index within the task)
  int p_task = blockIdx.x, p_q = 0, p_nt = 0, p_k0 = 0, issued = 0;
  auto load_task = [&]() {  // tasks with no tile (an empty row, no y_{k-1}) are skipped
    for (; p_task < n_tasks; p_task += gridDim.x) {
      const int a = p_task / n_chunks;
      p_k0 = __ldg(row_ptr + a);
      p_nt = __ldg(row_ptr + a + 1) - p_k0 + (has_prev ? 1 : 0);
      if (p_nt > 0) break;
    }
  };
  auto issue_next = [&]() {
    if (stall || p_task >= n_tasks) return;
    const int a = p_task / n_chunks, ch = p_task - a * n_chunks;
    const bool is_prev = p_q == p_nt - (has_prev ? 1 : 0) && has_prev;
    const int b = is_prev ? a : __ldg(col + p_k0 + p_q);
    const int st = issued % R;
    const uint32_t dst = smem_u32(smem + st * C::SB), bar = full(st);
    const float* src = (is_prev ? yprev : yin) + (int64_t)9 * b * s + (int64_t)ch * C::P;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    const int xb = NARROW ? 36 * s : C::XB;
    mbar_expect_tx(bar, xb + (is_prev ? 0 : C::HB));
    if (NARROW || s == C::P) {
      bulk_g2s(dst, src, xb, bar);  // the 9 rows are contiguous
    } else {
      for (int l = 0; l < 9; ++l) bulk_g2s(dst + l * C::P * 4, src + (int64_t)l * s, C::P * 4, bar);
    }
    if (!is_prev) bulk_g2s(dst + C::XB, hv + (int64_t)(p_k0 + p_q) * Layout<float, 9>::BS, C::HB, bar);
    ++issued;
    if (++p_q == p_nt) {
      p_task += gridDim.x;
      p_q = 0;
      load_task();
    }
  };
  if (lane == 0) {
    load_task();
    for (int j = 0; j < R; ++j) issue_next();
  }
  __syncwarp();

  double sum0 = 0.0, sum1 = 0.0;
  int it = 0;
  bool ok = true;
  uint32_t rdy = 0;  // stage it % R was found ready by the early test
  const int pl = 4 * lane;
  auto consumed = [&]() {
    // the warp is done with stage it % R: refill it with the tile R positions ahead
    __syncwarp();
    if (lane == 0) issue_next();
    ++it;
  };
  for (int task = blockIdx.x; task < n_tasks && ok; task += gridDim.x) {
    const int a = task / n_chunks, ch = task - a * n_chunks;
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    float2 acc[9][2];  // row i, probe v: acc_at_pp(acc, i, v)
#pragma unroll
    for (int i = 0; i < 9; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    for (int q = 0; q < k1 - k0; ++q) {
      const int st = it % R;
      if (!rdy) {
        ok = mbar_wait(full(st), (it / R) & 1);
        if (!ok) break;
      }
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      const unsigned char* base = smem + st * C::SB;
      spmm_tile_f2_pp(reinterpret_cast<const float*>(base), reinterpret_cast<const float*>(base + C::XB), P,
                      pl, acc);
      consumed();
    }
    if (!ok) break;
    float yp[9][4];
    if (has_prev) {
      const int st = it % R;
      if (!rdy) {
        ok = mbar_wait(full(st), (it / R) & 1);
        if (!ok) break;
      }
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      const float* X = reinterpret_cast<const float*>(smem + st * C::SB);
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        const float4 t = *reinterpret_cast<const float4*>(X + l * P + pl);
        yp[l][0] = t.x; yp[l][1] = t.y; yp[l][2] = t.z; yp[l][3] = t.w;
      }
      consumed();
    }
    const int p0 = ch * C::P + pl;
    if (NARROW && p0 >= s) continue;
    uint64_t sd = seed;
    int64_t rloc = (int64_t)9 * a;
    if (batch.atom_cl) {
      const int cl = __ldg(batch.atom_cl + a);
      sd = __ldg(batch.seed + cl);
      rloc = (int64_t)9 * (a - __ldg(batch.atom0 + cl));
    }
    // the task's partial sums, compensated; of narrow tasks in three floats, as good as the plain kernel's FP64 sums
    float cs0 = 0.f, cc0 = 0.f, cs1 = 0.f, cc1 = 0.f;
    Sum3 cs = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int64_t row = (int64_t)9 * a + i;
      float yo[4], r[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) yo[v] = alpha * acc_at_pp(acc, i, v);
      if (c_r != 0.f || direct) {
#pragma unroll
        for (int v = 0; v < 4; ++v) r[v] = tbk_probe_sign(sd, rloc + i, p0 + v);
      }
      if (c_r != 0.f) {
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[v] = fmaf(c_r, r[v], yo[v]);
      }
      if (has_prev) {
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[v] -= yp[i][v];
      }
      *reinterpret_cast<float4*>(yout + row * s + p0) = make_float4(yo[0], yo[1], yo[2], yo[3]);
      if (partials) {
        float xin[4];
        if (direct) {
#pragma unroll
          for (int v = 0; v < 4; ++v) xin[v] = r[v];
        } else {
          const float4 t = __ldg(reinterpret_cast<const float4*>(yin + row * s + p0));
          xin[0] = t.x; xin[1] = t.y; xin[2] = t.z; xin[3] = t.w;
        }
        float q0 = 0.f, q1 = 0.f;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          q0 = fmaf(yo[v], xin[v], q0);
          q1 = fmaf(yo[v], yo[v], q1);
        }
        if constexpr (NARROW) {
          sum3_add(cs, make_float2(q0, q1));
        } else {
          two_sum_acc(cs0, cc0, q0);
          two_sum_acc(cs1, cc1, q1);
        }
      }
    }
    if (partials) {
      sum0 += NARROW ? sum3_value(cs.h.x, cs.m.x, cs.l.x) : (double)cs0 + (double)cc0;
      sum1 += NARROW ? sum3_value(cs.h.y, cs.m.y, cs.l.y) : (double)cs1 + (double)cc1;
    }
    if (per_task && partials) {
      const double t = lanes_sum2(sum0, sum1, lane);
      if ((lane & 15) == 0) partials[2 * (int64_t)a + (lane >> 4)] = t;
      sum0 = sum1 = 0.0;
    }
  }
  if (!ok) {
    // let the copies in flight land before the CTA exits
    if (lane == 0) {
      atomicOr(err, 2);
      for (int j = it; j < issued; ++j) mbar_wait(full(j % R), (j / R) & 1);
    }
    return;
  }
  if (partials && !per_task) {
    const double t = lanes_sum2(sum0, sum1, lane);
    if ((lane & 15) == 0) partials[2 * blockIdx.x + (lane >> 4)] = t;
  }
}

// Sum of the consumer threads' partial sums into the CTA's slot (fixed order; the producer warp has
// returned or does not take part).
__device__ __forceinline__ void step_partials(double* __restrict__ partials, double sum0, double sum1, int warp,
                                              int lane, int nw) {
  __shared__ double red[2][32];
  const double a = lanes_sum2(sum0, sum1, lane);
  if ((lane & 15) == 0) red[lane >> 4][warp] = a;
  asm volatile("bar.sync 1, %0;" ::"r"(32 * nw) : "memory");
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += red[threadIdx.x][w];
    partials[2 * blockIdx.x + threadIdx.x] = t;
  }
}

// ---- one probe per lane: FP32 steps with little work per SM ------------------------------------------
//
// A task is a block row and a chunk of up to 512 probes; each consumer warp takes 32 probes, one per
// lane and all nine rows.  Where the chip is not full, a step lasts as long as one row does, and a
// row's time is that of a warp's instructions: a quarter of the self-fed kernel's per tile, with up
// to 8 tiles in flight instead of two.  A chunk is the whole panel width where that fits, so that a
// tile is one contiguous copy (nine row copies a tile cost 0.3 us more).  Per element the sums are
// the other kernels'.  The epilogue goes through shared memory to items of one row and four probes,
// so that panels are read and written 16 bytes at a time and the moment products add the same four
// probes as in the other kernels.  147 atoms x 128 probes: 8.3 us a step against 18.5 (self-fed
// kernel), 333 x 100: 9.7 against 22 (plain kernel, whose loads wait one after the other).
template <int NW>  // consumer warps at most: 4, 8 or 16
struct LaneCfg {
  static constexpr int R = NW == 16 ? 5 : 8;
  static constexpr int P = 32 * NW;
  static constexpr int XB = 9 * P * 4;
  static constexpr int HB = Layout<float, 9>::BS * 4;
  static constexpr int SB = ((XB + HB + 127) / 128) * 128;
  static constexpr int EB = 9 * 32 * 4;  // epilogue buffer of a warp
  static constexpr int SMEM = R * SB + NW * EB + 16 * R;
};

// ADJ: a step of the adjoint, with the further terms of `src` added in the fused adjoint kernel's order
// (y_k before y_prev, the others after) and no moment sums.  The other form asks for the CTAs per SM
// that shared memory gives: without the number the compiler took 80 registers and fetched less ahead (147 atoms x
// 200 probes 9.3 -> 10.6 us); with it the adjoint's, which needs 124, lost a tenth.
template <int NW, bool ADJ>
__global__ void __launch_bounds__(32 * (NW + 1), ADJ ? 0 : (NW == 4 ? 4 : (NW == 8 ? 2 : 1)))
cheb_step_lane(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const float* __restrict__ hv, const float* __restrict__ yin, const float* yprev, float* yout,
               const float alpha, const float c_r, const uint64_t seed, const int s, const int direct,
               const StepSources<float> src, double* __restrict__ partials, int* __restrict__ err,
               const int stall) {
  using C = LaneCfg<NW>;
  constexpr int R = C::R;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t bar0 = smem_u32(smem + R * C::SB + NW * C::EB);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (R + i); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x >> 5) - 1;
  const int n_chunks = (s + C::P - 1) / C::P, n_tasks = n_atoms * n_chunks;
  const int P = n_chunks == 1 ? s : C::P;  // floats between the rows of a tile
  if (threadIdx.x == 0) {
    for (int i = 0; i < R; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), nw);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();

  if (warp == nw) {
    // producer: lanes fetch the column indices 32 at a time, lane 0 waits for the stage, one copy per
    // lane (stall: a test of the bounded waits; nothing is copied, the consumers give up and report)
    int st = 0, ph = 1, issued = 0, ok = !stall;
    for (int task = blockIdx.x; task < n_tasks && ok; task += gridDim.x) {
      const int a = task / n_chunks, ch = task - a * n_chunks;
      const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
      const int wb = 4 * min(C::P, s - ch * C::P);  // bytes of a tile row
      for (int kb = k0; kb < k1 && ok; kb += 32) {
        const int mine = kb + lane < k1 ? __ldg(col + kb + lane) : 0;
        for (int k = kb; k < min(kb + 32, k1); ++k) {
          const int b = __shfl_sync(0xffffffffu, mine, k - kb);
          const uint32_t dst = smem_u32(smem + st * C::SB), bar = full(st);
          if (lane == 0) {
            ok = mbar_wait(empty(st), ph);
            if (ok) mbar_expect_tx(bar, 9 * wb + C::HB);
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
          const float* x = yin + (int64_t)9 * b * s + (int64_t)ch * C::P;
          if (lane == 9) bulk_g2s(dst + C::XB, hv + (int64_t)k * Layout<float, 9>::BS, C::HB, bar);
          if (n_chunks == 1) {
            if (lane == 0) bulk_g2s(dst, x, 9 * wb, bar);  // the 9 rows are contiguous
          } else if (lane < 9) {
            bulk_g2s(dst + lane * 4 * C::P, x + (int64_t)lane * s, wb, bar);
          }
          ++issued;
          if (++st == R) st = 0, ph ^= 1;
        }
      }
    }
    if (!ok && !stall && lane == 0) {
      // let the copies in flight land before the CTA exits
      atomicOr(err, 2);
      for (int j = (issued > R ? issued - R : 0); j < issued; ++j) mbar_wait(full(j % R), (j / R) & 1);
    }
    return;
  }

  float* ep = reinterpret_cast<float*>(smem + R * C::SB + warp * C::EB);  // 9 x 32
  const int pl = 32 * warp + lane;  // this lane's probe in the chunk
  // items of the epilogue: row irow[j], probes 4 igrp .. 4 igrp + 3 of the warp's 32
  const int igrp = lane & 7, irow = lane >> 3;  // item j: row irow + 4 j, j < 3
  // partial sums of all tasks of the CTA, in three floats: as good as the FP64 sums of the plain kernel
  Sum3 cs = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  int st = 0, ph = 0;
  bool ok = true;
  for (int task = blockIdx.x; task < n_tasks && ok; task += gridDim.x) {
    const int a = task / n_chunks, ch = task - a * n_chunks;
    const int k0 = __ldg(row_ptr + a), nb = __ldg(row_ptr + a + 1) - k0;
    const int p0 = ch * C::P + 32 * warp + 4 * igrp;  // the items' first probe
    // the items' y_prev and own y_in (ADJ: the source terms), fetched while the tiles stream
    float4 yp[3], xo[3], so[ADJ ? 3 : 1][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const bool has = irow + 4 * j < 9 && p0 < s;
      const int64_t off = ((int64_t)9 * a + irow + 4 * j) * s + p0;
      yp[j] = has && yprev ? *reinterpret_cast<const float4*>(yprev + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (ADJ) {
#pragma unroll
        for (int e = 0; e < 3; ++e)
          so[e][j] = has && src.p[e] ? __ldg(reinterpret_cast<const float4*>(src.p[e] + off)) : make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        xo[j] = has && partials && !direct ? *reinterpret_cast<const float4*>(yin + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    float2 acc[4];  // rows (0, 1), (2, 3), (4, 5), (6, 7)
    float acc8 = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = make_float2(0.f, 0.f);
    for (int q = 0; q < nb; ++q) {
      ok = mbar_wait(full(st), ph);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const float* X = reinterpret_cast<const float*>(smem + st * C::SB) + pl;
      const float* Hs = reinterpret_cast<const float*>(smem + st * C::SB + C::XB);
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        const float x = X[l * P];
        const float4 u0 = *reinterpret_cast<const float4*>(Hs + l * 12);
        const float4 u1 = *reinterpret_cast<const float4*>(Hs + l * 12 + 4);
        const float2 x2 = make_float2(x, x);
        acc[0] = __ffma2_rn(make_float2(u0.x, u0.y), x2, acc[0]);
        acc[1] = __ffma2_rn(make_float2(u0.z, u0.w), x2, acc[1]);
        acc[2] = __ffma2_rn(make_float2(u1.x, u1.y), x2, acc[2]);
        acc[3] = __ffma2_rn(make_float2(u1.z, u1.w), x2, acc[3]);
        acc8 = fmaf(Hs[l * 12 + 8], x, acc8);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(st));
      if (++st == R) st = 0, ph ^= 1;
    }
    if (!ok) break;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      ep[(2 * j) * 32 + lane] = alpha * acc[j].x;
      ep[(2 * j + 1) * 32 + lane] = alpha * acc[j].y;
    }
    ep[8 * 32 + lane] = alpha * acc8;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int row = irow + 4 * j;
      if (row >= 9 || p0 >= s) continue;
      const float4 t = *reinterpret_cast<const float4*>(ep + row * 32 + 4 * igrp);
      float yo[4] = {t.x, t.y, t.z, t.w}, r[4];
      if (c_r != 0.f || direct) {
#pragma unroll
        for (int v = 0; v < 4; ++v) r[v] = tbk_probe_sign(seed, (int64_t)9 * a + row, p0 + v);
      }
      if (c_r != 0.f) {
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[v] = fmaf(c_r, r[v], yo[v]);
      }
      auto add = [&](float c, const float4& x) {
        yo[0] = fmaf(c, x.x, yo[0]); yo[1] = fmaf(c, x.y, yo[1]);
        yo[2] = fmaf(c, x.z, yo[2]); yo[3] = fmaf(c, x.w, yo[3]);
      };
      if constexpr (ADJ) {
        if (src.c[0] != 0.f) add(src.c[0], so[0][j]);
      }
      if (yprev) {
        yo[0] -= yp[j].x; yo[1] -= yp[j].y; yo[2] -= yp[j].z; yo[3] -= yp[j].w;
      }
      if constexpr (ADJ) {
        if (src.c[1] != 0.f) add(src.c[1], so[1][j]);
        if (src.c[2] != 0.f) add(src.c[2], so[2][j]);
      }
      *reinterpret_cast<float4*>(yout + ((int64_t)9 * a + row) * s + p0) = make_float4(yo[0], yo[1], yo[2], yo[3]);
      if (!ADJ && partials) {
        const float xin[4] = {direct ? r[0] : xo[j].x, direct ? r[1] : xo[j].y, direct ? r[2] : xo[j].z,
                              direct ? r[3] : xo[j].w};
        float q0 = 0.f, q1 = 0.f;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          q0 = fmaf(yo[v], xin[v], q0);
          q1 = fmaf(yo[v], yo[v], q1);
        }
        sum3_add(cs, make_float2(q0, q1));
      }
    }
    __syncwarp();  // the buffer is free again
  }
  if (!ok) atomicOr(err, 2);
  if (!ADJ && partials)
    step_partials(partials, sum3_value(cs.h.x, cs.m.x, cs.l.x), sum3_value(cs.h.y, cs.m.y, cs.l.y), warp, lane, nw);
}

// ---- FP64 step by rows -------------------------------------------------------------------------------
//
// A warp takes 32 probes of ROWS (3 or 1) of the 9 rows of an atom, on its own, with the next block and
// tile loaded a block ahead.  A warp's FP64 FMA takes 64 cycles, and the SM about 19 for each when all four
// quarters issue them, so nothing but the
// even spread of the FMAs over the quarters counts; a warp of a third or a ninth of a row spreads them
// to within a few per cent (a row per three-warp CTA leaves every fourth quarter idle).  Narrow panels
// put several row groups into a warp.  200 atoms x 64 probes: 36 us a step against 125 with the plain
// kernel on 50 SMs, 2,000 x 128: 636 against 716, which is 18.4 cycles an FMA; at that rate 200 x 64 takes 27.
template <int ROWS>
__global__ void __launch_bounds__(128)
cheb_step_fp64(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const double* __restrict__ hv, const double* __restrict__ yin, const double* yprev, double* yout,
               const double alpha, const double c_r, const uint64_t seed, const int s, const int direct,
               const StepSources<double> src, double* __restrict__ partials, const int lp, const int n_sm) {
  constexpr int NG = 9 / ROWS, RS = Layout<double, 9>::RS, BS = Layout<double, 9>::BS;
  pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = 32 / lp;                   // row groups in a warp
  const int ngw = (NG + gw - 1) / gw;       // warps of an atom and chunk
  const int n_chunks = (s + 31) / 32;
  const int64_t units = (int64_t)n_atoms * n_chunks * ngw;
  double sum0 = 0.0, sum1 = 0.0;
  // long and short rows lie far apart in most listings: the CTAs that share an SM take their quarters in
  // opposite order
  const int quarter = (blockIdx.x / n_sm) & 1 ? 3 - warp : warp;
  for (int64_t u = (int64_t)quarter * gridDim.x + blockIdx.x; u < units; u += (int64_t)4 * gridDim.x) {
    const int64_t t = u / ngw;
    const int a = (int)(t / n_chunks), p0 = (int)(t - (int64_t)a * n_chunks) * 32 + lane % lp;
    const int g = (int)(u - t * ngw) * gw + lane / lp;
    if (lane / lp >= gw || g >= NG || p0 >= s) continue;
    int k = __ldg(row_ptr + a);
    const int k1 = __ldg(row_ptr + a + 1);
    double acc[ROWS], x[9], h[ROWS][9];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) acc[i] = 0.0;
    auto fetch = [&](int kk, int b, double (&xx)[9], double (&hh)[ROWS][9]) {
      const double* xb = yin + (int64_t)9 * b * s + p0;
      const double* hb = hv + (int64_t)kk * BS + ROWS * g * RS;
#pragma unroll
      for (int l = 0; l < 9; ++l) xx[l] = __ldg(xb + (int64_t)l * s);
#pragma unroll
      for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int l = 0; l < 9; ++l) hh[i][l] = __ldg(hb + i * RS + l);
    };
    int bn = k + 1 < k1 ? __ldg(col + k + 1) : 0;
    if (k < k1) fetch(k, __ldg(col + k), x, h);
    for (; k < k1; ++k) {
      double xn[9], hn[ROWS][9];
      if (k + 1 < k1) fetch(k + 1, bn, xn, hn);
      if (k + 2 < k1) bn = __ldg(col + k + 2);
#pragma unroll
      for (int l = 0; l < 9; ++l)
#pragma unroll
        for (int i = 0; i < ROWS; ++i) acc[i] = fma(h[i][l], x[l], acc[i]);
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        x[l] = xn[l];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) h[i][l] = hn[i][l];
      }
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const int64_t row = (int64_t)9 * a + ROWS * g + i, off = row * s + p0;
      double yo = alpha * acc[i], r = 0.0;
      if (c_r != 0.0 || direct) r = (double)tbk_probe_sign(seed, row, p0);
      if (c_r != 0.0) yo = fma(c_r, r, yo);
      if (yprev) yo -= yprev[off];
#pragma unroll
      for (int e = 0; e < 3; ++e)
        if (src.p[e]) yo = fma(src.c[e], __ldg(src.p[e] + off), yo);
      yout[off] = yo;
      if (partials) {
        sum0 = fma(yo, direct ? r : __ldg(yin + off), sum0);
        sum1 = fma(yo, yo, sum1);
      }
    }
  }
  if (partials) step_partials(partials, sum0, sum1, warp, lane, 4);
}

// ---- launch geometry ---------------------------------------------------------------------------

template <typename T, int B, bool P>
static int occupancy_simple() {
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cheb_step_kernel<T, B, P, false>, STEP_THREADS, 0);
  return n > 0 ? n : 1;
}

// two stages: 10 KB of ring per warp, so that the register limit (16 warps per SM), not shared
// memory (14 warps with three stages), sets the occupancy; measured 11 % faster on the batch
constexpr int SELF_R = 2;

static int occupancy_self() {
  using C = SelfCfg<SELF_R>;
  cudaFuncSetAttribute(cheb_step_self<SELF_R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  cudaFuncSetAttribute(cheb_step_self<SELF_R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cheb_step_self<SELF_R, false>, 32, C::SMEM);
  return n;
}

template <int CW, int D, bool DENSE = false>
static int occupancy_bulk() {
  using C = BulkCfg<CW, D>;
  cudaFuncSetAttribute(cheb_step_bulk<CW, D, DENSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cheb_step_bulk<CW, D, DENSE>, C::THREADS, C::SMEM);
  return n;
}

// three ring stages and at most 102 registers: four CTAs of the 512-probe kernel per SM (16
// consumer warps), 2.8 % faster per step than three CTAs with four stages at 128 registers
constexpr int BULK_D = 2;

int bulk_consumer_warps(const HOp& op, int s);
// Consumer warps of the TMA-fed kernel for this operator and probe count (0 = not eligible).
static int bulk_warps(const HOp& op, int s) {
  if (op.prec != TBK_MIXED || op.B != 9 || s % 128 != 0) return 0;
  if (s % 512 == 0) return 4;
  if (s % 256 == 0) return 2;
  return 1;
}

int bulk_consumer_warps(const HOp& op, int s) { return bulk_warps(op, s); }

// Consumer warps (probe chunk 128 cw per task) of the TMA-fed step for this operator: the tuned
// choice when tbk_autotune measured this shape, else the widest chunk.  Per-task partial sums
// (batches) keep the default layout.
static int chosen_cw(const tbk_ctx* ctx, const HOp& op, int s, int per_task) {
  const int cw = bulk_warps(op, s);
  if (!cw || per_task) return cw;
  const tbk_ctx::Tuned* t = find_tuned(ctx, op.n_rows, op.nnzb, s);
  return t && t->cw >= 1 && t->cw <= cw && s % (128 * t->cw) == 0 ? t->cw : cw;
}

template <int NW>
static int occupancy_lane() {
  cudaFuncSetAttribute(cheb_step_lane<NW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, LaneCfg<NW>::SMEM);
  cudaFuncSetAttribute(cheb_step_lane<NW, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, LaneCfg<NW>::SMEM);
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cheb_step_lane<NW, false>, 32 * (NW + 1), LaneCfg<NW>::SMEM);
  return n;
}

struct Occ {
  int simple = 0, bulk[5] = {0, 0, 0, 0, 0}, dense = 0, lane[3] = {0, 0, 0};
};

// Block of the plain kernel: `vec` probes per lane, rows in y.
static dim3 simple_block(int s, int vec) {
  const int lanes_needed = (s + vec - 1) / vec;
  int lanes = 1;  // a power of two, so that every warp of the CTA is complete
  while (lanes < lanes_needed && lanes < STEP_THREADS) lanes <<= 1;
  return dim3(lanes, STEP_THREADS / lanes);
}
static int64_t simple_tasks(const HOp& op, int s) {
  const int vec = op.prec == TBK_MIXED ? Vec16<float>::N : Vec16<double>::N;
  const dim3 b = simple_block(s, vec);
  return (int64_t)ceil_div(op.n_atoms, b.y) * ceil_div(s, b.x * vec);
}

bool tc_eligible(const HOp& op, int s);
void launch_step_tc(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G);

static int lane_class(int s);

// CTAs per SM of the step kernels on the context's device; the first call also sets their shared-memory limits.
// Nobody sees a device's numbers before all of them are there: contexts of several threads may come at once.
static const Occ& occupancies(const tbk_ctx* ctx) {
  static Occ occ[64];
  static std::once_flag once[64];
  const int dev = ctx->device < 0 || ctx->device >= 64 ? 0 : ctx->device;
  std::call_once(once[dev], [&] {
    Occ& o = occ[dev];
    int m = 1 << 30;
    m = std::min(m, std::min(occupancy_simple<float, 9, false>(), occupancy_simple<float, 9, true>()));
    m = std::min(m, std::min(occupancy_simple<float, 1, false>(), occupancy_simple<float, 1, true>()));
    m = std::min(m, std::min(occupancy_simple<double, 9, false>(), occupancy_simple<double, 9, true>()));
    m = std::min(m, std::min(occupancy_simple<double, 1, false>(), occupancy_simple<double, 1, true>()));
    o.simple = std::max(1, m);
    o.bulk[1] = occupancy_self();  // 128-probe tasks run on the self-fed kernel
    o.bulk[2] = occupancy_bulk<2, BULK_D>();
    o.dense = occupancy_bulk<2, BULK_D, true>();
    o.bulk[4] = occupancy_bulk<4, BULK_D>();
    o.lane[0] = occupancy_lane<4>();
    o.lane[1] = occupancy_lane<8>();
    o.lane[2] = occupancy_lane<16>();
  });
  return occ[dev];
}

// FP32 steps that the one-probe-per-lane kernel takes: up to 17 warps' work per SM, or any width beyond 128
// that is no multiple of 128 (whose tiles the other kernels would fetch row by row: 1,000 atoms x 196 probes 71 us a
// step against 33).  Measured us a step on 152 SMs, lane against self-fed kernel at 128 probes: 147 atoms 8.3
// (16.0), 333 atoms 9.6 (15.9), 700 atoms 16.4 (16.6); against cheb_step_bulk at 256: 147 atoms 10.1 (9.5).
static bool use_lane(const tbk_ctx* ctx, const HOp& op, int s) {
  if (op.prec != TBK_MIXED || op.B != 9) return false;
  if (s > 128) return s % 128 != 0;
  return (int64_t)op.n_atoms * ((s + 31) / 32) <= 17 * (int64_t)ctx->num_sms;
}
// The self-fed kernel with narrow tasks, where there is too much for the lane kernel: a warp per row whatever the
// probes, so that it loses to the plain kernel's several rows per warp on many rows of few.  us a step, narrow / plain:
// 4,000 atoms x 16 probes 40 / 55, 6,000 x 16 58 / 53, 10,000 x 16 93 / 54, x 20 93 / 98, 20,000 x 8 182 / 117, x 32 182 / 232.
static bool use_narrow(const tbk_ctx* ctx, const HOp& op, int s) {
  return op.prec == TBK_MIXED && op.B == 9 && s < 128 && (s > 16 || op.n_atoms <= 36 * ctx->num_sms);
}
// FP64 9x9 steps by rows: while the plain kernel's tasks take fewer than two rounds of its CTAs.  Beyond, its tiles of
// several rows and probes read less.  us a step, rows / plain: 1,000 atoms x 128 probes (0.8 rounds) 315 / 370, 3,000 x
// 64 (1.2) 500 / 541, 7,000 x 32 (1.4) 633 / 650; 10,000 x 32 (2.1) 911 / 886, 5,832 full rows x 64 (2.4) 1,102 /
// 1,040, 1,000 x 512 (3.3) 1,237 / 1,253, 10,000 x 128 (8) 3,408 / 3,274, x 512 (33) 13,609 / 12,834.
static bool use_rows64(const tbk_ctx* ctx, const HOp& op, int s) {
  return op.prec == TBK_FP64 && op.B == 9 && simple_tasks(op, s) < 2 * (int64_t)occupancies(ctx).simple * ctx->num_sms;
}

// Warps of an FP64 step by rows, and the rows a warp takes: one where three would leave SM quarters idle.
static int64_t fp64_units(const HOp& op, int s, int rows) {
  const int gw = 32 / std::min(32, s), ng = 9 / rows;
  return (int64_t)op.n_atoms * ((s + 31) / 32) * ((ng + gw - 1) / gw);
}
static int fp64_rows(const tbk_ctx* ctx, const HOp& op, int s) {
  return fp64_units(op, s, 3) >= 4 * (int64_t)ctx->num_sms ? 3 : 1;
}

// 256-probe tasks with 80 instead of 108 registers, so that seven CTAs per SM run instead of five: where five
// leave a second round.  us a step, five -> seven: 700 atoms 15.7 -> 16.7 and 850 19.6 -> 20.5 (8 bytes of
// spills), 1,000 23.2 -> 22.8, 1,200 28.3 -> 23.7, 3,000 64.4 -> 61.1 and 10,000 215 -> 195 (both with CTAs that
// stay); 126 stored steps on 1,000 atoms 3.45 -> 3.37 ms.
static bool dense_bulk(const tbk_ctx* ctx, const HOp& op, int s, int cw) {
  return cw == 2 && (int64_t)op.n_atoms * (s / 256) > 6 * ctx->num_sms;
}

int step_grid_ctas(tbk_ctx* ctx, const HOp& op, int s, int K, bool resident) {
  const Occ& o = occupancies(ctx);
  // every kernel loops over its tasks and none waits on another CTA, so any grid will do
  const int cw = chosen_cw(ctx, op, s, 0);
  if (resident) {
    // the tensor-core step (CTAs that set up their TMEM once) and the plain kernel, as many as fit
    const int64_t held = (int64_t)(cw && o.bulk[cw] > 0 ? o.bulk[cw] : o.simple) * ctx->num_sms;
    return (int)std::min(held, std::max(simple_tasks(op, s), cw ? (int64_t)op.n_atoms * (s / 128) : 0));
  }
  if (use_rows64(ctx, op, s))
    return (int)std::min<int64_t>((fp64_units(op, s, fp64_rows(ctx, op, s)) + 3) / 4, 4 * ctx->num_sms);
  if (use_lane(ctx, op, s))
    return (int)std::min<int64_t>((int64_t)op.n_atoms * ((s + 511) / 512), (int64_t)std::max(1, o.lane[lane_class(s)]) * ctx->num_sms);
  const bool narrow = use_narrow(ctx, op, s);
  if (!cw && !narrow) return (int)std::min((int64_t)o.simple * ctx->num_sms, simple_tasks(op, s));
  const int fed = cw && dense_bulk(ctx, op, s, cw) ? o.dense : (cw ? o.bulk[cw] : 0);
  const int per_sm = narrow && o.bulk[1] > 0 ? o.bulk[1] : (fed > 0 ? fed : o.simple);
  const int64_t tasks = cw ? (int64_t)op.n_atoms * (s / (128 * cw)) : op.n_atoms, held = (int64_t)per_sm * ctx->num_sms;
  // at most 256 MB of partial sums
  return (int)std::min<int64_t>(task_grid(tasks, held), std::max<int64_t>(held, ((int64_t)1 << 24) / std::max(1, K)));
}

template <typename T>
static StepSources<T> sources(const StepArgs& a) {
  StepSources<T> r;
  for (int e = 0; e < 3; ++e) {
    r.p[e] = (const T*)a.src[e];
    r.c[e] = (T)a.csrc[e];
  }
  return r;
}

template <typename T, int B>
static void launch_simple(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  const dim3 blk = simple_block(a.s, Vec16<T>::N);
  const T* hv = (const T*)op.hv;
  auto go = [&](auto kernel) {
    kernel<<<G, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, hv, (const T*)a.yin, (const T*)a.yprev, (T*)a.yout,
                                       (T)a.alpha, (T)a.c_r, a.seed, a.s, a.direct, sources<T>(a), a.partials);
  };
  if (a.src[0] || a.src[1] || a.src[2]) {
    // the FP64 adjoint of 1x1 operators; other kernels take the other ones
    TBK_CHECK_ARG((sizeof(T) == 8 && B == 1), "a plain step with further own-row terms");
    if constexpr (sizeof(T) == 8 && B == 1) go(cheb_step_kernel<T, B, false, true>);
  } else if (a.cur_is_probe) go(cheb_step_kernel<T, B, true, false>);
  else go(cheb_step_kernel<T, B, false, false>);
  post_launch(ctx, "cheb_step_kernel");
}

// The test hook that a TMA-fed step answers to, taken.
static int take_stall(tbk_ctx* ctx, const StepArgs& a) {
  int& hook = a.family == TBK_KERNEL_BACKWARD ? ctx->stall_next_adjoint : ctx->stall_next_step;
  const int stall = hook;
  hook = 0;
  return stall;
}

template <int CW, bool DENSE = false>
static void launch_bulk(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  using C = BulkCfg<CW, BULK_D>;
  launch_pdl(ctx, cheb_step_bulk<CW, BULK_D, DENSE>, G, C::THREADS, C::SMEM,
               op.n_atoms, op.row_ptr, op.col, (const float*)op.hv, (const float*)a.yin, (const float*)a.yprev,
               (float*)a.yout, (float)a.alpha, (float)a.c_r, a.seed, a.s, a.direct, a.partials, a.err, a.batch,
               a.per_task, take_stall(ctx, a));
  post_launch(ctx, "cheb_step_bulk");
}

template <bool NARROW>
static void launch_self(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  using C = SelfCfg<SELF_R>;
  launch_pdl(ctx, cheb_step_self<SELF_R, NARROW>, G, 32, C::SMEM,
               op.n_atoms, op.row_ptr, op.col, (const float*)op.hv, (const float*)a.yin, (const float*)a.yprev,
               (float*)a.yout, (float)a.alpha, (float)a.c_r, a.seed, a.s, a.direct, a.partials, a.err, a.batch,
               a.per_task, take_stall(ctx, a));
  post_launch(ctx, "cheb_step_self");
}

template <int NW>
static void launch_lane_nw(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  const int nw = std::min(NW, (a.s + 31) / 32);
  launch_pdl(ctx, a.adjoint ? cheb_step_lane<NW, true> : cheb_step_lane<NW, false>, G, 32 * (nw + 1), LaneCfg<NW>::SMEM,
             op.n_atoms, op.row_ptr, op.col, (const float*)op.hv, (const float*)a.yin, (const float*)a.yprev,
             (float*)a.yout, (float)a.alpha, (float)a.c_r, a.seed, a.s, a.direct, sources<float>(a), a.partials, a.err,
             take_stall(ctx, a));
  post_launch(ctx, "cheb_step_lane");
}

static int lane_class(int s) { return s <= 128 ? 0 : (s <= 256 ? 1 : 2); }  // 4, 8 or 16 warps

static void launch_lane(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  const int c = lane_class(a.s);
  if (c == 0) launch_lane_nw<4>(ctx, op, a, G);
  else if (c == 1) launch_lane_nw<8>(ctx, op, a, G);
  else launch_lane_nw<16>(ctx, op, a, G);
}

bool lane_adjoint_step(tbk_ctx* ctx, const HOp& op, const StepArgs& a) {
  if (!use_lane(ctx, op, a.s)) return false;
  KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
  launch_lane(ctx, op, a, step_grid_ctas(ctx, op, a.s));
  return true;
}

template <int ROWS>
static void launch_fp64(tbk_ctx* ctx, const HOp& op, const StepArgs& a, int G) {
  launch_pdl(ctx, cheb_step_fp64<ROWS>, G, 128, 0, op.n_atoms, op.row_ptr, op.col,
               (const double*)op.hv, (const double*)a.yin, (const double*)a.yprev, (double*)a.yout, a.alpha, a.c_r,
               a.seed, a.s, a.direct, sources<double>(a), a.partials, std::min(32, a.s), ctx->num_sms);
  post_launch(ctx, "cheb_step_fp64");
}

void launch_step(tbk_ctx* ctx, const HOp& op, const StepArgs& a) {
  KernelTimerScope timer(ctx, a.family);
  const int G = a.grid > 0 ? a.grid : step_grid_ctas(ctx, op, a.s, 0, a.force_simple || a.use_tc);
  if (a.use_tc && !a.cur_is_probe && a.err && !a.force_simple && !a.batch.atom_cl && !a.per_task &&
      tc_eligible(op, a.s)) {
    launch_step_tc(ctx, op, a, G);
    return;
  }
  const bool fed = !a.cur_is_probe && a.err && !a.force_simple && op.B == 9;  // a panel by bulk copies
  // (with an adjoint's own-row terms at every size: the plain kernel has none for 9x9 blocks)
  if (fed && op.prec == TBK_FP64 && (use_rows64(ctx, op, a.s) || a.src[0] || a.src[1] || a.src[2])) {
    if (fp64_rows(ctx, op, a.s) == 3) launch_fp64<3>(ctx, op, a, G);
    else launch_fp64<1>(ctx, op, a, G);
    return;
  }
  if (fed && !a.per_task && use_lane(ctx, op, a.s)) {
    launch_lane(ctx, op, a, G);
    return;
  }
  if (fed && use_narrow(ctx, op, a.s)) {
    launch_self<true>(ctx, op, a, G);
    return;
  }
  const int cw = chosen_cw(ctx, op, a.s, a.per_task);
  if (cw && !a.cur_is_probe && a.err && !a.force_simple && occupancies(ctx).bulk[cw] > 0) {
    if (cw == 4) launch_bulk<4>(ctx, op, a, G);
    else if (cw == 2 && dense_bulk(ctx, op, a.s, cw) && occupancies(ctx).dense > 0) launch_bulk<2, true>(ctx, op, a, G);
    else if (cw == 2) launch_bulk<2>(ctx, op, a, G);
    else launch_self<false>(ctx, op, a, G);
    return;
  }
  if (op.prec == TBK_MIXED) {
    if (op.B == 9) launch_simple<float, 9>(ctx, op, a, G); else launch_simple<float, 1>(ctx, op, a, G);
  } else {
    if (op.B == 9) launch_simple<double, 9>(ctx, op, a, G); else launch_simple<double, 1>(ctx, op, a, G);
  }
}

// A thread writes four probes of a row (16-byte stores), neighbouring threads neighbouring ones, over the rows' ends: a
// warp per row left most of its lanes idle on narrow panels.
template <typename T>
__global__ void __launch_bounds__(256)
scaled_probe_kernel(int64_t n_items, int groups, T c, uint64_t seed, T* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= n_items) return;
  const int64_t row = n_items <= 0xffffffffll ? (int64_t)((uint32_t)i / (uint32_t)groups) : i / groups;
  const int p = 4 * (int)(i - row * groups);
  T v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = tbk_probe_sign(seed, row, p + j) < 0.f ? -c : c;
  T* o = out + 4 * i;
  if constexpr (sizeof(T) == 4) {
    st16(o, v);
  } else {
    st16(o, v);
    st16(o + 2, v + 2);
  }
}

void launch_scaled_probe(tbk_ctx* ctx, const HOp& op, void* panel, double c, uint64_t seed, int s) {
  const int64_t n = op.n_rows * (s / 4);
  const unsigned grid = (unsigned)((n + 255) / 256);
  if (op.prec == TBK_MIXED)
    scaled_probe_kernel<float><<<grid, 256, 0, ctx->stream>>>(n, s / 4, (float)c, seed, (float*)panel);
  else
    scaled_probe_kernel<double><<<grid, 256, 0, ctx->stream>>>(n, s / 4, c, seed, (double*)panel);
  post_launch(ctx, "scaled_probe_kernel");
}

// ---- moment reduction ------------------------------------------------------------------------

// sums[2 j + c] = sum over CTAs of partials[(j * nctas + cta) * 2 + c], Kahan-compensated per
// thread over a fixed strided set, then a fixed-order tree.
__global__ void reduce_partials(const double* __restrict__ partials, int nctas, double* __restrict__ sums) {
  const int j = blockIdx.x;
  __shared__ double sh[2][256];
  double s0 = 0, c0 = 0, s1 = 0, c1 = 0;
  for (int t = threadIdx.x; t < nctas; t += blockDim.x) {
    const double* p = partials + ((int64_t)j * nctas + t) * 2;
    double y = p[0] - c0, u = s0 + y;
    c0 = (u - s0) - y;
    s0 = u;
    y = p[1] - c1;
    u = s1 + y;
    c1 = (u - s1) - y;
    s1 = u;
  }
  sh[0][threadIdx.x] = s0;
  sh[1][threadIdx.x] = s1;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sums[2 * j] = sh[0][0];
    sums[2 * j + 1] = sh[1][0];
  }
}

// Moments from the per-step sums (step j = 1..K stored at index j - 1):
//   direct:   mu_j = S0_j / s
//   doubling: mu_1 = S0_1 / s, mu_2j = 2 S1_j / s - mu_0, mu_2j-1 = 2 S0_j / s - mu_1 (j >= 2)
// (C_m C_n = (C_{m+n} + C_{|m-n|})/2).  mu_0 = n_rows exactly for +-1 probes.  flag = 1 when a
// panel norm exceeds ||r|| (a spectrum outside [-1, 1]) or a sum is not finite.
__global__ void finish_moments(const double* __restrict__ sums, int K, int order, int s,
                               int64_t n_rows, int direct, double* __restrict__ mom,
                               int* __restrict__ flag) {
  const double mu0 = (double)n_rows;
  const double inv_s = 1.0 / s;
  const double mu1 = K >= 1 ? sums[0] * inv_s : 0.0;
  for (int k = threadIdx.x; k < order; k += blockDim.x) {
    double v;
    if (k == 0) v = mu0;
    else if (direct) v = sums[2 * (k - 1)] * inv_s;
    else if (k == 1) v = mu1;
    else if ((k & 1) == 0) v = 2.0 * sums[2 * (k / 2 - 1) + 1] * inv_s - mu0;
    else v = 2.0 * sums[2 * ((k + 1) / 2 - 1)] * inv_s - mu1;
    mom[k] = v;
  }
  for (int j = threadIdx.x; j < K; j += blockDim.x) {
    const double e = sums[2 * j + 1] * inv_s, o = sums[2 * j];
    if (!(e <= mu0 * (1.0 + 1e-3)) || !isfinite(o)) atomicOr(flag, 1);
  }
}

// ---- per-probe moments -------------------------------------------------------------------------
//
// After step j, PD_BLOCKS row blocks each sum, for every probe i, the products of the new panel
// y_j with itself and with y_{j-1} (the probe block r for j = 1) over their rows:
//   part[(rb s + i) 2 + 0] = sum_rows y_j y_j   (direct: sum_rows r y_j),
//   part[(rb s + i) 2 + 1] = sum_rows y_j y_{j-1}.
// FP32 panels: products are summed in FP32 over runs of 32 rows, then in FP64.  A second kernel
// adds the row blocks in a fixed order, so the result does not depend on timing.
constexpr int PD_BLOCKS = 304;

template <typename T>
__global__ void __launch_bounds__(256)
probe_dots(int64_t n_rows, int s, int64_t rows_per_block, const T* __restrict__ y,
           const T* __restrict__ x, uint64_t seed, int direct, double* __restrict__ part) {
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
  const int64_t r1 = r0 + rows_per_block < n_rows ? r0 + rows_per_block : n_rows;
  for (int i = threadIdx.x; i < s; i += blockDim.x) {
    double d0 = 0.0, d1 = 0.0;
    for (int64_t b = r0; b < r1; b += 32) {
      const int64_t e = b + 32 < r1 ? b + 32 : r1;
      T t0 = T(0), t1 = T(0);
      for (int64_t row = b; row < e; ++row) {
        const T v = y[row * s + i];
        if (direct) {
          t0 += v * (T)tbk_probe_sign(seed, row, i);
        } else {
          const T u = x ? x[row * s + i] : (T)tbk_probe_sign(seed, row, i);
          t0 += v * v;
          t1 += v * u;
        }
      }
      d0 += (double)t0;
      d1 += (double)t1;
    }
    part[((int64_t)blockIdx.x * s + i) * 2] = d0;
    part[((int64_t)blockIdx.x * s + i) * 2 + 1] = d1;
  }
}

// dots[i 2 + c] = sum over the row blocks, in order, of part[(rb s + i) 2 + c]
__global__ void probe_dots_reduce(int nrb, int s, const double* __restrict__ part, double* __restrict__ dots) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= s) return;
  double a = 0.0, b = 0.0;
  for (int rb = 0; rb < nrb; ++rb) {
    a += part[((int64_t)rb * s + i) * 2];
    b += part[((int64_t)rb * s + i) * 2 + 1];
  }
  dots[2 * i] = a;
  dots[2 * i + 1] = b;
}

// per_probe[k s + i] = r_i^T C_k(H^) r_i from the dots of steps j = 1 .. K (dots[((j-1) s + i) 2
// + c]): mu_0 = n_rows; direct: mu_k = (r . y_k); doubling: mu_1 = y_1 . r, mu_2k = 2 y_k . y_k -
// mu_0, mu_2k-1 = 2 y_k . y_{k-1} - mu_1 (the identities the summed moments use).
__global__ void probe_moments_finish(const double* __restrict__ dots, int K, int order, int s,
                                     int64_t n_rows, int direct, double* __restrict__ per_probe) {
  const int64_t n = (int64_t)order * s;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(t / s), i = (int)(t - (int64_t)k * s);
    auto d = [&](int j, int c) { return dots[((int64_t)(j - 1) * s + i) * 2 + c]; };
    const double mu0 = (double)n_rows;
    double v;
    if (k == 0) v = mu0;
    else if (direct) v = d(k, 0);
    else if (k == 1) v = d(1, 1);
    else if ((k & 1) == 0) v = 2.0 * d(k / 2, 0) - mu0;
    else v = 2.0 * d((k + 1) / 2, 1) - d(1, 1);
    per_probe[t] = v;
  }
}

// ---- all steps of a small 1x1 operator in one launch (FP64) ----------------------------------------
//
// The probes do not meet until the moments are summed: a cluster of CTAs takes one probe through all steps,
// each with its share of the rows and the whole of y_j and y_{j-1} in shared memory; a new entry is stored in
// every CTA of the cluster, and a step ends with the cluster's barrier.  Rows are summed in the order of the
// step kernel.  A warp's FP64 instruction takes an SM 19 cycles: 10 per row and probe are the bound (0.6 us a
// step at 1,000 sites and 32 probes), then the chain of a row and the barrier.  Microseconds per step,
// a launch each -> so: 216 sites x 32 probes 6.2 -> 1.4, 1,000 x 32 8.2 -> 1.7, 1,000 x 512 18.9 -> 16.6,
// 2,744 x 64 10.3 -> 5.3, 5,832 x 64 16.4 -> 10.0, 10,648 x 4 7.1 -> 6.2, 10,648 x 512 138 -> 125.
constexpr int SWEEP_THREADS = 512;
constexpr int64_t SWEEP_ROWS = 11000;                   // two panels in shared memory
constexpr size_t SWEEP_PARTIALS = (size_t)56 << 20;     // bytes of partial sums: fit tbk_chebyshev_moments_noalloc's scratch
constexpr int SWEEP_FLUSH = 16;                         // steps whose sums wait in shared memory
constexpr int64_t SWEEP_SMEM = 220 << 10;               // beside them; with 4 KB more L1 is a tenth slower at 10,648 sites

// probe_panel: y_0, or NULL for the +-1 probes of the seed.  partials: two per CTA and step.  cap: blocks of
// the operator that fit in shared memory beside the panels; rows of a CTA's share beyond them stay in global memory
// and come from L2 in every step (the cluster's barrier drops what L1 holds), a lane walking its own row.
__global__ void __launch_bounds__(SWEEP_THREADS)
moments_sweep_b1(int n, int C, int cap, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                 const double* __restrict__ hv, const double* __restrict__ probe_panel, uint64_t seed, int s, int K,
                 double* __restrict__ partials) {
  extern __shared__ double ysm[];
  const int rank = blockIdx.x % C, probe = blockIdx.x / C;
  const int r0 = (int)((int64_t)n * rank / C), rows = (int)((int64_t)n * (rank + 1) / C) - r0;
  const int lane = threadIdx.x & 31, warps = blockDim.x / 32;
  __shared__ double sums[SWEEP_FLUSH][2][SWEEP_THREADS / 32];  // of each warp
  double* hs = ysm + 2 * n;
  int* cs = reinterpret_cast<int*>(hs + cap);
  int* rp = cs + cap;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    ysm[i] = probe_panel ? probe_panel[(int64_t)i * s + probe] : (double)tbk_probe_sign(seed, i, probe);
  const int k0 = __ldg(row_ptr + r0), nz = __ldg(row_ptr + r0 + rows) - k0;
  for (int i = threadIdx.x; i <= rows; i += blockDim.x) rp[i] = __ldg(row_ptr + r0 + i) - k0;
  const int staged = min(nz, cap);
  for (int k = threadIdx.x; k < staged; k += blockDim.x) {
    hs[k] = __ldg(hv + k0 + k);
    cs[k] = __ldg(col + k0 + k);
  }
  cluster_barrier();
  for (int j = 1; j <= K; ++j) {
    const double* in = ysm + ((j - 1) & 1) * n;
    double* out = ysm + (j & 1) * n;
    double s0 = 0.0, s1 = 0.0;
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      double acc = 0.0;
      const int k1 = rp[i + 1];
      if (k1 <= staged) {
#pragma unroll 4
        for (int k = rp[i]; k < k1; ++k) acc = fma(hs[k], in[cs[k]], acc);
      } else {
        for (int k = rp[i]; k < k1; ++k) acc = fma(__ldg(hv + k0 + k), in[__ldg(col + k0 + k)], acc);
      }
      const double y = j == 1 ? acc : 2.0 * acc - out[r0 + i];
      for (int c = 0; c < C; ++c) store_cluster(out + r0 + i, c, y);
      s0 = fma(y, in[r0 + i], s0);
      s1 = fma(y, y, s1);
    }
    const double a = lanes_sum2(s0, s1, lane);
    if ((lane & 15) == 0) sums[(j - 1) % SWEEP_FLUSH][lane >> 4][threadIdx.x >> 5] = a;
    cluster_barrier();
    if (j % SWEEP_FLUSH == 0 || j == K) {
      // the warps' sums of the last steps: eight threads add the (at most 16) of one
      const int j0 = (j - 1) / SWEEP_FLUSH * SWEEP_FLUSH;
      for (int e = threadIdx.x / 8; e < 2 * SWEEP_FLUSH; e += blockDim.x / 8) {
        const int w = threadIdx.x % 8;
        const bool has = j0 + e / 2 < j;
        double t = has && w < warps ? sums[e / 2][e & 1][w] : 0.0, err = 0.0;
        auto add = [&](double b) {  // t + b, its rounding error (TwoSum) to err
          const double u = t + b, z = u - t;
          err += (t - (u - z)) + (b - z);
          t = u;
        };
        if (has && w + 8 < warps) add(sums[e / 2][e & 1][w + 8]);
        for (int o = 4; o > 0; o >>= 1) {
          const double b = __shfl_xor_sync(0xffffffffu, t, o);
          err += __shfl_xor_sync(0xffffffffu, err, o);
          add(b);
        }
        if (has && w == 0) partials[2 * ((int64_t)(j0 + e / 2) * gridDim.x + blockIdx.x) + (e & 1)] = t + err;
      }
      __syncthreads();
    }
  }
}

// CTAs per probe (enough for the chip, at most a portable cluster) and threads per CTA (a row each).
static int sweep_cluster(const tbk_ctx* ctx, int s) {
  int c = 1;
  while (c < 8 && s * c < ctx->num_sms * 4 / 5) c *= 2;
  return c;
}
static int sweep_warps(const tbk_ctx* ctx, const HOp& op, int s) {
  return std::min(SWEEP_THREADS / 32, ceil_div(op.n_rows, 32 * sweep_cluster(ctx, s)));
}

static int sweep_partials(const tbk_ctx* ctx, int s) { return s * sweep_cluster(ctx, s); }

// Blocks that fit beside the panels and the row pointers.
static int64_t sweep_room(const HOp& op, int C) {
  return (SWEEP_SMEM - 16 * op.n_rows - 4 * (op.n_rows / C + 2)) / 12 - 1;
}

// Short rows always (us a step, sweep against a launch each: 10,648 sites of 7 blocks x 4 probes 6.4 / 7.1, x 512 126 /
// 138, although their blocks do not fit); longer ones where the blocks fit in shared memory (2,744 sites x 32 probes, 17
// blocks a row 5.8 / 10.3, 23 blocks, beyond it, 20.4 / 12.4; 5,832 x 512 of 143 blocks 4,599 / 744) and the chip is
// not full of FMAs anyway (216 sites x 512 probes, 36 blocks 17.5 / 18.6, 47 blocks 23.5 / 22.7; 1,000 x 512, 16
// blocks 28.4 / 26.8).
int sweep_ctas(const tbk_ctx* ctx, const HOp& op, int s, int K, int direct, bool per_probe, int flags) {
  if (op.B != 1 || op.prec != TBK_FP64 || K < 1 || direct || per_probe || (flags & TBK_PLAIN_KERNEL) ||
      op.n_rows > SWEEP_ROWS || s > 512 || 16 * (size_t)K * sweep_partials(ctx, s) > SWEEP_PARTIALS)
    return 0;
  const int C = sweep_cluster(ctx, s);
  const bool fits = op.nnzb <= C * sweep_room(op, C), small = s * op.nnzb <= (int64_t)30000 * ctx->num_sms;
  return op.nnzb <= 8 * op.n_rows || (fits && small) ? sweep_partials(ctx, s) : 0;
}

void launch_sweep(tbk_ctx* ctx, const HOp& op, const void* probe_panel, uint64_t seed, int s, int K,
                         double* partials) {
  KernelTimerScope timer(ctx, TBK_KERNEL_STEP);
  const int C = sweep_cluster(ctx, s), n = (int)op.n_rows;
  // panels, row pointers, and a quarter more blocks than the average share
  const int cap = (int)std::max<int64_t>(0, std::min(sweep_room(op, C), op.nnzb / C * 5 / 4 + 32)) & ~1;
  const size_t smem = 16 * (size_t)n + 4 * (n / C + 2) + 12 * (size_t)cap;
  TBK_CUDA(cudaFuncSetAttribute(moments_sweep_b1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SWEEP_SMEM));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(s * C);
  cfg.blockDim = dim3(32 * sweep_warps(ctx, op, s));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  TBK_CUDA(cudaLaunchKernelEx(&cfg, moments_sweep_b1, n, C, cap, op.row_ptr, op.col, (const double*)op.hv,
                              (const double*)probe_panel, seed, s, K, partials));
  post_launch(ctx, "moments_sweep_b1");
}

// ---- building blocks that allocate nothing (for the static-scratch entry point) --------------

// 9x9 blocks: a step on a panel takes a third of the time of one that regenerates every neighbour's probes.  1x1: the
// FP64 arithmetic hides the regeneration (us of seven steps, regenerated / from a panel: 17,576 sites x 16 probes 113 /
// 119, 216,000 x 128 of 168 blocks a row 32,472 / 32,505); FP32 from about eight blocks a row (216,000 x 128 of 7 blocks
// 1,004 / 1,006, 18 blocks 1,622 / 1,390, 77 blocks 4,812 / 3,318; 17,576 x 16 of 7 blocks 94 / 100).
bool probe_panel_pays(const HOp& op) { return op.B == 9 || (op.prec == TBK_MIXED && op.nnzb > 8 * op.n_rows); }

size_t mapped_h_bytes(const tbk_bsr* H, int prec) {
  const int bs = H->n_orb == 9 ? (prec == TBK_MIXED ? Layout<float, 9>::BS : Layout<double, 9>::BS) : 1;
  return (size_t)H->nnzb * bs * (prec == TBK_MIXED ? 4 : 8);
}

HOp prepare_hop_into(tbk_ctx* ctx, const tbk_bsr* H, double emin, double emax, int prec, void* dst, int* err) {
  TBK_CHECK_ARG(H != nullptr, "H is NULL");
  TBK_CHECK_ARG(H->n_orb == 1 || H->n_orb == 9, "n_orb must be 1 or 9");
  TBK_CHECK_ARG(H->n_atoms >= 1 && H->nnzb >= H->n_atoms, "empty or inconsistent matrix");
  TBK_CHECK_ARG(H->row_ptr && H->col && H->val, "NULL matrix array");
  TBK_CHECK_ARG(H->nnzb < INT32_MAX, "nnzb must be below 2^31");
  TBK_CHECK_ARG(std::isfinite(emin) && std::isfinite(emax) && emax > emin, "need emax > emin");
  TBK_CHECK_ARG(prec == TBK_MIXED || prec == TBK_FP64, "unknown precision");
  HOp op;
  op.n_atoms = H->n_atoms;
  op.B = H->n_orb;
  op.prec = prec;
  op.nnzb = H->nnzb;
  op.n_rows = (int64_t)H->n_atoms * H->n_orb;
  op.row_ptr = H->row_ptr;
  op.col = H->col;
  op.hv = dst;
  const double shift = 0.5 * (emax + emin), inv = 2.0 / (emax - emin);
  const int blk = MAP_THREADS, grid = map_grid(op);
  if (prec == TBK_MIXED) {
    if (op.B == 9)
      map_h_kernel<float, 9><<<grid, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, H->val, shift, inv, (float*)dst, err);
    else
      map_h_kernel<float, 1><<<grid, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, H->val, shift, inv, (float*)dst, err);
  } else {
    if (op.B == 9)
      map_h_kernel<double, 9><<<grid, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, H->val, shift, inv, (double*)dst, err);
    else
      map_h_kernel<double, 1><<<grid, blk, 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, H->val, shift, inv, (double*)dst, err);
  }
  post_launch(ctx, "map_h_kernel");
  return op;
}

void launch_partial_sums(tbk_ctx* ctx, const double* partials, int nctas, int steps, double* sums) {
  reduce_partials<<<steps, 256, 0, ctx->stream>>>(partials, nctas, sums);
  post_launch(ctx, "reduce_partials");
}

void launch_moment_reduction(tbk_ctx* ctx, const double* partials, int nctas, int K, int order, int s,
                             int64_t n_rows, int direct, double* sums, double* moments, int* flag) {
  if (K >= 1 && partials) launch_partial_sums(ctx, partials, nctas, K, sums);
  finish_moments<<<1, 256, 0, ctx->stream>>>(sums, K, order, s, n_rows, direct, moments, flag);
  post_launch(ctx, "finish_moments");
}

}  // namespace tbk

using namespace tbk;

namespace tbk {
// The moments sweep of tbk_chebyshev_moments; with per_probe, every step is followed by the
// per-probe dot products of its panels.  With probe_panel the probe block y_0 is that panel (the
// first step reads it as its source, the second as its y_{j-1}) and the moments divide by s_norm.
void moments_sweep(tbk_ctx* ctx, const tbk_bsr* H, double emin, double emax, uint64_t probe_seed,
                   int32_t n_probes, int32_t order, int32_t flags, double* moments, double* per_probe,
                   const void* probe_panel, int s_norm) {
  TBK_CHECK_ARG(order >= 1, "order must be >= 1");
  TBK_CHECK_ARG(n_probes >= 4 && n_probes % 4 == 0, "n_probes must be a positive multiple of 4");
  TBK_CHECK_ARG((flags & ~(TBK_FP64 | TBK_MOMENTS_DIRECT | TBK_PLAIN_KERNEL | TBK_TENSOR_CORES)) == 0,
                "unknown flag");
  const int prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  const int direct = (flags & TBK_MOMENTS_DIRECT) ? 1 : 0;
  TBK_CHECK_ARG(!probe_panel || (!direct && !per_probe), "a stored probe block takes doubled moments only");
  const int nrm = probe_panel && s_norm > 0 ? s_norm : n_probes;
  int* flag = (int*)scratch(ctx, WS_FLAGS, 64);
  TBK_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), ctx->stream));
  HOp op = prepare_hop(ctx, H, emin, emax, prec, WS_HHAT, flag);
  const int s = n_probes;
  const size_t esz = prec == TBK_MIXED ? 4 : 8;
  const size_t panel = (size_t)op.n_rows * s * esz;
  const int K = direct ? order - 1 : order / 2;   // steps: largest moment index 2K >= order - 1
  const int sweep = sweep_ctas(ctx, op, s, K, direct, per_probe != nullptr, flags);
  const int nctas = sweep ? sweep
                          : step_grid_ctas(ctx, op, s, K, (flags & (TBK_TENSOR_CORES | TBK_PLAIN_KERNEL)) != 0);
  double* partials = (double*)scratch(ctx, WS_PARTIALS, sizeof(double) * 2 * (size_t)std::max(1, K) * nctas);
  double* sums = (double*)scratch(ctx, WS_MISC, sizeof(double) * 2 * (size_t)std::max(1, K) + 64);
  if (sweep) launch_sweep(ctx, op, probe_panel, probe_seed, s, K, partials);
  void* A = K >= 1 && !sweep ? scratch(ctx, WS_PANEL0, panel) : nullptr;
  void* Bp = K >= 2 && !sweep ? scratch(ctx, WS_PANEL1, panel) : nullptr;
  // per-probe dots: row-block partials of one step, then K x s x 2 reduced dots
  const int64_t rpb = (op.n_rows + PD_BLOCKS - 1) / PD_BLOCKS;
  const int nrb = (int)((op.n_rows + rpb - 1) / rpb);
  double* pd_part = per_probe ? (double*)scratch(ctx, WS_PANEL2, sizeof(double) * 2 * (size_t)nrb * s) : nullptr;
  double* pd_dots = per_probe ? (double*)scratch(ctx, WS_SEGMENT, sizeof(double) * 2 * (size_t)std::max(1, K) * s)
                              : nullptr;
  void *cur = nullptr, *prev = nullptr;
  // y_0: the given panel, or one written into the second step's, or (NULL) regenerated by the first two steps
  void* y0 = probe_panel ? const_cast<void*>(probe_panel) : (probe_panel_pays(op) ? Bp : nullptr);
  for (int j = 1; j <= K && !sweep; ++j) {
    StepArgs a;
    a.seed = probe_seed;
    a.s = s;
    a.direct = direct;
    a.partials = partials + (size_t)(j - 1) * nctas * 2;
    a.err = flag;
    a.force_simple = (flags & TBK_PLAIN_KERNEL) ? 1 : 0;
    a.use_tc = (flags & TBK_TENSOR_CORES) ? 1 : 0;
    a.grid = nctas;
    if (j == 1) {
      // a further step follows: its panel holds the probe block until then
      if (y0 && !probe_panel) launch_scaled_probe(ctx, op, y0, 1.0, probe_seed, s);
      a.yin = y0;
      a.cur_is_probe = y0 ? 0 : 1;
      a.alpha = 1.0;
      a.yout = A;
      cur = A;
    } else if (j == 2) {
      a.yin = A;
      a.alpha = 2.0;
      if (y0) a.yprev = y0; else a.c_r = -1.0;
      a.yout = Bp;
      prev = A;
      cur = Bp;
    } else {
      a.yin = cur;
      a.yprev = prev;
      a.yout = prev;
      a.alpha = 2.0;
      std::swap(cur, prev);  // y_{j} now lives where y_{j-2} was
    }
    launch_step(ctx, op, a);
    if (per_probe) {
      // y_j at a.yout; y_{j-1} at a.yin (the probe block for j = 1)
      if (prec == TBK_MIXED)
        probe_dots<float><<<nrb, 256, 0, ctx->stream>>>(op.n_rows, s, rpb, (const float*)a.yout,
                                                        (const float*)a.yin, probe_seed, direct, pd_part);
      else
        probe_dots<double><<<nrb, 256, 0, ctx->stream>>>(op.n_rows, s, rpb, (const double*)a.yout,
                                                         (const double*)a.yin, probe_seed, direct, pd_part);
      post_launch(ctx, "probe_dots");
      probe_dots_reduce<<<ceil_div(s, 256), 256, 0, ctx->stream>>>(nrb, s, pd_part,
                                                                    pd_dots + (size_t)(j - 1) * 2 * s);
      post_launch(ctx, "probe_dots_reduce");
    }
  }
  launch_moment_reduction(ctx, partials, nctas, K, order, nrm, op.n_rows, direct, sums, moments, flag);
  if (per_probe) {
    const int64_t n = (int64_t)order * s;
    probe_moments_finish<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        pd_dots, K, order, s, op.n_rows, direct, per_probe);
    post_launch(ctx, "probe_moments_finish");
  }
  int hflag = 0;
  TBK_CUDA(cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  check_diagonal_flag(hflag);
  if (hflag & 2) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the recurrence kernel expired");
  if (hflag)
    throw Error(TBK_ERR_SPECTRUM, "a Chebyshev panel grew beyond ||r||: the spectrum of H is not "
                                  "inside [emin, emax]");
}
}  // namespace tbk

extern "C" int tbk_chebyshev_moments(tbk_ctx* ctx, const tbk_bsr* H, double emin, double emax,
                                     uint64_t probe_seed, int32_t n_probes, int32_t order,
                                     int32_t flags, double* moments) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr, "ctx is NULL");
  TBK_CHECK_ARG(moments != nullptr, "moments is NULL");
  DeviceGuard dg(ctx);
  moments_sweep(ctx, H, emin, emax, probe_seed, n_probes, order, flags, moments, nullptr);
  TBK_API_END
}

extern "C" int tbk_chebyshev_probe_moments(tbk_ctx* ctx, const tbk_bsr* H, double emin, double emax,
                                           uint64_t probe_seed, int32_t n_probes, int32_t order,
                                           int32_t flags, double* moments, double* per_probe) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr, "ctx is NULL");
  TBK_CHECK_ARG(per_probe != nullptr, "per_probe is NULL");
  DeviceGuard dg(ctx);
  double* mom = moments;
  if (!mom) mom = (double*)scratch(ctx, WS_COEF, sizeof(double) * (size_t)std::max(1, order));
  moments_sweep(ctx, H, emin, emax, probe_seed, n_probes, order, flags, mom, per_probe);
  TBK_API_END
}

extern "C" int tbk_test_step_grid(tbk_ctx* ctx, const tbk_bsr* H, int32_t n_probes, int32_t order, int32_t flags,
                                  int32_t* n_ctas) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr && H != nullptr && n_ctas != nullptr, "NULL argument");
  TBK_CHECK_ARG(H->n_orb == 1 || H->n_orb == 9, "n_orb must be 1 or 9");
  TBK_CHECK_ARG(H->n_atoms >= 1 && order >= 1 && n_probes >= 4 && n_probes % 4 == 0, "bad size");
  DeviceGuard dg(ctx);
  HOp op;
  op.B = H->n_orb;
  op.prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  op.n_atoms = H->n_atoms;
  op.n_rows = (int64_t)H->n_atoms * H->n_orb;
  op.nnzb = H->nnzb;
  *n_ctas = step_grid_ctas(ctx, op, n_probes, (flags & TBK_MOMENTS_DIRECT) ? order - 1 : order / 2,
                           (flags & (TBK_TENSOR_CORES | TBK_PLAIN_KERNEL)) != 0);
  TBK_API_END
}
