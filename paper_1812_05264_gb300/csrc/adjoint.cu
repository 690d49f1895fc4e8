// a9-a10: analytic derivative of the polynomial free-energy estimate (Sec. II.D, Eq.
// polynomial_response with S = I) and Hellmann-Feynman forces (Sec. II.A, Eq. observable).
//
// Omega^ = (1/s) sum_i r_i^T q(H^) r_i with q = sum_k c_k C_k, c_k = d_k beta_k[g].  Its gradient
// with respect to H, the bounds held fixed, is
//   G = (2/W)(1/s) sum_i sum_{j=0}^{p-2} y_ij x_ij^T,
//   y_j = C_j(H^) r,   x_j = (2 - delta_j0) b_{j+1},   b_m = sum_{k>=m} c_k U_{k-m}(H^) r,
// and b obeys the backward (Clenshaw) recurrence b_m = c_m r + 2 H^ b_{m+1} - b_{m+2}.  The
// backward sweep runs j = p-2 .. 0, adding y_j b_{j+1}^T on the block pattern and advancing b.
// The y_j are replayed from checkpoints kept every `seg` steps of a forward sweep; each segment
// is recomputed into a panel buffer just before its backward steps.
#include <algorithm>
#include <cmath>
#include <functional>
#include <type_traits>
#include <vector>

#include "adjoint_plan.cuh"
#include "bulk.cuh"
#include "cheb.cuh"
#include "model.cuh"
#include "sk.cuh"
#include "sums.cuh"

namespace tbk {

void coefficients(tbk_ctx* ctx, int fn, int p, double emin, double emax, double mu, double kT,
                  int damping, double* out);

// ---- sampled outer products for any probe count and precision -----------------------------------
//
// Gacc[k] += w * sum_probes y[a rows] (x) x[b rows]^T for every stored block k = (a, b); one writer per
// entry and launch, so the sums do not depend on timing.

// Row of stored block k (row_ptr[a] <= k < row_ptr[a + 1]), by the whole warp: 32 places at a time.
__device__ __forceinline__ int row_of_block(const int32_t* __restrict__ row_ptr, int n_atoms, int k, int lane) {
  int lo = 0, n = n_atoms;  // the row is in [lo, lo + n)
  while (n > 1) {
    const int step = (n + 31) / 32, at = lo + lane * step;
    const bool le = lane * step < n && __ldg(row_ptr + at) <= k;
    const int j = 31 - __clz((int)__ballot_sync(0xffffffffu, le));  // row_ptr[lo] <= k: lane 0 always
    n = min(step, n - j * step);
    lo += j * step;
  }
  return lo;
}

// 1x1 blocks: one warp per stored block.
template <typename T>
__global__ void __launch_bounds__(256)
sddmm_one(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
          const T* __restrict__ y, const T* __restrict__ x, int s, double w, double* __restrict__ Gacc,
          int64_t nnzb) {
  pdl_wait();
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= nnzb) return;
  const int lo = row_of_block(row_ptr, n_atoms, (int)k, lane), b = __ldg(col + k);
  T acc = T(0);
  for (int p = lane; p < s; p += 32)
    acc = fma(y[(int64_t)lo * s + p], x[(int64_t)b * s + p], acc);
  double v = (double)acc;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) Gacc[k] += w * v;
}

__device__ __forceinline__ float2 shfl_xor2(float2 v, int off) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off));
}
// Lane values of 2 N entries, (2 p, 2 p + 1) in v[p] -> the lanes' sum of entry e in each lane with e in its lowest
// bits: a butterfly reduce-scatter, each addition with its rounding errors.  A warp's FP64 addition takes the
// SM about 19 cycles.
template <int N>
__device__ __forceinline__ double butterfly_sum3(Sum3 (&v)[N], int lane) {
#pragma unroll
  for (int n = N / 2; n >= 1; n >>= 1) {
    const int off = 2 * n;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int p = 0; p < n; ++p) {
      const Sum3 give = up ? v[p] : v[p + n];
      if (up) v[p] = v[p + n];
      sum3_add(v[p], {shfl_xor2(give.h, off), shfl_xor2(give.m, off), shfl_xor2(give.l, off)});
    }
  }
  const bool odd = (lane & 1) != 0;
  auto mine = [&](float2 u) { return make_float2(odd ? u.y : u.x, 0.f); };
  auto other = [&](float2 u) { return make_float2(__shfl_xor_sync(0xffffffffu, odd ? u.x : u.y, 1), 0.f); };
  Sum3 t = {mine(v[0].h), mine(v[0].m), mine(v[0].l)};
  sum3_add(t, {other(v[0].h), other(v[0].m), other(v[0].l)});
  return sum3_value(t.h.x, t.m.x, t.l.x);
}
// The lanes' sum of entry `lane` of 27, through a 27 x 33 buffer of the warp: a lane adds the 32 values of its entry in
// a tree, two halves packed, without a butterfly's exchanges and selections.
__device__ __forceinline__ double transposed_sum3(const float (&v)[27], float (*buf)[33], int lane) {
#pragma unroll
  for (int e = 0; e < 27; ++e) buf[e][lane] = v[e];
  __syncwarp();
  const float* mine = buf[min(lane, 26)];
  Sum3 t[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    t[j].h = make_float2(mine[j], mine[j + 16]);
    two_sum(t[j].h, t[j].m, make_float2(mine[j + 8], mine[j + 24]));
    t[j].l = make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int n = 4; n >= 1; n >>= 1)
#pragma unroll
    for (int j = 0; j < n; ++j) sum3_add(t[j], t[j + n]);
  Sum3 r = {make_float2(t[0].h.x, 0.f), make_float2(t[0].m.x, 0.f), make_float2(t[0].l.x, 0.f)};
  sum3_add(r, {make_float2(t[0].h.y, 0.f), make_float2(t[0].m.y, 0.f), make_float2(t[0].l.y, 0.f)});
  return sum3_value(r.h.x, r.m.x, r.l.x);
}

// FP32 9x9 blocks: a warp takes three rows of a block, a lane probes lane, lane + 32, ... with 27 sums,
// the next 32 probes loaded ahead.  The lanes' sums have no fewer bits than FP64 ones.  333 atoms x 100 probes:
// 18 us against 233 for one warp per block that
// loaded as it went and added 81 FP64 butterflies (26 with all 81 sums in a warp, 12 warps per SM; 28 to
// 32 with a thread per entry and the tiles in shared memory, whose bandwidth then binds).  A whole call at 10,000
// x 100, us per order: 683 (674 with sums of two floats and a butterfly, 744 with those of three; six CTAs per SM
// 694, eight 791).
__global__ void __launch_bounds__(128, 7)
sddmm_rows32(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t nnzb,
             const float* __restrict__ y, const float* __restrict__ x, int s, double w,
             double* __restrict__ Gacc) {
  __shared__ float buf[4][27][33];
  pdl_wait();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= 3 * nnzb) return;
  const int k = (int)(gw / 3), g = (int)(gw - 3 * (int64_t)k);
  const int b = __ldg(col + k), a = row_of_block(row_ptr, n_atoms, k, lane);
  const float* yp = y + ((int64_t)9 * a + 3 * g) * s + lane;
  const float* xp = x + (int64_t)9 * b * s + lane;
  float acc[27], yv[3], xv[9];
#pragma unroll
  for (int e = 0; e < 27; ++e) acc[e] = 0.f;
  auto fetch = [&](int p, float (&yy)[3], float (&xx)[9]) {
    // past the last probe: zeros, which leave the sums as they are
    const bool in = p < s;
#pragma unroll
    for (int i = 0; i < 3; ++i) yy[i] = in ? __ldg(yp + (p - lane) + (int64_t)i * s) : 0.f;
#pragma unroll
    for (int l = 0; l < 9; ++l) xx[l] = in ? __ldg(xp + (p - lane) + (int64_t)l * s) : 0.f;
  };
  auto add = [&](const float (&yy)[3], const float (&xx)[9]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int l = 0; l < 9; ++l) acc[i * 9 + l] = fmaf(yy[i], xx[l], acc[i * 9 + l]);
  };
  fetch(lane, yv, xv);
  for (int p = lane; p - lane < s; p += 64) {
    float yn[3], xn[9];
    fetch(p + 32, yn, xn);
    add(yv, xv);
    fetch(p + 64, yv, xv);
    add(yn, xn);
  }
  const double sum = transposed_sum3(acc, buf[threadIdx.x >> 5], lane);
  if (lane < 27) atomicAdd(Gacc + (int64_t)k * 81 + 27 * g + lane, w * sum);
}

constexpr int OUT_STEPS = 64;  // steps per launch at most
struct OuterPanels {
  const float* y[OUT_STEPS];  // y_k, highest k first
  const float* x[OUT_STEPS];  // ybar_{k+1} (or b_{k+1})
};

// The same for several steps after them: a lane adds its 27 sums of each
// step to sums of three floats (13 packed operations for two entries), and one butterfly per launch adds those of
// the lanes.  A CTA is one block, so that its three warps find x in L1.  The loads' latency (12 warps per SM) and
// about 600 instructions a step bind; 168 registers are the limit, so that loads go 64 probes ahead (128: spills) and
// row offsets are formed on the way.  A whole call, us per order, 333 atoms x 100 probes: 32.8 (31.8 with sums of
// two floats, 37.1 with loads 128 ahead).
__global__ void __launch_bounds__(96, 4)
sddmm_steps32(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t nnzb,
              const __grid_constant__ OuterPanels wp, int nt, int last_is_y0, int s, double* __restrict__ Gacc) {
  pdl_wait();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= 3 * nnzb) return;
  const int k = (int)(gw / 3), g = (int)(gw - 3 * (int64_t)k);
  const int b = __ldg(col + k), a = row_of_block(row_ptr, n_atoms, k, lane);
  // byte offsets of the rows (panels are below 4 GB), so that a load needs no 64-bit arithmetic
  const uint32_t oy = 4u * ((9u * a + 3u * g) * s + lane), ox = 4u * (9u * b * s + lane), row = 4u * s;
  float acc[27], yv[2][3], xv[2][9];  // 64 probes ahead: with 128, spills take more than the latency
  Sum3 sum[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) sum[p].h = sum[p].m = sum[p].l = make_float2(0.f, 0.f);
  // probes p0 + 32 c + lane of step t; past the last probe zeros, which leave the sums as they are
  auto fetch = [&](int t, int p0, int c) {
    const char* Y = reinterpret_cast<const char*>(wp.y[t] + p0) + 128 * c;
    const char* X = reinterpret_cast<const char*>(wp.x[t] + p0) + 128 * c;
    auto at = [](const char* p, uint32_t o) { return __ldg(reinterpret_cast<const float*>(p + o)); };
    if (p0 + 32 * c + 32 <= s) {
#pragma unroll
      for (int i = 0; i < 3; ++i) yv[c][i] = at(Y, oy + i * row);
#pragma unroll
      for (int l = 0; l < 9; ++l) xv[c][l] = at(X, ox + l * row);
    } else {
      const bool in = p0 + 32 * c + lane < s;
#pragma unroll
      for (int i = 0; i < 3; ++i) yv[c][i] = in ? at(Y, oy + i * row) : 0.f;
#pragma unroll
      for (int l = 0; l < 9; ++l) xv[c][l] = in ? at(X, ox + l * row) : 0.f;
    }
  };
#pragma unroll
  for (int c = 0; c < 2; ++c)
    if (32 * c < s) fetch(0, 0, c);
  for (int t = 0; t < nt; ++t) {
#pragma unroll
    for (int e = 0; e < 27; ++e) acc[e] = 0.f;
    for (int p0 = 0; p0 < s; p0 += 64) {
      const bool more = p0 + 64 < s;
      const int tn = more ? t : t + 1, pn = more ? p0 + 64 : 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (p0 + 32 * c < s)
#pragma unroll
          for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int l = 0; l < 9; ++l) acc[i * 9 + l] = fmaf(yv[c][i], xv[c][l], acc[i * 9 + l]);
        if (tn < nt && pn + 32 * c < s) fetch(tn, pn, c);
      }
    }
    // the weight 2 is exact at any point: the sums hold half of what the launch adds, and y_0 enters with half
    if (last_is_y0 && t == nt - 1) {
#pragma unroll
      for (int e = 0; e < 27; ++e) acc[e] *= 0.5f;
    }
#pragma unroll
    for (int p = 0; p < 14; ++p) sum3_add(sum[p], make_float2(acc[2 * p], p < 13 ? acc[2 * p + 1] : 0.f));
  }
  const double v = butterfly_sum3(sum, lane);
  if (lane < 27) atomicAdd(Gacc + (int64_t)k * 81 + 27 * g + lane, 2.0 * v);
}

// FP64 9x9 blocks: a warp takes a block, 27 of its lanes three entries each over all probes (no sums
// across lanes), 32 probes of both tiles at a time through shared memory and the next 32 loaded ahead.
// Four sums per entry, over every fourth probe.  The FP64 rate binds (27 of 32 lanes at work); 200 atoms
// x 64 probes: 37 us against 161 with 81 butterflies per block.
__global__ void __launch_bounds__(128)
sddmm_rows64(int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t nnzb,
             const double* __restrict__ y, const double* __restrict__ x, int s, double w,
             double* __restrict__ Gacc) {
  __shared__ double ysh[4][9][33], xsh[4][9][33];
  pdl_wait();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (gw >= nnzb) return;
  const int k = (int)gw, i = lane / 3, l0 = 3 * (lane - 3 * i);  // entries (i, l0 .. l0 + 2), lanes below 27
  const int b = __ldg(col + k), a = row_of_block(row_ptr, n_atoms, k, lane);
  const double* ya = y + (int64_t)9 * a * s;
  const double* xb = x + (int64_t)9 * b * s;
  double yv[9], xv[9], acc[3][4];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int t = 0; t < 4; ++t) acc[j][t] = 0.0;
  auto fetch = [&](int p) {
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      yv[r] = p < s ? __ldg(ya + (int64_t)r * s + p) : 0.0;
      xv[r] = p < s ? __ldg(xb + (int64_t)r * s + p) : 0.0;
    }
  };
  fetch(lane);
  for (int p0 = 0; p0 < s; p0 += 32) {
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      ysh[warp][r][lane] = yv[r];
      xsh[warp][r][lane] = xv[r];
    }
    __syncwarp();
    fetch(p0 + 32 + lane);
    if (lane < 27) {
      const int n = min(32, s - p0);  // a multiple of 4
#pragma unroll 2
      for (int p = 0; p < n; p += 4)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const double yy = ysh[warp][i][p + t];
#pragma unroll
          for (int j = 0; j < 3; ++j) acc[j][t] = fma(yy, xsh[warp][l0 + j][p + t], acc[j][t]);
        }
    }
    __syncwarp();
  }
  if (lane < 27) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      atomicAdd(Gacc + (int64_t)k * 81 + 9 * i + l0 + j, w * ((acc[j][0] + acc[j][1]) + (acc[j][2] + acc[j][3])));
  }
}

// ---- fused Clenshaw step + sampled outer product (TMA-fed, FP32, 9x9 blocks, P = s) ------------
//
// For one backward index j and every block row a (one CTA task covers all s probes):
//   b_j[a]   = 2 sum_b H^_ab b_{j+1}[b] + c_j r[a] - b_{j+2}[a]          (skipped when bout = 0)
//   Gacc_ab += w sum_probes y_j[a] b_{j+1}[b]^T   for every neighbour block (a, b)
// The neighbour tiles b_{j+1}[b] and blocks H^_ab stream through a D-stage ring as in the
// forward step; the own-row tile y_j[a] is staged once per task.
// The 9x9 outer product of each tile is split into three groups of 3 rows, each taken by one
// consumer warp (in turn, so the load stays even): its 32 lanes cover interleaved 4-probe
// groups, and a butterfly reduce-scatter over the lanes leaves one entry per lane, added to the
// FP64 accumulator (one CTA owns each block, so each entry has one writer per launch).

template <int CW, bool SD = true>
struct SdCfg {
  static constexpr int D = SD ? 2 : 3;  // SD: 2 stages keep three CTAs within shared memory
  static constexpr int P = 128 * CW;
  static constexpr int XB = 9 * P * 4;
  static constexpr int HB = Layout<float, 9>::BS * 4;
  static constexpr int SB = ((XB + HB + 127) / 128) * 128;
  static constexpr int YB = SD ? ((XB + 127) / 128) * 128 : 0;
  static constexpr int SMEM = (D + 1) * SB + YB + 8 * (2 * D + 6);
  static constexpr int THREADS = 32 * (CW + 1);
};

// 32 lane partials per entry -> lane e holds the lane-sum of entry e.
__device__ __forceinline__ void butterfly32(float (&v)[32], int lane) {
#pragma unroll
  for (int off = 16, n = 32; off >= 1; off >>= 1, n >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int k = 0; k < n / 2; ++k) {
      const float send = up ? v[k] : v[k + n / 2];
      const float keep = up ? v[k + n / 2] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
}

// Rows 3g .. 3g+2 of the 9x9 outer product sum_p Y[i][p] X[l][p] over all P probes (lanes cover
// interleaved 4-probe groups): 27 entries, reduced over the lanes by one butterfly and added to
// the FP64 accumulator (one lane per entry).
template <int P>
__device__ __forceinline__ void sddmm_rows3(int g, const float* Y, const float* X, int lane, int64_t k,
                                            double w, double* __restrict__ Gacc) {
  // partial sums of entry (i - 3g) * 9 + l over this lane's probes; scalar accumulators keep the
  // kernel at 128 registers, so that three CTAs fit per SM
  float v1[27];
#pragma unroll
  for (int e = 0; e < 27; ++e) v1[e] = 0.f;
#pragma unroll 1
  for (int m = 0; m < P / 128; ++m) {
    const int pb = 4 * (lane + 32 * m);
    float yv[3][4];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float4 u = *reinterpret_cast<const float4*>(Y + (3 * g + i) * P + pb);
      yv[i][0] = u.x; yv[i][1] = u.y; yv[i][2] = u.z; yv[i][3] = u.w;
    }
#pragma unroll
    for (int l = 0; l < 9; ++l) {
      const float4 u = *reinterpret_cast<const float4*>(X + l * P + pb);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        float t = v1[i * 9 + l];
        t = fmaf(yv[i][0], u.x, t); t = fmaf(yv[i][1], u.y, t);
        t = fmaf(yv[i][2], u.z, t); t = fmaf(yv[i][3], u.w, t);
        v1[i * 9 + l] = t;
      }
    }
  }
  float v[32];
#pragma unroll
  for (int e = 0; e < 32; ++e) v[e] = e < 27 ? v1[e] : 0.f;
  butterfly32(v, lane);
  if (lane < 27)
    // fire-and-forget reduction: one writer per entry and launch, so the sum stays deterministic
    atomicAdd(Gacc + k * 81 + 27 * g + lane, w * (double)v[0]);
}

// SD = false: the Clenshaw step alone (the outer products are left to sddmm_window_g); the own-row
// tile y_j then streams through the ring like the other source terms.  SD = true: three CTAs of
// four consumer warps per SM, whose interleaving hides the latency of the outer product's
// reductions.  256 probes without them: five CTAs (128 registers) instead of the four of 150; us per forward
// and backward step 1,000 atoms 75.7 -> 73.1, 4,000 281 -> 275; six, with a stage less, 74.9 and 280.
template <int CW, bool SD>
__global__ void __launch_bounds__(32 * (CW + 1), SD || CW == 4 ? 3 : (CW == 2 ? 5 : 1))
clenshaw_sddmm_bulk(const int n_atoms, const int32_t* __restrict__ row_ptr,
                    const int32_t* __restrict__ col, const float* __restrict__ hv,
                    const float* __restrict__ bin, const float* bprev, float* bout,
                    const float* __restrict__ ypan, const float4 cf, const uint64_t seed,
                    const int s, const double w, double* __restrict__ Gacc, int* __restrict__ err,
                    const BatchRows batch, const float4* __restrict__ cf_cl,
                         const float* __restrict__ ym1, const float* __restrict__ yp1, const int y_first,
                    const int stall) {
  using C = SdCfg<CW, SD>;
  // every tile, the diagonal one included, streams through a ring of R = D + 1 stages
  constexpr int R = C::D + 1;
  extern __shared__ __align__(128) unsigned char smem[];
  float* Ys = reinterpret_cast<float*>(smem + R * C::SB);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + R * C::SB + C::YB);
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (R + i); };
  const uint32_t y_full = bar0 + 8u * (2 * R), y_empty = bar0 + 8u * (2 * R + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool has_prev = bprev != nullptr, has_out = bout != nullptr;
  constexpr bool y_tile = SD;  // the own-row tile y_j is staged once per task for the outer products
  if (threadIdx.x == 0) {
    for (int i = 0; i < R; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), CW);
    }
    mbar_init(y_full, 1);
    mbar_init(y_empty, CW);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();

  // own-row tiles streamed after the neighbour tiles, with the component of the (per-cluster)
  // coefficient vector that scales them: b_prev (-1), y_k (.y, when it is not staged), y_{k-1}
  // (.z), y_{k+1} (.w).  With per-cluster coefficients a tile is streamed whenever it is given.
  enum { X_PREV = 0, X_Y = 1, X_YM1 = 2, X_YP1 = 3 };
  const float* extra_src[4];
  int extra_kind[4];
  int n_extra = 0;
  if (has_out) {
    const bool any = cf_cl != nullptr;
    const bool y_own = !SD && ypan && (any || cf.y != 0.f);
    if (y_own && y_first) { extra_src[n_extra] = ypan; extra_kind[n_extra++] = X_Y; }
    if (has_prev) { extra_src[n_extra] = bprev; extra_kind[n_extra++] = X_PREV; }
    if (y_own && !y_first) { extra_src[n_extra] = ypan; extra_kind[n_extra++] = X_Y; }
    if (ym1 && (any || cf.z != 0.f)) { extra_src[n_extra] = ym1; extra_kind[n_extra++] = X_YM1; }
    if (yp1 && (any || cf.w != 0.f)) { extra_src[n_extra] = yp1; extra_kind[n_extra++] = X_YP1; }
  }
  if (warp == CW) {
    // (stall: a test of the bounded waits; nothing is copied, the consumers give up and report)
    if (lane == 0 && !stall) {
      int it = 0, y_it = 0;
      bool ok = true;
      for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
        const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
        if (y_tile) {
          ok = mbar_wait(y_empty, (y_it & 1) ^ 1);
          if (!ok) break;
          mbar_expect_tx(y_full, C::XB);
          bulk_g2s(smem_u32(Ys), ypan + (int64_t)9 * a * s, C::XB, y_full);
          ++y_it;
        }
        // after the neighbour tiles: the own-row tiles of b_prev, y_{k-1} and y_{k+1} (when used)
        const int nb = k1 - k0;
        const int nt = nb + n_extra;
        for (int q = 0; q < nt && ok; ++q) {
          const bool is_prev = q >= nb;
          const float* extra = is_prev ? extra_src[q - nb] : nullptr;
          const int b = is_prev ? a : __ldg(col + k0 + q);
          const int st = it % R;
          ok = mbar_wait(empty(st), ((it / R) & 1) ^ 1);
          if (!ok) break;
          const uint32_t dst = smem_u32(smem + st * C::SB), bar = full(st);
          ++it;
          const float* src = (is_prev ? extra : bin) + (int64_t)9 * b * s;
          mbar_expect_tx(bar, C::XB + (is_prev ? 0 : C::HB));
          bulk_g2s(dst, src, C::XB, bar);
          if (!is_prev) bulk_g2s(dst + C::XB, hv + (int64_t)(k0 + q) * Layout<float, 9>::BS, C::HB, bar);
        }
      }
      if (!ok) {
        // let the copies in flight land before the CTA exits
        atomicOr(err, 2);
        for (int j = (it > R ? it - R : 0); j < it; ++j) mbar_wait(full(j % R), (j / R) & 1);
        if (y_tile && y_it > 0) mbar_wait(y_full, (y_it - 1) & 1);
      }
    }
    return;
  }

  int it = 0, y_it = 0;
  bool ok = true;
  uint32_t rdy = 0;  // stage it % R was found ready by the early test
  const int pl = 4 * threadIdx.x;
  for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    // probe stream and cluster-local row of this atom; per-cluster coefficient in batches
    uint64_t sd = seed;
    int64_t rloc = (int64_t)9 * a;
    float4 cfa = cf;  // (probe, own y, y_{k-1}, y_{k+1}) coefficients of the source term
    if (batch.atom_cl) {
      const int cl = __ldg(batch.atom_cl + a);
      sd = __ldg(batch.seed + cl);
      rloc = (int64_t)9 * (a - __ldg(batch.atom0 + cl));
      if (cf_cl) cfa = cf_cl[cl];
    }
    if (y_tile) {
      ok = mbar_wait(y_full, y_it & 1);
      if (!ok) break;
    }
    float2 acc[9][2];  // row i, probe v: acc_at(acc, i, v)
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
      const float* X = reinterpret_cast<const float*>(base);
      if (has_out) spmm_tile_f2(X, reinterpret_cast<const float*>(base + C::XB), C::P, pl, acc);
      if constexpr (SD) {
        // row group g of this tile goes to warp (q + g + 1) mod CW: with 4 warps one warp rests
        // per tile, in turn
        for (int g = 0; g < 3; ++g)
          if ((q + g + 1) % CW == warp)
            sddmm_rows3<C::P>(g, Ys, X, lane, (int64_t)(k0 + q), w, Gacc);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(st));
      ++it;
    }
    if (!ok) break;
    if (!has_out) {
      if (y_tile) {
        __syncwarp();
        if (lane == 0) mbar_arrive(y_empty);
        ++y_it;
      }
      continue;
    }
    // y_out = 2 H^ b_in + cf.x r + cf.y y_own + (own-row tiles: -b_prev + cf.z y_{k-1} + cf.w y_{k+1})
    float yo[9][4];
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
      for (int v = 0; v < 4; ++v) yo[i][v] = 2.f * acc_at(acc, i, v);
    if (cfa.x != 0.f) {
#pragma unroll
      for (int i = 0; i < 9; ++i)
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[i][v] = fmaf(cfa.x, tbk_probe_sign(sd, rloc + i, pl + v), yo[i][v]);
    }
    if (y_tile && cfa.y != 0.f) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const float4 t = *reinterpret_cast<const float4*>(Ys + i * C::P + pl);
        yo[i][0] = fmaf(cfa.y, t.x, yo[i][0]); yo[i][1] = fmaf(cfa.y, t.y, yo[i][1]);
        yo[i][2] = fmaf(cfa.y, t.z, yo[i][2]); yo[i][3] = fmaf(cfa.y, t.w, yo[i][3]);
      }
    }
    for (int e = 0; e < n_extra; ++e) {
      const int st = it % R;
      if (!rdy) {
        ok = mbar_wait(full(st), (it / R) & 1);
        if (!ok) break;
      }
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      const float* X = reinterpret_cast<const float*>(smem + st * C::SB);
      const int kd = extra_kind[e];
      const float ce = kd == X_PREV ? -1.f : (kd == X_Y ? cfa.y : (kd == X_YM1 ? cfa.z : cfa.w));
      if (ce != 0.f) {  // a zero coefficient skips the tile (its rows may never have been formed)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const float4 t = *reinterpret_cast<const float4*>(X + i * C::P + pl);
          yo[i][0] = fmaf(ce, t.x, yo[i][0]); yo[i][1] = fmaf(ce, t.y, yo[i][1]);
          yo[i][2] = fmaf(ce, t.z, yo[i][2]); yo[i][3] = fmaf(ce, t.w, yo[i][3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty(st));
      ++it;
    }
    if (!ok) break;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int64_t row = (int64_t)9 * a + i;
      *reinterpret_cast<float4*>(bout + row * s + pl) = make_float4(yo[i][0], yo[i][1], yo[i][2], yo[i][3]);
    }
    if (y_tile) {
      __syncwarp();
      if (lane == 0) mbar_arrive(y_empty);
      ++y_it;
    }
  }
  if (!ok) atomicOr(err, 2);
}

// ---- outer products of a window of backward steps (TMA-fed, FP32, 9x9 blocks) ------------------
//
// Gacc_ab += w sum_{t < nw} sum_probes y_{k_t}[a] ybar_{k_t + 1}[b]^T for every stored block (a, b).
// Summing nw steps before the cross-lane reduction spreads its cost over nw block products.

struct WindowPanels {
  const float* y[SDW];  // y_{k_t} panels (n_rows x s)
  const float* x[SDW];  // ybar_{k_t + 1} panels
};

// One CTA task is one block row a.  Consumer warp (g, c) takes rows 3g .. 3g+2 of the block (27
// entries, one scalar sum each per lane) over probe chunk c (128 probes, 4 per lane), for g < 3
// and c < NC = P / 128.  The producer warp stages the window's own-row tiles y_{k_t}[a] once per
// block row and streams the neighbour tiles
// ybar_{k_t+1}[b] of every block through a D-stage ring read by all 3 NC warps.  Per block, each
// warp reduces its 27 sums over the lanes (one butterfly for all the window's steps) and warp
// (g, 0) adds the NC chunk partials in a fixed order and writes the 27 totals to the FP64
// accumulator: one writer per entry, so the result does not depend on timing.  (One warp holding
// all 81 entries, the earlier form, kept 6 consumer warps per SM at 128 probes: 2.80 ms per window
// on the 64-cluster batch against 2.02 ms.)
template <int NC>
struct WinGCfg {
  static constexpr int P = 128 * NC;
  static constexpr int NWARP = 3 * NC;  // consumer warps
  static constexpr int THREADS = 32 * (NWARP + 1);
  static constexpr int XB = 9 * P * 4;
  static constexpr int D = NC == 4 ? 6 : (NC == 1 ? 4 : 8);
  static constexpr int RED = 2 * 3 * NC * 32 * 4;  // [2 buffers][3 groups][NC chunks][32 lanes]
  static constexpr int NBAR = 2 * D + 2 + 12;
  static constexpr int SMEM = (SDW + D) * XB + RED + 8 * NBAR;
};

template <int NC>
__global__ void __launch_bounds__(32 * (3 * NC + 1), NC == 1 ? 5 : 1)
sddmm_window_g(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const WindowPanels wp, const int nw, const int s, const double w,
               double* __restrict__ Gacc, int* __restrict__ err, const BatchRows batch,
               const int32_t* __restrict__ kcl, const int k_lo) {
  using C = WinGCfg<NC>;
  constexpr int D = C::D, P = C::P, NWARP = C::NWARP;
  extern __shared__ __align__(128) unsigned char smem[];
  float* Yw = reinterpret_cast<float*>(smem);                       // SDW own-row tiles
  unsigned char* ring = smem + SDW * C::XB;                          // D neighbour tiles
  float* red = reinterpret_cast<float*>(smem + (SDW + D) * C::XB);   // [2][3][NC][32]
  const uint32_t bar0 = smem_u32(smem + (SDW + D) * C::XB + C::RED);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (D + i); };
  const uint32_t y_full = bar0 + 8u * (2 * D), y_empty = bar0 + 8u * (2 * D + 1);
  auto red_full = [&](int b, int g) { return bar0 + 8u * (2 * D + 2 + 3 * b + g); };
  auto red_empty = [&](int b, int g) { return bar0 + 8u * (2 * D + 8 + 3 * b + g); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < D; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), NWARP);
    }
    mbar_init(y_full, 1);
    mbar_init(y_empty, NWARP);
    for (int b = 0; b < 2; ++b)
      for (int g = 0; g < 3; ++g) {
        mbar_init(red_full(b, g), NC);
        mbar_init(red_empty(b, g), 1);
      }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();
  // steps of the window that take part for atom a
  auto atom_window = [&](int a) {
    return batch.atom_cl && kcl ? min(nw, max(0, __ldg(kcl + __ldg(batch.atom_cl + a)) - k_lo)) : nw;
  };

  if (warp == NWARP) {
    // producer warp: lane 0 issues the copies
    int it = 0, y_it = 0;
    bool ok = true;
    for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
      const int nwa = atom_window(a);
      if (nwa == 0) continue;
      if (lane == 0) ok = mbar_wait(y_empty, (y_it & 1) ^ 1);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      if (lane == 0) {
        mbar_expect_tx(y_full, nwa * C::XB);
        for (int t = 0; t < nwa; ++t)
          bulk_g2s(smem_u32(Yw + t * 9 * P), wp.y[t] + (int64_t)9 * a * s, C::XB, y_full);
      }
      ++y_it;
      if (lane == 0) {
        const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
        for (int q = k0; q < k1 && ok; ++q) {
          const int b = __ldg(col + q);
          for (int t = 0; t < nwa && ok; ++t) {
            const int st = it % D;
            ok = mbar_wait(empty(st), ((it / D) & 1) ^ 1);
            if (!ok) break;
            mbar_expect_tx(full(st), C::XB);
            bulk_g2s(smem_u32(ring + st * C::XB), wp.x[t] + (int64_t)9 * b * s, C::XB, full(st));
            ++it;
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    if (!ok && lane == 0) {
      atomicOr(err, 2);
      for (int j = (it > D ? it - D : 0); j < it; ++j) mbar_wait(full(j % D), (j / D) & 1);
      if (y_it > 0) mbar_wait(y_full, (y_it - 1) & 1);
    }
    return;
  }

  const int g = warp / NC, c = warp - g * NC;
  const int pl = 128 * c + 4 * lane;  // this lane's 4 probes
  int it = 0, y_it = 0, r_it = 0;
  bool ok = true;
  for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
    const int nwa = atom_window(a);
    if (nwa == 0) continue;
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    ok = mbar_wait(y_full, y_it & 1);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) break;
    for (int q = k0; q < k1; ++q) {
      float acc[27];
      // step t of the window for this block (first: the sums start here); false: a wait expired
      auto tile = [&](int t, auto first) {
        const int st = it % D;
        ok = mbar_wait(full(st), (it / D) & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return false;
        const float* X = reinterpret_cast<const float*>(ring + st * C::XB);
        const float* Y = Yw + t * 9 * P + 3 * g * P;
        float4 yv[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) yv[i] = *reinterpret_cast<const float4*>(Y + i * P + pl);
#pragma unroll
        for (int l = 0; l < 9; ++l) {
          const float4 xv = *reinterpret_cast<const float4*>(X + l * P + pl);
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            float u = decltype(first)::value ? yv[i].x * xv.x : fmaf(yv[i].x, xv.x, acc[i * 9 + l]);
            u = fmaf(yv[i].y, xv.y, u);
            u = fmaf(yv[i].z, xv.z, u); u = fmaf(yv[i].w, xv.w, u);
            acc[i * 9 + l] = u;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(st));
        ++it;
        return true;
      };
      if (nwa == SDW) {  // a full window: the step loop unrolled
        if (tile(0, std::true_type())) {
#pragma unroll
          for (int t = 1; t < SDW; ++t)
            if (!tile(t, std::false_type())) break;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 27; ++e) acc[e] = 0.f;
        for (int t = 0; t < nwa; ++t)
          if (!tile(t, std::false_type())) break;
      }
      if (!ok) break;
      // lanes -> lane e holds this chunk's sum of entry 27 g + e
      float v[32];
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = e < 27 ? acc[e] : 0.f;
      butterfly32(v, lane);
      if constexpr (NC == 1) {
        // one chunk: this warp alone holds the totals of its 27 entries (one writer per entry)
        if (lane < 27) atomicAdd(Gacc + (int64_t)q * 81 + 27 * g + lane, w * (double)v[0]);
        continue;
      }
      const int rb = r_it & 1, use = r_it >> 1;
      if (use > 0) {
        ok = mbar_wait(red_empty(rb, g), (use - 1) & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
      }
      float* R = red + (rb * 3 + g) * NC * 32;
      R[c * 32 + lane] = v[0];
      __syncwarp();
      if (lane == 0) mbar_arrive(red_full(rb, g));
      if (c == 0) {
        // fixed-order sum over the chunks, one writer per entry
        ok = mbar_wait(red_full(rb, g), use & 1);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (lane < 27) {
          float tsum = R[lane];
#pragma unroll
          for (int cc = 1; cc < NC; ++cc) tsum += R[cc * 32 + lane];
          atomicAdd(Gacc + (int64_t)q * 81 + 27 * g + lane, w * (double)tsum);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(red_empty(rb, g));
      }
      ++r_it;
    }
    if (!ok) break;
    __syncwarp();
    if (lane == 0) mbar_arrive(y_empty);
    ++y_it;
  }
  if (!ok) atomicOr(err, 2);
}

// ---- outer products of one or more steps, after them (FP32, 9x9 blocks, 128 or 256 probes) --------------
//
// Gacc_ab += sum_t w_t sum_probes y_t[a] x_t[b]^T, t in order, for every stored block (a, b): what the
// fused kernel adds inside its steps, with its additions (per lane over its interleaved 4-probe groups,
// a butterfly over the lanes, FP64 over the steps), so the result has its bits.  A warp holds all 81 sums
// of a block: 18 16-byte reads serve 324 FMAs where the fused kernel's three rows per warp read 12 for
// 108.  The next 128 probes (or the next step or block) of x come into each register as the rows are done
// with it: 8/9 of the FMAs cover their latency.  16 warps per SM of 121 registers at 128 probes, 12 of 168 at
// 256; what binds is the latency that these leave (issue 64 to 66 % busy, L1 54 to 60 %) and, at 128 probes, the
// butterfly (372 of 775 instructions a block and step).
// us per backward step with its outer products, fused -> a step kernel and these: 147 atoms x 128 probes
// 31 -> 11, 1,000 x 128 61 -> 30, 10,000 x 128 488 -> 263, 147 x 256 27 -> 15, 1,000 x 256 66 -> 58, 10,000
// x 256 548 -> 510.  At 512 probes both take the same (823 -> 836 at 10,000 atoms) and the fused kernel stays.
// 128 probes: a warp takes one block through all steps, the FP64 accumulator in registers; y_t[a] comes
// from L1, where the row's other blocks use it too.
__global__ void __launch_bounds__(128, 3)
outer_blocks(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
             const int64_t nnzb, const __grid_constant__ OuterPanels wp, const int nt, const int last_is_y0,
             double* __restrict__ Gacc) {
  constexpr int S = 128;
  pdl_wait();
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= nnzb) return;
  const int k = (int)gw, b = __ldg(col + k), a = row_of_block(row_ptr, n_atoms, k, lane);
  const int64_t offa = (int64_t)9 * a * S + 4 * lane, offb = (int64_t)9 * b * S + 4 * lane;
  double* g = Gacc + (int64_t)k * 81 + lane;
  double ga[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) ga[j] = lane < 27 ? g[27 * j] : 0.0;
  float4 x[9];
#pragma unroll
  for (int l = 0; l < 9; ++l) x[l] = __ldg(reinterpret_cast<const float4*>(wp.x[0] + offb + l * S));
  for (int t = 0; t < nt; ++t) {
    const float* yt = wp.y[t] + offa;
    const float* xn = wp.x[min(t + 1, nt - 1)] + offb;
    float4 y[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) y[i] = __ldg(reinterpret_cast<const float4*>(yt + i * S));
    float acc[81];
#pragma unroll
    for (int l = 0; l < 9; ++l) {
      const float4 u = x[l];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        float v = y[i].x * u.x;
        v = fmaf(y[i].y, u.y, v);
        v = fmaf(y[i].z, u.z, v); v = fmaf(y[i].w, u.w, v);
        acc[i * 9 + l] = v;
      }
      x[l] = __ldg(reinterpret_cast<const float4*>(xn + l * S));
    }
    const double w = last_is_y0 && t == nt - 1 ? 1.0 : 2.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float v[32];
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = e < 27 ? acc[27 * j + e] : 0.f;
      butterfly32(v, lane);
      ga[j] += w * (double)v[0];
    }
  }
  if (lane < 27) {
#pragma unroll
    for (int j = 0; j < 3; ++j) g[27 * j] = ga[j];
  }
}

// 256 probes: a CTA of NW warps takes a block row and stages y_t[a] in shared memory, two steps
// deep; a warp takes every NW-th block.
template <int NW>
__global__ void __launch_bounds__(32 * NW, 12 / NW)
outer_rows(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
            const __grid_constant__ OuterPanels wp, const int nt, const int last_is_y0, double* __restrict__ Gacc,
            int* __restrict__ err, const int stall) {
  constexpr int NC = 2, S = 128 * NC, XB = 9 * S * 4;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[4];
  const uint32_t full = smem_u32(bars), empty = full + 16;  // two each
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(full + 8 * i, 1);
      mbar_init(empty + 8 * i, NW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_wait();
  // tiles y_t[a] of the CTA's rows and steps, in order: number it in buffer it & 1
  const int rows = (n_atoms - blockIdx.x + gridDim.x - 1) / gridDim.x;
  const int n_tiles = rows * nt;
  // (stall: a test of the bounded waits; nothing is copied, the warps give up and report)
  auto issue = [&](int it) {
    if (stall) return;
    const int a = blockIdx.x + (it / nt) * gridDim.x;
    const uint32_t bar = full + 8 * (it & 1);
    mbar_expect_tx(bar, XB);
    bulk_g2s(smem_u32(smem + (it & 1) * XB), wp.y[it % nt] + (int64_t)9 * a * S, XB, bar);
  };
  if (threadIdx.x == 0) {
    issue(0);
    if (n_tiles > 1) issue(1);
  }
  bool ok = true;
  int it = 0;
  for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
    const int k0 = __ldg(row_ptr + a), nb = __ldg(row_ptr + a + 1) - k0;
    float4 x[9];
    if (warp < nb) {
      const float* x0 = wp.x[0] + (int64_t)9 * __ldg(col + k0 + warp) * S + 4 * lane;
#pragma unroll
      for (int l = 0; l < 9; ++l) x[l] = __ldg(reinterpret_cast<const float4*>(x0 + l * S));
    }
    for (int t = 0; t < nt; ++t, ++it) {
      ok = mbar_wait(full + 8 * (it & 1), (it >> 1) & 1);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const float* Y = reinterpret_cast<const float*>(smem + (it & 1) * XB) + 4 * lane;
      const double w = last_is_y0 && t == nt - 1 ? 1.0 : 2.0;
      for (int q = warp; q < nb; q += NW) {
        // where the next stage's x lies: this block's next probes, the next block, the next step
        const float* xq = wp.x[t] + (int64_t)9 * __ldg(col + k0 + q) * S + 4 * lane;
        const bool more = q + NW < nb;
        const float* xn = wp.x[more || t + 1 == nt ? t : t + 1] +
                          (int64_t)9 * __ldg(col + k0 + (more ? q + NW : warp)) * S + 4 * lane;
        float acc[81];
#pragma unroll
        for (int e = 0; e < 81; ++e) acc[e] = 0.f;
#pragma unroll 1
        for (int m = 0; m < NC; ++m) {
          float4 y[9];
#pragma unroll
          for (int i = 0; i < 9; ++i) y[i] = *reinterpret_cast<const float4*>(Y + i * S + 128 * m);
          const float* nx = m + 1 < NC ? xq + 128 * (m + 1) : xn;
#pragma unroll
          for (int l = 0; l < 9; ++l) {
            const float4 u = x[l];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              float v = acc[i * 9 + l];
              v = fmaf(y[i].x, u.x, v); v = fmaf(y[i].y, u.y, v);
              v = fmaf(y[i].z, u.z, v); v = fmaf(y[i].w, u.w, v);
              acc[i * 9 + l] = v;
            }
            x[l] = __ldg(reinterpret_cast<const float4*>(nx + l * S));
          }
        }
        double* g = Gacc + (int64_t)(k0 + q) * 81 + lane;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          float v[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] = e < 27 ? acc[27 * j + e] : 0.f;
          butterfly32(v, lane);
          // fire-and-forget: one writer per entry, its additions in program order
          if (lane < 27) atomicAdd(g + 27 * j, w * (double)v[0]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + 8 * (it & 1));
      if (threadIdx.x == 0 && it + 2 < n_tiles) {
        if (mbar_wait(empty + 8 * (it & 1), (it >> 1) & 1)) issue(it + 2);
        else atomicOr(err, 2);  // nothing is copied: the consumers give up in turn
      }
    }
  }
  if (!ok) {
    if (lane == 0) atomicOr(err, 2);
    // let the copies in flight land before the CTA exits
    if (threadIdx.x == 0 && !stall)
      for (int j = it; j < it + 2 && j < n_tiles; ++j) mbar_wait(full + 8 * (j & 1), (j >> 1) & 1);
  }
}

// ---- self-fed adjoint step for 128 probes (windowed schedule) ---------------------------------
//
// clenshaw_sddmm_bulk<1, false> with one warp per CTA and no producer warp: lane 0 keeps R tiles
// in flight (each row's neighbour tiles with their blocks, then its own-row source tiles) and
// refills a stage as soon as the warp is done with it, so more consumer warps fit per SM.
template <int R>
struct ClenSelfCfg {
  static constexpr int P = 128;
  static constexpr int XB = 9 * P * 4;
  static constexpr int HB = Layout<float, 9>::BS * 4;
  static constexpr int SB = ((XB + HB + 127) / 128) * 128;
  static constexpr int SMEM = R * SB + 8 * R;
};

template <int R>
__global__ void __launch_bounds__(32)
clenshaw_self(const int n_atoms, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
              const float* __restrict__ hv, const float* __restrict__ bin, const float* bprev, float* bout,
              const float* __restrict__ ypan, const float4 cf, const uint64_t seed, const int s,
              int* __restrict__ err, const BatchRows batch, const float4* __restrict__ cf_cl,
              const float* __restrict__ ym1, const float* __restrict__ yp1, const int y_first, const int stall) {
  using C = ClenSelfCfg<R>;
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t bar0 = smem_u32(smem + R * C::SB);
  auto full = [&](int i) { return bar0 + 8u * i; };
  const int lane = threadIdx.x;
  enum { X_PREV = 0, X_Y = 1, X_YM1 = 2, X_YP1 = 3 };
  const float* extra_src[4];
  int extra_kind[4];
  int n_extra = 0;
  {
    const bool any = cf_cl != nullptr;
    const bool y_own = ypan && (any || cf.y != 0.f);
    if (y_own && y_first) { extra_src[n_extra] = ypan; extra_kind[n_extra++] = X_Y; }
    if (bprev) { extra_src[n_extra] = bprev; extra_kind[n_extra++] = X_PREV; }
    if (y_own && !y_first) { extra_src[n_extra] = ypan; extra_kind[n_extra++] = X_Y; }
    if (ym1 && (any || cf.z != 0.f)) { extra_src[n_extra] = ym1; extra_kind[n_extra++] = X_YM1; }
    if (yp1 && (any || cf.w != 0.f)) { extra_src[n_extra] = yp1; extra_kind[n_extra++] = X_YP1; }
  }
  if (lane == 0) {
    for (int i = 0; i < R; ++i) mbar_init(full(i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  pdl_wait();
  int p_a = blockIdx.x, p_q = 0, p_k0 = 0, p_nb = 0, issued = 0;
  auto load_row = [&]() {  // rows with no tile (no stored block, no source term) are skipped
    for (; p_a < n_atoms; p_a += gridDim.x) {
      p_k0 = __ldg(row_ptr + p_a);
      p_nb = __ldg(row_ptr + p_a + 1) - p_k0;
      if (p_nb + n_extra > 0) break;
    }
  };
  // (stall: a test of the bounded waits; nothing is copied, the warp gives up and reports)
  auto issue_next = [&]() {
    if (stall || p_a >= n_atoms) return;
    const bool own = p_q >= p_nb;
    const int b = own ? p_a : __ldg(col + p_k0 + p_q);
    const float* src = (own ? extra_src[p_q - p_nb] : bin) + (int64_t)9 * b * s;
    const int st = issued % R;
    const uint32_t dst = smem_u32(smem + st * C::SB), bar = full(st);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(bar, C::XB + (own ? 0 : C::HB));
    bulk_g2s(dst, src, C::XB, bar);
    if (!own) bulk_g2s(dst + C::XB, hv + (int64_t)(p_k0 + p_q) * Layout<float, 9>::BS, C::HB, bar);
    ++issued;
    if (++p_q == p_nb + n_extra) {
      p_a += gridDim.x;
      p_q = 0;
      load_row();
    }
  };
  if (lane == 0) {
    load_row();
    for (int j = 0; j < R; ++j) issue_next();
  }
  __syncwarp();
  int it = 0;
  bool ok = true;
  uint32_t rdy = 0;  // stage it % R was found ready by the early test
  const int pl = 4 * lane;
  auto consumed = [&]() {
    __syncwarp();
    if (lane == 0) issue_next();
    ++it;
  };
  for (int a = blockIdx.x; a < n_atoms && ok; a += gridDim.x) {
    const int k0 = __ldg(row_ptr + a), k1 = __ldg(row_ptr + a + 1);
    uint64_t sd = seed;
    int64_t rloc = (int64_t)9 * a;
    float4 cfa = cf;
    if (batch.atom_cl) {
      const int cl = __ldg(batch.atom_cl + a);
      sd = __ldg(batch.seed + cl);
      rloc = (int64_t)9 * (a - __ldg(batch.atom0 + cl));
      if (cf_cl) cfa = cf_cl[cl];
    }
    float2 acc[9][2];
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
      spmm_tile_f2(reinterpret_cast<const float*>(base), reinterpret_cast<const float*>(base + C::XB), C::P,
                   pl, acc);
      consumed();
    }
    if (!ok) break;
    float yo[9][4];
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
      for (int v = 0; v < 4; ++v) yo[i][v] = 2.f * acc_at(acc, i, v);
    if (cfa.x != 0.f) {
#pragma unroll
      for (int i = 0; i < 9; ++i)
#pragma unroll
        for (int v = 0; v < 4; ++v) yo[i][v] = fmaf(cfa.x, tbk_probe_sign(sd, rloc + i, pl + v), yo[i][v]);
    }
    for (int e = 0; e < n_extra; ++e) {
      const int st = it % R;
      if (!rdy) {
        ok = mbar_wait(full(st), (it / R) & 1);
        if (!ok) break;
      }
      rdy = mbar_test(full((it + 1) % R), ((it + 1) / R) & 1);
      const float* X = reinterpret_cast<const float*>(smem + st * C::SB);
      const int kd = extra_kind[e];
      const float ce = kd == X_PREV ? -1.f : (kd == X_Y ? cfa.y : (kd == X_YM1 ? cfa.z : cfa.w));
      if (ce != 0.f) {  // a zero coefficient skips the tile (its rows may never have been formed)
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const float4 t = *reinterpret_cast<const float4*>(X + i * C::P + pl);
          yo[i][0] = fmaf(ce, t.x, yo[i][0]); yo[i][1] = fmaf(ce, t.y, yo[i][1]);
          yo[i][2] = fmaf(ce, t.z, yo[i][2]); yo[i][3] = fmaf(ce, t.w, yo[i][3]);
        }
      }
      consumed();
    }
    if (!ok) break;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int64_t row = (int64_t)9 * a + i;
      *reinterpret_cast<float4*>(bout + row * s + pl) = make_float4(yo[i][0], yo[i][1], yo[i][2], yo[i][3]);
    }
  }
  if (!ok && lane == 0) {
    // let the copies in flight land before the CTA exits
    atomicOr(err, 2);
    for (int j = it; j < issued; ++j) mbar_wait(full(j % R), (j / R) & 1);
  }
}

// two stages: ~21 warps per SM instead of 14 (shared memory sets the limit); measured 11 % faster
// on the batch than three stages
constexpr int CLEN_SELF_R = 2;

// tr[k] = index of block (b, a) for block k = (a, b) (the pattern is symmetric).
__global__ void transpose_map(int n_atoms, const int32_t* __restrict__ row_ptr,
                              const int32_t* __restrict__ col, int32_t* __restrict__ tr, int* err) {
  const int a = blockIdx.x * blockDim.y + threadIdx.y;
  if (a >= n_atoms) return;
  for (int k = row_ptr[a] + threadIdx.x; k < row_ptr[a + 1]; k += blockDim.x) {
    const int b = col[k];
    int lo = row_ptr[b], hi = row_ptr[b + 1] - 1, hit = -1;
    while (lo <= hi) {
      const int mid = (lo + hi) >> 1;
      const int c = col[mid];
      if (c == a) { hit = mid; break; }
      if (c < a) lo = mid + 1; else hi = mid - 1;
    }
    tr[k] = hit;
    if (hit < 0) atomicOr(err, 1);
  }
}

// G[k] = scale * (Gacc[k] + Gacc[tr[k]]^T) / 2
template <int B>
__global__ void symmetrize(int64_t nnzb, const int32_t* __restrict__ tr, const double* __restrict__ Gacc,
                           double scale, double* __restrict__ G) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nnzb * B * B) return;
  const int64_t k = t / (B * B);
  const int e = (int)(t - k * B * B), i = e / B, l = e - i * B;
  const int64_t kt = tr[k];
  G[t] = kt < 0 ? 0.0 : 0.5 * scale * (Gacc[t] + Gacc[kt * B * B + l * B + i]);
}

__device__ __forceinline__ double mi(double d, double L) { return L > 0.0 ? d - L * rint(d / L) : d; }

// tq[k] = <G_ab, dH_ab/dd> - <G_ba, dH_ba/dd>, d = R_b - R_a, for every off-diagonal block k = (a, b) whose
// transpose is stored, else 0 (SK model).  Since H_ba(-d) = H_ab(d)^T this is <G_ab + G_ba^T, dH_ab/dd>, and
// the transpose's value is its negative: one evaluation per pair.  The FP64 units (an SM takes about 19
// cycles for a warp's instruction) bind; forward-mode derivatives of all entries of every block by a thread that walks
// its own 648 bytes took 928 us at 10,000 atoms and 372 at 1,000 and 147; this 200, 58 and 29.
// A warp takes `rows` block rows, lists their pairs a < b, and stages G_ab + G_ba^T of 32 of them at a time
// (a stride of 81 doubles: no bank conflicts) for one thread each.
constexpr int BT_LIST = 128, BT_ROWS = 8;

__global__ void __launch_bounds__(32)
bond_terms(DevModel M, const double* __restrict__ pos, int n_atoms, const int32_t* __restrict__ row_ptr,
           const int32_t* __restrict__ col, const int32_t* __restrict__ tr, const double* __restrict__ G,
           double* __restrict__ tq, int rows) {
  __shared__ double S[32 * 81];
  __shared__ int rp[BT_ROWS + 1], list_k[BT_LIST], list_a[BT_LIST];
  const int lane = threadIdx.x;
  const int a0 = blockIdx.x * rows, nr = min(rows, n_atoms - a0);
  if (lane <= nr) rp[lane] = row_ptr[a0 + lane];
  __syncwarp();
  for (int base = rp[0]; base < rp[nr]; base += BT_LIST) {
    int n_list = 0;
    for (int k0 = base; k0 < min(base + BT_LIST, rp[nr]); k0 += 32) {
      const int k = k0 + lane;
      bool take = false;
      int a = 0;
      if (k < rp[nr]) {
        while (k >= rp[a + 1]) ++a;
        a += a0;
        const int b = col[k];
        const bool zero = b == a || tr[k] < 0;
        if (zero) tq[3 * (int64_t)k] = tq[3 * (int64_t)k + 1] = tq[3 * (int64_t)k + 2] = 0.0;
        take = !zero && b > a;
      }
      const unsigned m = __ballot_sync(0xffffffffu, take);
      if (take) {
        const int e = n_list + __popc(m & ((1u << lane) - 1));
        list_k[e] = k;
        list_a[e] = a;
      }
      n_list += __popc(m);
    }
    __syncwarp();
    for (int p0 = 0; p0 < n_list; p0 += 32) {
      const int np = min(32, n_list - p0);
#pragma unroll 8
      for (int p = 0; p < np; ++p) {
        const int k = list_k[p0 + p];
        const double* g = G + (int64_t)k * 81;
        const double* gt = G + (int64_t)__ldg(tr + k) * 81;
#pragma unroll
        for (int e = lane; e < 96; e += 32)
          if (e < 81) S[p * 81 + e] = __ldg(g + e) + __ldg(gt + (e % 9) * 9 + e / 9);
      }
      __syncwarp();
      if (lane < np) {
        const int k = list_k[p0 + lane], a = list_a[p0 + lane], b = col[k], kt = tr[k];
        double d[3], t[3];
        for (int c = 0; c < 3; ++c) d[c] = mi(pos[3 * b + c] - pos[3 * a + c], M.box[c]);
        const double* w = S + lane * 81;
        sk_bond_term(d, M.V, M.r0, M.decay, [&](int i, int j) { return w[9 * i + j]; }, t);
        for (int c = 0; c < 3; ++c) {
          tq[3 * (int64_t)k + c] = t[c];
          tq[3 * (int64_t)kt + c] = -t[c];
        }
      }
      __syncwarp();
    }
  }
}

// F_a = -dOmega/dR_a = sum over row a of tq: eight lanes per atom, fixed order.
__global__ void gather_forces(int n_atoms, const int32_t* __restrict__ row_ptr, const double* __restrict__ tq,
                              double* __restrict__ F) {
  const int a = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, sub = threadIdx.x & 7;
  double f[3] = {0.0, 0.0, 0.0};
  if (a < n_atoms)
    for (int k = row_ptr[a] + sub; k < row_ptr[a + 1]; k += 8)
      for (int c = 0; c < 3; ++c) f[c] += tq[3 * (int64_t)k + c];
#pragma unroll
  for (int d = 4; d >= 1; d /= 2)
    for (int c = 0; c < 3; ++c) f[c] += __shfl_xor_sync(0xffffffffu, f[c], d);
  if (a < n_atoms && sub == 0)
    for (int c = 0; c < 3; ++c) F[3 * a + c] = f[c];
}

bool fused_eligible(const HOp& op, int s, int plain);
// The adjoint of the doubled moments: mixed 9x9 at 128, 256 or 512 probes (fused kernels), FP64 always.
static bool doubled_eligible(const HOp& op, int s, int plain) {
  return fused_eligible(op, s, plain) || (!plain && op.prec == TBK_FP64);
}

bool fused_eligible(const HOp& op, int s, int plain) {
  return !plain && op.prec == TBK_MIXED && op.B == 9 && (s == 128 || s == 256 || s == 512);
}

template <int CW, bool SD>
static void launch_fused_cw(tbk_ctx* ctx, const HOp& op, const void* bin, const void* bprev, void* bout,
                            const void* ypan, float4 cf, uint64_t seed, int s, double w, double* Gacc,
                            int* err, const BatchRows& batch, const float4* cf_cl, const void* ym1,
                            const void* yp1, int y_first) {
  using C = SdCfg<CW, SD>;
  static int occ_dev[64] = {0};
  int& occ = occ_dev[ctx->device & 63];
  if (!occ) {
    TBK_CUDA(cudaFuncSetAttribute(clenshaw_sddmm_bulk<CW, SD>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    TBK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, clenshaw_sddmm_bulk<CW, SD>, C::THREADS, C::SMEM));
    TBK_CHECK_ARG(occ > 0, "fused adjoint kernel does not fit on this device");
  }
  const int G = task_grid(op.n_atoms, (int64_t)occ * ctx->num_sms);
  launch_pdl(ctx, clenshaw_sddmm_bulk<CW, SD>, G, C::THREADS, C::SMEM, op.n_atoms, op.row_ptr, op.col,
             (const float*)op.hv, (const float*)bin, (const float*)bprev, (float*)bout, (const float*)ypan, cf, seed, s, w,
             Gacc, err, batch, cf_cl, (const float*)ym1, (const float*)yp1, y_first, ctx->stall_next_adjoint);
  ctx->stall_next_adjoint = 0;
  post_launch(ctx, "clenshaw_sddmm_bulk");
}

// A backward step, fused with its outer products (Gacc) or alone (Gacc NULL).  y_first: alone, add the
// y_k term before y_prev as the fused kernel does.
void launch_fused(tbk_ctx* ctx, const HOp& op, const void* bin, const void* bprev, void* bout,
                  const void* ypan, float4 cf, uint64_t seed, int s, double w, double* Gacc,
                  int* err, const BatchRows& batch, const float4* cf_cl, const void* ym1,
                  const void* yp1, int y_first) {
  KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
  auto go = [&](auto cw, auto sd) {
    launch_fused_cw<decltype(cw)::value, decltype(sd)::value>(ctx, op, bin, bprev, bout, ypan, cf, seed, s, w,
                                                              Gacc, err, batch, cf_cl, ym1, yp1, y_first);
  };
  using T = std::true_type;
  using F = std::false_type;
  if (s == 512) Gacc ? go(std::integral_constant<int, 4>(), T()) : go(std::integral_constant<int, 4>(), F());
  else if (s == 256) Gacc ? go(std::integral_constant<int, 2>(), T()) : go(std::integral_constant<int, 2>(), F());
  else if (Gacc) go(std::integral_constant<int, 1>(), T());
  else {
    // the adjoint step alone at 128 probes: the self-fed single-warp kernel
    using C = ClenSelfCfg<CLEN_SELF_R>;
    static int occ_dev[64] = {0};
    int& occ = occ_dev[ctx->device & 63];
    if (!occ) {
      TBK_CUDA(cudaFuncSetAttribute(clenshaw_self<CLEN_SELF_R>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
      TBK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, clenshaw_self<CLEN_SELF_R>, 32, C::SMEM));
      TBK_CHECK_ARG(occ > 0, "self-fed adjoint kernel does not fit on this device");
    }
    const int G = task_grid(op.n_atoms, (int64_t)occ * ctx->num_sms);
    launch_pdl(ctx, clenshaw_self<CLEN_SELF_R>, G, 32, C::SMEM, op.n_atoms, op.row_ptr, op.col, (const float*)op.hv,
               (const float*)bin, (const float*)bprev, (float*)bout, (const float*)ypan, cf, seed, s, err, batch, cf_cl,
               (const float*)ym1, (const float*)yp1, y_first, ctx->stall_next_adjoint);
    ctx->stall_next_adjoint = 0;
    post_launch(ctx, "clenshaw_self");
  }
}

// A backward step whose outer products run later, with the fused kernel's additions.
static void launch_adjoint_step(tbk_ctx* ctx, const HOp& op, const void* bin, void* bprev, void* bout,
                                const void* ypan, float4 cf, uint64_t seed, int s, int* err, const void* ym1,
                                const void* yp1) {
  StepArgs a;
  a.seed = seed;
  a.s = s;
  a.yin = bin;
  a.yprev = bprev;
  a.yout = bout;
  a.alpha = 2.0;
  a.c_r = cf.x;
  a.src[0] = ypan;
  a.csrc[0] = cf.y;
  a.src[1] = ym1;
  a.csrc[1] = ym1 ? cf.z : 0.0;
  a.src[2] = yp1;
  a.csrc[2] = yp1 ? cf.w : 0.0;
  a.err = err;
  a.adjoint = 1;
  a.family = TBK_KERNEL_BACKWARD;
  if (lane_adjoint_step(ctx, op, a)) return;
  launch_fused(ctx, op, bin, bprev, bout, ypan, cf, seed, s, 0.0, nullptr, err, BatchRows(), nullptr, ym1, yp1, 1);
}

// Gacc += the outer products of nt steps (in order; the last one that of y_0 when last_is_y0).
template <int NW>
static void launch_outer_rows(tbk_ctx* ctx, const HOp& op, const OuterPanels& wp, int nt, int last_is_y0, double* Gacc,
                            int* err) {
  constexpr int SMEM = 2 * 9 * 256 * 4;
  static int occ_dev[64] = {0};
  int& occ = occ_dev[ctx->device & 63];
  if (!occ) {
    TBK_CUDA(cudaFuncSetAttribute(outer_rows<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    TBK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, outer_rows<NW>, 32 * NW, SMEM));
    TBK_CHECK_ARG(occ > 0, "outer-product kernel does not fit on this device");
  }
  launch_pdl(ctx, outer_rows<NW>, task_grid(op.n_atoms, (int64_t)occ * ctx->num_sms), 32 * NW, SMEM, op.n_atoms, op.row_ptr,
             op.col, wp, nt, last_is_y0, Gacc, err, ctx->stall_next_outer);
  ctx->stall_next_outer = 0;
}

static void launch_outer(tbk_ctx* ctx, const HOp& op, const OuterPanels& wp, int nt, int last_is_y0, int s,
                         double* Gacc, int* err) {
  KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
  if (s == 128)
    launch_pdl(ctx, outer_blocks, ceil_div(op.nnzb, 4), 128, 0, op.n_atoms, op.row_ptr, op.col, op.nnzb, wp, nt,
               last_is_y0, Gacc);
  else if (op.n_atoms <= ctx->num_sms)  // few rows: all 12 warps of an SM on one row
    launch_outer_rows<12>(ctx, op, wp, nt, last_is_y0, Gacc, err);
  else
    launch_outer_rows<4>(ctx, op, wp, nt, last_is_y0, Gacc, err);
  post_launch(ctx, "outer_products");
}

void launch_sddmm(tbk_ctx* ctx, const HOp& op, const void* y, const void* x, int s, double w, double* Gacc) {
  const bool f32 = op.prec == TBK_MIXED;
  if (op.B == 9) {
    if (f32)
      launch_pdl(ctx, sddmm_rows32, ceil_div(3 * op.nnzb, 4), 128, 0, op.n_atoms, op.row_ptr, op.col, op.nnzb,
                 (const float*)y, (const float*)x, s, w, Gacc);
    else
      launch_pdl(ctx, sddmm_rows64, ceil_div(op.nnzb, 4), 128, 0, op.n_atoms, op.row_ptr, op.col, op.nnzb,
                 (const double*)y, (const double*)x, s, w, Gacc);
  } else {
    const int grid = ceil_div(op.nnzb * 32, 256);
    if (f32)
      launch_pdl(ctx, sddmm_one<float>, grid, 256, 0, op.n_atoms, op.row_ptr, op.col, (const float*)y,
                 (const float*)x, s, w, Gacc, op.nnzb);
    else
      launch_pdl(ctx, sddmm_one<double>, grid, 256, 0, op.n_atoms, op.row_ptr, op.col, (const double*)y,
                 (const double*)x, s, w, Gacc, op.nnzb);
  }
  post_launch(ctx, "sddmm");
}

// Steps of the general adjoint whose outer products run together (0: after each step).  us per order of a whole call,
// after each step -> 16 together: 147 atoms x 36 probes 20.8 -> 18.8, 333 x 36 28.4 -> 25.6, 2,500 x 36 156 -> 141, 10,000
// x 36 594 -> 544, x 64 602 -> 551, 4,000 x 68 270 -> 252; 55 x 100 18.9 -> 17.8, 333 x 100 33.2 -> 32.8, 333 x 124 33.4
// -> 34.1, 700 x 100 61.3 -> 61.8, 4,000 x 100 276 -> 294, 10,000 x 124 689 -> 813; 147 x 200 26.0 -> 28.2, 333 x 384
// 68.7 -> 98.1: with more probes the lanes' sums are a smaller part, and the registers of the kept ones cost warps.
// The kernel's row offsets have 32 bits.
static int general_deferred_steps(const tbk_ctx* ctx, const HOp& op, int s) {
  const bool few = 10 * (int64_t)op.n_atoms <= 33 * (int64_t)ctx->num_sms;
  if (op.prec != TBK_MIXED || op.B != 9 || s > (few ? 128 : 96) || 4 * op.n_rows * s >= (int64_t)1 << 32) return 0;
  return 16;
}

static void launch_sddmm_steps(tbk_ctx* ctx, const HOp& op, const OuterPanels& wp, int nt, int last_is_y0, int s,
                               double* Gacc) {
  KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
  launch_pdl(ctx, sddmm_steps32, (unsigned)op.nnzb, 96, 0, op.n_atoms, op.row_ptr, op.col, op.nnzb, wp, nt,
             last_is_y0, s, Gacc);
  post_launch(ctx, "sddmm_steps32");
}

// ---- pieces shared with the batched driver -------------------------------------------------

void launch_symmetrize(tbk_ctx* ctx, int64_t nnzb, int B, const int32_t* tr, const double* Gacc, double scale,
                       double* G) {
  const int64_t tot = nnzb * B * B;
  if (B == 9)
    symmetrize<9><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(nnzb, tr, Gacc, scale, G);
  else
    symmetrize<1><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(nnzb, tr, Gacc, scale, G);
  post_launch(ctx, "symmetrize");
}

void launch_transpose_map(tbk_ctx* ctx, int n_atoms, const int32_t* row_ptr, const int32_t* col,
                          int32_t* tr, int* err) {
  transpose_map<<<ceil_div(n_atoms, 16), dim3(8, 16), 0, ctx->stream>>>(n_atoms, row_ptr, col, tr, err);
  post_launch(ctx, "transpose_map");
}

// G[k] = scale(cluster of row a) (Gacc[k] + Gacc[tr[k]]^T) / 2 for a merged batch.
__global__ void symmetrize_batched(int n_atoms, const int32_t* __restrict__ row_ptr,
                                   const int32_t* __restrict__ tr, const int32_t* __restrict__ atom_cl,
                                   const double* __restrict__ scale_cl, const double* __restrict__ Gacc,
                                   double* __restrict__ G) {
  const int a = blockIdx.x * blockDim.y + threadIdx.y;
  if (a >= n_atoms) return;
  const double sc = scale_cl[atom_cl[a]];
  for (int k = row_ptr[a]; k < row_ptr[a + 1]; ++k)
    for (int e = threadIdx.x; e < 81; e += blockDim.x) {
      const int i = e / 9, l = e - 9 * i;
      const int64_t kt = tr[k];
      G[(int64_t)k * 81 + e] = kt < 0 ? 0.0 : 0.5 * sc * (Gacc[(int64_t)k * 81 + e] + Gacc[kt * 81 + l * 9 + i]);
    }
}

void launch_symmetrize_batched(tbk_ctx* ctx, int n_atoms, const int32_t* row_ptr, const int32_t* tr,
                               const int32_t* atom_cl, const double* scale_cl, const double* Gacc,
                               double* G) {
  symmetrize_batched<<<ceil_div(n_atoms, 8), dim3(32, 8), 0, ctx->stream>>>(n_atoms, row_ptr, tr, atom_cl,
                                                                             scale_cl, Gacc, G);
  post_launch(ctx, "symmetrize_batched");
}

void launch_forces(tbk_ctx* ctx, const DevModel& M, const double* pos, int n_atoms, const int32_t* row_ptr,
                   const int32_t* col, const int32_t* tr, const double* G, double* tq, double* F) {
  // a warp per SM quarter, up to two rounds of 32 pairs each
  const int rows = std::max(1, std::min(BT_ROWS, ceil_div(n_atoms, 4 * ctx->num_sms)));
  bond_terms<<<ceil_div(n_atoms, rows), 32, 0, ctx->stream>>>(M, pos, n_atoms, row_ptr, col, tr, G, tq, rows);
  post_launch(ctx, "bond_terms");
  gather_forces<<<ceil_div(n_atoms, 16), 128, 0, ctx->stream>>>(n_atoms, row_ptr, tq, F);
  post_launch(ctx, "gather_forces");
}

template <int NC>
static void launch_window_g(tbk_ctx* ctx, const HOp& op, const WindowPanels& wp, int nw, int s, double w, double* Gacc, int* err, const BatchRows& batch,
                            const int32_t* kcl, int k_lo) {
  using C = WinGCfg<NC>;
  static int occ_dev[64] = {0};
  int& occ = occ_dev[ctx->device & 63];
  if (!occ) {
    TBK_CUDA(cudaFuncSetAttribute(sddmm_window_g<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    TBK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sddmm_window_g<NC>, C::THREADS, C::SMEM));
    TBK_CHECK_ARG(occ > 0, "windowed outer-product kernel does not fit on this device");
  }
  const int G = task_grid(op.n_atoms, (int64_t)occ * ctx->num_sms);
  launch_pdl(ctx, sddmm_window_g<NC>, G, C::THREADS, C::SMEM, op.n_atoms, op.row_ptr, op.col, wp, nw, s, w, Gacc, err, batch, kcl, k_lo);
  post_launch(ctx, "sddmm_window_g");
}

void launch_window(tbk_ctx* ctx, const HOp& op, const WindowPanels& wp, int nw, int s, double w, double* Gacc, int* err, const BatchRows& batch, const int32_t* kcl, int k_lo) {
  KernelTimerScope timer(ctx, TBK_KERNEL_WINDOW);
  TBK_CHECK_ARG(nw >= 1 && nw <= SDW && wp.y[0] != nullptr, "bad outer-product window");
  if (s == 512) launch_window_g<4>(ctx, op, wp, nw, s, w, Gacc, err, batch, kcl, k_lo);
  else if (s == 256) launch_window_g<2>(ctx, op, wp, nw, s, w, Gacc, err, batch, kcl, k_lo);
  else launch_window_g<1>(ctx, op, wp, nw, s, w, Gacc, err, batch, kcl, k_lo);
}

// ---- adjoint of the doubled moments (FP32 at 128, 256 and 512 probes, FP64) ---------------------
//
// The moments come from the doubling identities (C_m C_n = (C_{m+n} + C_{|m-n|})/2):
//   mu_2k = 2 e_k - mu_0,  mu_2k-1 = 2 o_k - mu_1,  e_k = <y_k, y_k>/s,  o_k = <y_k, y_{k-1}>/s,
// so Omega^ = sum_m c_m mu_m = const + sum_{k=1..K} (w_k e_k + v_k o_k),  K = floor(p/2), with
//   w_k = 2 c_2k (2k < p),  v_1 = c_1 - sum_{k>=2} c_{2k-1},  v_k = 2 c_{2k-1} (k >= 2, 2k-1 < p).
// Reverse-mode differentiation through y_{k+1} = 2 H^ y_k - y_{k-1} (y_1 = H^ y_0, y_0 = r):
//   ybar_K = g_K,  ybar_k = g_k + 2 H^ ybar_{k+1} - ybar_{k+2},
//   g_k = (2 w_k y_k + v_k y_{k-1} + v_{k+1} y_{k+1}) / s,
//   dOmega^/dH^ = sum_{k=1}^{K-1} 2 ybar_{k+1} y_k^T + ybar_1 y_0^T.
// This needs the y_k only up to K = p/2: half the forward, replay and backward work of the
// Clenshaw form of Eq. polynomial_response, for the same estimator and the same gradient.

// ybar_K = ca y_K + cb y_{K-1}, over all elements of the panels (four per thread).
template <typename T>
__global__ void ybar_init(int64_t n, T ca, const T* __restrict__ yk, T cb, const T* __restrict__ ykm1,
                          T* __restrict__ out) {
  const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  T v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = fma(ca, yk[i + j], cb * ykm1[i + j]);
#pragma unroll
  for (int j = 0; j < 4; ++j) out[i + j] = v[j];
}

// Steps whose outer products run together after them (0: fused into each step).  Up to 64, as long as
// their panels stay within 3/8 of L2, where the next kernel finds them; at 128 probes at least 8, since
// one warp per block then also saves the additions to Gacc.  us per step pair (forward and backward), fused
// and 1 / 2 / 4 / 8 steps: 2,000 atoms x 128 probes 120, 94 / 84 / 81 / 78; 10,000 x 128 584, 465 / 402 /
// 375 / 365; 2,000 x 256 160, 141 / 140 / 140 / 139; 10,000 x 256 750, 704 / 704 / 707 / 710; at 512
// probes 500 atoms 66.2 / 65.7, 1,000 atoms 119.1 / 119.4, 10,000 atoms 1147 / 1148.
static int deferred_steps(const tbk_ctx* ctx, const HOp& op, int s) {
  if (s == 512) return 0;
  const int64_t fit = ctx->l2_bytes * 3 / 8 / (2 * op.n_rows * s * 4);
  return (int)std::max<int64_t>(s == 128 ? 8 : 1, std::min<int64_t>(OUT_STEPS, fit));
}

// get_coefs() is called once every y_1 .. y_K has been formed for the first time (with
// `partials` != NULL those steps also wrote their moment partial sums at partials + 2 nctas (t-1),
// so the caller can finish the moments, solve for mu and return the coefficients c_0 .. c_{p-1}).
void adjoint_doubling(tbk_ctx* ctx, const HOp& op, uint64_t probe_seed, int s, int p,
                      const std::function<std::vector<double>()>& get_coefs, double* partials, int nctas,
                      int64_t max_panel_bytes, double* Gacc, int* err, int sched, const AdjBatch* bt,
                      const void* probe_panel, int s_norm) {
  TBK_CHECK_ARG(!(bt && probe_panel), "a batch regenerates its probes");
  // FP64: plain backward steps, each followed by its outer products
  const bool f64 = op.prec == TBK_FP64;
  const size_t esz = f64 ? 8 : 4;
  const bool windowed = sched == 1 && !f64;
  // fused schedule: steps whose outer products run after them in one launch (0: inside each step)
  int defer = sched == 0 && !f64 && !bt ? deferred_steps(ctx, op, s) : 0;
  // outer products on the tensor cores after each backward step, where that kernel applies
  const bool tensor = sched == 2 && !bt && !f64 && tc_sddmm_eligible(ctx, op, s, tc_sddmm_max_row(ctx, op));
  // a stored probe block y_0 (single system): read wherever the probe enters
  const bool r_panel = probe_panel != nullptr;
  const double nrm = r_panel && s_norm > 0 ? s_norm : s;
  const int K = bt ? (bt->K.empty() ? 0 : bt->K[0]) : p / 2;
  if (K < 1) {
    if (get_coefs) get_coefs();
    return;  // p = 1: the estimate does not depend on H
  }
  // atoms of the (order-sorted) clusters that take part in step t: a prefix of the merged rows
  auto active = [&](int t) {
    if (!bt) return op.n_atoms;
    int64_t r = 0;
    for (size_t ci = 0; ci < bt->K.size() && bt->K[ci] >= t; ++ci) r += bt->n_at[ci];
    return (int)r;
  };
  std::vector<double> w(K + 2, 0.0), v(K + 2, 0.0);
  // a batch brings its per-cluster coefficient table (filled by get_coefs() when given)
  bool have_coefs = bt != nullptr && !get_coefs;
  auto load_coefs = [&]() {
    const std::vector<double> c = get_coefs();
    have_coefs = true;
    if (bt) return;
    for (int k = 1; k <= K; ++k) {
      if (2 * k < p) w[k] = 2.0 * c[2 * k];
      if (k >= 2 && 2 * k - 1 < p) v[k] = 2.0 * c[2 * k - 1];
    }
    v[1] = p > 1 ? c[1] : 0.0;
    for (int k = 2; 2 * k - 1 < p; ++k) v[1] -= c[2 * k - 1];
  };
  auto ca = [&](int k) { return 2.0 * w[k] / nrm; };
  auto cb = [&](int k) { return v[k] / nrm; };
  auto cc = [&](int k) { return v[k + 1] / nrm; };

  const size_t panel = (size_t)op.n_rows * s * esz;
  size_t budget = max_panel_bytes > 0 ? (size_t)max_panel_bytes : panel_budget(ctx, WS_CHECKPOINTS);
  const int npan = K;  // y_1 .. y_K
  AdjointPlan plan;
  plan.npan = plan.seg = npan;
  plan.panel = panel;
  plan.windowed = windowed;
  plan.batch = bt != nullptr;
  if (defer > 0) {
    // as many ybar panels as fit beside the all-stored plan
    const int64_t room = (int64_t)(budget / panel) - (npan + 2) - 2;
    plan.defer = room < 0 ? 0 : (int)std::min<int64_t>(std::min(defer, K), room + 1);
  }
  // A batch's step t runs on the clusters with K_c >= t, a prefix of the merged rows, so its
  // all-stored plan can keep every y_j compactly: panel j holds the rows of the clusters still
  // running at step j - 1 (backward step j - 1 reads y_j on those rows, with a zero coefficient
  // for the clusters that stop there).  poff: byte offsets of P(0 .. npan) and E = y_{npan+1}.
  std::vector<size_t> poff;
  if (bt) {
    const size_t row_bytes = (size_t)op.B * s * esz;
    poff.resize((size_t)npan + 2);
    size_t o = 0;
    for (int i = 0; i <= npan + 1; ++i) {
      poff[i] = o;
      o += (size_t)active(std::max(i - 1, 0)) * row_bytes;
      o = (o + 255) & ~(size_t)255;
    }
    if (o + (size_t)plan.nx() * panel <= budget) plan.prefix_tail = o;
  }
  if (!plan.prefix_tail && plan.bytes() > budget && npan > 2) {
    plan.segment();
    if (plan.bytes() > budget)
      throw Error(TBK_ERR_OOM, "panel scratch budget of " + std::to_string(budget) +
                                   " bytes is below the checkpoint plan's " + std::to_string(plan.bytes()));
  }
  char* base = nullptr;
  while (!base) {
    try {
      base = (char*)scratch(ctx, WS_CHECKPOINTS, plan.bytes());
    } catch (const Error& e) {
      // the device could not map the plan after all: a smaller one
      if (e.code != TBK_ERR_OOM || !plan.shrink()) throw;
    }
  }
  const bool prefix = plan.prefix_tail > 0, all_stored = plan.nseg() <= 1;
  const size_t prefix_tail = plan.prefix_tail;
  const int NB = plan.nb(), seg = plan.seg, nseg = plan.nseg();
  const size_t n_seg_pan = (size_t)seg + 1, n_ckpt = plan.n_ckpt();
  defer = plan.defer;
  // P(0 .. npan + 1) of the prefix plan at poff, the full-size panels after them
  auto P = [&](size_t i) -> void* {
    if (!prefix) return base + i * panel;
    if (i <= (size_t)npan + 1) return base + poff[i];
    return base + prefix_tail + (i - ((size_t)npan + 2)) * panel;
  };
  auto CK = [&](int sg, int which) { return P(n_seg_pan + 2 * (size_t)sg + which); };
  void* E = P(n_seg_pan + n_ckpt);
  auto YB = [&](int j) { return P(n_seg_pan + n_ckpt + 1 + (size_t)(j % NB)); };
  void* R0 = bt ? P(n_seg_pan + n_ckpt + 1 + NB) : const_cast<void*>(probe_panel);
  const BatchRows br = bt ? bt->br : BatchRows();
  if (bt) {
    // the probe block of every cluster, and ybar = 0 on the rows of clusters not yet started
    // (their first backward step then reduces to ybar_K = g_K)
    launch_batch_probe_panel(ctx, op, br, s, R0);
    for (int j = 0; j < NB; ++j) TBK_CUDA(cudaMemsetAsync(YB(j), 0, panel, ctx->stream));
  }
  // y_0: the caller's or the batch's probe panel, else written just before the first step, in the first
  // segment at its place P(0) (where the last backward steps find it) and before that in E
  void* y0 = bt || r_panel ? R0 : E;
  auto forward_step = [&](int t, const void* yin, const void* yprev, void* yout, bool first_time) {
    HOp o = op;
    o.n_atoms = active(t);
    if (o.n_atoms <= 0) return;
    if (t == 1 && !bt && !r_panel) launch_scaled_probe(ctx, op, y0, 1.0, probe_seed, s);
    StepArgs a;
    a.seed = probe_seed;
    a.s = s;
    a.yin = t == 1 ? y0 : yin;
    a.alpha = t == 1 ? 1.0 : 2.0;
    if (t == 2) a.yprev = y0;
    else if (t >= 3) a.yprev = const_cast<void*>(yprev);
    a.yout = yout;
    a.err = err;
    a.batch = br;
    if (partials && first_time) {
      if (bt) {
        // per (atom, consumer warp) partial sums, reduced per cluster by the caller
        a.partials = partials + (size_t)(t - 1) * bt->pstride;
        a.per_task = 1;
      } else {
        a.partials = partials + (size_t)(t - 1) * nctas * 2;
        a.grid = nctas;
      }
    }
    launch_step(ctx, o, a);
  };
  if (!all_stored) {
    void *cur = nullptr, *prv = nullptr;
    const int last = seg * (nseg - 1);
    for (int t = 1; t <= last; ++t) {
      void* out = t == 1 ? P(0) : (t == 2 ? P(1) : prv);
      forward_step(t, cur, prv, out, true);
      prv = cur;
      cur = out;
      if (t % seg == 0) {
        const int sg = t / seg;
        TBK_CUDA(cudaMemcpyAsync(CK(sg, 0), prv, panel, cudaMemcpyDeviceToDevice, ctx->stream));
        TBK_CUDA(cudaMemcpyAsync(CK(sg, 1), cur, panel, cudaMemcpyDeviceToDevice, ctx->stream));
      }
    }
  }
  OuterPanels wait{};
  int n_wait = 0;
  int k = K;
  for (int sg = nseg - 1; sg >= -1 && k >= 0; --sg) {
    const int t0 = sg >= 0 ? 1 + seg * sg : 0;
    const int t1 = sg >= 0 ? std::min(npan, t0 + seg - 1) : 0;
    if (sg >= 0) {
      if (sg < nseg - 1) {
        // y_{t1+1} is the first panel of the segment just finished
        TBK_CUDA(cudaMemcpyAsync(E, P(1), panel, cudaMemcpyDeviceToDevice, ctx->stream));
      }
      const bool first_time = sg == nseg - 1;  // the last segment was never formed before
      if (sg == 0 && !bt && !r_panel) y0 = P(0);
      int t = t0;
      if (sg > 0) {
        TBK_CUDA(cudaMemcpyAsync(P(0), CK(sg, 1), panel, cudaMemcpyDeviceToDevice, ctx->stream));
        forward_step(t0, P(0), CK(sg, 0), P(1), first_time);
        ++t;
      }
      for (; t <= t1; ++t) {
        const int i = t - t0 + 1;
        forward_step(t, t == 1 ? nullptr : P(i - 1), t >= 3 ? P(i - 2) : nullptr, P(i), first_time);
      }
    }
    if (!have_coefs) load_coefs();
    // y_j for j in [t0 - 1, t1 + 1]
    auto Y = [&](int j) -> const void* {
      if (j == 0) return y0;
      if (j == t1 + 1) return E;
      return P(j - t0 + 1);
    };
    for (; k >= t0; --k) {
      HOp o = op;
      o.n_atoms = active(std::max(k, 1));
      if (k == K && !bt) {
        // ybar_K = g_K (y_{K+1} does not enter)
        const int64_t n = op.n_rows * s;
        const unsigned grid = (unsigned)((n + 1023) / 1024);
        if (f64)
          ybar_init<double><<<grid, 256, 0, ctx->stream>>>(n, ca(K), (const double*)Y(K), cb(K), (const double*)Y(K - 1),
                                                           (double*)YB(K));
        else
          ybar_init<float><<<grid, 256, 0, ctx->stream>>>(n, (float)ca(K), (const float*)Y(K), (float)cb(K),
                                                          (const float*)Y(K - 1), (float*)YB(K));
        post_launch(ctx, "ybar_init");
        continue;
      }
      if (f64) {
        // G += 2 y_k ybar_{k+1}^T (y_0 ybar_1^T last), then ybar_k = g_k + 2 H^ ybar_{k+1} - ybar_{k+2}
        {
          KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
          launch_sddmm(ctx, o, Y(k), YB(k + 1), s, k ? 2.0 : 1.0, Gacc);
        }
        if (k == 0) continue;
        StepArgs a;
        a.family = TBK_KERNEL_BACKWARD;
        a.seed = probe_seed;
        a.s = s;
        a.yin = YB(k + 1);
        a.yprev = k + 2 <= K ? YB(k + 2) : nullptr;
        a.yout = YB(k);
        a.src[0] = Y(k);
        a.csrc[0] = ca(k);
        a.src[1] = Y(k + 1);
        a.csrc[1] = cc(k);
        if (k == 1) {
          a.c_r = cb(1);
        } else {
          a.src[2] = Y(k - 1);
          a.csrc[2] = cb(k);
        }
        a.err = err;
        launch_step(ctx, o, a);
        continue;
      }
      if (k >= 1) {
        // ybar_k = g_k + 2 H^ ybar_{k+1} - ybar_{k+2}; fused: and G += 2 y_k ybar_{k+1}^T on the pattern
        // (the probe coefficient .x scales the regenerated y_0; a stored y_0 streams as y_{k-1})
        const bool r_gen = k == 1 && !r_panel;
        const float4 cf = bt ? make_float4(0.f, 0.f, 0.f, 0.f)
                             : make_float4(r_gen ? (float)cb(1) : 0.f, (float)ca(k), r_gen ? 0.f : (float)cb(k),
                                           (float)cc(k));
        const float4* cfk = bt ? bt->cft + (size_t)k * bt->K.size() : nullptr;
        if (defer) {
          launch_adjoint_step(ctx, o, YB(k + 1), k + 2 <= K ? YB(k + 2) : nullptr, YB(k), Y(k), cf, probe_seed, s, err,
                              (k >= 2 || r_panel) ? Y(k - 1) : nullptr, Y(k + 1));
          wait.y[n_wait] = (const float*)Y(k);
          wait.x[n_wait++] = (const float*)YB(k + 1);
          if (n_wait == defer) {
            launch_outer(ctx, o, wait, n_wait, 0, s, Gacc, err);
            n_wait = 0;
          }
          continue;
        }
        launch_fused(ctx, o, YB(k + 1), (k + 2 <= K || bt) ? YB(k + 2) : nullptr, YB(k), Y(k), cf, probe_seed, s,
                     2.0, (windowed || tensor) ? nullptr : Gacc, err, br, cfk,
                     (k >= 2 || r_panel) ? Y(k - 1) : nullptr, Y(k + 1), 0);
        // G += 2 y_k ybar_{k+1}^T on the pattern, on the tensor cores
        if (tensor) launch_tc_sddmm(ctx, o, Y(k), YB(k + 1), s, 2.0, Gacc, err);
        if (windowed && (k - 1) % SDW == 0 && k < K) {
          // G += 2 y_j ybar_{j+1}^T on the pattern for the window j = k .. min(k + SDW, K) - 1
          WindowPanels wp{};
          const int nw = std::min(SDW, K - k);
          for (int t = 0; t < nw; ++t) {
            wp.y[t] = (const float*)Y(k + t);
            wp.x[t] = (const float*)YB(k + t + 1);
          }
          launch_window(ctx, o, wp, nw, s, 2.0, Gacc, err, br, bt ? bt->d_K : nullptr, k);
        }
      } else if (defer) {
        wait.y[n_wait] = (const float*)Y(0);
        wait.x[n_wait++] = (const float*)YB(1);
        launch_outer(ctx, o, wait, n_wait, 1, s, Gacc, err);
      } else if (windowed) {
        // G += y_0 ybar_1^T
        WindowPanels wp{};
        wp.y[0] = (const float*)Y(0);
        wp.x[0] = (const float*)YB(1);
        launch_window(ctx, o, wp, 1, s, 1.0, Gacc, err, br, bt ? bt->d_K : nullptr, 0);
      } else if (tensor && r_panel) {
        // G += y_0 ybar_1^T with the caller's probe block
        launch_tc_sddmm(ctx, o, Y(0), YB(1), s, 1.0, Gacc, err);
      } else {
        launch_fused(ctx, o, YB(1), nullptr, nullptr, Y(0), make_float4(0.f, 0.f, 0.f, 0.f), probe_seed, s,
                     1.0, Gacc, err, br, nullptr, nullptr, nullptr, 0);
      }
    }
  }
}

}  // namespace tbk

using namespace tbk;

namespace tbk {
// The adjoint's outer-product schedule: TBK_WINDOWED or TBK_FUSED_ADJOINT when given, else what
// tbk_autotune measured for this shape, else fused.
int outer_schedule(const tbk_ctx* ctx, const HOp& op, int s, int flags) {
  if (flags & TBK_TC_OUTER) return 2;
  if (flags & TBK_WINDOWED) return 1;
  if (flags & TBK_FUSED_ADJOINT) return 0;
  const tbk_ctx::Tuned* t = find_tuned(ctx, op.n_rows, op.nnzb, s);
  return t ? t->windowed : 0;
}
}  // namespace tbk

extern "C" int tbk_density_and_forces(tbk_ctx* ctx, const tbk_bsr* H, const tbk_model* model,
                                      const double* pos, const double* box, double emin,
                                      double emax, uint64_t probe_seed, int32_t n_probes,
                                      int32_t order, double mu, double kT, int32_t damping,
                                      int32_t flags, int64_t max_panel_bytes, double* G,
                                      double* forces) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr, "ctx is NULL");
  TBK_CHECK_ARG(G || forces, "nothing to compute: G and forces are both NULL");
  TBK_CHECK_ARG(order >= 1, "order must be >= 1");
  TBK_CHECK_ARG(n_probes >= 4 && n_probes % 4 == 0, "n_probes must be a positive multiple of 4");
  TBK_CHECK_ARG((flags & ~(TBK_FP64 | TBK_PLAIN_KERNEL | TBK_WINDOWED | TBK_FUSED_ADJOINT | TBK_TC_OUTER)) == 0, "unknown flag");
  const int plain = (flags & TBK_PLAIN_KERNEL) ? 1 : 0;
  TBK_CHECK_ARG(kT > 0.0, "kT must be positive");
  DeviceGuard dg(ctx);
  const int prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  DevModel M{};
  if (forces) {
    M = upload_model(ctx, model, box, WS_TABLE);
    TBK_CHECK_ARG(M.kind == TBK_MODEL_SK, "forces need the Slater-Koster model");
    TBK_CHECK_ARG(pos != nullptr, "pos is NULL");
  }
  int* err = (int*)scratch(ctx, WS_FLAGS, 64);
  TBK_CUDA(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
  HOp op = prepare_hop(ctx, H, emin, emax, prec, WS_HHAT, err);
  const int p = order, s = n_probes, BB = op.B * op.B;
  const bool doubled = doubled_eligible(op, s, plain);
  const double W = emax - emin;

  // coefficients c_k = d_k beta_k[g] (device, then host for the per-step scalars)
  double* dcoef = (double*)scratch(ctx, WS_COEF, sizeof(double) * (size_t)p);
  coefficients(ctx, TBK_FN_FREE, p, emin, emax, mu, kT, damping, dcoef);
  std::vector<double> c(p);
  TBK_CUDA(cudaMemcpyAsync(c.data(), dcoef, sizeof(double) * p, cudaMemcpyDeviceToHost, ctx->stream));

  // transpose map of the pattern
  int32_t* tr = (int32_t*)scratch(ctx, WS_TRANSPOSE, sizeof(int32_t) * (size_t)op.nnzb);
  transpose_map<<<ceil_div(op.n_atoms, 16), dim3(8, 16), 0, ctx->stream>>>(op.n_atoms, op.row_ptr, op.col, tr, err);
  post_launch(ctx, "transpose_map");

  double* Gacc = (double*)scratch(ctx, WS_GACC, sizeof(double) * (size_t)op.nnzb * BB * 2);
  double* Gsym = Gacc + (size_t)op.nnzb * BB;
  TBK_CUDA(cudaMemsetAsync(Gacc, 0, sizeof(double) * (size_t)op.nnzb * BB, ctx->stream));

  const size_t esz = prec == TBK_MIXED ? 4 : 8;
  const size_t panel = (size_t)op.n_rows * s * esz;
  double scale = 2.0 / (W * s);
  if (doubled) {
    adjoint_doubling(ctx, op, probe_seed, s, p, [&]() { return c; }, nullptr, 0, max_panel_bytes, Gacc, err,
                       outer_schedule(ctx, op, s, flags), nullptr);
    scale = 2.0 / W;  // the 1/s of the moments is inside the source terms
  } else {
    // Panels y_1 .. y_{p-2} are needed in reverse order: all of them are kept when they fit the
    // budget, else segments of ~sqrt(2p) steps are replayed from checkpoints.
    const int npan = std::max(0, p - 2);  // y_1 .. y_{p-2}
    size_t budget = max_panel_bytes > 0 ? (size_t)max_panel_bytes : panel_budget(ctx, WS_CHECKPOINTS);
    int seg = std::max(1, npan);
    if ((size_t)(npan + 3) * panel > budget && npan > 2) {
      seg = std::max(2, (int)std::ceil(std::sqrt(2.0 * npan)));
      const size_t need = (size_t)(2 * ((npan + seg - 1) / seg) + seg + 3) * panel;
      if (need > budget)
        throw Error(TBK_ERR_OOM, "panel scratch budget of " + std::to_string(budget) +
                                     " bytes is below the checkpoint plan's " + std::to_string(need));
    }
    const int nseg = npan > 0 ? (npan + seg - 1) / seg : 0;
    const bool all_stored = nseg <= 1;
    // Scratch layout: P(0 .. seg) segment panels, P(seg+1 ..) checkpoints, then two b panels.
    // Segment sg covers y_j for j in [t0, t1], t0 = 1 + seg sg, t1 = min(p - 2, t0 + seg - 1),
    // and holds y_{t0 - 1 + i} at P(i).  Checkpoint sg (sg >= 1) is (y_{t0-2}, y_{t0-1}).
    const size_t n_seg_pan = (size_t)seg + 1;
    const size_t n_ckpt = all_stored ? 0 : 2 * (size_t)nseg;
    // b panels in a ring: two, or those of the steps whose outer products wait, as far as they fit
    int defer = all_stored && !plain && npan > 0 ? general_deferred_steps(ctx, op, s) : 0;
    defer = (int)std::max<int64_t>(0, std::min<int64_t>(std::min(defer, p - 1), (int64_t)(budget / panel) - (npan + 2)));
    if (defer < 8) defer = 0;
    size_t n_ring = defer ? (size_t)defer + 1 : 2;
    char* base = nullptr;
    try {
      base = (char*)scratch(ctx, WS_CHECKPOINTS, panel * (n_seg_pan + n_ckpt + n_ring));
    } catch (const Error& e) {
      // the device could not map that after all: with two b panels
      if (e.code != TBK_ERR_OOM || !defer) throw;
      defer = 0;
      n_ring = 2;
      base = (char*)scratch(ctx, WS_CHECKPOINTS, panel * (n_seg_pan + n_ckpt + n_ring));
    }
    auto P = [&](size_t i) { return (void*)(base + i * panel); };
    auto CK = [&](int sg, int which) { return P(n_seg_pan + 2 * (size_t)sg + which); };
    auto ring = [&](int i) { return P(n_seg_pan + n_ckpt + (size_t)((i + (int)n_ring) % (int)n_ring)); };
    int ib = 0;
    void* bcur = ring(ib);

    // y_t from y_{t-1} (yin) and y_{t-2} (yprev); y_0 is the probe block
    void* y0 = bcur;  // the probe block, written just before the first step (P(0) in the first segment)
    auto forward_step = [&](int t, const void* yin, const void* yprev, void* yout) {
      if (t == 1) launch_scaled_probe(ctx, op, y0, 1.0, probe_seed, s);
      StepArgs a;
      a.seed = probe_seed;
      a.s = s;
      a.yin = t == 1 ? y0 : yin;
      a.alpha = t == 1 ? 1.0 : 2.0;
      if (t == 2) a.yprev = y0;
      else if (t >= 3) a.yprev = const_cast<void*>(yprev);
      a.yout = yout;
      a.err = err;
      a.force_simple = plain;
      launch_step(ctx, op, a);
    };
    // Forward sweep to the last checkpoint, with two rotating panels.
    if (!all_stored) {
      void *cur = nullptr, *prv = nullptr;
      const int last = seg * (nseg - 1);
      for (int t = 1; t <= last; ++t) {
        void* out = t == 1 ? P(0) : (t == 2 ? P(1) : prv);
        forward_step(t, cur, prv, out);
        prv = cur;
        cur = out;
        if (t % seg == 0) {
          const int sg = t / seg;  // the segment starting at t0 = t + 1
          TBK_CUDA(cudaMemcpyAsync(CK(sg, 0), prv, panel, cudaMemcpyDeviceToDevice, ctx->stream));
          TBK_CUDA(cudaMemcpyAsync(CK(sg, 1), cur, panel, cudaMemcpyDeviceToDevice, ctx->stream));
        }
      }
    }
    // Backward sweep: b_{p-1} = c_{p-1} r, then for j = p-2 .. 0 add the y_j b_{j+1} term and
    // form b_j = c_j r + 2 H^ b_{j+1} - b_{j+2}.
    y0 = P(0);
    if (nseg == 0 && p >= 2) launch_scaled_probe(ctx, op, y0, 1.0, probe_seed, s);
    if (p >= 2) {
      launch_scaled_probe(ctx, op, bcur, c[p - 1], probe_seed, s);
      bool have_bprev = false;
      OuterPanels wait{};
      int n_wait = 0;
      int j = p - 2;
      for (int sg = nseg - 1; sg >= -1 && j >= 0; --sg) {
        const int t0 = sg >= 0 ? 1 + seg * sg : 0;
        const int t1 = sg >= 0 ? std::min(npan, t0 + seg - 1) : 0;
        if (sg >= 0) {
          int t = t0;
          if (sg > 0) {
            TBK_CUDA(cudaMemcpyAsync(P(0), CK(sg, 1), panel, cudaMemcpyDeviceToDevice, ctx->stream));
            forward_step(t0, P(0), CK(sg, 0), P(1));
            ++t;
          }
          for (; t <= t1; ++t) {
            const int i = t - t0 + 1;
            forward_step(t, t == 1 ? nullptr : P(i - 1), t >= 3 ? P(i - 2) : nullptr, P(i));
          }
        }
        for (; j >= t0; --j) {
          const void* yj = j == 0 ? y0 : P(j - t0 + 1);
          if (defer) {
            wait.y[n_wait] = (const float*)yj;
            wait.x[n_wait++] = (const float*)ring(ib);
            if (n_wait == defer || j == 0) {
              launch_sddmm_steps(ctx, op, wait, n_wait, j == 0, s, Gacc);
              n_wait = 0;
            }
          } else {
            KernelTimerScope timer(ctx, TBK_KERNEL_BACKWARD);
            launch_sddmm(ctx, op, yj, ring(ib), s, j == 0 ? 1.0 : 2.0, Gacc);
          }
          if (j >= 1) {
            StepArgs a;
            a.family = TBK_KERNEL_BACKWARD;
            a.seed = probe_seed;
            a.s = s;
            a.yin = ring(ib);
            a.alpha = 2.0;
            a.c_r = c[j];
            a.yprev = have_bprev ? ring(ib - 1) : nullptr;
            a.yout = ring(ib + 1);
            a.err = err;
            a.force_simple = plain;
            launch_step(ctx, op, a);
            ib = (ib + 1) % (int)n_ring;
            have_bprev = true;
          }
        }
      }
    }
  }
  // symmetrise and scale: G = scale sym(Gacc)
  double* Gout = G ? G : Gsym;
  const int64_t tot = op.nnzb * BB;
  if (op.B == 9)
    symmetrize<9><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(op.nnzb, tr, Gacc, scale, Gout);
  else
    symmetrize<1><<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(op.nnzb, tr, Gacc, scale, Gout);
  post_launch(ctx, "symmetrize");
  if (forces) {
    double* tq = (double*)scratch(ctx, WS_MISC, sizeof(double) * 3 * (size_t)op.nnzb);
    launch_forces(ctx, M, pos, op.n_atoms, op.row_ptr, op.col, tr, Gout, tq, forces);
  }
  int herr = 0;
  TBK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  check_diagonal_flag(herr);
  if (herr & 2) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the recurrence kernel expired");
  TBK_CHECK_ARG(herr == 0, "the block pattern is not symmetric");
  TBK_API_END
}

namespace tbk {
// The one-call energies and forces on the doubled-moment adjoint (fused-eligible shapes): the
// adjoint's forward sweep over y_1 .. y_{p/2} also yields the moments, so no separate moment pass
// runs.  probe_panel / s_norm: a stored probe block and its sample count (NULL / 0: the
// Rademacher probes regenerated from probe_seed, s of them).
void energies_and_forces_doubled(tbk_ctx* ctx, const tbk_bsr* H, const tbk_model* model, const double* pos,
                                 const double* box, double emin, double emax, uint64_t probe_seed, int s,
                                 int order, double n_electrons, double kT, int damping, int flags,
                                 int64_t max_panel_bytes, double* moments, double* observables, double* G,
                                 double* forces, const void* probe_panel, int s_norm) {
  const int prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  DevModel M{};
  if (forces) {
    M = upload_model(ctx, model, box, WS_TABLE);
    TBK_CHECK_ARG(M.kind == TBK_MODEL_SK, "forces need the Slater-Koster model");
    TBK_CHECK_ARG(pos != nullptr, "pos is NULL");
  }
  // err: bit 4 = a row has no diagonal block, bit 2 = a bounded wait expired, bit 1 = the pattern
  // is not symmetric; err[1] bit 1 = a panel outgrew ||r|| (the spectrum is not inside [emin, emax])
  int* err = (int*)scratch(ctx, WS_FLAGS, 64);
  TBK_CUDA(cudaMemsetAsync(err, 0, 2 * sizeof(int), ctx->stream));
  HOp op = prepare_hop(ctx, H, emin, emax, prec, WS_HHAT, err);
  const int p = order, BB = op.B * op.B;
  const int nrm = probe_panel && s_norm > 0 ? s_norm : s;
  const double W = emax - emin;
  int32_t* tr = (int32_t*)scratch(ctx, WS_TRANSPOSE, sizeof(int32_t) * (size_t)op.nnzb);
  launch_transpose_map(ctx, op.n_atoms, op.row_ptr, op.col, tr, err);
  double* Gacc = (double*)scratch(ctx, WS_GACC, sizeof(double) * (size_t)op.nnzb * BB * 2);
  double* Gsym = Gacc + (size_t)op.nnzb * BB;
  TBK_CUDA(cudaMemsetAsync(Gacc, 0, sizeof(double) * (size_t)op.nnzb * BB, ctx->stream));
  const int K = p / 2;
  const int nctas = step_grid_ctas(ctx, op, s, K);
  double* partials = (double*)scratch(ctx, WS_PARTIALS, sizeof(double) * 2 * (size_t)std::max(1, K) * nctas);
  // per-step sums, the solve's buffer (16-byte aligned), its result, the moments unless given
  const size_t nsums = 2 * (size_t)K + 64, nfermi = fermi_doubles(quad_nodes(p), p);
  double* sums = (double*)scratch(ctx, WS_SEGMENT, sizeof(double) * (nsums + nfermi + 16 + (size_t)p + 8));
  double* fbuf = sums + nsums;
  double* res = fbuf + nfermi;
  double* mom = moments ? moments : res + 16;
  double* dcoef = (double*)scratch(ctx, WS_COEF, sizeof(double) * (size_t)p);
  auto after_forward = [&]() {
    // moments from the doubling identities, then mu, Omega, E, N, then c_k = d_k beta_k[g](mu)
    launch_moment_reduction(ctx, partials, nctas, K, p, nrm, op.n_rows, 0, sums, mom, err + 1);
    fermi_enqueue(ctx, mom, p, emin, emax, n_electrons, 0.0, kT, damping, fbuf, res);
    double h[5];
    int herr[2] = {0, 0};
    TBK_CUDA(cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    TBK_CUDA(cudaMemcpyAsync(herr, err, sizeof(herr), cudaMemcpyDeviceToHost, ctx->stream));
    sync(ctx);
    check_diagonal_flag(herr[0]);
    if ((herr[0] | herr[1]) & 2) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the recurrence kernel expired");
    TBK_CHECK_ARG(herr[0] == 0, "the block pattern is not symmetric");
    if (herr[1])
      throw Error(TBK_ERR_SPECTRUM, "a Chebyshev panel grew beyond ||r||: the spectrum of H is not "
                                    "inside [emin, emax]");
    check_fermi_status(h[4], "n_electrons is outside the range of the estimated N(mu)");
    for (int i = 0; i < 4; ++i) observables[i] = h[i];
    coefficients(ctx, TBK_FN_FREE, p, emin, emax, h[0], kT, damping, dcoef);
    std::vector<double> c(p);
    TBK_CUDA(cudaMemcpyAsync(c.data(), dcoef, sizeof(double) * p, cudaMemcpyDeviceToHost, ctx->stream));
    sync(ctx);
    return c;
  };
  adjoint_doubling(ctx, op, probe_seed, s, p, after_forward, partials, nctas, max_panel_bytes, Gacc, err,
                   outer_schedule(ctx, op, s, flags), nullptr, probe_panel, s_norm);
  double* Gout = G ? G : Gsym;
  launch_symmetrize(ctx, op.nnzb, op.B, tr, Gacc, 2.0 / W, Gout);
  if (forces) {
    double* tq = (double*)scratch(ctx, WS_MISC, sizeof(double) * 3 * (size_t)op.nnzb);
    launch_forces(ctx, M, pos, op.n_atoms, op.row_ptr, op.col, tr, Gout, tq, forces);
  }
  int herr = 0;
  TBK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  check_diagonal_flag(herr);
  if (herr & 2) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the recurrence kernel expired");
  TBK_CHECK_ARG(herr == 0, "the block pattern is not symmetric");
}
}  // namespace tbk

// Energies and forces in one call: the adjoint's forward sweep over y_1 .. y_{p/2} also yields
// the (doubled) moments, so no separate moment pass is run.
extern "C" int tbk_energies_and_forces(tbk_ctx* ctx, const tbk_bsr* H, const tbk_model* model,
                                       const double* pos, const double* box, double emin,
                                       double emax, uint64_t probe_seed, int32_t n_probes,
                                       int32_t order, double n_electrons, double kT,
                                       int32_t damping, int32_t flags, int64_t max_panel_bytes,
                                       double* moments, double* observables, double* G,
                                       double* forces) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr && observables != nullptr, "NULL argument");
  TBK_CHECK_ARG(order >= 1, "order must be >= 1");
  TBK_CHECK_ARG(n_probes >= 4 && n_probes % 4 == 0, "n_probes must be a positive multiple of 4");
  TBK_CHECK_ARG((flags & ~(TBK_FP64 | TBK_PLAIN_KERNEL | TBK_WINDOWED | TBK_FUSED_ADJOINT | TBK_TC_OUTER)) == 0, "unknown flag");
  TBK_CHECK_ARG(kT > 0.0 && n_electrons >= 0.0, "kT must be positive and n_electrons >= 0");
  DeviceGuard dg(ctx);
  const int prec = (flags & TBK_FP64) ? TBK_FP64 : TBK_MIXED;
  const int plain = (flags & TBK_PLAIN_KERNEL) ? 1 : 0;
  HOp shape;
  shape.B = H ? H->n_orb : 0;
  shape.prec = prec;
  if (!H || !doubled_eligible(shape, n_probes, plain) || (prec == TBK_FP64 && !G && !forces)) {
    // the separate calls give the same results for the other shapes and precisions
    double* mom = moments ? moments : (double*)scratch(ctx, WS_SEGMENT, sizeof(double) * (size_t)order);
    int rc = tbk_chebyshev_moments(ctx, H, emin, emax, probe_seed, n_probes, order,
                                   flags & ~(TBK_WINDOWED | TBK_FUSED_ADJOINT | TBK_TC_OUTER), mom);
    if (rc != TBK_OK) throw Error(rc, tbk_last_error());
    rc = tbk_fermi_level(ctx, mom, order, emin, emax, n_electrons, 0.0, kT, damping, observables);
    if (rc != TBK_OK) throw Error(rc, tbk_last_error());
    if (G || forces) {
      rc = tbk_density_and_forces(ctx, H, model, pos, box, emin, emax, probe_seed, n_probes, order,
                                  observables[0], kT, damping, flags, max_panel_bytes, G, forces);
      if (rc != TBK_OK) throw Error(rc, tbk_last_error());
    }
    return TBK_OK;
  }
  energies_and_forces_doubled(ctx, H, model, pos, box, emin, emax, probe_seed, n_probes, order, n_electrons,
                              kT, damping, flags, max_panel_bytes, moments, observables, G, forces, nullptr, 0);
  TBK_API_END
}
