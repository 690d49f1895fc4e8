// a4: Chebyshev coefficients by Chebyshev-Gauss quadrature (Sec. II.B.1) and a8: chemical
// potential and observables from the moments (Sec. II.A Eqs. free_energy and density_matrix,
// with the traces replaced by the probe moments of Sec. II.C.2).
//
// With M nodes t_j = pi (j + 1/2)/M, x_j = cos t_j, e_j = emin (1 - x_j)/2 + emax (1 + x_j)/2:
//   alpha_k[h] = (2 - delta_k0)/M sum_j h(e_j) cos(k t_j),
// so any series sum_k d_k alpha_k[h] mu_k equals sum_j h(e_j) rho_j with the node weights
//   rho_j = (1/M) sum_k (2 - delta_k0) d_k mu_k cos(k t_j).
// The chemical-potential bisection therefore needs rho once and O(M) work per halving.
// cos(k t_j) = cos(pi m / (2M)) with m = k (2j + 1) mod 4M, read from a table of 4M entries.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace tbk {

__device__ __forceinline__ double fermi_fn(double e, double mu, double kT) {
  const double z = (e - mu) / kT;
  if (z > 0.0) {
    const double ez = exp(-z);
    return 2.0 * ez / (1.0 + ez);
  }
  return 2.0 / (1.0 + exp(z));
}
__device__ __forceinline__ double free_fn(double e, double mu, double kT) {
  const double u = -(e - mu) / kT;
  return -2.0 * kT * (fmax(u, 0.0) + log1p(exp(-fabs(u))));
}
__device__ __forceinline__ double node_energy(int j, int M, double emin, double emax) {
  const double x = cospi((j + 0.5) / M);
  return emin * (1.0 - x) * 0.5 + emax * (1.0 + x) * 0.5;
}

__device__ __forceinline__ double damp_factor(int k, int p, int damping) {
  if (damping != TBK_DAMP_JACKSON) return 1.0;
  // Jackson kernel (Weisse et al., Rev. Mod. Phys. 78, 275 (2006), Eq. 71) with N = p
  const double q = M_PI / (p + 1);
  return ((p - k + 1) * cos(q * k) + sin(q * k) / tan(q)) / (p + 1);
}

// ---- a4: coefficients ------------------------------------------------------------------------------

// The cosine table (4M entries) and h_j = h(e_j) at the M nodes, which the coefficient blocks read.
__global__ void coeff_setup(int fn, int M, double emin, double emax, double mu, double kT,
                            double* __restrict__ tab, double* __restrict__ hv) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < 4 * M) tab[j] = cospi((double)j / (2.0 * M));
  if (j >= M) return;
  const double e = node_energy(j, M, emin, emax);
  double h;
  if (fn == TBK_FN_FREE) h = free_fn(e, mu, kT);
  else {
    h = fermi_fn(e, mu, kT);
    if (fn == TBK_FN_ENERGY) h *= e;
  }
  hv[j] = h;
}

// One block per coefficient k.  The small coefficients of the tail are differences of large terms, so
// the order of this sum decides their last bits; it is kept fixed.
__global__ void coeff_kernel(int p, int M, int damping, const double* __restrict__ tab,
                             const double* __restrict__ hv, double* __restrict__ out) {
  __shared__ double red[32];
  const int k = blockIdx.x;
  const int period = 4 * M, step = (int)((2 * (int64_t)k * blockDim.x) % period);
  int m = (int)((int64_t)k * (2 * threadIdx.x + 1) % period);
  double s = 0.0, c = 0.0;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const double y = hv[j] * tab[m] - c, t = s + y;
    c = (t - s) - y;
    s = t;
    m += step;
    if (m >= period) m -= period;
  }
  const double tot = tbk_block_sum(s, red);
  if (threadIdx.x == 0) out[k] = (k == 0 ? 1.0 : 2.0) / M * tot * damp_factor(k, p, damping);
}

// ---- a8: chemical potential and observables --------------------------------------------------------
//
// Every problem (FermiJob) owns one buffer of fermi_doubles(M, p) doubles.  A solve is three launches
// for any number of problems (blockIdx.y = problem): the cosine table and the damped weights
// w_k = (2 - delta_k0) d_k mu_k; the node weights rho_j beside the node energies; the bisection.
struct FermiBuf {
  double* tab;       // 4M cosines
  double2* node;     // M pairs (e_j, rho_j)
  double* part;      // FERMI_PART partial sums, two sets used in turn
  unsigned* ctr;     // arrivals at the barrier of the CTAs that share the problem
  double* w;         // p weights
};
constexpr int FERMI_DEPTH = 5, FERMI_MIDS = (1 << FERMI_DEPTH) - 1;  // midpoints evaluated at once
constexpr int FERMI_THREADS = 256, FERMI_LANES = 1024, FERMI_PARTS = 16;
constexpr int FERMI_PART = 3 * FERMI_MIDS * FERMI_PARTS;  // >= 32 FERMI_MIDS

__device__ __forceinline__ FermiBuf fermi_buf(double* buf, int M) {
  return {buf, (double2*)(buf + 4 * (size_t)M), buf + 6 * (size_t)M, (unsigned*)(buf + 6 * (size_t)M + 2 * FERMI_PART),
          buf + 6 * (size_t)M + 2 * FERMI_PART + 2};
}
size_t fermi_doubles(int M, int p) { return 6 * (size_t)M + 2 * FERMI_PART + 2 + (size_t)p + (p & 1); }

__global__ void fermi_setup(const FermiJob one, const FermiJob* __restrict__ jobs,
                            const double* __restrict__ mom, int damping, double* __restrict__ buf) {
  const FermiJob j = jobs ? jobs[blockIdx.y] : one;
  const FermiBuf b = fermi_buf(buf + j.buf_off, j.M);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *b.ctr = 0;
  if (i < 4 * j.M) b.tab[i] = cospi((double)i / (2.0 * j.M));
  if (i < j.p) b.w[i] = (i == 0 ? 1.0 : 2.0) * damp_factor(i, j.p, damping) * mom[j.mom_off + i];
}

// Lanes that share two pairs of nodes: enough for `lanes` lanes in all if the problem were alone.  From its own
// size only, so that its sums do not depend on the problems that are solved with it.
__host__ __device__ inline int rho_groups(int M) { return (M / 2 + 1) / 2; }
__host__ __device__ inline int rho_lanes(int M, int lanes) {
  int S = 2;
  while (S < 32 && (int64_t)rho_groups(M) * S < lanes) S *= 2;
  return S;
}

// The node energies, and rho_j and rho_{M-1-j} from the even and the odd part of the sum over k
// (cos(k (pi - t)) = (-1)^k cos(k t): half the terms of two separate sums).  S lanes share the sums of
// two pairs of nodes, lane r takes k = r, r + S, ..., one parity per lane, each sum compensated, and so
// are the sums of the lanes.  The compensated chain
// is four dependent FP64 operations a term, 64 cycles each (an SM takes about 19 for a warp's when all four
// quarters are at them): one thread per node took 432 us at p = 2476 by latency alone; S lanes cut the chain until the issue rate binds.  Two pairs
// per lane: two chains in flight, and after the first exchange between lanes each has one pair to add.
__global__ void __launch_bounds__(32)
rho_kernel(const FermiJob one, const FermiJob* __restrict__ jobs, int lanes, double* __restrict__ buf) {
  const FermiJob job = jobs ? jobs[blockIdx.y] : one;
  const FermiBuf b = fermi_buf(buf + job.buf_off, job.M);
  const int M = job.M, p = job.p, S = rho_lanes(M, lanes);
  if (blockIdx.x * 32 / S >= rho_groups(M)) return;
  const int group = (blockIdx.x * 32 + threadIdx.x) / S, r = threadIdx.x % S;
  double s[2], e[2];
  unsigned m[2], step[2];
  const unsigned period = 4 * M;  // at most 2^26
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const unsigned odd = 2 * (2 * group + q) + 1;  // 2 j + 1; past the last pair: sums that are not used
    s[q] = e[q] = 0.0;
    step[q] = S * odd % period;
    m[q] = r * odd % period;
  }
#pragma unroll 2
  for (int k = r; k < p; k += S) {
    const double w = __ldg(b.w + k);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double y = w * __ldg(b.tab + m[q]) - e[q], t = s[q] + y;
      e[q] = (t - s[q]) - y;
      s[q] = t;
      m[q] += step[q];
      if (m[q] >= period) m[q] -= period;
    }
  }
  e[0] = -e[0];  // the sums are s + e
  e[1] = -e[1];
  // (s, e)[q] += (s2, e2) with the rounding error of s + s2 (TwoSum): rho_j carries one rounding of a sum
  auto add = [&](int q, double s2, double e2) {
    const double t = s[q] + s2, z = t - s[q];
    e[q] = (e[q] + e2) + ((s[q] - (t - z)) + (s2 - z));
    s[q] = t;
  };
  // lanes o apart add their sums; the first exchange leaves each with one of the two pairs
  int o = S / 2, pair = 2 * group;
  if (o >= 2) {
    const bool up = (r & o) != 0;
    const double s2 = __shfl_xor_sync(0xffffffffu, up ? s[0] : s[1], o), e2 = __shfl_xor_sync(0xffffffffu, up ? e[0] : e[1], o);
    if (up) {
      s[0] = s[1];
      e[0] = e[1];
      ++pair;
    }
    add(0, s2, e2);
    o >>= 1;
  }
  for (; o >= 2; o >>= 1) add(0, __shfl_xor_sync(0xffffffffu, s[0], o), __shfl_xor_sync(0xffffffffu, e[0], o));
  // an even lane holds the even part, the next the odd part; of those that hold the same pair one writes
  const bool writes = S == 2 || (r & ~1 & (S / 2 - 1)) == 0;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (q && S > 2) break;
    const double so = __shfl_xor_sync(0xffffffffu, s[q], 1), eo = __shfl_xor_sync(0xffffffffu, e[q], 1);
    if (r & 1) {
      s[q] = -s[q];
      e[q] = -e[q];
    }
    add(q, so, eo);
    const int j = pair + q, node = r & 1 ? M - 1 - j : j;
    if (j < M / 2 && writes)
      b.node[node] = make_double2(node_energy(node, M, job.emin, job.emax), (s[q] + e[q]) / M);
  }
}

// f(e) in a bisection sum.  Past 38 kT below mu, exp(z) < 2^-54 and f rounds to 2 exactly; past
// 80 kT above, f < 4e-35, far below the rounding that every rho_j carries.  Only the nodes between
// (about 1,200 whatever kT is, since M grows with W/kT) take the exponential and the division.
__device__ __forceinline__ double count_occupation(double e, double mu, double inv_kT) {
  const double z = (e - mu) * inv_kT;
  if (z <= -38.0) return 2.0;
  if (z >= 80.0) return 0.0;
  return 2.0 / (1.0 + exp(z));
}

// Bisection for N(mu) = n_e (skipped when n_e < 0), then Omega, E, N, by gridDim.x CTAs of one
// problem.  out = {mu, Omega, E, N, status}: status 1 when the bracket has no sign change, 2 when a
// wait expired.  The midpoints of the next `depth` halvings (nm = 2^depth - 1 of them) are evaluated
// at once, each by `parts` CTAs, and the halvings are then decided in order, so mu is the plain
// bisection's; one barrier for `depth` halvings.  N(mu) is summed as FERMI_LANES strided chains and
// a tree over them whatever the launch, and the observables over fixed runs of nodes, so that the results of a
// problem do not depend on the launch.  Latency binds: an FP64 operation
// takes 64 cycles or more and an occupation ~40 of them (45 halvings one after the other in one CTA: 0.65 ms
// at M = 504, 9.2 ms at M = 9904; this form 0.084 and 0.119 ms, of which the sums over 32 parts and the
// decisions were 0.02 and 0.05 more with every warp of every CTA at them).
__global__ void __launch_bounds__(FERMI_THREADS)
fermi_kernel(const FermiJob one, const FermiJob* __restrict__ jobs, int depth, int parts, double* __restrict__ buf,
             double* __restrict__ res) {
  __shared__ double red[32];
  __shared__ double cnt[FERMI_MIDS + 1];
  __shared__ double tree[16 * FERMI_MIDS];
  __shared__ double state[3];  // the bracket, and whether it is done
  __shared__ double my_mid;
  __shared__ double fs[FERMI_THREADS];
  const FermiJob job = jobs ? jobs[blockIdx.y] : one;
  const FermiBuf b = fermi_buf(buf + job.buf_off, job.M);
  double* out = res + 8 * (int64_t)blockIdx.y;
  const int M = job.M, ncta = gridDim.x, cta = blockIdx.x, tid = threadIdx.x;
  const double kT = job.kT, inv_kT = 1.0 / kT, W = job.emax - job.emin;
  int phase = 0;
  bool ok = true;
  // the chains of part pi (FERMI_LANES / parts of them), 32 of them summed into put[chain / 32]
  auto chains = [&](int pi, double mu, double* put) {
    const int span = FERMI_LANES / parts;
    if (span >= FERMI_THREADS) {  // a thread per chain, several times
      for (int g = 0; g < span; g += FERMI_THREADS) {
        const int t0 = pi * span + g + tid;
        double s = 0.0;
        for (int j = t0; j < M; j += FERMI_LANES) {
          const double2 n = __ldg(b.node + j);
          s = fma(count_occupation(n.x, mu, inv_kT), n.y, s);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) __stcg(put + (t0 >> 5), s);
      }
      return;
    }
    // several threads per chain take the occupations of consecutive links, the first one adds them
    const int rows = FERMI_THREADS / span, rr = tid / span, vt = tid - rr * span, t0 = pi * span + vt;
    double s = 0.0;
    for (int j0 = 0; j0 < M; j0 += rows * FERMI_LANES) {
      const int j = j0 + rr * FERMI_LANES + t0;
      fs[tid] = j < M ? count_occupation(__ldg(b.node + j).x, mu, inv_kT) : 0.0;
      __syncthreads();
      if (rr == 0)
        for (int q = 0; q < rows; ++q) {
          const int jj = j0 + q * FERMI_LANES + t0;
          if (jj < M) s = fma(fs[q * span + vt], __ldg(b.node + jj).y, s);
        }
      __syncthreads();
    }
    if (rr == 0) {
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if ((tid & 31) == 0) __stcg(put + (t0 >> 5), s);
    }
  };
  // cnt[q] = N(mid of q), q = 0 .. nm - 1, in every CTA
  auto evaluate = [&](int nm, auto mid_of) {
    double* part = b.part + (phase & 1) * FERMI_PART;
    if (ncta == 1) {
      for (int q = 0; q < nm; ++q) chains(0, mid_of(q), part + 32 * q);
      __threadfence_block();
      __syncthreads();
    } else {
      const int pi = cta / nm, q = cta - pi * nm;
      if (tid == 0) my_mid = mid_of(q);
      __syncthreads();
      if (pi < parts) chains(pi, my_mid, part + 32 * q);
      ok = ok && tbk_grid_wait(b.ctr, (unsigned)(ncta * (phase + 1)));
    }
    ++phase;
    // the tree over a midpoint's 32 sums, with all lanes at work on all midpoints: an SM takes 19 cycles for
    // a warp's FP64 addition
    for (int e = tid; e < 16 * nm; e += FERMI_THREADS) {
      const double* p = part + 2 * e - (e & 15);  // 32 (e / 16) + e % 16
      tree[e] = __ldcg(p) + __ldcg(p + 16);
    }
    __syncthreads();
    for (int o = 8; o > 0; o >>= 1) {
      for (int e = tid; e < o * nm; e += FERMI_THREADS) {
        const int q = e / o, i = e - q * o;
        const double t = tree[16 * q + i] + tree[16 * q + i + o];
        (o == 1 ? cnt[q] : tree[16 * q + i]) = t;
      }
      __syncthreads();
    }
  };
  double mu = job.mu_fixed, status = 0.0;
  if (job.n_e >= 0.0) {
    double lo = job.emin, hi = job.emax;
    evaluate(2, [&](int q) { return q ? hi : lo; });
    if (cnt[0] > job.n_e || cnt[1] < job.n_e) status = 1.0;
    __syncthreads();
    bool done = false;
    for (int it = 0; it < 200 && !done && ok; it += depth) {
      // heap order: node 1 is the midpoint of [lo, hi], node 2q that of the lower half below q
      evaluate((1 << depth) - 1, [&](int q) {
        double l = lo, h = hi;
        for (int bit = 30 - __clz(q + 1); bit >= 0; --bit) {
          const double mid = 0.5 * (l + h);
          if (((q + 1) >> bit) & 1) l = mid; else h = mid;
        }
        return 0.5 * (l + h);
      });
      if (tid == 0) {
        int node = 1;
        for (int d = 0; d < depth && it + d < 200 && !done; ++d) {
          const double mid = 0.5 * (lo + hi);
          const bool up = cnt[node - 1] < job.n_e;
          if (up) lo = mid; else hi = mid;
          node = 2 * node + (up ? 1 : 0);
          done = hi - lo < 1e-13 * W;
        }
        state[0] = lo;
        state[1] = hi;
        state[2] = done;
      }
      __syncthreads();
      lo = state[0];
      hi = state[1];
      done = state[2] != 0.0;
    }
    mu = 0.5 * (lo + hi);
  }
  // observables: runs of FERMI_THREADS nodes, of which a CTA takes every ncta-th; their number, and so the
  // order of the sums, follows from M alone
  const int runs = min((M + FERMI_THREADS - 1) / FERMI_THREADS, FERMI_PART / 3);
  double* part = b.part + (phase & 1) * FERMI_PART;
  for (int g = cta; g < runs; g += ncta) {
    double v[3] = {0.0, 0.0, 0.0};
    for (int j = g * FERMI_THREADS + tid; j < M; j += runs * FERMI_THREADS) {
      const double2 n = __ldg(b.node + j);
      const double f = fermi_fn(n.x, mu, kT);
      v[0] += free_fn(n.x, mu, kT) * n.y;
      v[1] += n.x * f * n.y;
      v[2] += f * n.y;
    }
    for (int q = 0; q < 3; ++q) {
      const double t = tbk_block_sum(v[q], red);
      if (tid == 0) __stcg(part + 3 * g + q, t);
    }
  }
  if (ncta > 1) ok = ok && tbk_grid_wait(b.ctr, (unsigned)(ncta * (phase + 1)));
  else __syncthreads();
  if (cta == 0 && tid < 96) {
    const int q = tid >> 5, lane = tid & 31;
    double t = 0.0;
    for (int i = lane; i < runs; i += 32) t += __ldcg(part + 3 * i + q);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) out[1 + q] = t;
    if (tid == 0) {
      out[0] = mu;
      out[4] = ok ? status : 2.0;
    }
  }
}

int quad_nodes(int p) { return std::max(4 * p, 256); }

// Enqueue the solves of n problems (jobs on the device, or `one` when NULL); M_max and p_max over
// them.  res: 8 doubles per problem.
static void fermi_launch(tbk_ctx* ctx, int n, const FermiJob& one, const FermiJob* d_jobs, int M_max, int p_max,
                         const double* moments, int damping, double* buf, double* res) {
  fermi_setup<<<dim3(ceil_div(std::max(4 * (int64_t)M_max, (int64_t)p_max), 256), n), 256, 0, ctx->stream>>>(
      one, d_jobs, moments, damping, buf);
  post_launch(ctx, "fermi_setup");
  // lanes of a problem: about eight warps per SM (the largest has fewer than twice that, or two per group)
  const int lanes = ctx->num_sms * 256, groups = rho_groups(M_max);
  const int64_t most = std::max<int64_t>(std::min<int64_t>((int64_t)groups * 32, 2 * (int64_t)lanes), 2 * (int64_t)groups);
  rho_kernel<<<dim3(ceil_div(most, 32), n), 32, 0, ctx->stream>>>(one, d_jobs, lanes, buf);
  post_launch(ctx, "rho_kernel");
  // CTAs per problem, as long as all problems fit the chip together: as many midpoints at once as
  // there is room for, then 4 to 16 CTAs per midpoint (one CTA per problem takes its midpoints one by
  // one).  Chains of one link are latency alone (M = 800: the call 120 us at depth 5 with 4 parts, 120 at
  // depth 4 and 124 at depth 5 with 8); longer ones want the CTAs for more parts instead (M = 9904, before the
  // sums were shared out: 300 us at depth 5, 171 us at 4 with twice the parts)
  int occ = 0;
  TBK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fermi_kernel, FERMI_THREADS, 0));
  const int room = occ * ctx->num_sms / n, links = ceil_div(M_max, FERMI_LANES);
  int depth = 1;
  const int depth_max = links > 1 ? FERMI_DEPTH - 1 : FERMI_DEPTH;
  while (depth < depth_max && (2 << depth) - 1 <= room) ++depth;
  const int nm = (1 << depth) - 1;
  int parts = links > 4 ? FERMI_PARTS : (links > 1 ? 8 : 4);
  while (parts > 1 && parts * nm > room) parts /= 2;
  const dim3 grid(room < 3 ? 1 : nm * parts, n);
  if (grid.x == 1) {
    fermi_kernel<<<grid, FERMI_THREADS, 0, ctx->stream>>>(one, d_jobs, 1, 1, buf, res);
  } else {
    // the CTAs of a problem wait for one another: a cooperative launch keeps them all resident
    FermiJob o = one;
    int d = depth;
    void* args[] = {&o, (void*)&d_jobs, &d, &parts, &buf, &res};
    TBK_CUDA(cudaLaunchCooperativeKernel((const void*)fermi_kernel, grid, dim3(FERMI_THREADS), args, 0, ctx->stream));
  }
  post_launch(ctx, "fermi_kernel");
}

void fermi_enqueue_batched(tbk_ctx* ctx, int n, const FermiJob* d_jobs, int M_max, int p_max, const double* moments,
                           int damping, double* buf, double* res) {
  fermi_launch(ctx, n, FermiJob(), d_jobs, M_max, p_max, moments, damping, buf, res);
}

void coefficients(tbk_ctx* ctx, int fn, int p, double emin, double emax, double mu, double kT,
                  int damping, double* out) {
  TBK_CHECK_ARG(p >= 1 && p <= (1 << 22), "order out of range");
  TBK_CHECK_ARG(fn == TBK_FN_FERMI || fn == TBK_FN_ENERGY || fn == TBK_FN_FREE, "unknown function");
  TBK_CHECK_ARG(damping == TBK_DAMP_NONE || damping == TBK_DAMP_JACKSON, "unknown damping");
  TBK_CHECK_ARG(kT > 0.0 && std::isfinite(kT), "kT must be positive");
  TBK_CHECK_ARG(emax > emin, "need emax > emin");
  const int M = quad_nodes(p);
  double* tab = (double*)scratch(ctx, WS_NODES, sizeof(double) * 5 * (size_t)M);
  double* hv = tab + 4 * (size_t)M;
  coeff_setup<<<ceil_div(4 * (int64_t)M, 256), 256, 0, ctx->stream>>>(fn, M, emin, emax, mu, kT, tab, hv);
  post_launch(ctx, "coeff_setup");
  coeff_kernel<<<p, 256, 0, ctx->stream>>>(p, M, damping, tab, hv, out);
  post_launch(ctx, "coeff_kernel");
}

// Enqueue the chemical-potential solve for one moment vector without synchronising: buf
// (fermi_doubles(quad_nodes(order), order) doubles, 16-byte aligned) and res (8 doubles: mu, Omega,
// E, N, status) are device buffers.
void fermi_enqueue(tbk_ctx* ctx, const double* moments, int order, double emin, double emax,
                   double n_electrons, double mu_fixed, double kT, int damping, double* buf, double* res) {
  TBK_CHECK_ARG(order >= 1 && order <= (1 << 22), "order out of range");
  TBK_CHECK_ARG(kT > 0.0 && std::isfinite(kT), "kT must be positive");
  TBK_CHECK_ARG(emax > emin, "need emax > emin");
  const int M = quad_nodes(order);
  const FermiJob j{M, order, emin, emax, n_electrons, mu_fixed, kT, 0, 0};
  fermi_launch(ctx, 1, j, nullptr, M, order, moments, damping, buf, res);
}

void check_fermi_status(double status, const char* no_bracket) {
  if (status == 2.0) throw Error(TBK_ERR_TIMEOUT, "a bounded wait in the chemical-potential solve expired");
  if (status != 0.0) throw Error(TBK_ERR_NOCONV, no_bracket);
}

}  // namespace tbk

using namespace tbk;

extern "C" int tbk_chebyshev_coefficients(tbk_ctx* ctx, int32_t fn, int32_t order, double emin,
                                          double emax, double mu, double kT, int32_t damping,
                                          double* out) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx && out, "NULL argument");
  DeviceGuard dg(ctx);
  coefficients(ctx, fn, order, emin, emax, mu, kT, damping, out);
  TBK_API_END
}

extern "C" int tbk_fermi_level(tbk_ctx* ctx, const double* moments, int32_t order, double emin,
                               double emax, double n_electrons, double mu_fixed, double kT,
                               int32_t damping, double* out) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx && moments && out, "NULL argument");
  TBK_CHECK_ARG(order >= 1 && order <= (1 << 22), "order out of range");
  TBK_CHECK_ARG(kT > 0.0 && std::isfinite(kT), "kT must be positive");
  TBK_CHECK_ARG(emax > emin, "need emax > emin");
  TBK_CHECK_ARG(damping == TBK_DAMP_NONE || damping == TBK_DAMP_JACKSON, "unknown damping");
  DeviceGuard dg(ctx);
  const int M = quad_nodes(order);
  const size_t nbuf = fermi_doubles(M, order);
  double* buf = (double*)scratch(ctx, WS_COEF, sizeof(double) * (nbuf + 8));
  double* res = buf + nbuf;
  fermi_enqueue(ctx, moments, order, emin, emax, n_electrons, mu_fixed, kT, damping, buf, res);
  double h[5];
  TBK_CUDA(cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  for (int i = 0; i < 4; ++i) out[i] = h[i];
  check_fermi_status(h[4], "n_electrons is outside the range of the estimated N(mu) on [emin, emax]");
  TBK_API_END
}
