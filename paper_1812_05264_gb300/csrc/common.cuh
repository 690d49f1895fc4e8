// Internal helpers shared by the libtbk translation units: the context, device scratch,
// error handling across the C ABI, and small device utilities.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/tbk.h"

namespace tbk {

struct Error : std::runtime_error {
  int code;
  Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

void set_error(const char* msg);

#define TBK_CHECK_ARG(cond, msg)                                              \
  do {                                                                        \
    if (!(cond)) throw ::tbk::Error(TBK_ERR_ARG, std::string(__func__) + ": " + (msg)); \
  } while (0)

#define TBK_CUDA(call)                                                        \
  do {                                                                        \
    cudaError_t _e = (call);                                                  \
    if (_e != cudaSuccess)                                                    \
      throw ::tbk::Error(_e == cudaErrorMemoryAllocation ? TBK_ERR_OOM : TBK_ERR_CUDA, \
                         std::string(#call) + ": " + cudaGetErrorString(_e)); \
  } while (0)

// Named scratch slots.  Each slot is a grow-only device buffer owned by the context.
enum Slot {
  WS_PANEL0 = 0, WS_PANEL1, WS_PANEL2, WS_PANEL3, WS_HHAT, WS_PARTIALS, WS_FLAGS, WS_COEF,
  WS_TABLE, WS_NODES, WS_CELLS, WS_CELLS2, WS_CELLS3, WS_LANCZOS, WS_GACC, WS_TRANSPOSE,
  WS_CHECKPOINTS, WS_SEGMENT, WS_MISC, WS_PROBES,
  WS_LOCAL0, WS_LOCAL1, WS_LOCAL2, WS_LOCAL3, WS_LOCAL4, WS_NSLOTS
};

}  // namespace tbk

struct tbk_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int num_sms = 0;
  int64_t l2_bytes = 0;
  int64_t launches = 0;
  void* slot_ptr[tbk::WS_NSLOTS] = {};
  size_t slot_bytes[tbk::WS_NSLOTS] = {};
  void* pinned = nullptr;        // small pinned host buffer for scalar read-back
  size_t pinned_bytes = 0;
  int stall_next_step = 0;       // test hook: the next TMA-fed step's producer issues no copies
  int stall_next_adjoint = 0;    // test hook: the same of the next TMA-fed adjoint step, fused or alone
  int stall_next_outer = 0;      // test hook: the same of the next outer_rows launch
  struct Tuned {                 // tbk_autotune's choices, per operator shape and probe count
    int64_t n_rows, nnzb;
    int s, cw, windowed;        // windowed: the outer-product schedule (0 fused, 1 windowed, 2 tensor cores)
  };
  std::vector<Tuned> tuned;
  int timed_mask = 0;            // bit f set: launches of kernel family f are bracketed by events
  std::vector<cudaEvent_t> timer_events;  // (begin, end) pairs
  std::vector<int> timer_family;          // family of each pair
  size_t timer_used = 0;                  // events in use
};

namespace tbk {

// Device scratch of at least `bytes` in slot s (contents undefined after growth).
void* scratch(tbk_ctx* ctx, Slot s, size_t bytes);
// Pinned host staging of at least `bytes`.
void* pinned(tbk_ctx* ctx, size_t bytes);
// Check the launch that was just enqueued and count it.
void post_launch(tbk_ctx* ctx, const char* what);
// Make ctx->device current for the scope.
struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(tbk_ctx* ctx);
  ~DeviceGuard();
};
void sync(tbk_ctx* ctx);
// The tuned choice for an operator of n_rows rows and nnzb blocks at s probes, or NULL.
const tbk_ctx::Tuned* find_tuned(const tbk_ctx* ctx, int64_t n_rows, int64_t nnzb, int s);
// Device bytes that slot s may grow to: what is free plus what s already holds, less a reserve
// of 2 GiB + 3 % of the device for everything else.
size_t panel_budget(tbk_ctx* ctx, Slot s);
// Brackets the launches of one kernel family with events on ctx->stream when that family is
// selected by tbk_kernel_timer (and the stream is not being captured into a graph).
struct KernelTimerScope {
  tbk_ctx* ctx = nullptr;
  KernelTimerScope(tbk_ctx* c, int kernel);
  ~KernelTimerScope();
};

// Launch with programmatic stream serialization: the launch is prepared while its predecessor in the
// stream runs and starts as that one's CTAs leave; the kernel must call pdl_wait() (bulk.cuh) before it
// touches anything.  2-3 us less a step in a chain of short launches.  (A predecessor that lets the
// next launch in while its own CTAs still run made it worse: the early CTAs double up on some SMs.
// 1,000 atoms x 256 probes 28.6 us a step against 23.4, 200 atoms x 64 in FP64 92 against 37.)
template <typename... P, typename... A>
inline void launch_pdl(tbk_ctx* ctx, void (*kernel)(P...), int grid, int threads, size_t smem, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  TBK_CUDA(cudaLaunchKernelEx(&cfg, kernel, (P)args...));
}

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

// One chemical-potential solve: M quadrature nodes, order p, moments at mom_off, its scratch of
// fermi_doubles(M, p) doubles at buf_off (even) of one buffer.  n_e < 0: mu_fixed is taken as mu.
struct FermiJob {
  int M, p;
  double emin, emax, n_e, mu_fixed, kT;
  int64_t mom_off, buf_off;
};
size_t fermi_doubles(int M, int p);
void fermi_enqueue(tbk_ctx* ctx, const double* moments, int order, double emin, double emax,
                   double n_electrons, double mu_fixed, double kT, int damping, double* buf, double* res);
void fermi_enqueue_batched(tbk_ctx* ctx, int n, const FermiJob* d_jobs, int M_max, int p_max, const double* moments,
                           int damping, double* buf, double* res);
// Throws for the status of a solve (res[4]): 1 = no sign change in the bracket, 2 = a wait expired.
void check_fermi_status(double status, const char* no_bracket);
int quad_nodes(int p);

}  // namespace tbk

#define TBK_API_BEGIN try {
#define TBK_API_END                                                           \
  }                                                                           \
  catch (const ::tbk::Error& e) {                                             \
    ::tbk::set_error(e.what());                                               \
    return e.code;                                                            \
  }                                                                           \
  catch (const std::exception& e) {                                           \
    ::tbk::set_error(e.what());                                               \
    return TBK_ERR_CUDA;                                                      \
  }                                                                           \
  ::tbk::set_error("");                                                       \
  return TBK_OK;

// ---------------------------------------------------------------------------------------
// Device utilities
// ---------------------------------------------------------------------------------------

// Rademacher probe entry for (row, probe): SplitMix64 output number (row * 2^32 + probe + 1)
// of a stream seeded with `seed` (Steele, Lea & Flood, OOPSLA 2014; mix64 finaliser of
// java.util.SplittableRandom).  Returns +1 or -1.
__device__ __forceinline__ float tbk_probe_sign(uint64_t seed, uint64_t row, uint64_t probe) {
  uint64_t z = seed + ((row << 32) + probe + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  return (z >> 63) ? -1.0f : 1.0f;
}

// Fixed-order block reduction of one double (blockDim.x a multiple of 32, <= 1024).
__device__ __forceinline__ double tbk_block_sum(double v, double* smem32) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) smem32[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (warp == 0) {
    t = lane < nwarps ? smem32[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;  // valid in thread 0
}

// Waits (one thread) until *p has reached target; what was written before it reached it is visible
// after.  Bounded: 0 when 2 s of the global timer went by, or after 2^26 polls.
__device__ __forceinline__ int tbk_spin_until(const unsigned* p, unsigned target) {
  uint64_t t0 = 0, t = 0;
  for (uint32_t i = 0;; ++i) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if ((int)(v - target) >= 0) return 1;
    if ((i & 1023u) == 1023u) {
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (!t0) t0 = t;
      if (t - t0 > 2000000000ull || i >= (1u << 26)) return 0;
    }
  }
}

// Barrier of the CTAs of one cooperative launch that share *ctr (zero before the first use): the
// n-th use waits for target = n * CTAs arrivals.  What a CTA wrote before is visible to the others
// after (read it past L1).  False in all threads of the CTA when the wait expired.
__device__ __forceinline__ bool tbk_grid_wait(unsigned* ctr, unsigned target) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    ok = tbk_spin_until(ctr, target);
  }
  return __syncthreads_and(ok) != 0;
}
