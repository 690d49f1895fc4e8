// a2: assemble the block-sparse Hamiltonian on the device (Sec. II.A: the NRL copper model is
// built from Slater-Koster two-centre blocks; Sec. IV: simple-cubic lattice test models).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "model.cuh"
#include "sk.cuh"

namespace tbk {

__device__ __forceinline__ double min_image(double d, double L) {
  return L > 0.0 ? d - L * rint(d / L) : d;
}

// Table models.
__global__ void assemble_table(DevModel M, const double* __restrict__ pos, int n_atoms,
                               const int32_t* __restrict__ row_ptr,
                               const int32_t* __restrict__ col, double* __restrict__ H,
                               int* __restrict__ err) {
  const int a = blockIdx.x * blockDim.y + threadIdx.y;  // block row per y-thread group
  if (a >= n_atoms) return;
  const int b_ = M.n_orb, bb = b_ * b_;
  for (int k = row_ptr[a] + threadIdx.x; k < row_ptr[a + 1]; k += blockDim.x) {
    const int b = col[k];
    double* out = H + (int64_t)k * bb;
    if (b == a) {
      for (int i = 0; i < bb; ++i) out[i] = 0.0;
      if (M.onsite_site)
        for (int i = 0; i < b_; ++i) out[i * b_ + i] += M.onsite_site[(int64_t)a * b_ + i];
      continue;
    }
    double d[3];
    for (int c = 0; c < 3; ++c) d[c] = min_image(pos[3 * b + c] - pos[3 * a + c], M.box[c]);
    int hit = -1;
    for (int t = 0; t < M.n_disp; ++t) {
      const double* q = M.disp + 3 * t;
      if (fabs(d[0] - q[0]) <= M.tol && fabs(d[1] - q[1]) <= M.tol && fabs(d[2] - q[2]) <= M.tol) {
        hit = t;
        break;
      }
    }
    if (hit < 0) {
      atomicExch(err, 1);
      for (int i = 0; i < bb; ++i) out[i] = 0.0;
    } else {
      for (int i = 0; i < bb; ++i) out[i] = M.blocks[(int64_t)hit * bb + i];
    }
  }
}

// The Slater-Koster model: H_ba = H_ab^T to the bit (each entry is a sum of products that change sign together,
// or not at all, with d), so a pair a < b is evaluated once, and its blocks written from shared memory with
// neighbouring lanes on neighbouring words.  A warp takes `rows` block rows and a lane one pair.  The FP64
// units bind (19 cycles of an SM for a warp's instruction): with a thread per block, writing it itself, 1,000
// atoms 51 us and 10,000 atoms 180; so 38 and 137, 147 atoms 51 and 20.
constexpr int AS_LIST = 128, AS_ROWS = 8;

// Index of column b in row a, or -1.
__device__ __forceinline__ int find_block(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int a, int b) {
  int lo = row_ptr[a], hi = row_ptr[a + 1];
  const int end = hi;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (col[mid] < b) lo = mid + 1; else hi = mid;
  }
  return lo < end && col[lo] == b ? lo : -1;
}

__global__ void __launch_bounds__(32)
assemble_sk(DevModel M, const double* __restrict__ pos, int n_atoms, const int32_t* __restrict__ row_ptr,
            const int32_t* __restrict__ col, double* __restrict__ H, int rows) {
  __shared__ double S[32 * 81];
  __shared__ int rp[AS_ROWS + 1], list_k[AS_LIST], list_t[AS_LIST], list_a[AS_LIST];
  const int lane = threadIdx.x, a0 = blockIdx.x * rows, nr = min(rows, n_atoms - a0);
  if (lane <= nr) rp[lane] = row_ptr[a0 + lane];
  __syncwarp();
  for (int base = rp[0]; base < rp[nr]; base += AS_LIST) {
    int n_list = 0;
    for (int k0 = base; k0 < min(base + AS_LIST, rp[nr]); k0 += 32) {
      const int k = k0 + lane;
      bool take = false;
      int a = 0, kt = -1;
      if (k < rp[nr]) {
        while (k >= rp[a + 1]) ++a;
        a += a0;
        const int b = col[k];
        if (b == a) {
          double* out = H + (int64_t)k * 81;
          for (int i = 0; i < 81; ++i) out[i] = 0.0;
          for (int i = 0; i < 9; ++i) out[10 * i] = M.onsite[sk_l(i)];
          if (M.onsite_site)
            for (int i = 0; i < 9; ++i) out[10 * i] += M.onsite_site[(int64_t)a * 9 + i];
        } else {
          // the block of (b, a), -1 where the pattern has none; below the diagonal the pair writes this
          // block if its search finds it (always, where columns ascend)
          kt = find_block(row_ptr, col, b, a);
          take = b > a || kt < 0 || find_block(row_ptr, col, a, b) != k;
          if (b < a) kt = -1;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, take);
      if (take) {
        const int e = n_list + __popc(m & ((1u << lane) - 1));
        list_k[e] = k;
        list_t[e] = kt;
        list_a[e] = a;
      }
      n_list += __popc(m);
    }
    __syncwarp();
    for (int p0 = 0; p0 < n_list; p0 += 32) {
      const int np = min(32, n_list - p0);
      if (lane < np) {
        const int a = list_a[p0 + lane], b = col[list_k[p0 + lane]];
        double d[3];
        for (int c = 0; c < 3; ++c) d[c] = min_image(pos[3 * b + c] - pos[3 * a + c], M.box[c]);
        sk_block(d, M.V, M.r0, M.decay, S + lane * 81);
      }
      __syncwarp();
      for (int p = 0; p < np; ++p) {
        const int k = list_k[p0 + p], kt = list_t[p0 + p];
#pragma unroll
        for (int e = lane; e < 96; e += 32) {
          if (e >= 81) continue;
          H[(int64_t)k * 81 + e] = S[p * 81 + e];
          if (kt >= 0) H[(int64_t)kt * 81 + e] = S[p * 81 + e % 9 * 9 + e / 9];
        }
      }
      __syncwarp();
    }
  }
}

DevModel upload_model(tbk_ctx* ctx, const tbk_model* model, const double* box, Slot slot) {
  TBK_CHECK_ARG(model != nullptr, "model is NULL");
  DevModel M{};
  M.kind = model->kind;
  M.n_orb = model->n_orb;
  TBK_CHECK_ARG(M.kind == TBK_MODEL_SK || M.kind == TBK_MODEL_TABLE, "unknown model kind");
  TBK_CHECK_ARG(M.n_orb == 1 || M.n_orb == 9, "n_orb must be 1 or 9");
  TBK_CHECK_ARG(M.kind != TBK_MODEL_SK || M.n_orb == 9, "the Slater-Koster model has 9 orbitals");
  for (int i = 0; i < 10; ++i) M.V[i] = model->sk_V[i];
  M.r0 = model->sk_r0;
  M.decay = model->sk_decay;
  for (int i = 0; i < 3; ++i) M.onsite[i] = model->onsite_spd[i];
  if (M.kind == TBK_MODEL_SK) TBK_CHECK_ARG(M.r0 > 0.0, "sk_r0 must be positive");
  for (int c = 0; c < 3; ++c) M.box[c] = box ? box[c] : 0.0;
  M.onsite_site = model->onsite_site;
  M.n_disp = 0;
  if (M.kind == TBK_MODEL_TABLE) {
    TBK_CHECK_ARG(model->n_disp >= 0 && (model->n_disp == 0 || (model->disp && model->disp_blocks)),
                  "table model needs disp and disp_blocks");
    M.n_disp = model->n_disp;
    M.tol = model->disp_tol > 0.0 ? model->disp_tol : 1e-6;
    const size_t bb = (size_t)M.n_orb * M.n_orb;
    const size_t bytes = sizeof(double) * (3 * (size_t)M.n_disp + bb * M.n_disp) + 16;
    double* dev = (double*)scratch(ctx, slot, bytes);
    TBK_CUDA(cudaMemcpyAsync(dev, model->disp, sizeof(double) * 3 * M.n_disp, cudaMemcpyHostToDevice, ctx->stream));
    TBK_CUDA(cudaMemcpyAsync(dev + 3 * M.n_disp, model->disp_blocks, sizeof(double) * bb * M.n_disp,
                             cudaMemcpyHostToDevice, ctx->stream));
    M.disp = dev;
    M.blocks = dev + 3 * M.n_disp;
  }
  return M;
}

}  // namespace tbk

using namespace tbk;

extern "C" int tbk_assemble_H(tbk_ctx* ctx, const tbk_model* model, const double* pos,
                              int32_t n_atoms, const double* box, const int32_t* row_ptr,
                              const int32_t* col, int64_t nnzb, double* H) {
  TBK_API_BEGIN
  TBK_CHECK_ARG(ctx != nullptr, "ctx is NULL");
  TBK_CHECK_ARG(n_atoms >= 0 && nnzb >= 0, "negative size");
  TBK_CHECK_ARG(n_atoms == 0 || (pos && row_ptr && col && H), "NULL array");
  DeviceGuard dg(ctx);
  DevModel M = upload_model(ctx, model, box, WS_TABLE);
  if (n_atoms == 0) return TBK_OK;
  int* err = (int*)scratch(ctx, WS_FLAGS, 64);
  TBK_CUDA(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
  if (M.kind == TBK_MODEL_SK) {
    const int rows = std::max(1, std::min(AS_ROWS, ceil_div(n_atoms, 4 * ctx->num_sms)));
    assemble_sk<<<ceil_div(n_atoms, rows), 32, 0, ctx->stream>>>(M, pos, n_atoms, row_ptr, col, H, rows);
    post_launch(ctx, "assemble_sk");
  } else {
    assemble_table<<<ceil_div(n_atoms, 16), dim3(8, 16), 0, ctx->stream>>>(M, pos, n_atoms, row_ptr, col, H, err);
    post_launch(ctx, "assemble_table");
  }
  int herr = 0;
  TBK_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  sync(ctx);
  TBK_CHECK_ARG(herr == 0, "a neighbour displacement matches no table entry");
  TBK_API_END
}
