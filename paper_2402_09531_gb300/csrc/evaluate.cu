// Evaluation of the kernel interpolant at new points (Sec. 2):
//   s(x_t) = sum_j phi(||x_t - x_j|| / sigma) c_j,  t = 1..n_t,
// the quantity whose error at test points is the prediction error of
// Sec. 6.2.  It is evaluated exactly: targets are blocked like leaves and
// every target block meets every source leaf in the kernel-summation engine
// (float32 tuned kernel or float64 generic kernel, by the plan's precision).
#include <algorithm>

#include "dwfmm_internal.cuh"

namespace dw {

namespace {

// Targets (row-major, leading dimension ld) -> blocks [G][d][m_pad]; padding
// slots repeat the block's first target.
__global__ void k_target_blocks(const double* t, int64_t nt, int64_t ld, int d, int m_pad, int G, double* blk) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<int64_t>(G) * m_pad) return;
  const int64_t g = i / m_pad;
  const int64_t src = i < nt ? i : g * m_pad;
  const int slot = static_cast<int>(i % m_pad);
  for (int k = 0; k < d; ++k) blk[(g * d + k) * m_pad + slot] = t[src * ld + k];
}

// All leaves for each of G rows, each row in `parts` pieces.
__global__ void k_full_lists(int G, int L, int parts, int32_t* rowptr, int32_t* col) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i <= static_cast<int64_t>(G) * parts)
    rowptr[i] = static_cast<int32_t>((i / parts) * L + (i % parts) * L / parts);
  if (i < static_cast<int64_t>(G) * L) col[i] = static_cast<int32_t>(i % L);
}

// The parts of every sum added in order.
template <typename T>
__global__ void k_eval_out(const T* out, int splits, int64_t split_stride, int64_t nt, int m_pad, int r0, int Rc,
                           double* y, int64_t ldy) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= nt * Rc) return;
  const int r = static_cast<int>(i / nt);
  const int64_t t = i % nt;
  const int64_t g = t / m_pad;
  const int slot = static_cast<int>(t % m_pad);
  const int64_t at = (g * kRC + r) * m_pad + slot;
  double v = static_cast<double>(out[at]);
  for (int p = 1; p < splits; ++p) v += static_cast<double>(out[p * split_stride + at]);
  y[(r0 + r) * ldy + t] = v;
}

// Workspaces are kept up to this size; a larger one is released after the call.
constexpr size_t kKeepBytes = size_t(256) << 20;

template <typename T>
void trim(DBuf<T>& b) {
  if (b.n * sizeof(T) > kKeepBytes) b.release();
}

}  // namespace

void evaluate(Plan& P, const double* tgt, int64_t nt, int64_t ldt, const double* c, int64_t ldc, double* out,
              int64_t ldo, int R) {
  cudaStream_t s = P.stream;
  const bool fp64 = P.prec == DWFMM_P_FP64;
  const int m = P.m_pad;
  const int G = static_cast<int>((nt + m - 1) / m);
  const int D = sum_padded_dim(P.d);
  if (!fp64 && D < 0) fail(DWFMM_ERR_INVALID_ARG, "evaluation in float32 needs d <= 20");
  P.ev_blk.alloc(static_cast<size_t>(G) * P.d * m);
  k_target_blocks<<<ceil_div(static_cast<int64_t>(G) * m, 256), 256, 0, s>>>(tgt, nt, ldt, P.d, m, G, P.ev_blk.p);
  ensure_workspace(P, fp64);
  const int64_t stride = static_cast<int64_t>(G) * kRC * m;
  // few target blocks leave most SMs idle: cut the sources into parts until
  // there are 8 CTAs for each SM (40 blocks of 256 targets against 131072
  // sites, d = 10 Gaussian: 3.50 ms in one part)
  const int splits = std::max(1, std::min({64, P.L, ceil_div(8 * sm_count(), G)}));
  // all leaves, for every block (float64) or as one row
  const int rows = fp64 ? G : 1, pieces = fp64 ? 1 : splits;
  P.ev_rows.alloc(static_cast<size_t>(rows) * pieces + 1);
  P.ev_col.alloc(static_cast<size_t>(rows) * P.L);
  k_full_lists<<<ceil_div(static_cast<int64_t>(rows) * std::max(P.L, pieces) + 1, 256), 256, 0, s>>>(
      rows, P.L, pieces, P.ev_rows.p, P.ev_col.p);
  if (fp64) {
    P.ev_out64.alloc(static_cast<size_t>(splits) * stride);
  } else {
    P.ev_blk32.alloc(static_cast<size_t>(G) * (D + 1) * m);
    launch_scaled_blocks(P.ev_blk.p, G, P.d, D, m, P.kernel, P.sigma, P.ev_blk32.p, s);
    P.ev_out32.alloc(static_cast<size_t>(splits) * stride);
  }
  for (int r0 = 0; r0 < R; r0 += kRC) {
    const int Rc = std::min(kRC, R - r0);
    launch_gather(P, c, ldc, r0, Rc, fp64, fp64 ? nullptr : P.xq32.p);
    if (fp64) {
      eval_f64(P, P.ev_blk.p, G, P.ev_rows.p, P.ev_col.p, splits, stride, Rc, P.ev_out64.p, s);
      k_eval_out<double><<<ceil_div(nt * Rc, 256), 256, 0, s>>>(P.ev_out64.p, splits, stride, nt, m, r0, Rc, out, ldo);
    } else {
      eval_f32(P, P.ev_blk32.p, G, P.ev_rows.p, P.ev_col.p, splits, stride, Rc, P.ev_out32.p, s);
      k_eval_out<float><<<ceil_div(nt * Rc, 256), 256, 0, s>>>(P.ev_out32.p, splits, stride, nt, m, r0, Rc, out, ldo);
    }
  }
  DW_CUDA(cudaGetLastError());
  DW_CUDA(cudaStreamSynchronize(s));
  trim(P.ev_blk);
  trim(P.ev_col);
  trim(P.ev_out64);
  trim(P.ev_blk32);
  trim(P.ev_out32);
}

}  // namespace dw
