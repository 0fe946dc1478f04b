// Kernel summation y_i = sum_j phi(||x_i - x_j|| / sigma) q_j of one target
// group over its list of source groups, one thread per target, sources staged
// through shared memory in chunks (the generic kernel, nearfield.cu).
#pragma once

#include "dwfmm_internal.cuh"

namespace dw {
namespace ks {

constexpr int kThreads = 128;
constexpr int kSrcChunk = 128;

// Rows of one side of a sum.
struct Side {
  int64_t gstride;   // elements between groups
  int ld;            // elements between coordinate rows (or rhs rows)
  const int32_t* count;
  int count_off;
  int count_const;   // used when count == nullptr
};

template <typename T, int KER>
__device__ __forceinline__ T phi_r2(T r2, T inv_sigma) {
  if (KER == DWFMM_K_GAUSS) return exp(T(-0.5) * r2 * inv_sigma * inv_sigma);
  const T s = sqrt(r2) * inv_sigma;
  if (KER == DWFMM_K_EXP) return exp(-s);
  const T t = T(1.7320508075688772) * s;
  return (T(1) + t) * exp(-t);
}

// Target i of group g against the entries rb .. re - 1 of its list, into out
// (the group's rows).  DM: compile-time bound on d (coordinates beyond d are
// zero, so the extra terms of the squared distance are exactly 0); RC:
// right-hand sides held in registers (rows beyond Rc are zero charges).  sc,
// sqs: DM and RC rows of kSrcChunk in shared memory.
template <typename T, int KER, int DM, int RC>
__device__ __forceinline__ void ksum_targets(int g, int i, int i_end, int rb, int re, const int32_t* col, int d,
                                             T inv_sigma, const T* tcoord, const Side& ts, const T* scoord,
                                             const Side& ss, const T* sq, int64_t sq_gstride, int sq_ld, T* out,
                                             int o_ld, int Rc, T* sc, T* sqs) {
  const int tcnt = ts.count ? ts.count[ts.count_off + g] : ts.count_const;
  T xt[DM];
#pragma unroll
  for (int k = 0; k < DM; ++k)
    xt[k] = (k < d && i < tcnt) ? tcoord[g * ts.gstride + static_cast<int64_t>(k) * ts.ld + i] : T(0);
  T acc[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) acc[r] = T(0);
  for (int e = rb; e < re; ++e) {
    const int s = col[e];
    const int scnt = ss.count ? ss.count[ss.count_off + s] : ss.count_const;
    for (int cb = 0; cb < scnt; cb += kSrcChunk) {
      const int cn = min(kSrcChunk, scnt - cb);
      __syncthreads();
      for (int idx = threadIdx.x; idx < DM * kSrcChunk; idx += kThreads) {
        const int k = idx / kSrcChunk, j = idx % kSrcChunk;
        sc[idx] = (j < cn && k < d) ? scoord[s * ss.gstride + static_cast<int64_t>(k) * ss.ld + cb + j] : T(0);
      }
      for (int idx = threadIdx.x; idx < RC * kSrcChunk; idx += kThreads) {
        const int r = idx / kSrcChunk, j = idx % kSrcChunk;
        sqs[idx] = (j < cn && r < Rc) ? sq[s * sq_gstride + static_cast<int64_t>(r) * sq_ld + cb + j] : T(0);
      }
      __syncthreads();
      for (int j = 0; j < cn; ++j) {
        T r2 = T(0);
#pragma unroll
        for (int k = 0; k < DM; ++k) {
          const T df = xt[k] - sc[k * kSrcChunk + j];
          r2 += df * df;
        }
        const T ph = phi_r2<T, KER>(r2, inv_sigma);
#pragma unroll
        for (int r = 0; r < RC; ++r) acc[r] += ph * sqs[r * kSrcChunk + j];
      }
    }
  }
  if (i < i_end) {
#pragma unroll
    for (int r = 0; r < RC; ++r)
      if (r < Rc) out[static_cast<int64_t>(r) * o_ld + i] = acc[r];
  }
}

}  // namespace ks
}  // namespace dw
