// Tuned float32 kernel summation for sm_103a: the P2P near field and the M2L
// couplings of the DW-FMM (Sec. 5.2), y_i = sum_j phi(|x_i - x_j| / sigma) q_j,
// where p2p_rot.cu and the tensor-core kernels do not apply, and direct sums.
//
// Design (one CTA per target group: a leaf, or a cluster's node set):
//  - Source blocks (scaled coordinates plus a norm row, then R charge rows)
//    are contiguous and 32-byte aligned in HBM, so each block is two 1-D TMA
//    bulk copies (cp.async.bulk, mbarrier completion) into a double-buffered
//    shared-memory stage; thread 0 issues, every thread waits with a bounded
//    try_wait loop that raises an error flag instead of hanging.
//  - Each thread owns TT targets; sources are read as float4 broadcasts from
//    shared memory, 4 sources per step.
//  - The kernel constants are folded into the coordinates when the source
//    blocks are built:
//      Gaussian:  x' = x sqrt(log2 e / (2 sigma^2)),  phi = ex2(2 x'.s' - |x'|^2 - |s'|^2)
//      exp:       x' = x log2 e / sigma,               phi = ex2(-|x' - s'|)
//      Matern:    x' = x sqrt3 / sigma,                phi = (1 + r') ex2(-r' log2 e)
//    so the Gaussian costs D FMAs, one add and one MUFU.EX2 per pair.
//  - Arithmetic is packed: fma/add/sub.f32x2 (two lanes per instruction) for
//    distances and accumulation; charges are interleaved per source.
//  - Per source block the contributions are summed in float32 partials, then
//    folded into per-target running sums with Kahan compensation (kept in
//    shared memory).
#include <atomic>
#include <cstdint>

#include "dwfmm_internal.cuh"
#include "sum_f32.cuh"

namespace dw {

namespace {

using namespace sk;

// One CTA per target group and part of its list (the whole CTA is the group):
// part p writes at out + p * split_stride.
template <int D, int RC, int KER>
__global__ void __launch_bounds__(kThreadsMax, 3) k_sum_f32(SumArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[2];
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int tile_base = 0;
  const Grp G{static_cast<int>(threadIdx.x), static_cast<int>(blockDim.x), 0};
  // the parts' boundaries are read, not computed: any arithmetic on them takes
  // the list walk out of the uniform registers (31 more registers a thread)
  if (a.entry_t) {   // one entry's sum
    const int e = static_cast<int>(blockIdx.x);
    (void)sum_block<D, RC, KER>(a, a.entry_t[2 * e] - a.entry_off, e, e + 1, a.out + e * a.out_gstride, G, smem, full,
                                tile_base);
    return;
  }
  const int part = static_cast<int>(blockIdx.y);
  const int g = a.first + static_cast<int>(blockIdx.x);
  const int row = a.first_row + static_cast<int>(blockIdx.x) * a.row_step + part;
  const int rb = a.rowptr[row], re = a.rowptr[row + 1];
  (void)sum_block<D, RC, KER>(a, g, rb, re, a.out + part * a.split_stride + g * a.out_gstride, G, smem, full,
                              tile_base);
}

// Rows of `parts` equal pieces of every list (rows * parts + 1 boundaries).
__global__ void k_part_rows(const int32_t* rowptr, int rows, int parts, int32_t* out) {
  const int t = static_cast<int>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t > rows * parts) return;
  const int g = t < rows * parts ? t / parts : rows - 1, p = t < rows * parts ? t % parts : parts;
  const int64_t len = rowptr[g + 1] - rowptr[g];
  out[t] = rowptr[g] + static_cast<int32_t>((len * p) / parts);
}

// out[g][r][i] = the parts' sums added in order, compensated (r < Rc).
__global__ void k_add_parts(const float* part, int splits, int64_t stride, int groups, int ld, int Rc, float* out) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= static_cast<int64_t>(groups) * Rc * ld) return;
  const int64_t gr = t / ld;
  const int64_t at = ((gr / Rc) * kRC + gr % Rc) * ld + t % ld;
  float s = part[at], c = 0.0f;
  for (int p = 1; p < splits; ++p) {
    const float y = part[p * stride + at] - c, z = s + y;
    c = (z - s) - y;
    s = z;
  }
  out[at] = s;
}

// out[g][r][i] = the sums of row g's entries [entry][Rc][ld], in list order,
// with the compensation of sum_block.
__global__ void k_fold_entries(const float* part, const int32_t* rowptr, int groups, int ld, int Rc, float* out) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= static_cast<int64_t>(groups) * Rc * ld) return;
  const int i = static_cast<int>(t % ld);
  const int64_t gr = t / ld;
  const int r = static_cast<int>(gr % Rc);
  const int g = static_cast<int>(gr / Rc);
  const int64_t at = static_cast<int64_t>(r) * ld + i, step = static_cast<int64_t>(Rc) * ld;
  float acc = 0.0f, c = 0.0f;
  const int re = rowptr[g + 1];
  for (int e = rowptr[g]; e < re; e += 8) {
    float w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = e + u < re ? part[(e + u) * step + at] : 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (e + u >= re) break;
      const float y = w[u] - c, s = acc + y;
      c = (s - acc) - y;
      acc = s;
    }
  }
  out[(static_cast<int64_t>(g) * kRC + r) * ld + i] = acc;
}

// Row layout [g][16][ld] -> interleaved [g][ld][RC] (first RC rows).
__global__ void k_interleave(const float* src, int64_t groups, int ld, int RC, float* dst) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= groups * ld * RC) return;
  interleave_elem(src, ld, RC, dst, t);
}

// Scaled source blocks [g][D+1][ld] from float64 coordinates [g][d][ld].
__global__ void k_scaled_blocks(const double* src, int64_t groups, int d, int D, int ld, int kernel,
                                double sigma, float* dst) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= groups * ld) return;
  const int64_t g = t / ld;
  const int i = static_cast<int>(t % ld);
  double scale;
  if (kernel == DWFMM_K_GAUSS) scale = sqrt(1.4426950408889634 / (2.0 * sigma * sigma));
  else if (kernel == DWFMM_K_EXP) scale = 1.4426950408889634 / sigma;
  else scale = 1.7320508075688772 / sigma;
  double n2 = 0.0;
  for (int k = 0; k < D; ++k) {
    const double v = k < d ? src[(g * d + k) * ld + i] * scale : 0.0;
    const float f = static_cast<float>(v);
    dst[(g * (D + 1) + k) * ld + i] = f;
    n2 += static_cast<double>(f) * static_cast<double>(f);
  }
  dst[(g * (D + 1) + D) * ld + i] = static_cast<float>(n2);
}

// Couplings of small node sets: one CTA per target cluster, one node and one
// share of the list per thread (thread (t, sub) takes the entries sub, sub +
// nsub, ...), so that 10 nodes do not leave 22 lanes of a warp idle.  Each
// entry's n terms are summed in float32, entries and threads with
// compensation.  The blocks are read through L1 (the lanes of a share read the
// same words).  10 nodes, d = 8, N = 100003, 4 right-hand sides: 131 us with one
// CTA of 32 threads a cluster, 36 us; 20 nodes, d = 16, N = 50021: 184, 98 us.
struct SmallArgs {
  const float* nodes;      // scaled blocks [c][D + 1][ld]
  const float* mom;        // [c][16][ld], zero beyond n
  float* loc;
  const int32_t* rowptr;
  const int32_t* col;
  int first, n, ld, Rc;
};

constexpr int kSmallThreads = 128;
constexpr int kSmallNodes = 32;   // padded nodes

template <int D, int RC, int KER>
__global__ void __launch_bounds__(kSmallThreads) k_m2l_small(const SmallArgs a) {
  __shared__ float red[2][RC][kSmallThreads];
  const int g = a.first + static_cast<int>(blockIdx.x);
  const int tid = static_cast<int>(threadIdx.x);
  const int nsub = kSmallThreads / a.n;
  const int sub = tid / a.n, t = tid - sub * a.n;
  const int ld = a.ld, n4 = (a.n + 3) & ~3;
  const int rb = a.rowptr[g], re = sub < nsub ? a.rowptr[g + 1] : rb;
  const float* tb = a.nodes + static_cast<int64_t>(g) * (D + 1) * ld + t;
  u64 x2[D], nt2;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float v = KER == DWFMM_K_GAUSS ? 2.0f * tb[k * ld] : tb[k * ld];
    x2[k] = pk2(v, v);
  }
  nt2 = pk2(-tb[D * ld], -tb[D * ld]);
  float s[RC], c[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) s[r] = c[r] = 0.0f;
  for (int e = rb + sub; e < re; e += nsub) {
    const int64_t src = a.col[e];
    const float* sb = a.nodes + src * (D + 1) * ld;
    const float* q = a.mom + src * kRC * ld;
    u64 acc[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = 0ull;
    for (int j = 0; j < n4; j += 4) {
      u64 e0, e1;
      if (KER == DWFMM_K_GAUSS) {
        const ulonglong2 ns = *reinterpret_cast<const ulonglong2*>(sb + D * ld + j);
        e0 = fsub2(nt2, ns.x);
        e1 = fsub2(nt2, ns.y);
      } else {
        e0 = e1 = 0ull;
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const ulonglong2 sv = *reinterpret_cast<const ulonglong2*>(sb + k * ld + j);
        if (KER == DWFMM_K_GAUSS) {
          e0 = ffma2(x2[k], sv.x, e0);
          e1 = ffma2(x2[k], sv.y, e1);
        } else {
          const u64 d0 = fsub2(x2[k], sv.x), d1 = fsub2(x2[k], sv.y);
          e0 = ffma2(d0, d0, e0);
          e1 = ffma2(d1, d1, e1);
        }
      }
      float p0, p1, p2, p3;
      up2(e0, p0, p1);
      up2(e1, p2, p3);
      const u64 f0 = pk2(phi_scaled<KER>(p0), phi_scaled<KER>(p1)), f1 = pk2(phi_scaled<KER>(p2), phi_scaled<KER>(p3));
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(q + r * ld + j);
        acc[r] = ffma2(f0, qv.x, acc[r]);
        acc[r] = ffma2(f1, qv.y, acc[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      float v0, v1;
      up2(acc[r], v0, v1);
      const float y = (v0 + v1) - c[r], z = s[r] + y;
      c[r] = (z - s[r]) - y;
      s[r] = z;
    }
  }
#pragma unroll
  for (int r = 0; r < RC; ++r) {
    red[0][r][tid] = s[r];
    red[1][r][tid] = c[r];
  }
  __syncthreads();
  for (int o = tid; o < a.n * a.Rc; o += kSmallThreads) {
    const int r = o / a.n, i = o - r * a.n;
    float v = red[0][r][i], w = red[1][r][i];
    for (int u = 1; u < nsub; ++u) {
      const float y = red[0][r][u * a.n + i] - (red[1][r][u * a.n + i] + w), z = v + y;
      w = (z - v) - y;
      v = z;
    }
    a.loc[(static_cast<int64_t>(g) * kRC + r) * ld + i] = v;
  }
}

template <int D, int RC>
void m2l_small_kernel(int kernel, const SmallArgs& a, int groups, cudaStream_t s) {
  if (kernel == DWFMM_K_EXP) k_m2l_small<D, RC, DWFMM_K_EXP><<<groups, kSmallThreads, 0, s>>>(a);
  else if (kernel == DWFMM_K_MATERN32) k_m2l_small<D, RC, DWFMM_K_MATERN32><<<groups, kSmallThreads, 0, s>>>(a);
  else k_m2l_small<D, RC, DWFMM_K_GAUSS><<<groups, kSmallThreads, 0, s>>>(a);
}

template <int D>
void m2l_small_rc(int kernel, int RC, const SmallArgs& a, int groups, cudaStream_t s) {
  if (RC <= 1) m2l_small_kernel<D, 1>(kernel, a, groups, s);
  else if (RC <= 4) m2l_small_kernel<D, 4>(kernel, a, groups, s);
  else if (RC <= 8) m2l_small_kernel<D, 8>(kernel, a, groups, s);
  else m2l_small_kernel<D, 16>(kernel, a, groups, s);
}

void m2l_small(Plan& P, int D, int RC, int Rc, int first) {
  const SmallArgs a{P.d_ynodek.p, P.mom32.p, P.loc32.p, P.d_far_rowptr.p, P.d_far_col.p, first, P.n, P.n_pad, Rc};
  const int groups = P.C - first;
  switch (D) {
    case 4: m2l_small_rc<4>(P.kernel, RC, a, groups, P.stream); break;
    case 8: m2l_small_rc<8>(P.kernel, RC, a, groups, P.stream); break;
    case 10: m2l_small_rc<10>(P.kernel, RC, a, groups, P.stream); break;
    case 12: m2l_small_rc<12>(P.kernel, RC, a, groups, P.stream); break;
    case 16: m2l_small_rc<16>(P.kernel, RC, a, groups, P.stream); break;
    default: m2l_small_rc<20>(P.kernel, RC, a, groups, P.stream); break;
  }
}

template <int D, int RC>
void launch_kernel_type(int kernel, SumArgs a, int groups, int threads, size_t smem, cudaStream_t s) {
  switch (kernel) {
    case DWFMM_K_EXP:
      k_sum_f32<D, RC, DWFMM_K_EXP><<<dim3(groups, a.parts), threads, smem, s>>>(a);
      break;
    case DWFMM_K_MATERN32:
      k_sum_f32<D, RC, DWFMM_K_MATERN32><<<dim3(groups, a.parts), threads, smem, s>>>(a);
      break;
    default:
      k_sum_f32<D, RC, DWFMM_K_GAUSS><<<dim3(groups, a.parts), threads, smem, s>>>(a);
  }
}

template <int D>
void launch_rc(int kernel, int RC, SumArgs a, int groups, int threads, size_t smem, cudaStream_t s) {
  if (RC <= 1) launch_kernel_type<D, 1>(kernel, a, groups, threads, smem, s);
  else if (RC <= 4) launch_kernel_type<D, 4>(kernel, a, groups, threads, smem, s);
  else if (RC <= 8) launch_kernel_type<D, 8>(kernel, a, groups, threads, smem, s);
  else launch_kernel_type<D, 16>(kernel, a, groups, threads, smem, s);
}

template <int D>
void set_attrs() {
  const int big = 200 * 1024;
#define DW_ATTR(RC)                                                                                           \
  cudaFuncSetAttribute(k_sum_f32<D, RC, DWFMM_K_EXP>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);      \
  cudaFuncSetAttribute(k_sum_f32<D, RC, DWFMM_K_MATERN32>, cudaFuncAttributeMaxDynamicSharedMemorySize, big); \
  cudaFuncSetAttribute(k_sum_f32<D, RC, DWFMM_K_GAUSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  DW_ATTR(1)
  DW_ATTR(4)
  DW_ATTR(8)
  DW_ATTR(16)
#undef DW_ATTR
}

int padded_dim(int d) {
  if (d <= 4) return 4;
  if (d <= 8) return 8;
  if (d <= 10) return 10;
  if (d <= 12) return 12;
  if (d <= 16) return 16;
  if (d <= 20) return 20;
  return -1;
}

int padded_rc(int Rc) { return Rc <= 1 ? 1 : Rc <= 4 ? 4 : Rc <= 8 ? 8 : 16; }

void dispatch(int D, int kernel, int RC, SumArgs a, int groups, int threads, size_t smem, cudaStream_t s) {
  switch (D) {
    case 4: launch_rc<4>(kernel, RC, a, groups, threads, smem, s); break;
    case 8: launch_rc<8>(kernel, RC, a, groups, threads, smem, s); break;
    case 10: launch_rc<10>(kernel, RC, a, groups, threads, smem, s); break;
    case 12: launch_rc<12>(kernel, RC, a, groups, threads, smem, s); break;
    case 16: launch_rc<16>(kernel, RC, a, groups, threads, smem, s); break;
    default: launch_rc<20>(kernel, RC, a, groups, threads, smem, s); break;
  }
}

// Devices whose kernel attributes are set.  Atomic: host threads may make
// their first call on a device at the same time (both then set the same
// attributes, which is harmless).
std::atomic<uint64_t> g_attrs_dev{0};

constexpr size_t kEntryPartsBytes = size_t(256) << 20;   // one sum per near entry

void ensure_attrs() {
  const uint64_t bit = device_bit();
  if (g_attrs_dev.load() & bit) return;
  set_attrs<4>();
  set_attrs<8>();
  set_attrs<10>();
  set_attrs<12>();
  set_attrs<16>();
  set_attrs<20>();
  DW_CUDA(cudaGetLastError());
  g_attrs_dev.fetch_or(bit);
}

// Scaled blocks for the current tree: leaf sites and cluster nodes.
void ensure_scaled(Plan& P, int D) {
  if (P.dpad == D && P.d_ptsk.p && P.d_ynodek.p) return;
  const int64_t nl = static_cast<int64_t>(P.L) * (D + 1) * P.m_pad;
  const int64_t nc = static_cast<int64_t>(P.C) * (D + 1) * P.n_pad;
  P.d_ptsk.alloc(nl);
  P.d_ynodek.alloc(nc);
  k_scaled_blocks<<<ceil_div(static_cast<int64_t>(P.L) * P.m_pad, 256), 256, 0, P.stream>>>(
      P.d_pts64.p, P.L, P.d, D, P.m_pad, P.kernel, P.sigma, P.d_ptsk.p);
  k_scaled_blocks<<<ceil_div(static_cast<int64_t>(P.C) * P.n_pad, 256), 256, 0, P.stream>>>(
      P.d_ynode64.p, P.C, P.d, D, P.n_pad, P.kernel, P.sigma, P.d_ynodek.p);
  DW_CUDA(cudaGetLastError());
  P.dpad = D;
}

size_t stage_bytes(int D, int RC, int ld) {
  const size_t comp = static_cast<size_t>(kTT) * (RC >= 2 ? RC / 2 : 1) * kThreadsMax * sizeof(unsigned long long);
  return 2 * static_cast<size_t>((D + 1) * ld + RC * ld) * sizeof(float) + comp;
}

}  // namespace

int sum_padded_dim(int d) { return padded_dim(d); }
int sum_padded_rc(int r) { return padded_rc(r); }
size_t sum_stage_bytes(int D, int RC, int ld) { return stage_bytes(D, RC, ld); }
void ensure_sum_attrs() { ensure_attrs(); }

void launch_sum_f32(int D, int kernel, int RC, const SumArgs& a, int groups, int threads, size_t smem,
                    cudaStream_t s) {
  if (groups > 0) dispatch(D, kernel, RC, a, groups, threads, smem, s);
}

void launch_interleave(const float* src, int64_t groups, int ld, int RC, float* dst, cudaStream_t s) {
  const int64_t nq = groups * ld * RC;
  if (nq > 0) k_interleave<<<ceil_div(nq, 256), 256, 0, s>>>(src, groups, ld, RC, dst);
}

void launch_scaled_blocks(const double* src, int64_t groups, int d, int D, int ld, int kernel, double sigma,
                          float* dst, cudaStream_t s) {
  if (groups > 0)
    k_scaled_blocks<<<ceil_div(groups * ld, 256), 256, 0, s>>>(src, groups, d, D, ld, kernel, sigma, dst);
}

// rot: each unordered pair once (rot_ready).  The charges are in P.xq32, but for
// 9..16 right-hand sides of MIXED plans.
bool p2p_f32_tuned(Plan& P, int Rc, bool rot, bool steady, cudaStream_t s) {
  const int D = padded_dim(P.d);
  if (D < 0) return false;
  const int RC = padded_rc(Rc);
  const size_t smem = stage_bytes(D, RC, P.m_pad);
  if (smem > 200 * 1024) return false;
  ensure_attrs();
  ensure_scaled(P, D);
  // the tree build made the scaled blocks on P.stream; the side stream waits
  if (s != P.stream) {
    DW_CUDA(cudaEventRecord(P.ev_scaled, P.stream));
    DW_CUDA(cudaStreamWaitEvent(s, P.ev_scaled, 0));
  }
  if (rot) {
    P.near_engine = 2;
    near_rot(P, D, Rc, s);
    P.near_parts = 2;
    DW_CUDA(cudaGetLastError());
    return true;
  }
  // MIXED plans with 9..16 right-hand sides: contraction on the tensor cores,
  // each unordered near pair once where the symmetric kernel applies
  P.near_engine = 4;
  if (P.prec == DWFMM_P_MIXED && RC == 16 && near_sym_tc(P, D, Rc, s)) return true;
  P.near_engine = 3;
  if (P.prec == DWFMM_P_MIXED && RC == 16)   // the gather leaves these to the kernels that read them
    launch_interleave(P.xb32.p, P.L, P.m_pad, RC, P.xq32.p, s);
  if (P.prec == DWFMM_P_MIXED && RC == 16 &&
      sum_tc(D, P.kernel, P.d_ptsk.p, static_cast<int64_t>(D + 1) * P.m_pad, P.d_ptsk.p,
             static_cast<int64_t>(D + 1) * P.m_pad, P.xq32.p, P.L, P.bq32, P.ynear32.p,
             static_cast<int64_t>(kRC) * P.m_pad, P.d_near_rowptr.p, P.d_near_col.p, P.d_count.p, P.L - 1, 0, 0,
             P.L, P.m_pad, Rc, P.gauss_fact, P.d_err.p, s))
    return true;
  P.near_engine = 2;
  SumArgs a{};
  a.tgt = P.d_ptsk.p;
  a.tgt_gstride = static_cast<int64_t>(D + 1) * P.m_pad;
  a.src = P.d_ptsk.p;
  a.src_gstride = a.tgt_gstride;
  a.q = P.xq32.p;
  a.q_gstride = static_cast<int64_t>(RC) * P.m_pad;
  a.out = P.ynear32.p;
  a.out_gstride = static_cast<int64_t>(kRC) * P.m_pad;
  a.rowptr = P.d_near_rowptr.p;
  a.col = P.d_near_col.p;
  a.count = P.d_count.p;
  a.count_off = P.L - 1;
  a.count_const = 0;
  a.first = 0;
  a.ld = P.m_pad;
  a.Rc = Rc;
  a.err = P.d_err.p;
  const int threads = std::min(kThreadsMax, round_up(ceil_div(P.m_pad, kTT), 32));
  // few leaves: their lists in up to 16 parts, until every SM has 4 CTAs
  // (d = 10 Gaussian, N = 3362, 12 right-hand sides, 16 leaves: the product
  // took 177 us in one part, 45 us in 16)
  const int splits = std::max(1, std::min(16, 4 * sm_count() / P.L));
  const size_t col = static_cast<size_t>(P.nnear) * P.m_pad;   // one sum per entry
  const size_t most = kEntryPartsBytes / (col * sizeof(float));
  const int64_t part = static_cast<int64_t>(P.L) * a.out_gstride;
  if (steady && splits > 1 && most >= static_cast<size_t>(Rc) &&
      P.grow(P.entry_parts32, col * P.work_cols(Rc, RC, most))) {
    // every entry's sum by itself, then in list order with the compensation
    // that one CTA per leaf would carry: the same bits, on all SMs
    // (N = 3001, d = 16: 174 us with 32 CTAs)
    a.entry_t = P.d_near_pairs.p;
    a.entry_off = P.L - 1;
    a.out_gstride = static_cast<int64_t>(Rc) * P.m_pad;
    a.out = P.entry_parts32.p;
    dispatch(D, P.kernel, RC, a, static_cast<int>(P.nnear), threads, smem, s);
    k_fold_entries<<<ceil_div(static_cast<int64_t>(P.L) * Rc * P.m_pad, 128), 128, 0, s>>>(
        P.entry_parts32.p, P.d_near_rowptr.p, P.L, P.m_pad, Rc, P.ynear32.p);
  } else if (splits > 1 && !steady && (P.part_rows.p || !capturing(P.stream)) &&
             P.grow(P.near_parts32, static_cast<size_t>(splits) * part)) {
    if (!P.part_rows.p) {   // once per tree, outside a capture
      P.part_rows.alloc(static_cast<size_t>(P.L) * splits + 1);
      k_part_rows<<<ceil_div(static_cast<int64_t>(P.L) * splits + 1, 256), 256, 0, s>>>(P.d_near_rowptr.p, P.L, splits,
                                                                                       P.part_rows.p);
    }
    a.rowptr = P.part_rows.p;
    a.row_step = a.parts = splits;
    a.split_stride = part;
    a.out = P.near_parts32.p;
    dispatch(D, P.kernel, RC, a, P.L, threads, smem, s);
    k_add_parts<<<ceil_div(static_cast<int64_t>(P.L) * Rc * P.m_pad, 256), 256, 0, s>>>(
        P.near_parts32.p, splits, a.split_stride, P.L, P.m_pad, Rc, P.ynear32.p);
  } else {
    dispatch(D, P.kernel, RC, a, P.L, threads, smem, s);
  }
  DW_CUDA(cudaGetLastError());
  return true;
}

// Every target block against every source leaf in float32 (exact evaluation),
// the sources in `parts` parts; part p writes at out + p * split_stride.
// tgtk: scaled target blocks; rowptr, col: one row of all leaves, cut into the
// parts.
void eval_f32(Plan& P, const float* tgtk, int G, const int32_t* rowptr, const int32_t* col,
              int parts, int64_t split_stride, int Rc, float* out, cudaStream_t s) {
  const int D = padded_dim(P.d);
  const int RC = padded_rc(Rc);
  ensure_attrs();
  ensure_scaled(P, D);
  SumArgs a{};
  a.tgt = tgtk;
  a.tgt_gstride = static_cast<int64_t>(D + 1) * P.m_pad;
  a.src = P.d_ptsk.p;
  a.src_gstride = a.tgt_gstride;
  a.q = P.xq32.p;
  a.q_gstride = static_cast<int64_t>(RC) * P.m_pad;
  a.out = out;
  a.out_gstride = static_cast<int64_t>(kRC) * P.m_pad;
  a.rowptr = rowptr;
  a.col = col;
  a.row_step = 0;
  a.parts = parts;
  a.split_stride = split_stride;
  a.count = P.d_count.p;
  a.count_off = P.L - 1;
  a.ld = P.m_pad;
  a.Rc = Rc;
  a.err = P.d_err.p;
  const int threads = std::min(kThreadsMax, round_up(ceil_div(P.m_pad, kTT), 32));
  dispatch(D, P.kernel, RC, a, G, threads, stage_bytes(D, RC, P.m_pad), s);
  DW_CUDA(cudaGetLastError());
}

namespace {

// The ordered-pair tensor-core M2L (every far block, both orderings):
// interleaved moments, then the kernel-summation engine on node sets.
bool m2l_ordered_tc(Plan& P, int D, int Rc) {
  const int first = (1 << P.jmin) - 1;
  P.momq32.alloc(static_cast<size_t>(P.C) * P.n_pad * kRC);
  const int64_t nq = static_cast<int64_t>(P.C) * P.n_pad * 16;
  k_interleave<<<ceil_div(nq, 256), 256, 0, P.stream>>>(P.mom32.p, P.C, P.n_pad, 16, P.momq32.p);
  // own charge-block scratch: the near field runs concurrently on the side stream
  return sum_tc(D, P.kernel, P.d_ynodek.p, static_cast<int64_t>(D + 1) * P.n_pad, P.d_ynodek.p,
                static_cast<int64_t>(D + 1) * P.n_pad, P.momq32.p, P.C, P.bqm32, P.loc32.p,
                static_cast<int64_t>(kRC) * P.n_pad, P.d_far_rowptr.p, P.d_far_col.p, nullptr, 0, P.n, first,
                P.C - first, P.n_pad, Rc, P.gauss_fact, P.d_err.p, P.stream);
}

}  // namespace

// MIXED plans with 9..16 right-hand sides have two tensor-core M2L engines
// (every ordered far pair, TF32 hi/lo; each unordered pair once, FP16 hi/lo
// with fixed-point transposed sums).  Unless the caller chose one, the
// first such matvec of a tree times both on the plan's moments buffer (set
// to zero; values do not change the time) before the near field starts,
// and the faster is kept for the tree.  Not while the stream is being
// captured or the phase timers run (the ordered engine then).
void m2l_autotune(Plan& P, int Rc) {
  if (P.prec != DWFMM_P_MIXED || Rc < 9 || Rc > 16 || P.m2l_pref >= 0 || P.m2l_tuned >= 0) return;
  if (P.jmin > P.J || P.tm.on) return;
  if (capturing(P.stream)) return;
  const int D = padded_dim(P.d);
  if (D < 0 || stage_bytes(D, 16, P.n_pad) > 200 * 1024) return;
  ensure_attrs();
  ensure_scaled(P, D);
  DW_CUDA(cudaMemsetAsync(P.mom32.p, 0, static_cast<size_t>(P.C) * kRC * P.n_pad * sizeof(float), P.stream));
  cudaEvent_t e0, e1, e2;
  DW_CUDA(cudaEventCreate(&e0));
  DW_CUDA(cudaEventCreate(&e1));
  DW_CUDA(cudaEventCreate(&e2));
  DW_CUDA(cudaEventRecord(e0, P.stream));
  const bool sym = m2l_sym_tc(P, D, Rc, P.stream);
  DW_CUDA(cudaEventRecord(e1, P.stream));
  const bool ord = m2l_ordered_tc(P, D, Rc);
  DW_CUDA(cudaEventRecord(e2, P.stream));
  DW_CUDA(cudaEventSynchronize(e2));
  float ms_sym = 0.f, ms_ord = 0.f;
  DW_CUDA(cudaEventElapsedTime(&ms_sym, e0, e1));
  DW_CUDA(cudaEventElapsedTime(&ms_ord, e1, e2));
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaEventDestroy(e2);
  P.m2l_tune_ms[0] = sym ? ms_sym : -1.0;
  P.m2l_tune_ms[1] = ord ? ms_ord : -1.0;
  P.m2l_tuned = (sym && (!ord || ms_sym < ms_ord)) ? 3 : 2;
}

bool m2l_f32_tuned(Plan& P, int Rc, bool steady) {
  const int D = padded_dim(P.d);
  if (D < 0) return false;
  const int RC = padded_rc(Rc);
  const size_t smem = stage_bytes(D, RC, P.n_pad);
  if (smem > 200 * 1024) return false;
  ensure_attrs();
  ensure_scaled(P, D);
  if (P.prec == DWFMM_P_MIXED && RC == 16) {
    const int want = P.m2l_pref >= 0 ? P.m2l_pref : (P.m2l_tuned >= 0 ? P.m2l_tuned : 2);
    if (want == 3 && m2l_sym_tc(P, D, Rc, P.stream)) {
      P.m2l_engine = 3;
      return true;
    }
    if (m2l_ordered_tc(P, D, Rc)) {
      P.m2l_engine = 2;
      return true;
    }
  }
  const int first = (1 << P.jmin) - 1;
  if (P.n_pad <= kSmallNodes && !steady) {
    P.m2l_engine = 1;
    m2l_small(P, D, RC, Rc, first);
    DW_CUDA(cudaGetLastError());
    return true;
  }
  P.momq32.alloc(static_cast<size_t>(P.C) * P.n_pad * kRC);
  const int64_t nq = static_cast<int64_t>(P.C) * P.n_pad * RC;
  k_interleave<<<ceil_div(nq, 256), 256, 0, P.stream>>>(P.mom32.p, P.C, P.n_pad, RC, P.momq32.p);
  P.m2l_engine = 1;
  SumArgs a{};
  a.tgt = P.d_ynodek.p;
  a.tgt_gstride = static_cast<int64_t>(D + 1) * P.n_pad;
  a.src = P.d_ynodek.p;
  a.src_gstride = a.tgt_gstride;
  a.q = P.momq32.p;
  a.q_gstride = static_cast<int64_t>(RC) * P.n_pad;
  a.out = P.loc32.p;
  a.out_gstride = static_cast<int64_t>(kRC) * P.n_pad;
  a.rowptr = P.d_far_rowptr.p;
  a.col = P.d_far_col.p;
  a.count = nullptr;
  a.count_off = 0;
  a.count_const = P.n;
  a.first = a.first_row = first;
  a.ld = P.n_pad;
  a.Rc = Rc;
  a.err = P.d_err.p;
  const int threads = std::min(kThreadsMax, round_up(ceil_div(P.n_pad, kTT), 32));
  dispatch(D, P.kernel, RC, a, P.C - first, threads, smem, P.stream);
  DW_CUDA(cudaGetLastError());
  return true;
}

}  // namespace dw
