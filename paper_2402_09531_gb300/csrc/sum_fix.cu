// Float64 near field and couplings with fixed-point kernel values: the tree's
// records and the launches (kernels in sum_fix.cuh, format in fix64.cuh).
#include <algorithm>
#include <cmath>

#include "sum_fix.cuh"

namespace dw {

namespace {

using namespace fx;

// Records [group][ld][2 * DM] of points [group][d][ld]: limbs of each
// coordinate relative to the root box's lower corner.
__global__ void k_fix_records(const double* pts, int64_t groups, int d, int DM, int ld, const double* lo0, int F,
                              int2* rec) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= groups * ld * DM) return;
  const int k = static_cast<int>(t % DM);
  const int64_t gi = t / DM;
  int2 v = make_int2(0, 0);
  if (k < d) {
    const int i = static_cast<int>(gi % ld);
    const int64_t g = gi / ld;
    const s64 u = static_cast<s64>(to_units(pts[(g * d + k) * ld + i], F) - to_units(lo0[k], F));
    v = make_int2(static_cast<int>(u >> 30), static_cast<int>(u & 0x3fffffff));
  }
  rec[t] = v;
}

// out[g][r][i] = sum over parts of part[p][g][r][i] in part order (r < Rc).
__global__ void k_fix_parts(const double* part, int splits, int64_t stride, int64_t n, int64_t o_gstride, int o_ld,
                            int Rc, double* out) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  if (static_cast<int>((t % o_gstride) / o_ld) >= Rc) return;
  double acc = 0.0;
  for (int p = 0; p < splits; ++p) acc += part[p * stride + t];
  out[t] = acc;
}

int padded_d(int d) { return d <= 4 ? 4 : d <= 8 ? 8 : d <= 10 ? 10 : d <= 12 ? 12 : 16; }
int padded_r(int r) { return r <= 1 ? 1 : r <= 4 ? 4 : 16; }

void dispatch(int kernel, int d, int RC, const FixArgs& a, int ctas, cudaStream_t s) {
  if (ctas <= 0) return;
  if (kernel == DWFMM_K_EXP) launch_fix_exp(d, RC, a, ctas, s);
  else if (kernel == DWFMM_K_MATERN32) launch_fix_matern(d, RC, a, ctas, s);
  else launch_fix_gauss(d, RC, a, ctas, s);
}

void dispatch_sym(int kernel, int d, int RC, const FixSymArgs& a, int chunks, cudaStream_t s) {
  if (kernel == DWFMM_K_EXP) launch_fix_sym_exp(d, RC, a, chunks, s);
  else if (kernel == DWFMM_K_MATERN32) launch_fix_sym_matern(d, RC, a, chunks, s);
  else launch_fix_sym_gauss(d, RC, a, chunks, s);
}

// Passes of tp targets and threads per target for groups of n points: the
// fewest passes that leave the fewest of the 128 threads without a target
// (n = 98: 4 passes of 25 with 5 threads each use 123 of them, one pass 98).
void shape(FixArgs& a, int n) {
  double best = 0.0;
  for (int p = ceil_div(n, fx::kThreads); p <= ceil_div(n, fx::kThreads) + 4; ++p) {
    const int tp = ceil_div(n, p), nsub = fx::kThreads / tp;
    if (nsub > 5 && p > 1) break;
    const double use = static_cast<double>(n) * nsub / (p * fx::kThreads);
    if (use > best * 1.08) {
      best = use;
      a.passes = p;
      a.tp = tp;
      a.nsub = nsub;
    }
  }
}

// Chunks of the upper rows for the symmetric form; false when it does not
// apply: leaves below a warp's width (the lanes of a turn would share a
// target) or above 128 slots (twice the shared memory, half the CTAs of an SM), or a
// list that is not symmetric.  Up to 4 right-hand sides it is the faster form (1: 5.2 against
// 9.8 ms at N = 65536, d = 8; 4: 7.1 against 11.3 ms); 16 would need their
// sums for both sides in registers.
bool sym_ready(Plan& P) {
  if (P.fx_sym >= 0) return P.fx_sym == 1;
  if (capturing(P.stream)) return false;
  P.fx_sym = 0;
  if (P.m_pad > fx::kThreads || P.sym_nup <= 0) return false;
  // a warp takes 64 sources at a time; 8 such batches where that still leaves
  // every SM 32 warps, fewer on small trees
  const int64_t per_sm = P.sym_nup * P.m_pad / 64 / (32 * sm_count());
  P.fx_batches = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(8, per_sm)));
  if (!row_chunks(P, fx::kThreads / 32 * 64 * P.fx_batches, 32, P.fx_rows)) return false;
  P.fx_sym = 1;
  return true;
}

constexpr size_t kSymMaxBytes = size_t(8) << 30;   // partial sums of the symmetric form

}  // namespace

bool fix_ready(Plan& P) {
  if (P.fx_state >= 0) return P.fx_state == 1;
  if (capturing(P.stream)) return false;   // the records are built outside a capture
  P.fx_state = 0;
  if (P.d > fx::kMaxD || P.N == 0) return false;
  double longest = 0.0;
  for (int k = 0; k < P.d; ++k) longest = std::max(longest, P.h_hi0[k] - P.h_lo0[k]);
  // nodes of a cluster with a widened degenerate edge may pass the box by 1e-12 max(1, longest)
  const double guard = 2e-12 * std::max(1.0, longest);
  double d2 = 0.0;
  for (int k = 0; k < P.d; ++k) {
    const double e = P.h_hi0[k] - P.h_lo0[k] + guard;
    d2 += e * e;
  }
  const double diag = std::sqrt(d2) * (1.0 + 1e-6);
  if (!(diag > 1e-150 && diag < 1e150)) return false;
  P.fx_F = fx::units_exponent(diag);
  if (!fx::make_consts(P.kernel, P.sigma, P.fx_F, P.fx_c)) return false;
  const int DM = padded_d(P.d);
  const int64_t nl = static_cast<int64_t>(P.L) * P.m_pad, nc = static_cast<int64_t>(P.C) * P.n_pad;
  try {
    P.fx_pts.alloc(nl * 2 * DM);
    P.fx_nodes.alloc(nc * 2 * DM);
  } catch (const ApiError& e) {   // no memory for the records: the float64 unit, for this tree
    if (e.status != DWFMM_ERR_OOM) throw;
    P.fx_pts.release();
    P.fx_nodes.release();
    return false;
  }
  if (!P.fx_table.p) {
    fx::u64 t[fx::kTable];
    fx::make_table(t);
    P.fx_table.alloc(fx::kTable);
    DW_CUDA(cudaMemcpyAsync(P.fx_table.p, t, sizeof(t), cudaMemcpyHostToDevice, P.stream));
  }
  k_fix_records<<<ceil_div(nl * DM, 256), 256, 0, P.stream>>>(P.d_pts64.p, P.L, P.d, DM, P.m_pad, P.d_lo.p, P.fx_F,
                                                              reinterpret_cast<int2*>(P.fx_pts.p));
  k_fix_records<<<ceil_div(nc * DM, 256), 256, 0, P.stream>>>(P.d_ynode64.p, P.C, P.d, DM, P.n_pad, P.d_lo.p, P.fx_F,
                                                              reinterpret_cast<int2*>(P.fx_nodes.p));
  DW_CUDA(cudaGetLastError());
  (void)sym_ready(P);
  P.fx_state = 1;
  return true;
}

bool near_fix(Plan& P, int Rc, cudaStream_t s) {
  P.near_parts = 0;
  if (P.fx_state != 1) return false;
  const int RC = padded_r(Rc);
  size_t most = 0;   // columns of partial sums
  if (P.fx_sym == 1 && RC <= 4)
    most = kSymMaxBytes / ((static_cast<size_t>(P.fx_rows.n) + P.sym_nup) * P.m_pad * sizeof(double));
  const size_t cols = P.work_cols(Rc, RC, most);
  if (most >= static_cast<size_t>(Rc) && P.grow(P.sym_pf, P.fx_rows.n * cols * P.m_pad) &&
      P.grow(P.sym_pt, P.sym_nup * cols * P.m_pad)) {
    FixSymArgs b{};
    b.rec = reinterpret_cast<const int4*>(P.fx_pts.p);
    b.charge = P.xb64.p;
    b.table = P.fx_table.p;
    b.c = P.fx_c;
    b.count = P.d_count.p + P.L - 1;
    b.chunk_t = P.fx_rows.t.p;
    b.chunk_ptr = P.fx_rows.ptr.p;
    b.uprow = P.sym_uprow.p;
    b.up_s = P.sym_s.p;
    b.ld = P.m_pad;
    b.Rc = Rc;
    b.cmax = P.fx_rows.cmax;
    b.batches = P.fx_batches;
    b.pf = P.sym_pf.p;
    b.pt = P.sym_pt.p;
    dispatch_sym(P.kernel, P.d, RC, b, P.fx_rows.n, s);
    P.near_parts = 1;
    P.near_engine = 1;
    return true;
  }
  P.near_engine = 0;
  FixArgs a{};
  a.rec = reinterpret_cast<const int4*>(P.fx_pts.p);
  a.table = P.fx_table.p;
  a.c = P.fx_c;
  a.rowptr = P.d_near_rowptr.p;
  a.col = P.d_near_col.p;
  a.ld = P.m_pad;
  a.Rc = Rc;
  a.count = P.d_count.p;
  a.count_off = P.L - 1;
  a.charge = P.xb64.p;
  a.q_gstride = static_cast<int64_t>(kRC) * P.m_pad;
  a.o_gstride = a.q_gstride;
  int cmax = 1;
  for (int l = 0; l < P.L; ++l) cmax = std::max(cmax, P.h_count[P.L - 1 + l]);
  shape(a, cmax);
  // few leaves: their lists are cut into parts, so that every SM has CTAs
  const int want = 8 * sm_count();
  a.splits = 1;
  if (P.L * a.passes < want) a.splits = std::min(16, ceil_div(want, P.L * a.passes));
  const int64_t stride = static_cast<int64_t>(P.L) * a.o_gstride;
  if (a.splits > 1 && !P.grow(P.near_parts64, static_cast<size_t>(a.splits) * stride)) a.splits = 1;
  const int ctas = P.L * a.passes * a.splits;
  if (a.splits == 1) {
    a.out = P.ynear64.p;
    dispatch(P.kernel, P.d, RC, a, ctas, s);
  } else {
    a.out = P.near_parts64.p;
    a.split_stride = stride;
    dispatch(P.kernel, P.d, RC, a, ctas, s);
    k_fix_parts<<<ceil_div(stride, 256), 256, 0, s>>>(P.near_parts64.p, a.splits, stride, stride, a.o_gstride, P.m_pad,
                                                      Rc, P.ynear64.p);
  }
  return true;
}

bool m2l_fix(Plan& P, int Rc) {
  if (P.fx_state != 1) return false;
  const int RC = padded_r(Rc);
  const int first = (1 << P.jmin) - 1, groups = P.C - first;
  FixArgs a{};
  a.rec = reinterpret_cast<const int4*>(P.fx_nodes.p);
  a.table = P.fx_table.p;
  a.c = P.fx_c;
  a.rowptr = P.d_far_rowptr.p;
  a.col = P.d_far_col.p;
  a.first = first;
  a.ld = P.n_pad;
  a.Rc = Rc;
  a.count_const = P.n;
  a.charge = P.mom64.p;
  a.q_gstride = static_cast<int64_t>(kRC) * P.n_pad;
  a.o_gstride = a.q_gstride;
  a.out = P.loc64.p;
  a.splits = 1;
  shape(a, P.n);
  // node sets small enough for four threads a target: whole sets per thread
  const int cap = RC > 4 ? 64 : 128;
  if (a.nsub >= 4 && P.n <= 32) a.group_entries = std::max(1, std::min(2 * a.nsub, cap / P.n));
  dispatch(P.kernel, P.d, RC, a, groups * a.passes, P.stream);
  return true;
}

}  // namespace dw
