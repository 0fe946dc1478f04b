// Far-field phases of the DW-FMM matvec (Sec. 5.2, Eq. (5.4) with the
// two-scale relation of the nested cluster bases).
//
// With mu_c = P_c^T x (Legendre moments), m_c = V^{-T} mu_c (charges at the
// nodes a_c(xi_alpha)), l_c = sum_{s in far(c)} S_{c,s} m_s (potentials at
// the nodes) and lambda_c = V^{-1} l_c + T_c lambda_parent (Legendre
// coefficients of the local expansion), the far-field part of y is
// P_leaf lambda_leaf.  With T_c = V^{-1} B_c, B_c[alpha][alpha'] =
// p_hat_alpha'(a_parent^{-1}(a_c(xi_alpha))):
//   P2M:  mu_leaf[b]   = sum_{i in leaf} p_hat_b(a_leaf^{-1} x_i) x_i
//   M2M:  mu_p[b]      = sum_{c child} sum_a p_hat_b(a_p^{-1} y^c_a) m_c[a]
//   L2L:  l_c[a]      += sum_b lambda_p[b] p_hat_b(a_p^{-1} y^c_a)
//   L2P:  y_i          = sum_b lambda_leaf[b] p_hat_b(a_leaf^{-1} x_i)
// P2M and M2M are one kernel (Legendre moments of a box from point charges,
// then V^{-T}); L2L, V^{-1} and (on the leaf level) L2P are one kernel.
#include <algorithm>
#include <atomic>

#include "dwfmm_internal.cuh"
#include "p2p_rot.cuh"
#include "sum_f32.cuh"

namespace dw {

namespace {

constexpr int kFarThreads = 128;
constexpr size_t kFarMaxSmem = 200 * 1024;
constexpr int kAcceptChunk = 32;               // farfield_smem_need: the limit on index sets
constexpr size_t kFarTableBytes = 40 * 1024;   // Legendre tables of a chunk of points

// Stride of a point's Legendre table (odd: consecutive points fall into
// different banks); its last used slot holds 1, the value of a missing factor.
__host__ __device__ constexpr int far_stride(int lsum) { return (lsum + 1) | 1; }

// Points per chunk of tables.
template <typename T>
__host__ __device__ constexpr int far_points(int lsum) {
  const int most = static_cast<int>(kFarTableBytes / sizeof(T)) / far_stride(lsum);
  return most >= kFarThreads ? kFarThreads : most >= 64 ? 64 : 32;
}

// Shared memory of both passes: tables, two arrays of n_pad x RC, the threads'
// partial sums (a chunk's charges in the same place), the multi-indices.  The
// CTAs run beside the near field's, in what those leave of an SM.
template <typename T>
constexpr size_t far_smem(int lsum, int n, int n_pad, int nnz, int RC) {
  const int pc = far_points<T>(lsum);
  return (static_cast<size_t>(pc) * far_stride(lsum) + (2 * static_cast<size_t>(n_pad) + kFarThreads) * RC) *
             sizeof(T) +
         static_cast<size_t>(n) * nnz * sizeof(int16_t);
}

// Order of the sums.  STEADY: one thread a row of results, its terms in order,
// and P_j by its division, then the factor sqrt(2j+1): what the conjugate
// gradient iterations repeat bit for bit (apply_op in solve.cu).  Otherwise
// several threads a row and the recurrence from a table (d = 16, 20 indices,
// float32: 6 levels up 84 us in order, 50 us so).

// p_hat_j(t) = sqrt(2j+1) P_j(2t-1), j = 1 .. deg, into row[j]; not in order: by
// the normalised recurrence p_{j+1} = a_j u p_j - b_j p_{j-1} (a division and a
// root are ~20 instructions each on a float64 unit of 2 a clock).
template <typename T, bool STEADY>
__device__ __forceinline__ void legendre_row(const ExpDev& e, T t, int deg, T* row) {
  const T u = T(2) * t - T(1);
  if constexpr (STEADY) {
    T pm = T(1), pc = u;
    row[1] = u * sqrt(T(3));
    for (int j = 1; j < deg; ++j) {
      const T pn = (T(2 * j + 1) * u * pc - T(j) * pm) / T(j + 1);
      row[j + 1] = pn * sqrt(T(2 * j + 3));
      pm = pc;
      pc = pn;
    }
  } else {
    T prev = T(1), cur = static_cast<T>(e.leg64[0].x) * u;
    row[1] = cur;
    for (int j = 1; j < deg; ++j) {
      const double2 c = e.leg64[j];
      const T next = static_cast<T>(c.x) * u * cur - static_cast<T>(c.y) * prev;
      row[j + 1] = next;
      prev = cur;
      cur = next;
    }
  }
}

// Legendre tables of cn points at t = (y - lo) iext, one point and dimension
// per thread and step.  Only dimensions with a degree above 0 are looked at,
// and degree 0 is not stored (a factor never names it).  point(p): the point's
// first coordinate; ys: between coordinates.
template <typename T, bool STEADY, class F>
__device__ __forceinline__ void fill_tables(const ExpDev& e, int cn, int ys, const T* lo, const T* iext, T* tab,
                                            F point) {
  const int LS = far_stride(e.lsum);
  const int tid = static_cast<int>(threadIdx.x);
  for (int p = tid; p < cn; p += kFarThreads) tab[p * LS + e.lsum] = T(1);
  for (int q = tid; q < cn * e.nact; q += kFarThreads) {
    const int m = q / cn, p = q - m * cn;
    const int k = e.act[m];
    const T t = (point(p)[static_cast<int64_t>(k) * ys] - lo[k]) * iext[k];
    legendre_row<T, STEADY>(e, t, e.qk[k], tab + p * LS + e.loff[k]);
  }
}

// Basis value of the multi-index with factors fac[0..nnz) at a point's table.
template <typename T>
__device__ __forceinline__ T basis_value(const T* tab, const int16_t* fac, int nnz) {
  T v = tab[fac[0]];
  for (int z = 1; z < nnz; ++z) v *= tab[fac[z]];
  return v;
}

// Multi-indices in shared memory, missing factors pointing at the slot of 1.
__device__ __forceinline__ void load_factors(const ExpDev& e, int16_t* fac) {
  for (int i = threadIdx.x; i < e.n * e.nnz_max; i += kFarThreads) {
    const int16_t f = e.fac[i];
    fac[i] = f < 0 ? static_cast<int16_t>(e.lsum) : f;
  }
}

// Threads over `rows` results: one thread a row (in order), or thread (row, sub)
// sums the terms sub, sub + nsub, ..., and `reduce` adds a row's sums; small
// index sets (10 indices are common) leave most of the CTA idle with one thread
// a row.
template <typename T, bool STEADY>
struct Split {
  int per, row, sub, nsub;
  bool on;
  __device__ __forceinline__ explicit Split(int rows) {
    per = rows < kFarThreads ? rows : kFarThreads;
    nsub = STEADY ? 1 : kFarThreads / per;
    sub = static_cast<int>(threadIdx.x) / per;
    row = static_cast<int>(threadIdx.x) - sub * per;
    on = sub < nsub;
  }
};

// dst[a][r] = load(a, r) for a < rows: every load of a thread starts before its
// first store, which the compiler could not move them past (16 right-hand sides
// one load after the other cost 5 us a level; d = 4, N = 12857, 16 right-hand
// sides, float32 downward pass: 109 us, 52 us with all of them in flight).
template <typename T, int RC, class F>
__device__ __forceinline__ void stage(int rows, T* dst, F load) {
  for (int a = threadIdx.x; a < rows; a += kFarThreads) {
    T v[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) v[r] = load(a, r);
#pragma unroll
    for (int r = 0; r < RC; ++r) dst[a * RC + r] = v[r];
  }
}

// put(row, r, value) for every row and right-hand side; red: RC x kFarThreads
// (neighbouring threads in neighbouring banks, and neighbouring rows written
// together).
template <typename T, int RC, class S, class F>
__device__ __forceinline__ void reduce(const S& s, const T (&acc)[RC], T* red, F put) {
  if (s.nsub == 1) {   // the thread's sums are the row's
    if (s.on) {
#pragma unroll
      for (int r = 0; r < RC; ++r) put(s.row, r, acc[r]);
    }
    return;
  }
  __syncthreads();
  if (s.on) {
#pragma unroll
    for (int r = 0; r < RC; ++r) red[r * kFarThreads + threadIdx.x] = acc[r];
  }
  __syncthreads();
  if (s.on)
    for (int r = s.sub; r < RC; r += s.nsub) {
      T v = red[r * kFarThreads + s.row];
      for (int u = 1; u < s.nsub; ++u) v += red[r * kFarThreads + u * s.per + s.row];
      put(s.row, r, v);
    }
}

// Moments of cluster g, then m = V^{-T} mu, for the right-hand sides r0 .. r0 +
// RC - 1 (rows beyond Rc zero).
//  leaf mode:     sources = the leaf's sites, charges = right-hand sides.
//  children mode: sources = nodes of both children, charges = their m.
template <typename T, int RC, bool STEADY>
__device__ __forceinline__ void moments_body(const ExpDev& e, int g, int leaf_mode, int L, const int32_t* count,
                                             const T* pts, int m_pad, const T* xb, const T* ynode,
                                             const T* lo_all, const T* iext_all, const T* vinv, int r0, int Rc, T* mom) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = e.n, np = e.n_pad, d = e.d, nnz = e.nnz_max;
  const int LS = far_stride(e.lsum), PC = far_points<T>(e.lsum);
  T* tab = reinterpret_cast<T*>(smem_raw);     // [PC][LS]
  T* mu = tab + PC * LS;                       // [n_pad][RC]
  T* red = mu + 2 * np * RC;                   // [kFarThreads][RC]
  T* qs = red;                                 // [PC][RC], before the reduction
  int16_t* fac = reinterpret_cast<int16_t*>(red + kFarThreads * RC);
  const T* lo = lo_all + static_cast<int64_t>(g) * d;
  const T* iext = iext_all + static_cast<int64_t>(g) * d;
  const int leaf = g - (L - 1);
  const int S = leaf_mode ? count[g] : 2 * n;
  load_factors(e, fac);
  auto point = [&](int p) -> const T* {
    if (leaf_mode) return pts + static_cast<int64_t>(leaf) * d * m_pad + p;
    const int ch = p >= n ? 1 : 0;
    return ynode + static_cast<int64_t>(2 * g + 1 + ch) * d * np + (p - ch * n);
  };
  auto charge = [&](int p, int r) -> T {
    if (r0 + r >= Rc) return T(0);
    if (leaf_mode) return xb[(static_cast<int64_t>(leaf) * kRC + r0 + r) * m_pad + p];
    const int ch = p >= n ? 1 : 0;
    return mom[(static_cast<int64_t>(2 * g + 1 + ch) * kRC + r0 + r) * np + (p - ch * n)];
  };
  for (int ab = 0; ab < n; ab += kFarThreads) {
    const int rows = min(kFarThreads, n - ab);
    const Split<T, STEADY> s(rows);
    T acc[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = T(0);
    for (int cb = 0; cb < S; cb += PC) {
      const int cn = min(PC, S - cb);
      __syncthreads();
      fill_tables<T, STEADY>(e, cn, leaf_mode ? m_pad : np, lo, iext, tab, [&](int p) { return point(cb + p); });
      stage<T, RC>(cn, qs, [&](int p, int r) { return charge(cb + p, r); });
      __syncthreads();
      if (s.on) {
        const int16_t* f = fac + (ab + s.row) * nnz;
        for (int p = s.sub; p < cn; p += s.nsub) {
          const T b = basis_value<T>(tab + p * LS, f, nnz);
#pragma unroll
          for (int r = 0; r < RC; ++r) acc[r] += b * qs[p * RC + r];
        }
      }
    }
    reduce<T, RC>(s, acc, red, [&](int a, int r, T v) { mu[(ab + a) * RC + r] = v; });
  }
  __syncthreads();
  // m = V^{-T} mu
  for (int ab = 0; ab < n; ab += kFarThreads) {
    const int rows = min(kFarThreads, n - ab);
    const Split<T, STEADY> s(rows);
    T acc[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = T(0);
    if (s.on)
      for (int b = s.sub; b < n; b += s.nsub) {
        const T v = vinv[b * np + ab + s.row];
#pragma unroll
        for (int r = 0; r < RC; ++r) acc[r] += v * mu[b * RC + r];
      }
    reduce<T, RC>(s, acc, red, [&](int a, int r, T v) {
      mom[(static_cast<int64_t>(g) * kRC + r0 + r) * np + ab + a] = r0 + r < Rc ? v : T(0);
    });
  }
  for (int q = threadIdx.x; q < (np - n) * RC; q += kFarThreads)
    mom[(static_cast<int64_t>(g) * kRC + r0 + q / (np - n)) * np + n + q % (np - n)] = T(0);
}

// One cluster per CTA, RC right-hand sides in registers.  Bound by latency (a
// few thousand clocks a level) and, at float64, by the unit's 2 multiply-adds a
// clock: d = 4, N = 4096 float64, 10 indices, 1 right-hand side, 4 levels:
// 164 us with 16 right-hand sides' sums in 10 threads, 34 us with one side's
// in 120.
template <typename T, int RC, bool STEADY>
__global__ void __launch_bounds__(kFarThreads)
k_moments(ExpDev e, int first, int leaf_mode, int L, const int32_t* count, const T* pts, int m_pad,
          const T* xb, const T* ynode, const T* lo_all, const T* iext_all, const T* vinv, int r0, int Rc,
          T* mom) {
  moments_body<T, RC, STEADY>(e, first + blockIdx.x, leaf_mode, L, count, pts, m_pad, xb, ynode, lo_all, iext_all, vinv,
                      r0, Rc, mom);
}

// Downward pass on cluster g of level `level`, right-hand sides r0 .. r0 + RC - 1:
//   l_g += B_g lambda_parent  (if level > jmin), lambda_g = V^{-1} l_g,
//   and on the leaf level y_far = P_leaf lambda_leaf.
// vinvt: the transpose of V^{-1} (consecutive threads read consecutive entries).
template <typename T, int RC, bool STEADY>
__device__ __forceinline__ void downward_body(const ExpDev& e, int g, int level, int jmin, int J, int L,
                                              const int32_t* count, const T* pts, int m_pad, const T* ynode,
                                              const T* lo_all, const T* iext_all, const T* loc, T* lco,
                                              const T* vinvt, int r0, int Rc, T* yfar) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = e.n, np = e.n_pad, d = e.d, nnz = e.nnz_max;
  const int LS = far_stride(e.lsum), PC = far_points<T>(e.lsum);
  T* tab = reinterpret_cast<T*>(smem_raw);     // [PC][LS]
  T* lamp = tab + PC * LS;                     // [n_pad][RC]
  T* lsm = lamp + np * RC;                     // [n_pad][RC]
  T* red = lsm + np * RC;                      // [kFarThreads][RC]
  int16_t* fac = reinterpret_cast<int16_t*>(red + kFarThreads * RC);
  load_factors(e, fac);
  auto of = [&](const T* x, int c) {
    return [=](int a, int r) { return r0 + r < Rc ? x[(static_cast<int64_t>(c) * kRC + r0 + r) * np + a] : T(0); };
  };
  stage<T, RC>(n, lsm, of(loc, g));
  if (level > jmin) {
    const int p = (g - 1) / 2;
    stage<T, RC>(n, lamp, of(lco, p));
    const T* lo = lo_all + static_cast<int64_t>(p) * d;
    const T* iext = iext_all + static_cast<int64_t>(p) * d;
    const T* yn = ynode + static_cast<int64_t>(g) * d * np;
    for (int ab = 0; ab < n; ab += PC) {
      const int rows = min(PC, n - ab);
      __syncthreads();
      fill_tables<T, STEADY>(e, rows, np, lo, iext, tab, [&](int a) { return yn + ab + a; });
      __syncthreads();
      const Split<T, STEADY> s(rows);
      T acc[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) acc[r] = T(0);
      if (s.on)
        for (int b = s.sub; b < n; b += s.nsub) {
          const T v = basis_value<T>(tab + s.row * LS, fac + b * nnz, nnz);
#pragma unroll
          for (int r = 0; r < RC; ++r) acc[r] += v * lamp[b * RC + r];
        }
      reduce<T, RC>(s, acc, red, [&](int a, int r, T v) { lsm[(ab + a) * RC + r] += v; });
    }
  }
  __syncthreads();
  // lambda_g = V^{-1} l_g  (into lamp)
  for (int ab = 0; ab < n; ab += kFarThreads) {
    const int rows = min(kFarThreads, n - ab);
    const Split<T, STEADY> s(rows);
    T acc[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = T(0);
    if (s.on)
      for (int b = s.sub; b < n; b += s.nsub) {
        const T v = vinvt[b * np + ab + s.row];
#pragma unroll
        for (int r = 0; r < RC; ++r) acc[r] += v * lsm[b * RC + r];
      }
    reduce<T, RC>(s, acc, red, [&](int a, int r, T v) {
      lamp[(ab + a) * RC + r] = v;
      if (level < J) lco[(static_cast<int64_t>(g) * kRC + r0 + r) * np + ab + a] = v;
    });
  }
  if (level < J) return;
  // L2P on the leaf's sites
  const int leaf = g - (L - 1);
  const int cnt = count[g];
  const T* lo = lo_all + static_cast<int64_t>(g) * d;
  const T* iext = iext_all + static_cast<int64_t>(g) * d;
  const T* pp = pts + static_cast<int64_t>(leaf) * d * m_pad;
  for (int ib = 0; ib < cnt; ib += PC) {
    const int rows = min(PC, cnt - ib);
    __syncthreads();
    fill_tables<T, STEADY>(e, rows, m_pad, lo, iext, tab, [&](int i) { return pp + ib + i; });
    __syncthreads();
    const Split<T, STEADY> s(rows);
    T acc[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = T(0);
    if (s.on)
      for (int b = s.sub; b < n; b += s.nsub) {
        const T v = basis_value<T>(tab + s.row * LS, fac + b * nnz, nnz);
#pragma unroll
        for (int r = 0; r < RC; ++r) acc[r] += v * lamp[b * RC + r];
      }
    reduce<T, RC>(s, acc, red, [&](int i, int r, T v) {
      if (r0 + r < Rc) yfar[(static_cast<int64_t>(leaf) * kRC + r0 + r) * m_pad + ib + i] = v;
    });
  }
}

template <typename T, int RC, bool STEADY>
__global__ void __launch_bounds__(kFarThreads)
k_downward(ExpDev e, int first, int level, int jmin, int J, int L, const int32_t* count,
           const T* pts, int m_pad, const T* ynode, const T* lo_all, const T* iext_all,
           const T* loc, T* lco, const T* vinvt, int r0, int Rc, T* yfar) {
  downward_body<T, RC, STEADY>(e, first + blockIdx.x, level, jmin, J, L, count, pts, m_pad, ynode, lo_all, iext_all, loc,
                       lco, vinvt, r0, Rc, yfar);
}

// ---- many problems in one launch (batches) --------------------------------
// Work item = (problem, cluster); every problem's arrays come from its entry
// of the problem table.

__device__ __forceinline__ int level_of(int g) { return 31 - __clz(g + 1); }

// Up to 4 right-hand sides in registers, or up to 16.
template <bool STEADY>
__device__ __forceinline__ void moments_item(const ProbF32& p, int c) {
  const int leaf = level_of(c) == p.J;
  if (p.R <= 4)
    moments_body<float, 4, STEADY>(p.e, c, leaf, p.L, p.count, p.pts, p.m_pad, p.xb, p.ynode, p.lo, p.iext, p.vinv, 0, p.R,
                           p.mom);
  else
    moments_body<float, 16, STEADY>(p.e, c, leaf, p.L, p.count, p.pts, p.m_pad, p.xb, p.ynode, p.lo, p.iext, p.vinv, 0, p.R,
                            p.mom);
}

template <bool STEADY>
__device__ __forceinline__ void downward_item(const ProbF32& p, int c) {
  if (p.R <= 4)
    downward_body<float, 4, STEADY>(p.e, c, level_of(c), p.jmin, p.J, p.L, p.count, p.pts, p.m_pad, p.ynode, p.lo, p.iext,
                            p.loc, p.lco, p.vinvt, 0, p.R, p.yfar);
  else
    downward_body<float, 16, STEADY>(p.e, c, level_of(c), p.jmin, p.J, p.L, p.count, p.pts, p.m_pad, p.ynode, p.lo, p.iext,
                             p.loc, p.lco, p.vinvt, 0, p.R, p.yfar);
}

template <bool STEADY>
__global__ void __launch_bounds__(kFarThreads)
k_moments_batched(const ProbF32* probs, const int2* work) {
  const int2 w = work[blockIdx.x];
  moments_item<STEADY>(probs[w.x], w.y);
}

template <bool STEADY>
__global__ void __launch_bounds__(kFarThreads)
k_downward_batched(const ProbF32* probs, const int2* work) {
  const int2 w = work[blockIdx.x];
  downward_item<STEADY>(probs[w.x], w.y);
}

// Problem of a global leaf (binary search in the leaf offsets).
__device__ __forceinline__ int problem_of(const int* leaf_off, int P, int gl) {
  int lo = 0, hi = P - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (leaf_off[mid] <= gl) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Element t of the gathered right-hand sides xb[leaf][r][ld] (t < Ltot * 16 * ld).
__device__ __forceinline__ void gather_elem(const ProbF32* probs, const int* leaf_off, int P, int ld, float* xb,
                                            int64_t t) {
  const int i = static_cast<int>(t % ld);
  const int64_t lr = t / ld;
  const int r = static_cast<int>(lr % kRC);
  const int gl = static_cast<int>(lr / kRC);
  const int pi = problem_of(leaf_off, P, gl);
  const ProbF32& p = probs[pi];
  const int c = p.L - 1 + (gl - leaf_off[pi]);
  float v = 0.0f;
  if (r < p.R && i < p.count[c]) v = static_cast<float>(p.x[static_cast<int64_t>(r) * p.ldx + p.perm[p.begin[c] + i]]);
  xb[t] = v;
}

__global__ void k_gather_batched(const ProbF32* probs, const int* leaf_off, int P, int Ltot, int ld, float* xb) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= static_cast<int64_t>(Ltot) * kRC * ld) return;
  gather_elem(probs, leaf_off, P, ld, xb, t);
}

// Running sum: float32 values with compensation (the float64 unit is too
// narrow for a conversion and an addition per value), float64 values plainly.
template <typename T>
struct Running;
template <>
struct Running<float> {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float y = v - c, t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return static_cast<double>(s) - static_cast<double>(c); }
};
template <>
struct Running<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double value() const { return s; }
};

// Part p of np of the near-field sums of one site: every np-th chunk sum of its
// leaf's row (c0 .. c1 - 1) and a range of the transposed sums of its nlo lower
// entries, `at` + index * step each.  Loads go out eight at a time.
template <typename T>
__device__ __forceinline__ double near_part(const T* pf, int c0, int c1, const T* pt, const int32_t* lo_slot, int nlo,
                                            int e_base, int64_t at, int64_t step, int p, int np) {
  Running<T> acc;
  for (int e = c0 + p; e < c1; e += 4 * np) {
    T w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = e + u * np < c1 ? pf[(e + u * np) * step + at] : T(0);
#pragma unroll
    for (int u = 0; u < 4; ++u) acc.add(w[u]);
  }
  int k = static_cast<int>((static_cast<int64_t>(nlo) * p) / np);
  const int ke = static_cast<int>((static_cast<int64_t>(nlo) * (p + 1)) / np);
  for (; k < ke; k += 8) {
    T w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = k + u < ke ? pt[(lo_slot[k + u] - e_base) * step + at] : T(0);
#pragma unroll
    for (int u = 0; u < 8; ++u) acc.add(w[u]);
  }
  return acc.value();
}

constexpr int kPartThreads = 512;

// y = near + far of right-hand side r of global leaf gl, written to the
// caller's order, by `threads` threads (a divisor of kPartThreads; the parts of
// the near-field sums are those of kPartThreads threads whatever it is, so the
// result does not depend on it).  part: kPartThreads doubles of shared memory
// when threads = kPartThreads.
template <int THREADS>
__device__ __forceinline__ void scatter_row(const ProbF32& p, int lo_leaf, int gl, int r, int ld,
                                            const BatchParts& bp, const float* ynear, const float* yfar, double* part) {
  const int leaf = gl - lo_leaf;
  const int c = p.L - 1 + leaf;
  const int cnt = p.count[c];
  const int np = kPartThreads / ld;
  const int tid = static_cast<int>(threadIdx.x);
  const int64_t at = static_cast<int64_t>(r) * ld, step = static_cast<int64_t>(p.rc) * ld;
  int c0 = 0, c1 = 0, k0 = 0, nlo = 0;
  if (p.pf) {
    c0 = bp.chunk_ptr[gl] - p.chunk0;
    c1 = bp.chunk_ptr[gl + 1] - p.chunk0;
    k0 = bp.lorow[gl];
    nlo = bp.lorow[gl + 1] - k0;
  }
  auto near = [&](int q, int i) {
    return near_part<float>(p.pf, c0, c1, p.pt, bp.lo_slot + k0, nlo, p.e_base, at + i, step, q, np);
  };
  auto put = [&](int i, double v) {
    const int64_t t = (static_cast<int64_t>(gl) * kRC + r) * ld + i;
    if (!p.pf) v = static_cast<double>(ynear[t]);
    if (p.jmin <= p.J) v += static_cast<double>(yfar[t]);
    p.y[static_cast<int64_t>(r) * p.ldy + p.perm[p.begin[c] + i]] = v;
  };
  if constexpr (THREADS == kPartThreads) {
    const int q = tid / ld, i = tid - q * ld;
    double v = 0.0;
    if (p.pf && q < np && i < cnt) v = near(q, i);
    part[tid] = v;
    __syncthreads();
    if (tid < cnt) {
      for (int u = 1; u < np; ++u) v += part[u * ld + tid];
      put(tid, v);
    }
  } else {
    for (int i = tid; i < cnt; i += THREADS) {
      double v = 0.0;
      if (p.pf) {
        v = near(0, i);
        for (int u = 1; u < np; ++u) v += near(u, i);
      }
      put(i, v);
    }
  }
}

__global__ void __launch_bounds__(kPartThreads)
k_scatter_batched(const ProbF32* probs, const int* leaf_off, int P, int Rmax, int ld, BatchParts bp, const float* ynear,
                  const float* yfar) {
  __shared__ double part[kPartThreads];
  const int gl = static_cast<int>(blockIdx.x) / Rmax, r = static_cast<int>(blockIdx.x) % Rmax;
  const int pi = problem_of(leaf_off, P, gl);
  const ProbF32& p = probs[pi];
  if (r >= p.R) return;
  scatter_row<kPartThreads>(p, leaf_off[pi], gl, r, ld, bp, ynear, yfar, part);
}

// A batch without such sums, or with leaves too wide for kPartThreads: one
// thread per element (t < Ltot * 16 * ld).
__global__ void k_scatter_rows(const ProbF32* probs, const int* leaf_off, int P, int Ltot, int ld, const float* ynear,
                               const float* yfar) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= static_cast<int64_t>(Ltot) * kRC * ld) return;
  const int i = static_cast<int>(t % ld);
  const int64_t lr = t / ld;
  const int r = static_cast<int>(lr % kRC);
  const int gl = static_cast<int>(lr / kRC);
  const int pi = problem_of(leaf_off, P, gl);
  const ProbF32& p = probs[pi];
  const int c = p.L - 1 + (gl - leaf_off[pi]);
  if (r >= p.R || i >= p.count[c]) return;
  double v = static_cast<double>(ynear[t]);
  if (p.jmin <= p.J) v += static_cast<double>(yfar[t]);
  p.y[static_cast<int64_t>(r) * p.ldy + p.perm[p.begin[c] + i]] = v;
}

// ---------------------------------------------------------------------------
// Persistent batch matvec: the whole fused matvec of a batch as one
// cooperative launch (every CTA resident at once).  Phases, each ended by a
// grid-wide barrier (one arrival counter per phase, bounded wait):
//   gather | interleave of the near-field charges, P2M of the leaves |
//   M2M, one phase per height | interleave of the moments | the couplings
//   (M2L, work queue) | L2L and L2P, one phase per level | the rest of the
//   near field | scatter.
// The near field (P2P) needs only the gathered charges, so from the second
// barrier on a CTA that has done its share of a far-field phase takes
// near-field target groups from a work queue while it waits for the others:
// the short phases of the coarse levels no longer leave SMs idle, and all
// right-hand-side classes share one queue (no tail per class).  Near-field
// and coupling target groups run on groups of gs threads (several per CTA:
// the tuned width), each group with its own stages and stage barriers,
// taking items on its own until its queue is empty or its barrier completes;
// the summation order inside a target group is that of k_sum_f32, so the
// result equals the launch-per-phase matvec bit for bit.
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A barrier waits at most this long with nothing to do (every CTA is
// resident, so the others only have their share of one phase left).
constexpr uint64_t kPersistWaitNs = 4000000000ull;

template <int D, int KER>
__device__ __forceinline__ bool persist_sum_item(const PersistSeg* segs, int nseg, int idx, const sk::Grp& G,
                                                 unsigned char* sm, uint64_t* full, int& tiles) {
  int s = 0;
  while (s + 1 < nseg && idx >= segs[s].count) {
    idx -= segs[s].count;
    ++s;
  }
  const PersistSeg& sg = segs[s];
  if (sg.by_pair) {   // the whole CTA is the group
    float* rsm = reinterpret_cast<float*>(sm);
    if (sg.rc <= 1) rot::rot_chunk<D, 1, KER>(sg.r, idx, rsm);
    else if (sg.rc <= 4) rot::rot_chunk<D, 4, KER>(sg.r, idx, rsm);
    else rot::rot_chunk<D, 8, KER>(sg.r, idx, rsm);
    return true;
  }
  const int g = sg.a.first + idx;
  const int rb = sg.a.rowptr[g], re = sg.a.rowptr[g + 1];
  float* out = sg.a.out + g * sg.a.out_gstride;
  switch (sg.rc) {
    case 1: return sk::sum_block<D, 1, KER>(sg.a, g, rb, re, out, G, sm, full, tiles);
    case 4: return sk::sum_block<D, 4, KER>(sg.a, g, rb, re, out, G, sm, full, tiles);
    case 8: return sk::sum_block<D, 8, KER>(sg.a, g, rb, re, out, G, sm, full, tiles);
    default: return sk::sum_block<D, 16, KER>(sg.a, g, rb, re, out, G, sm, full, tiles);
  }
}

// Shared state of a persistent CTA: stage barriers and completed-stage counts
// of up to four groups, the item each group took, a broadcast word.
struct PShared {
  uint64_t full[kPersistThreads / 32][2];
  int tiles[kPersistThreads / 32];
  int item[kPersistThreads / 32];
  int flag;
};

// Summation items from a queue (head `head`, `total` items): every group of
// gs threads takes target groups one at a time and sums them, on its own,
// until the queue is empty or, if `stop` is given, the barrier counter *stop
// has reached gridDim.x (checked by the group's first thread between items).
// 0: the queue is empty; 1: stopped by the barrier; -1: a copy wait gave up
// (error flag set).
template <int D, int KER>
__device__ __noinline__ int persist_drain(const PersistSeg* segs, int nseg, int total, unsigned* head, int gs,
                                          int gbytes, unsigned char* smem, PShared& sh, const unsigned* stop) {
  const int gid = static_cast<int>(threadIdx.x) / gs;
  const sk::Grp G{static_cast<int>(threadIdx.x) % gs, gs, 1 + gid};
  unsigned char* gsm = smem + static_cast<size_t>(gid) * gbytes;
  int tiles = sh.tiles[gid];
  bool ok = true, empty = false;
  for (;;) {
    if (G.tid == 0) {
      int it = -1;   // -1: the barrier is complete
      if (!stop || ld_acquire_gpu(stop) < gridDim.x) it = static_cast<int>(atomicAdd(head, 1u));
      sh.item[gid] = it;
    }
    sk::grp_sync(G);
    const int it = sh.item[gid];
    sk::grp_sync(G);   // read by every thread before the next item overwrites it
    if (it < 0) break;
    if (it >= total) {
      empty = true;
      break;
    }
    if (!persist_sum_item<D, KER>(segs, nseg, it, G, gsm, sh.full[gid], tiles)) {
      ok = false;
      break;
    }
  }
  if (G.tid == 0) sh.tiles[gid] = tiles;
  const int bad = __syncthreads_or(!ok);
  const int emp = __syncthreads_or(empty);
  return bad ? -1 : (emp ? 0 : 1);
}

// Arrive at barrier `ph` and wait until every CTA has; meanwhile, if `near`,
// the CTA's groups take near-field items from their queue until the barrier
// completes or the queue is empty.  False when the wait gave up (error flag
// 4) or a copy wait did.
template <int D, int KER>
__device__ __noinline__ bool persist_barrier(const PersistArgs& pa, int ph, bool near, bool& near_left, unsigned char* smem,
                                PShared& sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(pa.sync + ph, 1u);
  }
  uint64_t t0 = threadIdx.x == 0 ? global_ns() : 0;
  for (;;) {
    if (threadIdx.x == 0) {
      const bool all = ld_acquire_gpu(pa.sync + ph) >= gridDim.x;
      sh.flag = all ? 1 : (global_ns() - t0 > kPersistWaitNs ? 2 : 0);
    }
    __syncthreads();
    const int f = sh.flag;
    __syncthreads();
    if (f == 1) break;
    if (f == 2) {
      if (threadIdx.x == 0) atomicExch(pa.err, 4);
      return false;
    }
    if (near && near_left) {
      const int r = persist_drain<D, KER>(pa.near, pa.nnear, pa.near_total, pa.sync + kPersistSync - 2,
                                          pa.gs_near, pa.near_group_bytes, smem, sh, pa.sync + ph);
      if (r < 0) return false;
      if (r == 0) near_left = false;
      if (threadIdx.x == 0) t0 = global_ns();
      continue;
    }
    if (threadIdx.x == 0) __nanosleep(256);
  }
  // the other CTAs' writes are now visible; order them before this CTA's
  // bulk copies (async proxy) as well
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncthreads();
  return true;
}

__device__ __forceinline__ void persist_up_items(const PersistArgs& pa, int h) {
  for (int i = static_cast<int>(blockIdx.x); i < pa.up_cnt[h]; i += static_cast<int>(gridDim.x)) {
    const int2 w = pa.work[pa.up_off[h] + i];
    moments_item<false>(pa.probs[w.x], w.y);
    __syncthreads();
  }
}

__device__ __forceinline__ void persist_down_items(const PersistArgs& pa, int j) {
  for (int i = static_cast<int>(blockIdx.x); i < pa.down_cnt[j]; i += static_cast<int>(gridDim.x)) {
    const int2 w = pa.work[pa.down_off[j] + i];
    downward_item<false>(pa.probs[w.x], w.y);
    __syncthreads();
  }
}

__device__ __forceinline__ void persist_interleave(const PersistSeg* segs, int nseg, int64_t t0, int64_t stride) {
  for (int s = 0; s < nseg; ++s) {
    const PersistSeg& sg = segs[s];
    const int ld = sg.a.ld;
    const int64_t n = static_cast<int64_t>(sg.groups) * ld * sg.rc;
    const float* src = sg.ilv_src + static_cast<int64_t>(sg.a.first) * kRC * ld;
    float* dst = const_cast<float*>(sg.a.q) + static_cast<int64_t>(sg.a.first) * sg.rc * ld;
    for (int64_t t = t0; t < n; t += stride) sk::interleave_elem(src, ld, sg.rc, dst, t);
  }
}

template <int D, int KER>
__global__ void __launch_bounds__(kPersistThreads, 3) k_batch_persistent(const __grid_constant__ PersistArgs pa) {
  extern __shared__ __align__(128) unsigned char psm[];
  __shared__ PShared sh;
  if (threadIdx.x == 0) {
    for (int k = 0; k < kPersistThreads / 32; ++k) {
      sk::mbar_init(&sh.full[k][0], 1);
      sk::mbar_init(&sh.full[k][1], 1);
      sh.tiles[k] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  int ph = 0;
  bool near_left = pa.near_total > 0;
  // gather
  const int64_t nel = static_cast<int64_t>(pa.Ltot) * kRC * pa.ld;
  if (pa.io)
    for (int64_t t = t0; t < nel; t += stride) gather_elem(pa.probs, pa.leaf_off, pa.P, pa.ld, pa.xb, t);
  if (!persist_barrier<D, KER>(pa, ph++, false, near_left, psm, sh)) return;
  // near-field charges; P2M of the leaves
  persist_interleave(pa.near, pa.nnear, t0, stride);
  if (pa.nup > 0) persist_up_items(pa, 0);
  if (!persist_barrier<D, KER>(pa, ph++, false, near_left, psm, sh)) return;
  // M2M by height
  for (int h = 1; h < pa.nup; ++h) {
    persist_up_items(pa, h);
    if (!persist_barrier<D, KER>(pa, ph++, true, near_left, psm, sh)) return;
  }
  // M2L
  if (pa.m2l_total > 0) {
    persist_interleave(pa.m2l, pa.nm2l, t0, stride);
    if (!persist_barrier<D, KER>(pa, ph++, true, near_left, psm, sh)) return;
    if (persist_drain<D, KER>(pa.m2l, pa.nm2l, pa.m2l_total, pa.sync + kPersistSync - 1, pa.gs_m2l,
                              pa.m2l_group_bytes, psm, sh, nullptr) < 0)
      return;
    if (!persist_barrier<D, KER>(pa, ph++, true, near_left, psm, sh)) return;
  }
  // L2L / L2P by level
  for (int j = 0; j < pa.ndown; ++j) {
    persist_down_items(pa, j);
    if (!persist_barrier<D, KER>(pa, ph++, true, near_left, psm, sh)) return;
  }
  // the rest of the near field
  if (near_left && persist_drain<D, KER>(pa.near, pa.nnear, pa.near_total, pa.sync + kPersistSync - 2, pa.gs_near,
                                          pa.near_group_bytes, psm, sh, nullptr) < 0)
    return;
  if (!persist_barrier<D, KER>(pa, ph++, false, near_left, psm, sh)) return;
  if (!pa.io) return;
  for (int gl = static_cast<int>(blockIdx.x); gl < pa.Ltot; gl += static_cast<int>(gridDim.x)) {
    const int pi = problem_of(pa.leaf_off, pa.P, gl);
    const ProbF32& p = pa.probs[pi];
    for (int r = 0; r < p.R; ++r)
      scatter_row<kPersistThreads>(p, pa.leaf_off[pi], gl, r, pa.ld, pa.parts, pa.ynear, pa.yfar, nullptr);
  }
}

// x (caller order, column-major) -> xb[leaf][r][m_pad] for the columns
// [r0, r0 + Rc), rows up to `rows` (the rest of them zero); xq, if given: the
// same values interleaved, [leaf][m_pad][rows].
template <typename T>
__global__ void k_gather(const double* x, int64_t ldx, int r0, int Rc, int rows, const int32_t* perm,
                         const int32_t* begin, const int32_t* count, int L, int m_pad, T* xb, T* xq) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t total = static_cast<int64_t>(L) * rows * m_pad;
  if (t >= total) return;
  const int i = static_cast<int>(t % m_pad);
  const int64_t lr = t / m_pad;
  const int r = static_cast<int>(lr % rows);
  const int leaf = static_cast<int>(lr / rows);
  const int c = L - 1 + leaf;
  T v = T(0);
  if (r < Rc && i < count[c]) v = static_cast<T>(x[static_cast<int64_t>(r0 + r) * ldx + perm[begin[c] + i]]);
  xb[(static_cast<int64_t>(leaf) * kRC + r) * m_pad + i] = v;
  if (xq) xq[(static_cast<int64_t>(leaf) * m_pad + i) * rows + r] = v;
}

// Scatter of the symmetric near fields: y = the row's chunk sums and the
// transposed sums of its lower entries, plus the far field.  One CTA per leaf
// and right-hand side; its threads' groups of m_pad take parts of both lists
// (added in order), so that a short tree still has enough loads in flight: the
// reads are rows of m_pad values all over the entries.  d = 8, N = 100003, 4
// right-hand sides: 220 us with one thread per value and float64 additions.
template <typename T>
__global__ void __launch_bounds__(kPartThreads)
k_scatter_parts(double* y, int64_t ldy, int r0, int Rc, const int32_t* perm, const int32_t* begin,
                const int32_t* count, int L, int m_pad, int ldp, const int32_t* chunk_ptr, const int32_t* lorow,
                const int32_t* lo_slot, const T* pf, const T* pt, const T* yfar, int has_far) {
  __shared__ double part[kPartThreads];
  const int tid = static_cast<int>(threadIdx.x);
  const int leaf = static_cast<int>(blockIdx.x) / Rc, r = static_cast<int>(blockIdx.x) % Rc;
  const int c = L - 1 + leaf;
  const int cnt = count[c];
  const int np = kPartThreads / ldp;
  const int p = tid / ldp, i = tid - p * ldp;
  const int k0 = lorow[leaf];
  double v = 0.0;
  if (p < np && i < cnt)
    v = near_part<T>(pf, chunk_ptr[leaf], chunk_ptr[leaf + 1], pt, lo_slot + k0, lorow[leaf + 1] - k0, 0,
                     static_cast<int64_t>(r) * ldp + i, static_cast<int64_t>(Rc) * ldp, p, np);
  part[tid] = v;
  __syncthreads();
  if (tid >= cnt) return;
  for (int u = 1; u < np; ++u) v += part[u * ldp + tid];
  if (has_far) v += static_cast<double>(yfar[(static_cast<int64_t>(leaf) * kRC + r) * m_pad + tid]);
  y[static_cast<int64_t>(r0 + r) * ldy + perm[begin[c] + tid]] = v;
}

template <typename T>
__global__ void k_scatter(double* y, int64_t ldy, int r0, int Rc, const int32_t* perm,
                          const int32_t* begin, const int32_t* count, int L, int m_pad,
                          const T* ynear, const T* yfar, int has_far) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t total = static_cast<int64_t>(L) * Rc * m_pad;
  if (t >= total) return;
  const int i = static_cast<int>(t % m_pad);
  const int64_t lr = t / m_pad;
  const int r = static_cast<int>(lr % Rc);
  const int leaf = static_cast<int>(lr / Rc);
  const int c = L - 1 + leaf;
  if (i >= count[c]) return;
  const int64_t o = (static_cast<int64_t>(leaf) * kRC + r) * m_pad + i;
  double v = static_cast<double>(ynear[o]);
  if (has_far) v += static_cast<double>(yfar[o]);
  y[static_cast<int64_t>(r0 + r) * ldy + perm[begin[c] + i]] = v;
}

template <typename T>
struct Bufs {
  T *xb, *ynear, *yfar, *mom, *loc, *lco;
  const T *pts, *ynode, *lo, *iext, *vinv, *vinvt;
};

template <typename T>
Bufs<T> bufs(Plan& P);

template <>
Bufs<double> bufs<double>(Plan& P) {
  return Bufs<double>{P.xb64.p,   P.ynear64.p, P.yfar64.p,  P.mom64.p,  P.loc64.p, P.lco64.p,
                      P.d_pts64.p, P.d_ynode64.p, P.d_lo.p, P.d_iext.p, P.d_vinv.p, P.d_vinvt.p};
}
template <>
Bufs<float> bufs<float>(Plan& P) {
  return Bufs<float>{P.xb32.p,   P.ynear32.p, P.yfar32.p,  P.mom32.p,   P.loc32.p,  P.lco32.p,
                     P.d_pts32.p, P.d_ynode32.p, P.d_lo32.p, P.d_iext32.p, P.d_vinv32.p, P.d_vinvt32.p};
}

// Upward passes (levels J .. jmin) or downward passes (jmin .. J).
template <typename T, int RC, bool STEADY>
int far_levels(Plan& P, bool up, int Rc) {
  cudaStream_t s = P.stream;
  const Bufs<T> B = bufs<T>(P);
  const ExpDev e = P.exp_dev();
  const int J = P.J, L = P.L;
  const size_t smem = far_smem<T>(e.lsum, e.n, e.n_pad, e.nnz_max, RC);
  static std::atomic<uint64_t> done{0};
  const uint64_t bit = device_bit();
  if (!(done.load() & bit)) {   // large index sets
    DW_CUDA(cudaFuncSetAttribute(k_moments<T, RC, STEADY>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFarMaxSmem));
    DW_CUDA(cudaFuncSetAttribute(k_downward<T, RC, STEADY>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFarMaxSmem));
    done.fetch_or(bit);
  }
  int launches = 0;
  for (int i = 0; i <= J - P.jmin; ++i) {
    const int j = up ? J - i : P.jmin + i;
    const int first = (1 << j) - 1;
    for (int r0 = 0; r0 < Rc; r0 += RC, ++launches) {
      if (up)
        k_moments<T, RC, STEADY><<<1 << j, kFarThreads, smem, s>>>(e, first, j == J, L, P.d_count.p, B.pts, P.m_pad, B.xb,
                                                           B.ynode, B.lo, B.iext, B.vinv, r0, Rc, B.mom);
      else
        k_downward<T, RC, STEADY><<<1 << j, kFarThreads, smem, s>>>(e, first, j, P.jmin, J, L, P.d_count.p, B.pts, P.m_pad,
                                                            B.ynode, B.lo, B.iext, B.loc, B.lco, B.vinvt, r0, Rc,
                                                            B.yfar);
    }
  }
  return launches;
}

// The right-hand sides a thread keeps: the padded count, or fewer at a time
// where an index set of hundreds of entries needs the shared memory.
template <typename T, bool STEADY>
int far_levels_rc(Plan& P, bool up, int Rc) {
  auto fits = [&](int RC) { return far_smem<T>(P.lsum, P.n, P.n_pad, P.nnz_max, RC) <= kFarMaxSmem; };
  if (Rc > 8 && fits(16)) return far_levels<T, 16, STEADY>(P, up, Rc);
  if (Rc > 4 && fits(8)) return far_levels<T, 8, STEADY>(P, up, Rc);
  if (Rc > 1 && fits(4)) return far_levels<T, 4, STEADY>(P, up, Rc);
  return far_levels<T, 1, STEADY>(P, up, Rc);
}

template <typename T>
int far_pass(Plan& P, bool up, int Rc, bool steady) {
  if (steady) return far_levels_rc<T, true>(P, up, Rc);
  return far_levels_rc<T, false>(P, up, Rc);
}

template <typename T>
void farfield_impl(Plan& P, int Rc, bool steady) {
  if (P.jmin > P.J) {  // no admissible block: the far field is empty (the scatter does not read it)
    P.far_engine = sizeof(T) == 8 ? 0 : 1;
    return;
  }
  cudaStream_t s = P.stream;
  // one or two right-hand sides leave the tensor tile of 16 columns empty: the
  // CUDA cores take half as many launches, with work that fits the sides given
  // (d = 16, 20 indices, N = 50021, 7 levels up and down: 375 us on the tensor
  // cores; the error against float64 is 0.3 to 0.6 times as large, too)
  if (sizeof(T) == 4 && (Rc > 2 || steady) && farfield_tc_eligible(P)) {
    P.far_engine = 2;
    farfield_tc(P, Rc, steady);
    return;
  }
  P.far_engine = sizeof(T) == 8 ? 0 : 1;
  timer_begin(P, 1, s);
  int launches = far_pass<T>(P, true, Rc, steady);
  timer_end(P, 1, s, launches);
  timer_begin(P, 2, s);
  launch_m2l(P, Rc, sizeof(T) == 8, steady);
  timer_end(P, 2, s, 1);
  timer_begin(P, 3, s);
  launches = far_pass<T>(P, false, Rc, steady);
  timer_end(P, 3, s, launches);
  DW_CUDA(cudaGetLastError());
}

}  // namespace

size_t farfield_smem_need(const Plan& P, bool fp64) {
  const size_t es = fp64 ? 8 : 4;
  const size_t a = (static_cast<size_t>(kAcceptChunk) * P.lsum + kAcceptChunk * kRC + static_cast<size_t>(P.n_pad) * kRC) * es;
  const size_t b = (2 * static_cast<size_t>(P.n_pad) * kRC + static_cast<size_t>(kFarThreads) * P.lsum) * es;
  return std::max(a, b);
}

void launch_gather(Plan& P, const double* x, int64_t ldx, int r0, int Rc, bool fp64, float* xq) {
  const int rows = fp64 ? Rc : sum_padded_rc(Rc);
  const int64_t total = static_cast<int64_t>(P.L) * rows * P.m_pad;
  if (fp64)
    k_gather<double><<<ceil_div(total, 256), 256, 0, P.stream>>>(x, ldx, r0, Rc, rows, P.d_perm.p, P.d_begin.p,
                                                                 P.d_count.p, P.L, P.m_pad, P.xb64.p, nullptr);
  else
    k_gather<float><<<ceil_div(total, 256), 256, 0, P.stream>>>(x, ldx, r0, Rc, rows, P.d_perm.p, P.d_begin.p,
                                                                P.d_count.p, P.L, P.m_pad, P.xb32.p, xq);
  DW_CUDA(cudaGetLastError());
}

void launch_scatter(Plan& P, double* y, int64_t ldy, int r0, int Rc, bool fp64) {
  const int64_t total = static_cast<int64_t>(P.L) * Rc * P.m_pad;
  const int has_far = P.jmin <= P.J;
  const int grid = ceil_div(total, 256);
  if (P.near_parts == 1)
    k_scatter_parts<double><<<P.L * Rc, kPartThreads, 0, P.stream>>>(
        y, ldy, r0, Rc, P.d_perm.p, P.d_begin.p, P.d_count.p, P.L, P.m_pad, P.m_pad, P.fx_rows.ptr.p, P.sym_lorow.p,
        P.sym_loslot.p, P.sym_pf.p, P.sym_pt.p, P.yfar64.p, has_far);
  else if (P.near_parts == 2)
    k_scatter_parts<float><<<P.L * Rc, kPartThreads, 0, P.stream>>>(
        y, ldy, r0, Rc, P.d_perm.p, P.d_begin.p, P.d_count.p, P.L, P.m_pad, round_up(P.rot.cmax, 8), P.rot.ptr.p, P.sym_lorow.p,
        P.sym_loslot.p, P.rot_pf.p, P.rot_pt.p, P.yfar32.p, has_far);
  else if (fp64)
    k_scatter<double><<<grid, 256, 0, P.stream>>>(y, ldy, r0, Rc, P.d_perm.p, P.d_begin.p, P.d_count.p, P.L, P.m_pad,
                                                  P.ynear64.p, P.yfar64.p, has_far);
  else
    k_scatter<float><<<grid, 256, 0, P.stream>>>(y, ldy, r0, Rc, P.d_perm.p, P.d_begin.p, P.d_count.p, P.L, P.m_pad,
                                                 P.ynear32.p, P.yfar32.p, has_far);
  DW_CUDA(cudaGetLastError());
}

void batch_far_attrs() {
  const int big = 200 * 1024;
  DW_CUDA(cudaFuncSetAttribute(k_moments_batched<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  DW_CUDA(cudaFuncSetAttribute(k_downward_batched<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  DW_CUDA(cudaFuncSetAttribute(k_moments_batched<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  DW_CUDA(cudaFuncSetAttribute(k_downward_batched<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
}

// One problem's shared memory in the batched passes (moments_item, downward_item).
size_t batch_far_smem(int lsum, int n, int n_pad, int nnz, int R) {
  return far_smem<float>(lsum, n, n_pad, nnz, R <= 4 ? 4 : 16);
}

size_t batch_far_need(int lsum, int n_pad) {
  const size_t a = (static_cast<size_t>(kAcceptChunk) * lsum + kAcceptChunk * kRC + static_cast<size_t>(n_pad) * kRC) * 4;
  const size_t b = (2 * static_cast<size_t>(n_pad) * kRC + static_cast<size_t>(kFarThreads) * lsum) * 4;
  return std::max(a, b);
}

void launch_moments_batched(const ProbF32* probs, const int2* work, int items, size_t smem, bool steady, cudaStream_t s) {
  if (items <= 0) return;
  if (steady) k_moments_batched<true><<<items, kFarThreads, smem, s>>>(probs, work);
  else k_moments_batched<false><<<items, kFarThreads, smem, s>>>(probs, work);
}

void launch_downward_batched(const ProbF32* probs, const int2* work, int items, size_t smem, bool steady, cudaStream_t s) {
  if (items <= 0) return;
  if (steady) k_downward_batched<true><<<items, kFarThreads, smem, s>>>(probs, work);
  else k_downward_batched<false><<<items, kFarThreads, smem, s>>>(probs, work);
}

void launch_gather_batched(const ProbF32* probs, const int* leaf_off, int P, int Ltot, int ld, float* xb,
                           cudaStream_t s) {
  const int64_t total = static_cast<int64_t>(Ltot) * kRC * ld;
  k_gather_batched<<<ceil_div(total, 256), 256, 0, s>>>(probs, leaf_off, P, Ltot, ld, xb);
}

void launch_scatter_batched(const ProbF32* probs, const int* leaf_off, int P, int Ltot, int ld, int Rmax,
                            const BatchParts& parts, const float* ynear, const float* yfar, cudaStream_t s) {
  if (parts.chunk_ptr) {
    k_scatter_batched<<<Ltot * Rmax, kPartThreads, 0, s>>>(probs, leaf_off, P, Rmax, ld, parts, ynear, yfar);
    return;
  }
  const int64_t total = static_cast<int64_t>(Ltot) * kRC * ld;
  k_scatter_rows<<<ceil_div(total, 256), 256, 0, s>>>(probs, leaf_off, P, Ltot, ld, ynear, yfar);
}

size_t persist_group_bytes(int D, int RC, int ld, int threads) { return sk::group_stage_bytes(D, RC, ld, threads); }

namespace {

template <int D>
const void* persist_fn_d(int kernel) {
  switch (kernel) {
    case DWFMM_K_EXP: return reinterpret_cast<const void*>(k_batch_persistent<D, DWFMM_K_EXP>);
    case DWFMM_K_MATERN32: return reinterpret_cast<const void*>(k_batch_persistent<D, DWFMM_K_MATERN32>);
    default: return reinterpret_cast<const void*>(k_batch_persistent<D, DWFMM_K_GAUSS>);
  }
}

const void* persist_fn(int D, int kernel) {
  switch (D) {
    case 4: return persist_fn_d<4>(kernel);
    case 8: return persist_fn_d<8>(kernel);
    case 10: return persist_fn_d<10>(kernel);
    case 12: return persist_fn_d<12>(kernel);
    case 16: return persist_fn_d<16>(kernel);
    default: return persist_fn_d<20>(kernel);
  }
}

template <int D>
cudaError_t persist_launch_d(int kernel, const cudaLaunchConfig_t& cfg, const PersistArgs& pa) {
  switch (kernel) {
    case DWFMM_K_EXP: return cudaLaunchKernelEx(&cfg, k_batch_persistent<D, DWFMM_K_EXP>, pa);
    case DWFMM_K_MATERN32: return cudaLaunchKernelEx(&cfg, k_batch_persistent<D, DWFMM_K_MATERN32>, pa);
    default: return cudaLaunchKernelEx(&cfg, k_batch_persistent<D, DWFMM_K_GAUSS>, pa);
  }
}

}  // namespace

int persist_blocks_per_sm(int D, int kernel, size_t smem) {
  const void* f = persist_fn(D, kernel);
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, kPersistThreads, smem) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_batch_persistent(int D, int kernel, const PersistArgs& pa, int grid, size_t smem,
                                    cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(kPersistThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  switch (D) {
    case 4: return persist_launch_d<4>(kernel, cfg, pa);
    case 8: return persist_launch_d<8>(kernel, cfg, pa);
    case 10: return persist_launch_d<10>(kernel, cfg, pa);
    case 12: return persist_launch_d<12>(kernel, cfg, pa);
    case 16: return persist_launch_d<16>(kernel, cfg, pa);
    default: return persist_launch_d<20>(kernel, cfg, pa);
  }
}

void launch_farfield(Plan& P, int Rc, bool fp64, bool steady) {
  if (fp64) farfield_impl<double>(P, Rc, steady);
  else farfield_impl<float>(P, Rc, steady);
}

}  // namespace dw
