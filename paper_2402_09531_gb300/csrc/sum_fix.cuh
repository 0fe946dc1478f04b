// Float64 kernel summation with kernel values from the integer pipes
// (fix64.cuh), one translation unit per kernel function (sum_fix_exp.cu,
// sum_fix_matern.cu, sum_fix_gauss.cu).  Charges and sums are float64.
//
// k_fix_sum: one CTA per (target group, pass of up to 128 targets, part of the
// list).  A thread owns one target; groups of at most 64 targets are shared by
// several threads, which take every nsub-th source (or, for short source
// groups, every nsub-th group).  Sources and charges are rows in HBM and come
// in by cp.async one stage ahead.  Bound by the wide products (32 lanes a clock
// on an SM) for a few right-hand sides, beyond that by the float64 unit's 2
// multiply-adds a clock, one for each pair and side; the two share an issue port
// (32 multiply-adds alone take a warp 512 clocks, 116 products 58, both 610).
// d = 10 Gaussian, N = 12289, 16 right-hand sides, the whole product: 34.6 ms with
// kernel values from the float64 unit, 5.0 ms; its 2.4e9 multiply-adds take 4.1.
// Charges and sums in fixed point would take 3.2 ms there, but keep a term only to
// 2^-55 of the largest one, not of itself.
#pragma once

#include <atomic>
#include <type_traits>

#include "fix64.cuh"

namespace dw {
namespace fx {

constexpr int kThreads = 128;
constexpr int kFoldStages = 4;   // stages summed before the running sums take them

template <int RC>
constexpr int stage_cap() { return RC > 4 ? 64 : 128; }

// Table, two stages of records (2 DM ints per point: limb pairs, zero beyond
// d) and charges (RC rows), running sums of RC rows.
template <int DM, int RC>
constexpr size_t fix_smem() {
  return kTable * sizeof(u64) + 2 * static_cast<size_t>(stage_cap<RC>()) * (2 * DM * sizeof(int) + RC * sizeof(double)) +
         (RC > 4 ? static_cast<size_t>(RC) * kThreads * sizeof(double) : 0);
}

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

__device__ __forceinline__ void cp8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// phi of one target (limbs x) and P source records, `stride` int4 apart.
template <int KER, int DM, int P>
__device__ __forceinline__ void pair_phi(const int (&xh)[DM], const int (&xl)[DM], const int4* rec, int stride,
                                         const Consts& c, const u64* table, double (&out)[P]) {
  u64 A[P], C[P];
  s64 B[P];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    A[q] = C[q] = 0;
    B[q] = 0;
#pragma unroll
    for (int k = 0; k < DM; k += 2) {
      const int4 v = rec[q * stride + (k >> 1)];
      const int h0 = xh[k] - v.x, l0 = xl[k] - v.y, h1 = xh[k + 1] - v.z, l1 = xl[k + 1] - v.w;
      A[q] += static_cast<u64>(static_cast<s64>(h0) * h0);
      B[q] += static_cast<s64>(h0) * l0;
      C[q] += static_cast<u64>(static_cast<s64>(l0) * l0);
      A[q] += static_cast<u64>(static_cast<s64>(h1) * h1);
      B[q] += static_cast<s64>(h1) * l1;
      C[q] += static_cast<u64>(static_cast<s64>(l1) * l1);
    }
  }
  phi64<KER, P>(A, B, C, c, table, out);
}

template <int KER, int DM, int RC>
__global__ void __launch_bounds__(kThreads, RC > 4 ? 3 : 4) k_fix_sum(const FixArgs a) {
  constexpr int CAP = stage_cap<RC>();
  constexpr int RV = DM / 2;   // int4 per record
  extern __shared__ __align__(16) unsigned char smem[];
  u64* table = reinterpret_cast<u64*>(smem);
  int4* srec = reinterpret_cast<int4*>(smem + kTable * sizeof(u64));   // [2][CAP][RV]
  double* sq = reinterpret_cast<double*>(srec + 2 * CAP * RV);         // [2][RC][CAP]
  double* sacc = sq + 2 * CAP * RC;                                    // [RC][kThreads] if RC > 4

  const int part = static_cast<int>(blockIdx.x) % a.splits;
  const int gp = static_cast<int>(blockIdx.x) / a.splits;
  const int pass = gp % a.passes;
  const int g = a.first + gp / a.passes;
  const int r0 = a.rowptr[g], len = a.rowptr[g + 1] - r0;
  const int rb = r0 + static_cast<int>((static_cast<int64_t>(len) * part) / a.splits);
  const int re = r0 + static_cast<int>((static_cast<int64_t>(len) * (part + 1)) / a.splits);
  const int t0 = pass * a.tp;
  const int t_end = min(a.ld, t0 + a.tp);
  double* out = a.out + part * a.split_stride + g * a.o_gstride;

  for (int i = threadIdx.x; i < kTable; i += kThreads) table[i] = a.table[i];
  const int sub = static_cast<int>(threadIdx.x) / a.tp;
  const int i = t0 + static_cast<int>(threadIdx.x) % a.tp;
  const bool on = sub < a.nsub && i < t_end;
  int xh[DM], xl[DM];
  {
    const int4* tr = a.rec + (static_cast<int64_t>(g) * a.ld + (on ? i : 0)) * RV;
#pragma unroll
    for (int k = 0; k < DM; k += 2) {
      const int4 v = tr[k >> 1];
      xh[k] = v.x;
      xl[k] = v.y;
      xh[k + 1] = v.z;
      xl[k + 1] = v.w;
    }
  }
  // sums of a few stages, and the running sums that take them: many short sums
  // lose less than a long one, and what is added to the running sums is little
  double acc[RC], tot[RC > 4 ? 1 : RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) acc[r] = 0.0;
  if constexpr (RC > 4) {
#pragma unroll
    for (int r = 0; r < RC; ++r) sacc[r * kThreads + threadIdx.x] = 0.0;
  } else {
#pragma unroll
    for (int r = 0; r < RC; ++r) tot[r] = 0.0;
  }
  int staged = 0;
  auto fold = [&]() {
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      if (r >= a.Rc) break;
      if constexpr (RC > 4) sacc[r * kThreads + threadIdx.x] += acc[r];
      else tot[r] += acc[r];
      acc[r] = 0.0;
    }
  };

  // P sources j, j + dj, ... of the buffer: kernel values, and their products
  // (columns in eights, then fours, then twos up to Rc: the branches are between
  // blocks that the compiler can interleave with the integer work)
  auto values = [&](auto& p, int buf, int j, int dj) {
    constexpr int P = sizeof(p) / sizeof(double);
    pair_phi<KER, DM, P>(xh, xl, srec + (buf * CAP + j) * RV, dj * RV, a.c, table, p);
  };
  auto add = [&](const auto& p, int buf, int j, int dj) {
    constexpr int P = sizeof(p) / sizeof(double);
    const double* q = sq + buf * CAP * RC + j;
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      if ((r == 2 || r == 8 || r == 12) && r >= a.Rc) break;
#pragma unroll
      for (int u = 0; u < P; ++u) acc[r] = fma(p[u], q[r * CAP + u * dj], acc[r]);
    }
  };
  // two sources at a time, the next two's values on the integer pipes while the
  // float64 unit adds the last two's
  auto terms = [&](int buf, int j0, int dj, int j1) {
    int j = j0;
    if (j + dj < j1) {
      double p[2], pn[2];
      values(p, buf, j, dj);
      for (j += 2 * dj; j + dj < j1; j += 2 * dj) {
        values(pn, buf, j, dj);
        add(p, buf, j - 2 * dj, dj);
        p[0] = pn[0];
        p[1] = pn[1];
      }
      add(p, buf, j - 2 * dj, dj);
    }
    if (j < j1) {
      double p[1];
      values(p, buf, j, dj);
      add(p, buf, j, dj);
    }
  };
  // cn slots of source group s from slot cb (rows are multiples of 8 slots)
  auto load = [&](int buf, int s, int cb, int cn) {
    const int4* rsrc = a.rec + (static_cast<int64_t>(s) * a.ld + cb) * RV;
    int4* rdst = srec + buf * CAP * RV;
    for (int k = threadIdx.x; k < cn * RV; k += kThreads) cp16(rdst + k, rsrc + k);
    const double* qsrc = a.charge + s * a.q_gstride + cb;
    double* qdst = sq + buf * CAP * RC;
    for (int k = threadIdx.x; k < a.Rc * (CAP / 2); k += kThreads) {
      const int r = k / (CAP / 2), j = k % (CAP / 2) * 2;
      if (j < cn) cp16(qdst + r * CAP + j, qsrc + static_cast<int64_t>(r) * a.ld + j);
    }
    cp_commit();
  };

  if (a.group_entries > 0) {
    // short source groups (one size): group_entries of them a stage
    const int n = a.count_const;
    const int ge = a.group_entries;
    auto load_entries = [&](int buf, int e) {
      const int ne = min(ge, re - e);
      const int per = n * RV;
      for (int k = threadIdx.x; k < ne * per; k += kThreads) {
        const int en = k / per;
        cp16(srec + buf * CAP * RV + k, a.rec + static_cast<int64_t>(a.col[e + en]) * a.ld * RV + (k - en * per));
      }
      if (static_cast<int>(threadIdx.x) < ne * n) {   // at most CAP slots
        const int en = static_cast<int>(threadIdx.x) / n;
        const double* qsrc = a.charge + a.col[e + en] * a.q_gstride + (static_cast<int>(threadIdx.x) - en * n);
        double* qdst = sq + buf * CAP * RC + threadIdx.x;
        for (int r = 0; r < a.Rc; ++r) cp8(qdst + r * CAP, qsrc + static_cast<int64_t>(r) * a.ld);
      }
      cp_commit();
    };
    if (rb < re) load_entries(0, rb);
    int buf = 0;
    for (int e = rb; e < re; e += ge, buf ^= 1) {
      cp_wait_all();
      __syncthreads();
      if (e + ge < re) load_entries(buf ^ 1, e + ge);
      const int ne = min(ge, re - e);
      for (int en = on ? sub : ne; en < ne; en += a.nsub) terms(buf, en * n, 1, en * n + n);
      if (++staged % kFoldStages == 0) fold();
    }
  } else {
    int e = rb, cb = 0, buf = 0;
    auto count = [&](int en) { return a.count ? a.count[a.count_off + a.col[en]] : a.count_const; };
    int cnt = e < re ? count(e) : 0;
    if (e < re) load(0, a.col[e], 0, min(CAP, cnt));
    while (e < re) {
      const int cn = min(CAP, cnt - cb);
      int ne = e, ncb = cb + CAP, ncnt = cnt;
      if (ncb >= cnt) {
        ncb = 0;
        if (++ne < re) ncnt = count(ne);
      }
      cp_wait_all();
      __syncthreads();
      if (ne < re) load(buf ^ 1, a.col[ne], ncb, min(CAP, ncnt - ncb));
      if (on) terms(buf, sub, a.nsub, cn);
      if (++staged % kFoldStages == 0) fold();
      e = ne;
      cb = ncb;
      cnt = ncnt;
      buf ^= 1;
    }
  }
  fold();

  if constexpr (RC > 4) {
    if (a.nsub > 1) __syncthreads();
  } else {
    if (a.nsub > 1) {   // the stages become the partial sums of the target's threads
      __syncthreads();
      double* red = reinterpret_cast<double*>(srec);
#pragma unroll
      for (int r = 0; r < RC; ++r) red[r * kThreads + threadIdx.x] = tot[r];
      sacc = red;
      __syncthreads();
    }
  }
  if (!on || sub > 0) return;
#pragma unroll
  for (int r = 0; r < RC; ++r) {
    if (r >= a.Rc) break;
    double v;
    if (RC > 4 || a.nsub > 1) {
      v = sacc[r * kThreads + threadIdx.x];
      for (int u = 1; u < a.nsub; ++u) v += sacc[r * kThreads + threadIdx.x + u * a.tp];
    } else {
      v = tot[RC > 4 ? 0 : r];
    }
    out[static_cast<int64_t>(r) * a.ld + i] = v;
  }
}

// Each unordered pair of near leaves once (leaves of 32 to 128 sites, up to 4
// right-hand sides): a CTA takes target leaf T and a chunk of the sources of
// its upper entries (T, S >= T), laid end to end.  A warp holds 64 sources, 2
// per lane, and turns over T's sites: at step s lane l meets target l + s
// (modulo T's size, which is at least the warp's width), so the lanes' targets
// differ and each adds to its target's sum in shared memory without atomics,
// while the sources' sums stay in registers.  No lane idles on a ragged leaf:
// the turn takes exactly T's size, and the sources are a stream.  Bound by the
// wide products, beyond 2 right-hand sides with the float64 unit close behind.
// d = 8 Matern, 1 right-hand side, N = 262144, the whole product: 440 ms with kernel
// values from the float64 unit (each pair once, too) -> 43.2 ms.
template <int DM>
constexpr int sym_stride() { return DM == 10 ? 20 : 2 * DM + 4; }   // ints, 4 mod 8: no bank conflicts

template <int DM, int RC>
constexpr size_t fix_sym_smem(int ld) {
  return kTable * sizeof(u64) + static_cast<size_t>(ld) * sym_stride<DM>() * sizeof(int) +
         static_cast<size_t>(1 + kThreads / 32) * RC * ld * sizeof(double);
}

template <int KER, int DM, int RC>
__global__ void __launch_bounds__(kThreads) k_fix_sym(const FixSymArgs a) {
  constexpr int TS = sym_stride<DM>(), RV = DM / 2, NW = kThreads / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int ld = a.ld;
  u64* table = reinterpret_cast<u64*>(smem);
  double* facc = reinterpret_cast<double*>(table + kTable);            // [NW][RC][ld]
  double* tq = facc + NW * RC * ld;                                    // [RC][ld]
  int* trec = reinterpret_cast<int*>(tq + RC * ld);                    // [ld][TS]
  const int chunk = blockIdx.x;
  const int T = a.chunk_t[chunk];
  const int c = a.count[T];
  const int e0 = a.uprow[T], ne = a.uprow[T + 1] - e0;
  const int warp = static_cast<int>(threadIdx.x) >> 5, lane = static_cast<int>(threadIdx.x) & 31;
  const int per = NW * 64 * a.batches;                                 // sources per chunk
  const int first = (chunk - a.chunk_ptr[T]) * per;

  for (int i = threadIdx.x; i < kTable; i += kThreads) table[i] = a.table[i];
  for (int i = threadIdx.x; i < c * RV; i += kThreads)
    *reinterpret_cast<int4*>(trec + (i / RV) * TS + (i % RV) * 4) = a.rec[static_cast<int64_t>(T) * ld * RV + i];
  for (int i = threadIdx.x; i < a.Rc * ld; i += kThreads) tq[i] = a.charge[static_cast<int64_t>(T) * kRC * ld + i];
  for (int i = threadIdx.x; i < NW * RC * ld; i += kThreads) facc[i] = 0.0;
  __syncthreads();
  double* fw = facc + warp * RC * ld;

  for (int b = 0; b < a.batches; ++b) {
    const int base = first + (b * NW + warp) * 64;
    if (base >= ne * a.cmax) break;
    int sh[2][DM], sl[2][DM];
    double q[2][RC];
    int ent[2], slot[2];   // entry of the source, -1: nothing to write
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = base + u * 32 + lane;
      const int en = j / a.cmax;
      slot[u] = j - en * a.cmax;
      int S = T;
      bool ok = en < ne;
      if (ok) {
        S = a.up_s[e0 + en];
        ok = slot[u] < a.count[S];
      }
      ent[u] = ok && S != T ? e0 + en : -1;
      const int at = ok ? slot[u] : 0;
      const int4* rec = a.rec + (static_cast<int64_t>(S) * ld + at) * RV;
#pragma unroll
      for (int k = 0; k < DM; k += 2) {
        const int4 v = rec[k >> 1];
        sh[u][k] = v.x;
        sl[u][k] = v.y;
        sh[u][k + 1] = v.z;
        sl[u][k + 1] = v.w;
      }
#pragma unroll
      for (int r = 0; r < RC; ++r)
        q[u][r] = ok && r < a.Rc ? a.charge[(static_cast<int64_t>(S) * kRC + r) * ld + at] : 0.0;
    }
    double tr[2][RC];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int r = 0; r < RC; ++r) tr[u][r] = 0.0;
    int t = lane;
    for (int s = 0; s < c; ++s) {
      u64 A[2] = {0, 0}, C[2] = {0, 0};
      s64 B[2] = {0, 0};
      double p[2];
      const int4* rec = reinterpret_cast<const int4*>(trec + t * TS);
#pragma unroll
      for (int k = 0; k < DM; k += 2) {
        const int4 v = rec[k >> 1];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int h0 = sh[u][k] - v.x, l0 = sl[u][k] - v.y, h1 = sh[u][k + 1] - v.z, l1 = sl[u][k + 1] - v.w;
          A[u] += static_cast<u64>(static_cast<s64>(h0) * h0);
          B[u] += static_cast<s64>(h0) * l0;
          C[u] += static_cast<u64>(static_cast<s64>(l0) * l0);
          A[u] += static_cast<u64>(static_cast<s64>(h1) * h1);
          B[u] += static_cast<s64>(h1) * l1;
          C[u] += static_cast<u64>(static_cast<s64>(l1) * l1);
        }
      }
      phi64<KER, 2>(A, B, C, a.c, table, p);
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        if (r % 2 == 0 && r >= a.Rc) break;   // columns in twos
        double f = fw[r * ld + t];
        const double x = r < a.Rc ? tq[r * ld + t] : 0.0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          f = fma(p[u], q[u][r], f);
          tr[u][r] = fma(p[u], x, tr[u][r]);
        }
        fw[r * ld + t] = f;
      }
      if (++t >= c) t -= c;
      __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (ent[u] < 0) continue;
#pragma unroll
      for (int r = 0; r < RC; ++r)
        if (r < a.Rc) a.pt[(static_cast<int64_t>(ent[u]) * a.Rc + r) * ld + slot[u]] = tr[u][r];
    }
  }
  __syncthreads();
  double* pf = a.pf + static_cast<int64_t>(chunk) * a.Rc * ld;
  for (int i = threadIdx.x; i < a.Rc * ld; i += kThreads) {
    double v = facc[i];
#pragma unroll
    for (int w = 1; w < NW; ++w) v += facc[w * RC * ld + i];
    pf[i] = v;
  }
}

template <int KER, int DM, int RC>
void launch_sym(const FixSymArgs& a, int chunks, cudaStream_t s) {
  const size_t smem = fix_sym_smem<DM, RC>(a.ld);
  if (fix_sym_smem<DM, RC>(kThreads) > 48 * 1024) {
    static std::atomic<uint64_t> done{0};
    const uint64_t bit = device_bit();
    if (!(done.load() & bit)) {
      DW_CUDA(cudaFuncSetAttribute(k_fix_sym<KER, DM, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(fix_sym_smem<DM, RC>(kThreads))));
      done.fetch_or(bit);
    }
  }
  k_fix_sym<KER, DM, RC><<<chunks, kThreads, smem, s>>>(a);
}

template <int KER, int DM>
void launch_sym_rc(int RC, const FixSymArgs& a, int chunks, cudaStream_t s) {
  if (RC <= 1) launch_sym<KER, DM, 1>(a, chunks, s);
  else launch_sym<KER, DM, 4>(a, chunks, s);
}

template <int KER>
void launch_sym_d(int d, int RC, const FixSymArgs& a, int chunks, cudaStream_t s) {
  if (d <= 4) launch_sym_rc<KER, 4>(RC, a, chunks, s);
  else if (d <= 8) launch_sym_rc<KER, 8>(RC, a, chunks, s);
  else if (d <= 10) launch_sym_rc<KER, 10>(RC, a, chunks, s);
  else if (d <= 12) launch_sym_rc<KER, 12>(RC, a, chunks, s);
  else launch_sym_rc<KER, 16>(RC, a, chunks, s);
}

template <int KER, int DM, int RC>
void launch_fix(const FixArgs& a, int ctas, cudaStream_t s) {
  constexpr size_t smem = fix_smem<DM, RC>();
  if (smem > 48 * 1024) {
    static std::atomic<uint64_t> done{0};
    const uint64_t bit = device_bit();
    if (!(done.load() & bit)) {
      DW_CUDA(cudaFuncSetAttribute(k_fix_sum<KER, DM, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(smem)));
      done.fetch_or(bit);
    }
  }
  k_fix_sum<KER, DM, RC><<<ctas, kThreads, smem, s>>>(a);
}

template <int KER, int DM>
void launch_fix_rc(int RC, const FixArgs& a, int ctas, cudaStream_t s) {
  if (RC <= 1) launch_fix<KER, DM, 1>(a, ctas, s);
  else if (RC <= 4) launch_fix<KER, DM, 4>(a, ctas, s);
  else launch_fix<KER, DM, 16>(a, ctas, s);
}

template <int KER>
void launch_fix_d(int d, int RC, const FixArgs& a, int ctas, cudaStream_t s) {
  if (d <= 4) launch_fix_rc<KER, 4>(RC, a, ctas, s);
  else if (d <= 8) launch_fix_rc<KER, 8>(RC, a, ctas, s);
  else if (d <= 10) launch_fix_rc<KER, 10>(RC, a, ctas, s);
  else if (d <= 12) launch_fix_rc<KER, 12>(RC, a, ctas, s);
  else launch_fix_rc<KER, 16>(RC, a, ctas, s);
}

}  // namespace fx
}  // namespace dw
