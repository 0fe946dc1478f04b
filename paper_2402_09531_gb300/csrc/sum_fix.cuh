// Float64 kernel summation in fixed point (fix64.cuh), one translation unit
// per kernel function (sum_fix_exp.cu, sum_fix_matern.cu, sum_fix_gauss.cu).
//
// k_fix_sum: one CTA per (target group, pass of up to 128 targets, part of the
// list).  A thread owns one target; groups of at most 64 targets are shared by
// several threads, which take every nsub-th source (or, for short source
// groups, every nsub-th group).  Sources and charges are contiguous records in
// HBM and come in by cp.async one stage ahead.  Bound by the wide products
// (32 lanes a clock on an SM).  d = 10 Gaussian near field, N = 12289, 16
// right-hand sides: 29.7 -> 3.1 ms; couplings of the d = 8 Matern tree at
// N = 262144 (10 nodes a cluster): 26.7 -> 0.33 ms (a float64 warp there had
// 10 of its 32 lanes at work).
#pragma once

#include <atomic>
#include <type_traits>

#include "fix64.cuh"
#include "ksum.cuh"

namespace dw {
namespace fx {

constexpr int kThreads = ks::kThreads;

template <int RC>
constexpr int stage_cap() { return RC > 4 ? 64 : 128; }

// Records: 2 * DM ints per point (limb pairs, zero beyond d); charges: RC
// limb pairs per point.  pts_stage * DM: see fix_smem.
template <int DM, int RC>
constexpr size_t fix_smem() {
  return kTable * sizeof(u64) + 2 * static_cast<size_t>(stage_cap<RC>()) * (2 * DM + 2 * RC) * sizeof(int) +
         (RC > 4 ? static_cast<size_t>(RC) * kThreads * sizeof(double) : 0);
}

struct Limbs {
  int h, l;
};

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
                                         const Consts& c, const u64* table, u64 (&out)[P]) {
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
  phi56<KER, P>(A, B, C, c, table, out);
}

// (hh, m) += phi q: hh counts 2^(e - 55), m 2^(e - 83); the product of the two
// low limbs (below 2^(e - 57), signed) is left out.
__device__ __forceinline__ void mac(u64 p, int qh, int ql, s64& hh, s64& m) {
  const int ph = static_cast<int>(p >> 28), pl = static_cast<int>(p) & 0xfffffff;
  hh += static_cast<s64>(ph) * qh;
  m += static_cast<s64>(ph) * ql;
  m += static_cast<s64>(pl) * qh;
}

__device__ __forceinline__ double flush(s64& hh, s64& m, double scale, double acc) {
  const s64 v = hh + ((m + (1ll << 27)) >> 28);
  hh = m = 0;
  return fma(static_cast<double>(v), scale, acc);
}

template <int KER, int DM, int RC>
__global__ void __launch_bounds__(kThreads, RC > 4 ? 3 : 4) k_fix_sum(const FixArgs a) {
  constexpr int CAP = stage_cap<RC>();
  constexpr int RV = DM / 2;   // int4 per record
  extern __shared__ __align__(16) unsigned char smem[];
  u64* table = reinterpret_cast<u64*>(smem);
  int4* srec = reinterpret_cast<int4*>(smem + kTable * sizeof(u64));   // [2][CAP][RV]
  int2* sq = reinterpret_cast<int2*>(srec + 2 * CAP * RV);             // [2][CAP][RC]
  double* sacc = reinterpret_cast<double*>(sq + 2 * CAP * RC);         // [RC][kThreads] if RC > 4

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

  if (*a.flag) {   // a charge the format does not take (not finite, below 2^-960): float64
    double* sc = reinterpret_cast<double*>(smem);
    ks::ksum_targets<double, KER, DM, RC>(g, t0 + static_cast<int>(threadIdx.x), t_end, rb, re, a.col, a.d, a.inv_sigma,
                                          a.coord, a.side, a.coord, a.side, a.charge, a.q_gstride, a.ld, out, a.ld,
                                          a.Rc, sc, sc + DM * ks::kSrcChunk);
    return;
  }

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
  s64 hh[RC], mm[RC];
  double acc[RC > 4 ? 1 : RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) hh[r] = mm[r] = 0;
  if constexpr (RC > 4) {
#pragma unroll
    for (int r = 0; r < RC; ++r) sacc[r * kThreads + threadIdx.x] = 0.0;
  } else {
#pragma unroll
    for (int r = 0; r < RC; ++r) acc[r] = 0.0;
  }

  // sources j and (if P = 2) j + dj of the buffer
  auto term = [&](auto np, int buf, int j, int dj) {
    constexpr int P = decltype(np)::value;
    u64 p[P];
    pair_phi<KER, DM, P>(xh, xl, srec + (buf * CAP + j) * RV, dj * RV, a.c, table, p);
#pragma unroll
    for (int u = 0; u < P; ++u) {
      const int2* q = sq + (buf * CAP + j + u * dj) * RC;
      if constexpr (RC == 1) {
        const int2 v = q[0];
        mac(p[u], v.x, v.y, hh[0], mm[0]);
      } else {
#pragma unroll
        for (int r = 0; r < RC; r += 2) {
          const int4 v = *reinterpret_cast<const int4*>(q + r);
          mac(p[u], v.x, v.y, hh[r], mm[r]);
          mac(p[u], v.z, v.w, hh[r + 1], mm[r + 1]);
        }
      }
    }
  };
  auto terms = [&](int buf, int j0, int dj, int j1) {
    int j = j0;
    for (; j + dj < j1; j += 2 * dj) term(std::integral_constant<int, 2>{}, buf, j, dj);
    if (j < j1) term(std::integral_constant<int, 1>{}, buf, j, dj);
  };
  auto flush_all = [&](int s) {
    const double* sc = a.qscale + static_cast<int64_t>(s) * kRC;
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      if constexpr (RC > 4) {
        double* p = sacc + r * kThreads + threadIdx.x;
        *p = flush(hh[r], mm[r], sc[r], *p);
      } else {
        acc[r] = flush(hh[r], mm[r], sc[r], acc[r]);
      }
    }
  };
  // cn slots of source group s from slot cb into buffer slots at `at`
  auto load = [&](int buf, int at, int s, int cb, int cn) {
    const int4* rsrc = a.rec + (static_cast<int64_t>(s) * a.ld + cb) * RV;
    int4* rdst = srec + (buf * CAP + at) * RV;
    for (int k = threadIdx.x; k < cn * RV; k += kThreads) cp16(rdst + k, rsrc + k);
    const int2* qsrc = a.q + (static_cast<int64_t>(s) * a.ld + cb) * RC;
    int2* qdst = sq + (buf * CAP + at) * RC;
    if constexpr (RC == 1) {
      for (int k = threadIdx.x; k < cn; k += kThreads) cp8(qdst + k, qsrc + k);
    } else {
      for (int k = threadIdx.x; k < cn * (RC / 2); k += kThreads) cp16(qdst + 2 * k, qsrc + 2 * k);
    }
  };

  if (a.group_entries > 0) {
    // short source groups (one size): group_entries of them a stage
    const int n = a.side.count_const;
    const int ge = a.group_entries;
    auto load_entries = [&](int buf, int e) {
      const int ne = min(ge, re - e);
      const int per = n * RV;
      for (int k = threadIdx.x; k < ne * per; k += kThreads) {
        const int en = k / per;
        cp16(srec + buf * CAP * RV + k, a.rec + static_cast<int64_t>(a.col[e + en]) * a.ld * RV + (k - en * per));
      }
      const int perq = n * RC;
      for (int k = threadIdx.x; k < ne * perq; k += kThreads) {
        const int en = k / perq;
        cp8(sq + buf * CAP * RC + k, a.q + static_cast<int64_t>(a.col[e + en]) * a.ld * RC + (k - en * perq));
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
      for (int en = on ? sub : ne; en < ne; en += a.nsub) {
        terms(buf, en * n, 1, en * n + n);
        flush_all(a.col[e + en]);
      }
    }
  } else {
    int e = rb, cb = 0, buf = 0;
    auto count = [&](int en) {
      return a.side.count ? a.side.count[a.side.count_off + a.col[en]] : a.side.count_const;
    };
    int cnt = e < re ? count(e) : 0;
    if (e < re) {
      load(0, 0, a.col[e], 0, min(CAP, cnt));
      cp_commit();
    }
    while (e < re) {
      const int s = a.col[e];
      const int cn = min(CAP, cnt - cb);
      int ne = e, ncb = cb + CAP, ncnt = cnt;
      if (ncb >= cnt) {
        ncb = 0;
        if (++ne < re) ncnt = count(ne);
      }
      cp_wait_all();
      __syncthreads();
      if (ne < re) {
        load(buf ^ 1, 0, a.col[ne], ncb, min(CAP, ncnt - ncb));
        cp_commit();
      }
      if (on) {
        terms(buf, sub, a.nsub, cn);
        flush_all(s);
      }
      e = ne;
      cb = ncb;
      cnt = ncnt;
      buf ^= 1;
    }
  }

  if constexpr (RC > 4) {
    if (a.nsub > 1) __syncthreads();
  } else {
    if (a.nsub > 1) {   // the stages become the partial sums of the target's threads
      __syncthreads();
      double* red = reinterpret_cast<double*>(srec);
#pragma unroll
      for (int r = 0; r < RC; ++r) red[r * kThreads + threadIdx.x] = acc[r];
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
      v = acc[RC > 4 ? 0 : r];
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
// wide products.  d = 8 Matern, 1 right-hand side, N = 262144: 412 ms (float64,
// each pair once) -> 48 ms; N = 65536: 10.3 ms with k_fix_sum, 5.8 ms here.
template <int DM>
constexpr int sym_stride() { return DM == 10 ? 20 : 2 * DM + 4; }   // ints, 4 mod 8: no bank conflicts

template <int DM, int RC>
constexpr size_t fix_sym_smem(int ld) {
  return kTable * sizeof(u64) + static_cast<size_t>(ld) * (sym_stride<DM>() + 2 * RC) * sizeof(int) +
         static_cast<size_t>(kThreads / 32) * RC * ld * (2 * sizeof(s64) + sizeof(double));
}

template <int KER, int DM, int RC>
__global__ void __launch_bounds__(kThreads) k_fix_sym(const FixSymArgs a) {
  constexpr int TS = sym_stride<DM>(), RV = DM / 2, NW = kThreads / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int ld = a.ld;
  u64* table = reinterpret_cast<u64*>(smem);
  longlong2* facc = reinterpret_cast<longlong2*>(table + kTable);      // [NW][RC][ld] (hh, m)
  double* dacc = reinterpret_cast<double*>(facc + NW * RC * ld);       // [NW][RC][ld]
  int* trec = reinterpret_cast<int*>(dacc + NW * RC * ld);             // [ld][TS]
  int* tq = trec + ld * TS;                                            // [ld][2 RC]
  const int chunk = blockIdx.x;
  const int T = a.chunk_t[chunk];
  const int c = a.count[T];
  const int e0 = a.uprow[T], ne = a.uprow[T + 1] - e0;
  const int warp = static_cast<int>(threadIdx.x) >> 5, lane = static_cast<int>(threadIdx.x) & 31;
  const int per = NW * 64 * a.batches;                                 // sources per chunk
  const int first = (chunk - a.chunk_ptr[T]) * per;
  double* pf = a.pf + static_cast<int64_t>(chunk) * a.Rc * ld;

  if (*a.flag) {   // a charge the format does not take (not finite, below 2^-960): float64
    auto phi = [&](int g, int i, int h, int j) {
      double r2 = 0.0;
      for (int k = 0; k < a.d; ++k) {
        const double df = a.coord[(static_cast<int64_t>(g) * a.d + k) * ld + i] -
                          a.coord[(static_cast<int64_t>(h) * a.d + k) * ld + j];
        r2 += df * df;
      }
      return ks::phi_r2<double, KER>(r2, a.inv_sigma);
    };
    const int last = min(first + per, ne * a.cmax);
    for (int i = threadIdx.x; i < c; i += kThreads)
      for (int r = 0; r < a.Rc; ++r) {
        double v = 0.0;
        for (int j = first; j < last; ++j) {
          const int S = a.up_s[e0 + j / a.cmax], slot = j % a.cmax;
          if (slot < a.count[S]) v += phi(T, i, S, slot) * a.charge[(static_cast<int64_t>(S) * kRC + r) * ld + slot];
        }
        pf[static_cast<int64_t>(r) * ld + i] = v;
      }
    for (int j = first + static_cast<int>(threadIdx.x); j < last; j += kThreads) {
      const int e = e0 + j / a.cmax, slot = j % a.cmax, S = a.up_s[e];
      if (S == T || slot >= a.count[S]) continue;
      for (int r = 0; r < a.Rc; ++r) {
        double v = 0.0;
        for (int i = 0; i < c; ++i) v += phi(T, i, S, slot) * a.charge[(static_cast<int64_t>(T) * kRC + r) * ld + i];
        a.pt[(static_cast<int64_t>(e) * a.Rc + r) * ld + slot] = v;
      }
    }
    return;
  }

  for (int i = threadIdx.x; i < kTable; i += kThreads) table[i] = a.table[i];
  for (int i = threadIdx.x; i < c * RV; i += kThreads)
    *reinterpret_cast<int4*>(trec + (i / RV) * TS + (i % RV) * 4) = a.rec[static_cast<int64_t>(T) * ld * RV + i];
  for (int i = threadIdx.x; i < c * RC; i += kThreads)
    reinterpret_cast<int2*>(tq)[i] = a.q[static_cast<int64_t>(T) * ld * RC + i];
  for (int i = threadIdx.x; i < NW * RC * ld; i += kThreads) {
    facc[i] = make_longlong2(0, 0);
    dacc[i] = 0.0;
  }
  __syncthreads();
  longlong2* fw = facc + warp * RC * ld;
  double* dw = dacc + warp * RC * ld;
  double scale[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) scale[r] = a.qscale[r];
  auto drain = [&]() {   // the target sums hold at most 128 terms
    for (int i = lane; i < RC * ld; i += 32) {
      const longlong2 v = fw[i];
      s64 hh = v.x, m = v.y;
      dw[i] = flush(hh, m, a.qscale[i / ld], dw[i]);
      fw[i] = make_longlong2(0, 0);
    }
    __syncwarp();
  };

  for (int b = 0; b < a.batches; ++b) {
    const int base = first + (b * NW + warp) * 64;
    if (base >= ne * a.cmax) break;
    int sh[2][DM], sl[2][DM], qh[2][RC], ql[2][RC];
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
      const int64_t at = static_cast<int64_t>(S) * ld + (ok ? slot[u] : 0);
#pragma unroll
      for (int k = 0; k < DM; k += 2) {
        const int4 v = a.rec[at * RV + (k >> 1)];
        sh[u][k] = v.x;
        sl[u][k] = v.y;
        sh[u][k + 1] = v.z;
        sl[u][k + 1] = v.w;
      }
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        const int2 v = ok ? a.q[at * RC + r] : make_int2(0, 0);
        qh[u][r] = v.x;
        ql[u][r] = v.y;
      }
    }
    s64 th[2][RC], tm[2][RC];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int r = 0; r < RC; ++r) th[u][r] = tm[u][r] = 0;
    int t = lane;
    for (int s = 0; s < c; ++s) {
      u64 A[2] = {0, 0}, C[2] = {0, 0}, p[2];
      s64 B[2] = {0, 0};
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
      phi56<KER, 2>(A, B, C, a.c, table, p);
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        longlong2 f = fw[r * ld + t];
        const int2 q = reinterpret_cast<const int2*>(tq)[t * RC + r];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          mac(p[u], qh[u][r], ql[u][r], reinterpret_cast<s64&>(f.x), reinterpret_cast<s64&>(f.y));
          mac(p[u], q.x, q.y, th[u][r], tm[u][r]);
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
        if (r < a.Rc)
          a.pt[(static_cast<int64_t>(ent[u]) * a.Rc + r) * ld + slot[u]] = flush(th[u][r], tm[u][r], scale[r], 0.0);
    }
    if (b & 1) drain();
  }
  drain();
  __syncthreads();
  for (int i = threadIdx.x; i < a.Rc * ld; i += kThreads) {
    double v = dacc[i];
#pragma unroll
    for (int w = 1; w < NW; ++w) v += dacc[w * RC * ld + i];
    pf[i] = v;
  }
}

template <int KER, int DM, int RC>
void launch_sym(const FixSymArgs& a, int chunks, cudaStream_t s) {
  const size_t smem = fix_sym_smem<DM, RC>(a.ld);
  if (fix_sym_smem<DM, RC>(ks::kThreads) > 48 * 1024) {
    static std::atomic<uint64_t> done{0};
    const uint64_t bit = device_bit();
    if (!(done.load() & bit)) {
      DW_CUDA(cudaFuncSetAttribute(k_fix_sym<KER, DM, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(fix_sym_smem<DM, RC>(ks::kThreads))));
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
